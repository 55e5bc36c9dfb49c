"""GPU parity of the PCA temporal analysis (covariance, Jacobi eigensolver with an
FP64-accurate refinement, projection energy) against the FP64 oracle.

Bars: the energy image E within relative L2 1e-4; eigenvalues within 1e-6 of
the largest eigenvalue (absolute; the covariance is accumulated from float32
fields, whose own error is ~3e-7 relative).
"""
import numpy as np
import pytest

from oracle import hv_oracle as O
from paper_2508_03911_gb300 import hv, synth
from tests._util import oracle_params, rel_l2, to_device, to_hv

pytestmark = pytest.mark.gpu

IMAGE_TOL = 1e-4
LAM_TOL = 1e-6


def gpu_pca(frames, p):
    import torch
    n, H, W = frames.shape
    bits = 8 if frames.dtype == np.uint8 else 16
    r = hv.Renderer(W, H, bits, n)
    try:
        hv.hv_set_params(r.h, to_hv(p))
        wf = r.window_floats()
        assert wf == H * W
        out = torch.zeros(n * wf, dtype=torch.float32, device="cuda")
        assert r.push(to_device(frames)) == hv.HV_OK
        nw = 0
        while True:
            k = r.render(out[nw * wf:])
            nw += k
            if k == 0:
                break
        torch.cuda.synchronize()
        lam = hv.hv_pca_eigenvalues(r.h, p["T"])
        return out.cpu().numpy()[: nw * wf].reshape(nw, H, W), lam
    finally:
        r.close()


def oracle_windows(frames, p):
    starts = O.window_starts(frames.shape[0], p["T"], p["stride"])
    res = []
    for s in starts:
        U = np.stack([O.spatial(O.convert(f), p) for f in frames[s:s + p["T"]]])
        res.append(O.pca(U, p["pca_lo"], p["pca_hi"]))
    return res


@pytest.mark.parametrize("H,W,T,S,lohi,spatial", [
    (64, 64, 32, 32, (2, 8), "fresnel"),      # the paper's PCA 32/32 shape, small frame
    (32, 64, 64, 16, (1, 5), "asp"),          # overlapping windows
    (64, 32, 32, 48, (3, 32), "none"),        # stride beyond the window, band to the end
    (128, 128, 256, 256, (2, 64), "asp"),     # the PCA workload's window shape, smaller frame
])
def test_pca_parity(H, W, T, S, lohi, spatial):
    n = T + S + 7
    fr = synth.random_frames(n, H, W, 12, seed=H + T + S)
    p = oracle_params(spatial=spatial, z_m=0.4, temporal="pca", T=T, stride=S, pca_lo=lohi[0],
                      pca_hi=lohi[1], H=H, W=W)
    img, lam = gpu_pca(fr, p)
    ref = oracle_windows(fr, p)
    assert img.shape[0] == len(ref)
    for w, rw in enumerate(ref):
        e = rel_l2(img[w], rw["E"])
        assert e <= IMAGE_TOL, (w, e)
    lam_ref = ref[-1]["lam"]
    assert np.max(np.abs(lam - lam_ref)) <= LAM_TOL * lam_ref[0]
    assert np.all(np.diff(lam) <= 0)


def test_pca_long_windows_pipelined():
    """Five overlapping long windows (T = 128, S = 64) in one render: the eigensolvers run on
    streams of their own beside later windows' covariances and earlier windows' projections,
    the windows taking turns at as many buffer sets as eigensolvers fit the device; every
    window's image and the last window's eigenvalues against the oracle."""
    H = W = 64
    T, S = 128, 64
    fr = synth.random_frames(T + 4 * S + 9, H, W, 12, seed=77)
    p = oracle_params(spatial="asp", z_m=0.4, temporal="pca", T=T, stride=S, pca_lo=2, pca_hi=64, H=H, W=W)
    img, lam = gpu_pca(fr, p)
    ref = oracle_windows(fr, p)
    assert img.shape[0] == len(ref) == 5
    for w, rw in enumerate(ref):
        e = rel_l2(img[w], rw["E"])
        assert e <= IMAGE_TOL, (w, e)
    lam_ref = ref[-1]["lam"]
    assert np.max(np.abs(lam - lam_ref)) <= LAM_TOL * lam_ref[0]


def test_pca_windows_of_512_frames_pipelined():
    """Three windows in one render where one eigensolver runs at a time, all on the same
    scratch (T = 512, cooperative): the covariance of the next window, beside it, touches none of
    it. All components but the first, the static part's, whose eigenvalue stands far apart."""
    H = W = 64
    T, S = 512, 256
    fr = synth.random_frames(T + 2 * S, H, W, 12, seed=78)
    p = oracle_params(spatial="none", temporal="pca", T=T, stride=S, pca_lo=2, pca_hi=T, H=H, W=W)
    img, lam = gpu_pca(fr, p)
    ref = oracle_windows(fr, p)
    assert img.shape[0] == len(ref) == 3
    for w, rw in enumerate(ref):
        e = rel_l2(img[w], rw["E"])
        assert e <= IMAGE_TOL, (w, e)
    lam_ref = ref[-1]["lam"]
    assert np.max(np.abs(lam - lam_ref)) <= LAM_TOL * lam_ref[0]


@pytest.mark.parametrize("precision,tol", [("split_bf16", 1e-4), ("bf16", 5e-2)])
@pytest.mark.parametrize("H,W,T", [(64, 64, 64), (128, 64, 256), (64, 128, 128)])
def test_pca_tensor_core_covariance(precision, tol, H, W, T):
    """Covariance on the tensor cores (tcgen05, BF16 or split-BF16 inputs, FP32
    accumulation): E against the FP64 oracle; the error is printed per case."""
    n = T + 5
    fr = synth.random_frames(n, H, W, 12, seed=H * 3 + T + len(precision))
    p = oracle_params(spatial="fresnel", z_m=0.3, temporal="pca", T=T, stride=T, pca_lo=2,
                      pca_hi=min(T, 40), H=H, W=W)
    import torch
    r = hv.Renderer(W, H, 16, n)
    try:
        hv.hv_set_params(r.h, to_hv(p, precision=precision))
        out = torch.zeros(n * H * W, dtype=torch.float32, device="cuda")
        assert r.push(to_device(fr)) == hv.HV_OK
        nw = r.render(out)
        torch.cuda.synchronize()
        lam = hv.hv_pca_eigenvalues(r.h, T)
        img = out.cpu().numpy()[: nw * H * W].reshape(nw, H, W)
    finally:
        r.close()
    ref = oracle_windows(fr, p)
    e = rel_l2(img[0], ref[0]["E"])
    el = float(np.max(np.abs(lam - ref[0]["lam"])) / ref[0]["lam"][0])
    print(f"{precision} {H}x{W} T={T}: E rel L2 {e:.3e}, lam max err / lam1 {el:.3e}")
    assert e <= tol
    assert el <= tol


@pytest.fixture(scope="module")
def pca_scene_window():
    sc = synth.build(synth.scene_pca())
    fr = synth.frames(sc, 0, 256)
    p = oracle_params(spatial="asp", z_m=0.40, temporal="pca", T=256, stride=256, pca_lo=2,
                      pca_hi=64, H=512, W=512)
    U = np.stack([O.spatial(O.convert(f), p) for f in fr])
    return fr, p, {(2, 64): O.pca(U, 2, 64), (2, 9): O.pca(U, 2, 9)}


def cut_gaps(lam, lo, hi):
    """Relative eigenvalue gaps (in units of lam_1) at the two cuts of the sub-basis
    lo..hi (1-based): lam_{lo-1} - lam_lo (none for lo = 1) and lam_hi - lam_{hi+1}."""
    g = []
    if lo > 1:
        g.append((lam[lo - 2] - lam[lo - 1]) / lam[0])
    if hi < len(lam):
        g.append((lam[hi - 1] - lam[hi]) / lam[0])
    return g


def gpu_pca_window(fr, p, precision):
    """One window of N x N frames through the C ABI: (energy image, eigenvalues)."""
    import torch
    T, N = p["T"], p["H"]
    r = hv.Renderer(N, N, 16, T)
    try:
        hv.hv_set_params(r.h, to_hv(p, precision=precision))
        out = torch.zeros(N * N, dtype=torch.float32, device="cuda")
        assert r.push(to_device(fr)) == hv.HV_OK
        assert r.render(out) == 1
        torch.cuda.synchronize()
        lam = hv.hv_pca_eigenvalues(r.h, T)
        return out.cpu().numpy().reshape(N, N), lam
    finally:
        r.close()


@pytest.mark.parametrize("T,H,W", [(32, 64, 64), (64, 32, 64), (128, 64, 64), (256, 64, 64)])
def test_pca_rank_deficient_windows(T, H, W):
    """Windows of six distinct images (every other eigenvalue is 0): the eigenvalues of the
    exact integer covariance, and the whole band's energy, which is sum_t |u_t|^2 where the
    eigenvectors are unitary. These are products of float32 rotations, about 8 sweeps of T - 1
    of them in each column, unitary to 8 T 2^-24 / 2 at worst: 6e-5 for T = 256."""
    rng = np.random.default_rng(T)
    base = rng.integers(0, 4096, (6, H, W), dtype=np.uint16)
    fr = base[rng.integers(0, 6, 2 * T)]
    p = oracle_params(spatial="none", temporal="pca", T=T, stride=T, pca_lo=1, pca_hi=T, H=H, W=W)
    img, lam = gpu_pca(fr, p)
    assert img.shape[0] == 2
    x = fr.reshape(2, T, H * W).astype(np.float64)
    for w in range(2):
        e = (x[w] ** 2).sum(0).reshape(H, W)
        assert np.max(np.abs(img[w] - e) / e) <= 6e-5
    ref = np.linalg.eigvalsh(x[1] @ x[1].T)[::-1]
    assert np.max(np.abs(lam - ref)) <= LAM_TOL * ref[0]


def test_pca_batched_many_windows():
    """Short windows are batched: all windows of one render in one launch per kernel
    (one CTA per window for the eigensolver), overlapping and non-overlapping.

    The frames come from the Doppler scene, whose spectrum separates the sub-basis
    2..3 from its neighbours by >= 1e-2 lam_1. The projector onto the sub-basis then
    moves by about |dC| / gap (Davis-Kahan) ~ 1e-5 under the float32 covariance
    error, inside the 1e-4 bar. White-noise frames leave gaps of ~1e-5 lam_1 at
    most band edges, where no float32 covariance pins the sub-space to 1e-4."""
    for (N, T, S, n) in [(64, 32, 32, 32 * 40 + 5), (32, 64, 16, 64 + 16 * 70)]:
        fr = synth.frames(synth.build(synth.scene_pca(N=N)), 0, n)
        H = W = N
        p = oracle_params(spatial="fresnel", z_m=0.3, temporal="pca", T=T, stride=S, pca_lo=2,
                          pca_hi=3, H=H, W=W)
        img, lam = gpu_pca(fr, p)
        ref = oracle_windows(fr, p)
        assert img.shape[0] == len(ref) > 32
        for w in range(len(ref)):
            e = rel_l2(img[w], ref[w]["E"])
            assert e <= IMAGE_TOL, (w, e)
        assert np.max(np.abs(lam - ref[-1]["lam"])) <= LAM_TOL * ref[-1]["lam"][0]


@pytest.mark.parametrize("precision,tol", [("fp32", IMAGE_TOL), ("split_bf16", IMAGE_TOL),
                                           ("bf16", 5e-2)])
def test_pca_scene_window_full_size(pca_scene_window, precision, tol):
    """One window of the PCA workload: 512x512 12-bit frames, ASP z = 0.40 m,
    T = 256, per covariance precision.

    The workload's sub-basis 2..64 cuts the noise bulk of the spectrum, where
    lam_64 - lam_65 is ~1e-9 lam_1: below 1e-6 lam_1 that cut is "parity
    ambiguous" (several sub-bases are correct), so there the eigenvalues (unique)
    and the total energy sum_p E = sum_j lam_j (unique to within the gap) are
    compared, and E itself only as a valid result. The sub-basis 2..9 ends at a
    clear gap (~6e-3 lam_1), asserted first: there E is unique and held to the bar."""
    fr, p, refs = pca_scene_window
    for (lo, hi), ref in refs.items():
        q = dict(p, pca_lo=lo, pca_hi=hi)
        img, lam = gpu_pca_window(fr, q, precision)
        gaps = cut_gaps(ref["lam"], lo, hi)
        e = rel_l2(img, ref["E"])
        el = float(np.max(np.abs(lam - ref["lam"])) / ref["lam"][0])
        tot = abs(float(img.sum(dtype=np.float64)) - float(ref["lam"][lo - 1:hi].sum())) / float(
            ref["lam"][lo - 1:hi].sum())
        ambiguous = min(gaps) <= 1e-6
        print(f"scene {precision} {lo}..{hi}: cut gaps {['%.1e' % g for g in gaps]} lam_1"
              f"{' (parity ambiguous)' if ambiguous else ''}; E rel L2 {e:.3e}, total energy "
              f"{tot:.2e}, lam max err / lam1 {el:.3e}")
        assert el <= max(LAM_TOL, tol)
        assert tot <= max(10 * IMAGE_TOL, tol)
        assert e <= tol
        if (lo, hi) == (2, 9):
            assert not ambiguous


def test_pca_full_range_16bit_fresnel_long_window():
    """512x512 frames at the full 16-bit range through the unnormalised Fresnel
    transform, T = 128: diagonal covariance entries reach ~3e19, so products of
    two of them exceed the float32 range. The float32 phase of the eigensolver
    works on C scaled by a power of two; without that its rotation tests overflow.
    Sub-basis 2..9, whose cuts sit at clear gaps (asserted)."""
    sc = synth.build(synth.scene_pca(N=512, bits=16))
    fr = synth.frames(sc, 0, 128)
    assert fr.max() == 65535
    p = oracle_params(spatial="fresnel", z_m=0.25, temporal="pca", T=128, stride=128, pca_lo=2,
                      pca_hi=9, H=512, W=512)
    U = np.stack([O.spatial(O.convert(f), p) for f in fr])
    ref = O.pca(U, 2, 9)
    del U
    assert float(np.max(np.real(np.diag(ref["C"])))) > 1.9e19
    assert min(cut_gaps(ref["lam"], 2, 9)) > 1e-6
    for precision in ("fp32", "split_bf16"):
        img, lam = gpu_pca_window(fr, p, precision)
        e = rel_l2(img, ref["E"])
        el = float(np.max(np.abs(lam - ref["lam"])) / ref["lam"][0])
        print(f"16-bit Fresnel {precision}: E rel L2 {e:.3e}, lam max err / lam1 {el:.3e}")
        assert np.all(np.isfinite(img)) and np.all(np.isfinite(lam))
        assert e <= IMAGE_TOL
        # split-BF16 covariance: the eigenvalue bar of the other split-BF16 cases
        assert el <= (LAM_TOL if precision == "fp32" else max(LAM_TOL, IMAGE_TOL))


def test_pca_rejects_unbuilt_precisions_and_bad_basis():
    r = hv.Renderer(64, 64, 16, 8)
    try:
        for kw in (dict(pca_lo=0), dict(pca_hi=33), dict(pca_lo=5, pca_hi=4), dict(T=16)):
            p = oracle_params(temporal="pca", T=32, stride=32, pca_lo=2, pca_hi=8, H=64, W=64)
            p.update(kw)
            with pytest.raises(hv.HvError):
                hv.hv_set_params(r.h, to_hv(p))
    finally:
        r.close()


@pytest.mark.parametrize("T,bar", [(32, 1.9e-7), (64, 2.2e-7), (128, 2.35e-7), (256, 2.6e-7)])
def test_rounding_of_the_sub_basis(T, bar):
    """Energy of all components of noise but the first, against float64: what thousands of float32
    rotations leave of the eigenvectors' orthogonality. The frames are fixed and the arithmetic
    deterministic; the mean over three windows is 1.7, 1.9, 2.0 and 2.1e-7 with c^2 + s^2 and |ph|
    scaled to 1, and was 2.1, 2.5, 2.7 and 3.0e-7 (2.1 to 3.2e-7 with correctly rounded roots and
    quotients)."""
    N = 64
    err = []
    for seed in range(3):
        fr = np.random.default_rng(100 * T + seed).integers(0, 4096, (T, N, N)).astype(np.uint16)
        p = oracle_params(spatial="none", temporal="pca", T=T, stride=T, pca_lo=2, pca_hi=T, H=N, W=N)
        img, _ = gpu_pca_window(fr, p, "fp32")
        x = fr.reshape(T, N * N).astype(np.float64)
        _, v = np.linalg.eigh(x @ x.T)
        err.append(rel_l2(img, ((v[:, :-1].T @ x) ** 2).sum(0).reshape(N, N)))
    assert np.mean(err) <= bar, err

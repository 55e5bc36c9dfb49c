"""Host code of the library against a CUDA runtime that only writes calls down: the order of
copies on several streams, scratch after an allocation that failed, calls that failed half way."""
import pytest

from tests._fake_cuda import run, unordered_copies

RING = """
import numpy as np
W = H = 64
r = hv.Renderer(W, H, 8, 16)
r.set_params(W, H, spatial="asp", T=8, stride=4, fs=20000.0, band=(1, 2))
g = hv.hv_group_open([r.h], use_graph=%(graph)s)
out = Dev((8, H, W), 4)
host = np.zeros((8, H, W), np.uint8)
log()
assert hv.hv_render_group(g, [Dev((12, H, W), 1)], [out]) == [2]
assert r.push(host, async_=True) == hv.HV_OK     # frames 12 .. 19, slots 12 .. 15, 0 .. 3
assert r.render(out) == 2
assert r.push(host, async_=True) == hv.HV_OK     # frames 20 .. 27: over the group's 8 .. 11
r.render(out)
print(json.dumps(log()))
"""


def test_pushes_follow_the_copy_of_a_groups_last_frames():
    """A group step of 12 frames copies the four that the next window reads again into slots 8
    .. 11 of the input ring, behind its images; a later push from the host overwrites the
    slots on the copy stream."""
    for graph in (False, True):
        assert unordered_copies(run(RING % dict(graph=graph))) == []


SWEEP = """
import numpy as np
N, MB = 512, 1 << 20
r = hv.Renderer(N, N, 16, 256)
r.set_params(N, N, spatial="asp", T=128, stride=128, fs=20000.0, band=(1, 2))
fr, out = Dev((128, N, N), 2), Dev((1, N, N), 4)
def render():
    log()
    assert r.push(fr) == hv.HV_OK and r.render(out) == 1
    return [l[1:] for l in log() if l[0] == "scratch"]
before = render()
fake.fake_fail_malloc(%(least)d * MB, 1 << 40, %(times)d)
try:
    hv.hv_focus_sweep(r.h, Dev((64, N, N), 2), np.linspace(0.1, 0.6, 64), Dev((64, 64), 4))
    status = 0
except hv.HvError as e:
    status = e.status
fake.fake_fail_malloc(0, 0, 0)
print(json.dumps([status, before, render()]))
"""


@pytest.mark.parametrize("least,times,status", [(400, 1, 0), (100, 2, -4)])
def test_renders_after_a_sweep_without_memory(least, times, status):
    """A sweep of 64 holograms of 512 x 512 asks for 512 MB where a render has 256. With memory
    for fewer images, and without any for it, a later render's launches stay in their scratch."""
    got, before, after = run(SWEEP % dict(least=least, times=times))
    assert got == status
    for launches in (before, after):
        assert len(launches) >= 3
        for w, h, n, spatial, room1, room2 in launches:
            assert room1 >= n * w * (h // 2 + 1) * 8 and room2 >= n * w * h * 8


def test_features_as_a_handles_first_call():
    """Settings are applied by the call itself: the launch size follows from them."""
    assert run("""
r = hv.Renderer(256, 256, 16, 256)
r.set_params(256, 256, spatial="asp", T=16, stride=16, fs=20000.0, band=(1, 2))
log()
hv.hv_af_features(r.h, Dev((200, 256, 256), 2), Dev((200, 128, 128), 2))
print(json.dumps([l[3] for l in log() if l[0] == "scratch"]))
""") == [200, 200]


FAILED_STEP = """
W = H = 64
rs = [hv.Renderer(W, H, 8, 16) for _ in range(2)]
for r in rs:
    r.set_params(W, H, spatial="asp", T=8, stride=4, fs=20000.0, band=(1, 2))
g = hv.hv_group_open([r.h for r in rs], use_graph=%(graph)s)
fr, outs = [Dev((12, H, W), 1) for _ in rs], [Dev((8, H, W), 4) for _ in rs]
log()
fake.fake_fail_launch(b"k_stft", 1)
try:
    hv.hv_render_group(g, fr, outs)
    failed = False
except hv.HvError:
    failed = True
copied = sum(l[4] for l in log() if l[0] == "copy" and fr[0].p <= l[3] < fr[0].p + 12 * W * H)
pushed = [r.stats()["frames_pushed"] for r in rs]
windows = [r.render(o) for r, o in zip(rs, outs)]
print(json.dumps([failed, pushed, copied // (W * H), windows]))
"""


def test_a_failed_group_step_keeps_no_frames_it_has_not():
    """The first member's STFT does not launch. Without a graph its frames are queued all the
    same, copied, and a render takes them; of a graph nothing runs, so no member has frames."""
    assert run(FAILED_STEP % dict(graph=False)) == [True, [12, 0], 12, [2, 0]]
    assert run(FAILED_STEP % dict(graph=True)) == [True, [0, 0], 0, [0, 0]]


SHORT = """
MB = 1 << 20
r = hv.Renderer(%(side)d, %(side)d, 16, %(cap)d)
r.set_params(%(side)d, %(side)d, fs=20000.0, band=(1, 2), moments=("M0", "M1"), %(kw)s)
out = Dev((64, 2, %(side)d, %(side)d), 4)
assert r.push(Dev((%(cap)d, %(side)d, %(side)d), 2)) == hv.HV_OK
log()
fake.fake_fail_malloc(%(low)d, %(high)d, 100)
nw = r.render(out)
lines = log()
print(json.dumps([nw, [l[2] // MB for l in lines if l[0] == "malloc"], [l[3] for l in lines if l[0] == "scratch"]]))
"""


def test_overlapping_windows_tuned_without_memory_for_the_trial():
    """No memory for the images that the STFT kernels are timed with (64 windows of two images):
    the default kernel renders."""
    nw, _, _ = run(SHORT % dict(side=256, cap=1024, low=64 * 2 * 65536 * 4, high=64 * 2 * 65536 * 4,
                                kw='spatial="none", T=128, stride=16, tuned=1'))
    assert nw == 57


def test_default_launches_without_64_mb():
    """Where 64 MB of fields a launch do not fit, 32 MB do: 16 frames of 512 x 512."""
    nw, sizes, frames = run(SHORT % dict(side=512, cap=200, low=60 << 20, high=300 << 20,
                                         kw='spatial="asp", T=128, stride=128'))
    assert nw == 1 and sizes.count(32) == 2 and max(frames) == 16


def test_fused_transform_takes_no_scratch_for_launches_side_by_side():
    """One launch for all frames: 64 MB, a launch's frames, and not four times that."""
    _, sizes, _ = run(SHORT % dict(side=256, cap=480, low=1, high=0,
                                   kw='spatial="fresnel", T=128, stride=128, spatial_kernel="fused"'))
    assert 64 in sizes and 256 not in sizes


def test_tuning_record_names_the_kernels_that_run():
    """Selections that other kernels serve, and windows that overlap."""
    assert run("""
got = []
for kw in (dict(spatial_kernel="persistent"), dict(spatial_kernel="cluster"), dict(stft_kernel="window_wide"),
           dict(stft_kernel="window_pipelined"), dict(stft_kernel="window_tma"), dict(stft_kernel="window", stride=64),
           dict(stride=64), dict()):
    r = hv.Renderer(256, 256, 16, 256)
    r.set_params(256, 256, **dict(dict(spatial="asp", T=128, stride=128, fs=20000.0, band=(1, 2)), **kw))
    assert r.push(Dev((256, 256, 256), 2)) == hv.HV_OK
    r.render(Dev((4, 1, 256, 256), 4))
    t = hv.hv_get_tuning(r.h)
    got.append([t["spatial_kernel"], t["stft_kernel"]])
print(json.dumps(got))
""") == [[1, 2], [2, 2], [1, 2], [1, 2], [1, 2], [1, 1], [1, 1], [1, 2]]


def test_tables_after_an_allocation_that_failed():
    """Larger frames whose tables do not fit, then smaller ones: the tables are allocated again."""
    status, null = run("""
MB = 1 << 20
r = hv.Renderer(1024, 1024, 8, 16)
def use(side):
    r.set_params(side, side, spatial="asp", T=8, stride=8, fs=20000.0, band=(1, 2))
    assert r.push(Dev((8, side, side), 1)) == hv.HV_OK
    return r.render(Dev((1, 1, side, side), 4))
assert use(512) == 1
fake.fake_fail_malloc(16 * MB, 17 * MB, 1)  # two tables of 1024 x 1024 values and the chirps
try:
    use(1024)
    status = 0
except hv.HvError as e:
    status = e.status
log()
assert use(256) == 1
print(json.dumps([status, sum(1 for l in log() if l[0] == "copy" and l[2] < 4096)]))
""")
    assert status == -4 and null == 0


def test_a_sweep_after_one_without_memory_for_its_tables():
    """The transfer functions of the sweep before the failed one are gone: formed again."""
    status, copied = run("""
import numpy as np
N = 256
r = hv.Renderer(N, N, 16, 4)
r.set_params(N, N, spatial="asp", T=8, stride=8, fs=20000.0, band=(1, 2))
fr, out = Dev((4, N, N), 2), Dev((4, 512), 4)
table = N * (N // 2 + 1) * 8
def sweep(nz):
    log()
    hv.hv_focus_sweep(r.h, fr, np.linspace(0.1, 0.6, nz), out)
    return sum(l[4] for l in log() if l[0] == "copy")
sweep(8)
assert sweep(8) == 0
fake.fake_fail_malloc(512 * table, 512 * table, 1)
try:
    sweep(512)
    status = 0
except hv.HvError as e:
    status = e.status
print(json.dumps([status, sweep(8) // table]))
""")
    assert status == -4 and copied == 8


def test_settings_whose_tuning_failed_flush_the_queue():
    """A window half of whose frames were propagated with the settings before: all of them are
    again, also where the autotuner found no memory and the call before said so."""
    status, frames = run("""
MB, N = 1 << 20, 512
r = hv.Renderer(N, N, 16, 64)
kw = dict(spatial="asp", T=32, stride=16, fs=20000.0, band=(1, 2))
out = Dev((1, 1, N, N), 4)
r.set_params(N, N, **kw)
assert r.push(Dev((64, N, N), 2)) == hv.HV_OK and r.render(out) == 1
r.set_params(N, N, z=0.2, tuned=1, **kw)
fake.fake_fail_malloc(30 * MB, 1 << 40, 1000)
try:
    r.render(out)
    status = 0
except hv.HvError as e:
    status = e.status
fake.fake_fail_malloc(0, 0, 0)
before = r.stats()["frames_propagated"]
assert r.render(out) == 1
print(json.dumps([status, r.stats()["frames_propagated"] - before]))
""")
    assert status == -4 and frames == 32

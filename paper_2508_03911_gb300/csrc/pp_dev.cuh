// pp_dev.cuh -- block-wide FFT stages over strips of lines staged in shared memory: the
// column passes of the fused transform (k_spatial_pp.cu) and the network input's passes
// (k_features.cu).
#pragma once
#include "fft_dev.cuh"

namespace hv {

// Strips of 16 lines of length L (8 at 1024), NT threads.
template <int L>
struct PpCfg {
  static constexpr int BT = L >= 1024 ? 8 : 16;
  static constexpr int NT = FftThreads<L, BT>::value;  // L for 64 <= L <= 512, 512 at 1024
  static_assert(L % NT == 0 && NT % BT == 0, "threads cover the elements of a line");
};

// ------------------------------------------------ stage inputs and epilogues

// Element t of line b from the FFT buffer.
template <int LD>
struct SmemSrc {
  static constexpr bool kAliasesBuf = true;
  const float2* buf;
  __device__ __forceinline__ float2 operator()(int t, int b) const { return buf[t * LD + b]; }
};

// Element t (row y) of column b from a staged raw strip [y][BT], converted to
// complex; with the Fresnel chirp cy[y] * cx (cx: this thread's column factor).
template <bool U8, bool CHIRP, int BT, bool ALIAS = false>
struct RawSrc {
  static constexpr bool kAliasesBuf = ALIAS;  // staged inside the FFT buffer: read all before writing
  const unsigned char* raw;
  const float2* cy;
  float2 cx;
  __device__ __forceinline__ float2 operator()(int t, int b) const {
    const float v = U8 ? float(raw[t * BT + b]) : float(reinterpret_cast<const uint16_t*>(raw)[t * BT + b]);
    if constexpr (CHIRP) return cscale(cmul(cy[t], cx), v);
    return make_float2(v, 0.f);
  }
};

// Bin k of line b straight to global memory at out[k * stride + b].
struct GlobalOut {
  static constexpr bool kSyncFirst = false;
  static constexpr bool kJFast = false;
  float2* out;
  uint32_t stride;
  __device__ __forceinline__ void operator()(int b, int k, float2 v) const { out[size_t(k) * stride + b] = v; }
};

// One Stockham stage of span NS over the strip's lines (thread layout and index
// rules of fft_dev.cuh), and recursively the rest. The first stage reads
// through `src`, later ones the buffer (row stride LD); twiddles come from the shared table
// tws[e] = exp(-2 pi i e / L). The last stage hands bin k of line b to epi.
// With an epilogue of kJFast, the last stage maps threads bin-fastest (b = idx / NB,
// j = idx % NB) and takes its twiddles from twl[(m - 1) NS + j] (contiguous in j).
// Barrier between stages: the whole CTA (BAR = 0), or named barrier BAR over the
// pass's NT threads (warp-specialised kernels whose other warps do not take part).
template <int BAR, int NT>
__device__ __forceinline__ void pp_sync() {
  if constexpr (BAR == 0) __syncthreads();
  else asm volatile("bar.sync %0, %1;\n" ::"n"(BAR), "n"(NT) : "memory");
}

template <int L, int NS, int DIR, class Src, class Epi, int LD, int BAR>
__device__ __forceinline__ void pp_stages(const Src& src, float2* buf, const float2* tws, const Epi& epi,
                                          const float2* twl = nullptr) {
  using C = PpCfg<L>;
  // row stride LD = 16 (TMA-staged strips): with lines fastest, a warp's stage accesses
  // are two contiguous 128-byte runs
  constexpr int NT = C::NT, BT = C::BT;
  constexpr int REM = L / NS;
  constexpr int R = BlockRadix<REM, L, BT, NT>::value;
  constexpr int NB = L / R;
  static_assert((BT * NB) % NT == 0, "thread count must divide the butterflies");
  constexpr int ITEMS = BT * NB / NT;
  constexpr bool LAST = NS * R == L;
  constexpr bool JF = LAST && Epi::kJFast;
  float2 v[ITEMS][R];
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int idx = threadIdx.x + it * NT;
    const int b = JF ? idx / NB : idx % BT, j = JF ? idx % NB : idx / BT;
#pragma unroll
    for (int m = 0; m < R; ++m) v[it][m] = src(j + m * NB, b);
    if constexpr (NS > 1) {
      const int jm = j % NS;
#pragma unroll
      for (int m = 1; m < R; ++m) {
        float2 w = JF ? twl[(m - 1) * NS + jm] : tws[jm * m * (L / (NS * R))];
        if constexpr (DIR > 0) w.y = -w.y;
        v[it][m] = cmul(v[it][m], w);
      }
    }
    dft<R, DIR>(v[it]);
  }
  if constexpr (LAST) {
    if constexpr (Epi::kSyncFirst) pp_sync<BAR, NT>();  // every read of buf is done
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const int idx = threadIdx.x + it * NT;
      const int b = JF ? idx / NB : idx % BT, j = JF ? idx % NB : idx / BT;
#pragma unroll
      for (int m = 0; m < R; ++m) epi(b, j + m * NB, v[it][m]);
    }
  } else {
    if constexpr (Src::kAliasesBuf) pp_sync<BAR, NT>();
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const int idx = threadIdx.x + it * NT;
      const int b = idx % BT, j = idx / BT;
      const int base = (j / NS) * NS * R + (j % NS);
#pragma unroll
      for (int m = 0; m < R; ++m) buf[(base + m * NS) * LD + b] = v[it][m];
    }
    pp_sync<BAR, NT>();
    SmemSrc<LD> s{buf};
    pp_stages<L, NS * R, DIR, SmemSrc<LD>, Epi, LD, BAR>(s, buf, tws, epi, twl);
  }
}

}  // namespace hv

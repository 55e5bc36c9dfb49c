// k_features.cu -- the autofocus network's input from raw frames of sides 64 .. 1024: the
// centred spectrum's 2 x 2 blocks as log1p(mean |F|) (DC bin as 0), standardised over the
// frame and rounded to bfloat16.
//
//   columns  raw [y][x] -> column FFT of 16 real columns (8 of 1024 points) -> S1 [ky][x]
//   rows     S1 row ky -> row FFT. Widths up to 256: the cells and the frame's (sum v,
//            sum v^2) from the registers of the last stage; wider frames store the spectrum
//            and bin it in a kernel of its own.
//
// Persistent CTAs that stage their next strip by cp.async while they transform one, over all
// H rows and with the transforms of a real column one at a time: 512 holograms of 256 x 256 in
// 68 + 145 us, bound by issue and the stages' barriers. Half of the spectrum, from two real
// columns to a complex line, with the mirrored cells from the same |F|, took 37 + 71, but a
// bfloat16 result turns a float32 error into a whole unit where a value lies near the middle of
// two, and that carries into the network: 6,330 of 8.4 million inputs differed from the float64
// result's bfloat16 instead of 4,650, and the network's answer was 7.7e-5 off instead of 6.1e-5.
#include <cuda_bf16.h>

#include "pp_dev.cuh"
#include "hv_internal.h"
#include "../../include/hv.h"

namespace hv {

namespace {

enum FeaturePass { COLS, CELLS, ROWS };

template <int L>
struct FeatCfg : PpCfg<L> {
  static constexpr int LD = PpCfg<L>::BT + 1;
  static constexpr size_t BUF = size_t(L) * LD * sizeof(float2);
  static constexpr size_t RAW = size_t(L) * PpCfg<L>::BT * 2;  // one uint16 strip
  static constexpr size_t TW = size_t(L) * sizeof(float2);
};

__device__ __forceinline__ void cpa8(void* s, const void* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(static_cast<unsigned>(__cvta_generic_to_shared(s))),
               "l"(g)
               : "memory");
}
__device__ __forceinline__ void cpa16(void* s, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(static_cast<unsigned>(__cvta_generic_to_shared(s))),
               "l"(g)
               : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cpa_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Bin k of line b straight to global memory at out[b * stride + k], with the
// last stage's threads laid out along the bins (consecutive lanes hold
// consecutive bins of one line, so the stores are coalesced).
struct RowOut {
  static constexpr bool kSyncFirst = false;
  static constexpr bool kJFast = true;
  float2* out;
  uint32_t stride;
  __device__ __forceinline__ void operator()(int b, int k, float2 v) const { out[size_t(b) * stride + k] = v; }
};

// Cells from bins handed out bin-fastest with 16 butterflies per
// line (lanes 0-15: row b, lanes 16-31: row b + 1; bins j + 16 m): the 2 x 2 block
// of unshifted bins (even ky, even kx) sits in lanes j, j ^ 1, j ^ 16, j ^ 17. The
// lane with even j of the even row writes log1p(mean |F|) (DC bin as 0) at the
// block's centred position and adds it to its running (sum v, sum v^2).
struct CellsOut {
  static constexpr bool kSyncFirst = false;
  static constexpr bool kJFast = true;
  float* cells;      // this frame's [H/2][W/2]
  uint32_t ky0;      // unshifted row of the strip's first line
  uint32_t W, H;
  float* s;          // s[0] += v, s[1] += v^2
  __device__ __forceinline__ void operator()(int b, int k, float2 v) const {
    const uint32_t ky = ky0 + uint32_t(b);
    float a = (ky | uint32_t(k)) ? sqrtf(fmaf(v.x, v.x, v.y * v.y)) : 0.f;
    a += __shfl_xor_sync(0xffffffffu, a, 1);
    a += __shfl_xor_sync(0xffffffffu, a, 16);
    if (((threadIdx.x & 31) & 17) == 0) {  // even bin, even row
      const float c = log1pf(0.25f * a);
      const uint32_t r = ((ky + H / 2) & (H - 1)) >> 1, q = ((uint32_t(k) + W / 2) & (W - 1)) >> 1;
      cells[size_t(r) * (W / 2) + q] = c;
      s[0] += c;
      s[1] = fmaf(c, c, s[1]);
    }
  }
};

// Span NS and radix R of the last stage of the pass (the BlockRadix chain).
template <int L, int BT, int NT>
struct LastStage {
  static constexpr int radix(int rem) {
    return (rem % 16 == 0 && (BT * (L / 16)) % NT == 0 && BT * (L / 16) >= NT) ? 16
           : (rem % 8 == 0 ? 8 : (rem % 4 == 0 ? 4 : 2));
  }
  static constexpr int ns() {
    int ns = 1;
    while (ns * radix(L / ns) < L) ns *= radix(L / ns);
    return ns;
  }
  static constexpr int NS = ns();
  static constexpr int R = L / NS;
};

// Raw strip: rows 0..L-1, columns s0..s0+BT-1 of frame i -> dst [y][BT], in 16-byte pieces
// (8-byte ones where a row segment is shorter: uint8 at BT = 8); pixel by pixel where the
// frames are not 16-byte aligned.
template <int L>
__device__ __forceinline__ void prefetch_raw(const SpatialArgs& a, int i, int s0, unsigned char* dst) {
  using C = FeatCfg<L>;
  const int bpp = a.in_kind == IN_U8 ? 1 : 2;
  const int seg = C::BT * bpp;  // bytes of one row segment: 8, 16 or 32
  const size_t rslot = (a.raw.slot0 + uint32_t(i)) % a.raw.cap;
  const unsigned char* src = static_cast<const unsigned char*>(a.raw.base) + (rslot * size_t(a.W) * L + s0) * bpp;
  const size_t row = size_t(a.W) * bpp;
  if (reinterpret_cast<uintptr_t>(a.raw.base) & 15) {
    for (int e = threadIdx.x; e < L * C::BT; e += C::NT) {
      const int y = e / C::BT, b = e % C::BT;
      if (bpp == 1) dst[e] = src[y * row + b];
      else reinterpret_cast<uint16_t*>(dst)[e] = reinterpret_cast<const uint16_t*>(src + y * row)[b];
    }
  } else if (seg >= 16) {
    const int pieces = seg / 16;
    for (int e = threadIdx.x; e < L * pieces; e += C::NT) {
      const int y = e / pieces, q = e % pieces;
      cpa16(dst + y * seg + q * 16, src + y * row + q * 16);
    }
  } else {
    for (int y = threadIdx.x; y < L; y += C::NT) cpa8(dst + y * seg, src + y * row);
  }
  cpa_commit();
}

// Complex strip: line b of the strip is src[b * L + t], t = 0..L-1 -> buf[t][b].
template <int L>
__device__ __forceinline__ void prefetch_lines(const float2* src, float2* dst) {
  using C = FeatCfg<L>;
#pragma unroll
  for (int t = threadIdx.x; t < L; t += C::NT)
#pragma unroll
    for (int b = 0; b < C::BT; ++b) cpa8(&dst[t * C::LD + b], &src[b * L + t]);
  cpa_commit();
}

template <int L, FeaturePass PASS>
__global__ void __launch_bounds__(FeatCfg<L>::NT, (L <= 256 ? 768 / L : 1))
    k_feature_pass(SpatialArgs a, int nitems, int strip_log2) {
  using C = FeatCfg<L>;
  extern __shared__ __align__(16) unsigned char smem[];
  float2* tws = reinterpret_cast<float2*>(smem);
  float2* twl = reinterpret_cast<float2*>(smem + C::TW);  // rows: last-stage twiddles by (m, j)
  unsigned char* body = smem + (PASS == COLS ? C::TW : 2 * C::TW);
  float2* buf0 = reinterpret_cast<float2*>(body);
  // columns: one FFT buffer and two raw staging buffers; rows: two FFT buffers
  float2* buf1 = reinterpret_cast<float2*>(body + C::BUF);
  unsigned char* raw0 = body + C::BUF;
  unsigned char* raw1 = body + C::BUF + C::RAW;
  const int tid = threadIdx.x;
  const int smask = (1 << strip_log2) - 1;
  const bool u8 = a.in_kind == IN_U8;
  const float2* twg = PASS == COLS ? a.tw_h : a.tw_w;
  for (int e = tid; e < L; e += C::NT) tws[e] = __ldg(&twg[e]);
  if constexpr (PASS != COLS) {
    using LS = LastStage<L, C::BT, C::NT>;
    for (int e = tid; e < (LS::R - 1) * LS::NS; e += C::NT) {
      const int m = e / LS::NS + 1, jm = e % LS::NS;
      twl[e] = __ldg(&twg[jm * m * (L / (LS::NS * LS::R))]);
    }
  }
  auto issue = [&](int it, int cur) {
    const int i = it >> strip_log2, s0 = (it & smask) * C::BT;
    if constexpr (PASS == COLS) prefetch_raw<L>(a, i, s0, cur == 0 ? raw0 : raw1);
    else prefetch_lines<L>(a.scratch1 + size_t(i) * L * a.H + size_t(s0) * L, cur == 0 ? buf0 : buf1);
  };

  int item = blockIdx.x;
  if (item < nitems) issue(item, 0);
  for (int k = 0; item < nitems; ++k, item += gridDim.x) {
    const int cur = k & 1;
    const int i = item >> strip_log2, s0 = (item & smask) * C::BT;
    cpa_wait_all();
    __syncthreads();  // this item's input resident; the other buffer is free
    const int nxt = item + gridDim.x;
    if (nxt < nitems) issue(nxt, cur ^ 1);
    if constexpr (PASS == COLS) {
      // S1[ky][x]: bin ky of column s0 + b at s1[ky * W + s0 + b]
      const GlobalOut out{a.scratch1 + size_t(i) * a.H * a.W + s0, a.W};
      const unsigned char* raw = cur == 0 ? raw0 : raw1;
      const float2 none = make_float2(0.f, 0.f);
      using Src8 = RawSrc<true, false, C::BT>;
      using Src16 = RawSrc<false, false, C::BT>;
      if (u8) pp_stages<L, 1, -1, Src8, GlobalOut, C::LD, 0>(Src8{raw, nullptr, none}, buf0, tws, out);
      else pp_stages<L, 1, -1, Src16, GlobalOut, C::LD, 0>(Src16{raw, nullptr, none}, buf0, tws, out);
    } else {
      // the strip's spectra are dead once staged: drop their L2 lines unwritten
      const char* st = reinterpret_cast<const char*>(a.scratch1 + size_t(i) * L * a.H + size_t(s0) * L);
      for (int e = tid; e < C::BT * L * 8 / 128; e += C::NT)
        asm volatile("discard.global.L2 [%0], 128;\n" ::"l"(st + size_t(e) * 128) : "memory");
      float2* buf = cur == 0 ? buf0 : buf1;
      const SmemSrc<C::LD> src{buf};
      if constexpr (PASS == ROWS) {
        // spectrum [ky][kx]: bin kx of row s0 + b, stored from the registers of the last
        // stage (threads along kx there)
        float2* out = static_cast<float2*>(a.tq.base) + size_t(i) * a.H * a.W + size_t(s0) * a.W;
        pp_stages<L, 1, -1, SmemSrc<C::LD>, RowOut, C::LD, 0>(src, buf, tws, RowOut{out, a.W}, twl);
      } else {
        float acc[2] = {0.f, 0.f};
        const CellsOut out{a.cells + size_t(i) * (a.H / 2) * (a.W / 2), uint32_t(s0), a.W, a.H, acc};
        pp_stages<L, 1, -1, SmemSrc<C::LD>, CellsOut, C::LD, 0>(src, buf, tws, out, twl);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
          acc[1] += __shfl_xor_sync(0xffffffffu, acc[1], o);
        }
        __shared__ float red[2][C::NT / 32];
        if ((tid & 31) == 0) {
          red[0][tid >> 5] = acc[0];
          red[1][tid >> 5] = acc[1];
        }
        __syncthreads();
        if (tid < 2) {
          double t = 0.0;
#pragma unroll
          for (int w = 0; w < C::NT / 32; ++w) t += red[tid][w];
          atomicAdd(&a.tam_acc[size_t(i) * a.tam_stride + tid], t);
        }
      }
    }
  }
  cpa_wait_all();
}

template <int L, FeaturePass PASS>
cudaError_t launch_pass(const SpatialArgs& a, uint32_t lines, cudaStream_t s) {
  using C = FeatCfg<L>;
  const size_t smem = PASS == COLS ? C::TW + C::BUF + 2 * C::RAW : 2 * C::TW + 2 * C::BUF;
  auto kern = k_feature_pass<L, PASS>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  int per_sm = 0, dev = 0, nsm = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, C::NT, smem);
  if (e != cudaSuccess) return e;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  int strip_log2 = 0;
  while ((uint32_t(C::BT) << strip_log2) < lines) ++strip_log2;
  const int nitems = int(a.n) << strip_log2;
  int grid = per_sm * nsm;
  if (grid > nitems) grid = nitems;
  if (grid < 1) grid = 1;
  kern<<<grid, C::NT, smem, s>>>(a, nitems, strip_log2);
  return cudaGetLastError();
}

template <FeaturePass PASS>
cudaError_t pass_by_len(const SpatialArgs& a, cudaStream_t s) {
  const uint32_t L = PASS == COLS ? a.H : a.W, lines = PASS == COLS ? a.W : a.H;
  if constexpr (PASS != ROWS) {
    switch (L) {
      case 64: return launch_pass<64, PASS>(a, lines, s);
      case 128: return launch_pass<128, PASS>(a, lines, s);
      case 256: return launch_pass<256, PASS>(a, lines, s);
    }
  }
  if constexpr (PASS != CELLS) {
    switch (L) {
      case 512: return launch_pass<512, PASS>(a, lines, s);
      case 1024: return launch_pass<1024, PASS>(a, lines, s);
    }
  }
  return cudaErrorInvalidValue;
}

constexpr int FT_NT = 512;

// Binned log-magnitude of cell (r, c): the centred spectrum's 2 x 2 block
// rows 2r, 2r+1 and columns 2c, 2c+1; centred row y is unshifted row
// (y + H/2) mod H. The DC bin counts as zero (the mean is removed).
__device__ __forceinline__ float cell_value(const float2* F, uint32_t W, uint32_t H, uint32_t r, uint32_t c) {
  float m = 0.f;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const uint32_t y = (2 * r + a + H / 2) & (H - 1);
      const uint32_t x = (2 * c + b + W / 2) & (W - 1);
      const float2 v = F[size_t(y) * W + x];
      if (x | y) m += sqrtf(fmaf(v.x, v.x, v.y * v.y));
    }
  return log1pf(0.25f * m);
}

// One CTA per frame: mean and deviation of the cells in float64, then the
// standardised cells rounded to bfloat16 (nearest, ties to even).
__global__ void __launch_bounds__(FT_NT) k_af_features(const float2* spec, uint32_t W, uint32_t H,
                                                       __nv_bfloat16* out) {
  const uint32_t f = blockIdx.x;
  const float2* F = spec + size_t(f) * W * H;
  const uint32_t cw = W / 2, ncell = (W / 2) * (H / 2);
  // a thread's few cells summed in float32 (values below ~20), the block in float64
  float f1 = 0.f, f2 = 0.f;
  for (uint32_t e = threadIdx.x; e < ncell; e += FT_NT) {
    const float v = cell_value(F, W, H, e / cw, e % cw);
    f1 += v;
    f2 = fmaf(v, v, f2);
  }
  double s1 = f1, s2 = f2;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
  }
  __shared__ double red[2][FT_NT / 32];
  __shared__ float stat[2];
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = s1;
    red[1][threadIdx.x >> 5] = s2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t1 = 0.0, t2 = 0.0;
    for (int w = 0; w < FT_NT / 32; ++w) {
      t1 += red[0][w];
      t2 += red[1][w];
    }
    const double mean = t1 / ncell;
    const double var = t2 / ncell - mean * mean;
    stat[0] = float(mean);
    stat[1] = var > 0.0 ? float(1.0 / sqrt(var)) : 0.f;
  }
  __syncthreads();
  const float mean = stat[0], inv = stat[1];
  __nv_bfloat16* o = out + size_t(f) * ncell;
  for (uint32_t e = threadIdx.x; e < ncell; e += FT_NT)
    o[e] = __float2bfloat16_rn((cell_value(F, W, H, e / cw, e % cw) - mean) * inv);
}

// The network input from precomputed cells, one CTA per frame: the frame's mean
// and deviation from its float64 sums (once), then (v - mean) / deviation rounded
// to bfloat16 (as k_af_features).
__global__ void __launch_bounds__(FT_NT) k_af_standardize(const float* cells, const double* sums, uint32_t stride,
                                                         uint32_t ncell, __nv_bfloat16* out) {
  const uint32_t f = blockIdx.x;
  __shared__ float stat[2];
  if (threadIdx.x == 0) {
    const double mean = sums[size_t(f) * stride] / ncell;
    const double var = sums[size_t(f) * stride + 1] / ncell - mean * mean;
    stat[0] = float(mean);
    stat[1] = var > 0.0 ? float(1.0 / sqrt(var)) : 0.f;
  }
  __syncthreads();
  const float m = stat[0], inv = stat[1];
  const float* c = cells + size_t(f) * ncell;
  __nv_bfloat16* o = out + size_t(f) * ncell;
  for (uint32_t e = threadIdx.x; e < ncell; e += FT_NT) o[e] = __float2bfloat16_rn((c[e] - m) * inv);
}

}  // namespace

cudaError_t launch_features(const SpatialArgs& a0, void* out_bf16, cudaStream_t s) {
  if (a0.n == 0) return cudaSuccess;
  SpatialArgs a = a0;
  const uint32_t cells = (a.W / 2) * (a.H / 2);
  __nv_bfloat16* out = static_cast<__nv_bfloat16*>(out_bf16);
  cudaError_t e = pass_by_len<COLS>(a, s);
  if (e != cudaSuccess) return e;
  if (a.W > 256) {
    a.tq = RingRef{a.scratch2, a.n, 0};
    e = pass_by_len<ROWS>(a, s);
    if (e != cudaSuccess) return e;
    k_af_features<<<a.n, FT_NT, 0, s>>>(a.scratch2, a.W, a.H, out);
    return cudaGetLastError();
  }
  // scratch2: the cells [n][H/2][W/2] (floats), then their (sum, sum of squares)
  a.cells = reinterpret_cast<float*>(a.scratch2);
  a.tam_acc = reinterpret_cast<double*>(a.scratch2 + (size_t(a.n) * cells + 1) / 2);
  a.tam_stride = 2;
  e = cudaMemsetAsync(a.tam_acc, 0, size_t(a.n) * 2 * sizeof(double), s);
  if (e == cudaSuccess) e = pass_by_len<CELLS>(a, s);
  if (e != cudaSuccess) return e;
  k_af_standardize<<<a.n, FT_NT, 0, s>>>(a.cells, a.tam_acc, a.tam_stride, cells, out);
  return cudaGetLastError();
}

}  // namespace hv

// k_spatial_strip.cu -- the spatial transform (Sec. III-B.1) of frames with sides 64
// .. 1024 as three (ASP) or two (Fresnel) passes of 1-D FFTs whose operands go from
// global memory straight to registers and back:
//
//   columns  raw [y][x] -> column FFT -> S1 [ky][x]. ASP: two real columns are one
//            complex line, the two spectra separated in registers after, and only
//            ky = 0 .. H/2 stored (a real column's spectrum is Hermitian). Fresnel:
//            one column times the chirp per line, every ky stored.
//   rows     ASP: S1 row ky -> row FFT W(kx); IFFT(W H) is row ky of S2, and row H - ky
//            is conj(IFFT(W conj(H))): the spectrum there is conj(W(-kx)), and H(ky, kx)
//            depends on kx^2 and ky^2 only. So H/2 + 1 forward and H inverse row FFTs a
//            frame. Fresnel: S1 row ky -> row FFT -> time queue [ky][kx].
//   columns  ASP: S2 [ky][x] -> column IFFT -> time queue [y][x].
//
// Every FFT is two register stages (radices 8 x 8 .. 32 x 32) with one exchange
// through shared memory between them. A column CTA takes BT neighbouring lines, lines
// fastest across lanes, so that a load or store of one row is BT x 8 contiguous
// bytes; a row FFT is carried by 8, 16 or 32 lanes of one warp, which then needs no
// CTA barrier. Nothing is staged: the up to 32 loads that feed a thread's first stage
// are all in flight at once, and several CTAs per SM overlap one another's loads,
// arithmetic and stores.
//
// Bound by memory: ASP moves 2 + 4 | 4 + 8 | 8 + 8 bytes per 16-bit pixel (34 against the
// 42 of passes over full spectra). Us a frame in large launches, against the persistent
// block-wide passes that staged each strip of 16 lines in shared memory (two strips per
// CTA, so one or two CTAs per SM from 512 points on): 256 x 256 ASP 0.53 -> 0.37, Fresnel
// 0.33 -> 0.31; 512 x 512 3.14 -> 1.89 and 1.65 -> 1.36; 1024 x 1024 17.0 -> 8.9 and
// 8.4 -> 6.1; 128 x 128 0.139 -> 0.107 and 0.081 -> 0.083. Callers with more frames than one
// launch takes queue up to four launches side by side: 0.34 and 0.27, 1.74 and 1.21, 9.6 and
// 5.6 for runs of 4,096, 1,024 and 256 frames of 256, 512 and 1024 (with float32 constants in
// the 32-point DFT, further off, 1.73 and 1.21, 9.4 and 5.5).
#include "strip_dev.cuh"
#include "hv_internal.h"
#include "../../include/hv.h"

namespace hv {

namespace {

// Column FFT of raw strips. ASP: BT lines of two columns, S1 [0 .. H/2][W];
// Fresnel: BT lines of one column, S1 [H][W].
template <int L, bool ASP>
__global__ void __launch_bounds__(ColCfg<L>::NT, ColCfg<L>::CTAS) k_strip_cols(SpatialArgs a, uint32_t nitems,
                                                                              uint32_t strips) {
  using C = ColCfg<L>;
  extern __shared__ __align__(16) unsigned char smem[];
  float2* buf = reinterpret_cast<float2*>(smem);
  float2* tw = buf + C::ROWS * C::BT;
  load_stage_twiddles<C::R1, C::NTW, C::NT>(tw, a.tw_h);
  const int b = threadIdx.x % C::BT, t = threadIdx.x / C::BT;
  const uint32_t W = a.W;
  for (uint32_t item = blockIdx.x; item < nitems; item += gridDim.x) {
    const uint32_t i = item / strips, s = item % strips;
    const size_t frame = ((a.raw.slot0 + i) % a.raw.cap) * size_t(W) * L;
    float2 v[C::I1][C::R1];
    load_raw_strip<L, ASP>(a, frame, s, t, b, v);
    col_stage1<L, -1>(v, buf, t, b);
    float2 u[C::I2][C::R2];
    col_stage2<L, -1>(u, buf, tw, t, b);
    if constexpr (!ASP) {
      float2* out = a.scratch1 + size_t(i) * L * W + size_t(s) * C::BT + b;
#pragma unroll
      for (int it = 0; it < C::I2; ++it)
#pragma unroll
        for (int m = 0; m < C::R2; ++m) out[size_t(col_j2<L>(t, it) + C::R1 * m) * W] = u[it][m];
    } else {
      float2* out = a.scratch1 + size_t(i) * (L / 2 + 1) * W + size_t(s) * (2 * C::BT) + 2 * b;
      auto put = [&](int k, float2 z, float2 w) {
        *reinterpret_cast<float4*>(out + size_t(k) * W) = unpack_pair(z, w);
      };
      if constexpr (C::I2 == 2) {
        if (t != 0) {
          // bins t + R1 m in u[0][m], their mirrors (R1 - t) + R1 (R2 - 1 - m) in u[1]
#pragma unroll
          for (int m = 0; m < C::R2 / 2; ++m) {
            put(t + C::R1 * m, u[0][m], u[1][C::R2 - 1 - m]);
            put(C::R1 - t + C::R1 * m, u[1][m], u[0][C::R2 - 1 - m]);
          }
        } else {
          // bins R1 m mirror R1 (R2 - m); bins R1 / 2 + R1 m mirror R1 / 2 + R1 (R2 - 1 - m)
          put(0, u[0][0], u[0][0]);
#pragma unroll
          for (int m = 1; m <= C::R2 / 2; ++m) put(C::R1 * m, u[0][m], u[0][C::R2 - m]);
#pragma unroll
          for (int m = 0; m < C::R2 / 2; ++m) put(C::R1 / 2 + C::R1 * m, u[1][m], u[1][C::R2 - 1 - m]);
        }
      } else {
        __syncthreads();  // every second-stage read is done
#pragma unroll
        for (int m = 0; m < C::R2; ++m) buf[(t + C::R1 * m) * C::BT + b] = u[0][m];
        __syncthreads();
#pragma unroll 4
        for (int k = t; k <= L / 2; k += C::NJ) put(k, buf[k * C::BT + b], buf[((L - k) & (L - 1)) * C::BT + b]);
      }
    }
  }
}

// Column IFFT of strips of S2 [ky][x] -> time queue [y][x].
template <int L>
__global__ void __launch_bounds__(ColCfg<L>::NT, ColCfg<L>::CTAS) k_strip_icols(SpatialArgs a, uint32_t nitems,
                                                                               uint32_t strips) {
  using C = ColCfg<L>;
  extern __shared__ __align__(16) unsigned char smem[];
  float2* buf = reinterpret_cast<float2*>(smem);
  float2* tw = buf + C::ROWS * C::BT;
  load_stage_twiddles<C::R1, C::NTW, C::NT>(tw, a.tw_h);
  const int b = threadIdx.x % C::BT, t = threadIdx.x / C::BT;
  const uint32_t W = a.W;
  for (uint32_t item = blockIdx.x; item < nitems; item += gridDim.x) {
    const uint32_t i = item / strips, s = item % strips;
    const float2* in = a.scratch2 + size_t(i) * L * W + size_t(s) * C::BT + b;
    float2 v[C::I1][C::R1];
#pragma unroll
    for (int it = 0; it < C::I1; ++it)
#pragma unroll
      for (int m = 0; m < C::R1; ++m) v[it][m] = in[size_t(t + C::NJ * it + (L / C::R1) * m) * W];
    col_stage1<L, +1>(v, buf, t, b);
    float2 u[C::I2][C::R2];
    col_stage2<L, +1>(u, buf, tw, t, b);
    float2* out = static_cast<float2*>(a.tq.base) + ((a.tq.slot0 + i) % a.tq.cap) * size_t(L) * W + size_t(s) * C::BT + b;
#pragma unroll
    for (int it = 0; it < C::I2; ++it)
#pragma unroll
      for (int m = 0; m < C::R2; ++m) __stcs(&out[size_t(col_j2<L>(t, it) + C::R1 * m) * W], u[it][m]);
  }
}

// ASP rows: S1 rows 0 .. H/2 of n frames -> S2 rows 0 .. H - 1. Rows 0 and H / 2 are
// their own mirrors (their W is Hermitian in kx, so both products give the same row);
// a last warp with a row too many repeats the last row. Neither needs a branch. Up to 256
// points W stays in registers for the second product; from 512 points on it would take 64
// more of them, and the forward FFT is done again instead (the row is an L1 or L2 hit): a
// sixth more arithmetic for 20 resident warps per SM instead of 12 (us a frame: 512 x 512
// 0.85 -> 0.77, 1024 x 1024 3.70 -> 3.36).
template <int L>
__global__ void __launch_bounds__(RowCfg<L>::NT, RowCfg<L>::ASP_CTAS) k_strip_rows_asp(SpatialArgs a, uint32_t nrows) {
  using C = RowCfg<L>;
  extern __shared__ __align__(16) unsigned char smem[];
  float2* tw = reinterpret_cast<float2*>(smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, jl = lane % C::LP, sub = lane / C::LP;
  float2* rowp = tw + C::NTW + (warp * C::RPW + sub) * C::RS;
  load_stage_twiddles<C::R1, C::NTW, C::NT>(tw, a.tw_w);
  __syncthreads();
  const uint32_t H = a.H, HR = H / 2 + 1;
  for (uint32_t r0 = (blockIdx.x * C::NW + warp) * C::RPW; r0 < nrows; r0 += gridDim.x * C::NW * C::RPW) {
    const uint32_t row = r0 + sub < nrows ? r0 + sub : nrows - 1;
    const uint32_t i = row / HR, ky = row % HR;
    const float2* in = a.scratch1 + size_t(row) * L + jl;
    const float2* h = a.asp_h + size_t(ky) * L + jl;
    float2* out = a.scratch2 + size_t(i) * H * L + jl;
    if constexpr (C::AGAIN) {
#pragma unroll 1
      for (int conj = 0; conj < 2; ++conj) {
        const float sign = conj ? -1.f : 1.f;
        float2 v[C::R1];
#pragma unroll
        for (int m = 0; m < C::R1; ++m) v[m] = in[C::LP * m];
        strip_row_fft<L, -1>(v, rowp, tw, jl);
#pragma unroll
        for (int m = 0; m < C::R1; ++m) {
          const float2 w = __ldg(&h[C::LP * m]);
          v[m] = cmul(v[m], make_float2(w.x, sign * w.y));
        }
        strip_row_fft<L, +1>(v, rowp, tw, jl);
        float2* o = out + size_t(conj ? (H - ky) & (H - 1) : ky) * L;
#pragma unroll
        for (int m = 0; m < C::R1; ++m) o[C::LP * m] = make_float2(v[m].x, sign * v[m].y);
      }
    } else {
      float2 v[C::R1], u[C::R1];
#pragma unroll
      for (int m = 0; m < C::R1; ++m) v[m] = in[C::LP * m];
      strip_row_fft<L, -1>(v, rowp, tw, jl);
#pragma unroll
      for (int m = 0; m < C::R1; ++m) u[m] = cmul(v[m], __ldg(&h[C::LP * m]));
      strip_row_fft<L, +1>(u, rowp, tw, jl);
#pragma unroll
      for (int m = 0; m < C::R1; ++m) out[size_t(ky) * L + C::LP * m] = u[m];
#pragma unroll
      for (int m = 0; m < C::R1; ++m) {
        // read again (an L1 hit): kept from the first product it would cost 2 R1 registers
        float2 w;
        asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];\n" : "=f"(w.x), "=f"(w.y) : "l"(&h[C::LP * m]) : "memory");
        w.y = -w.y;
        u[m] = cmul(v[m], w);
      }
      strip_row_fft<L, +1>(u, rowp, tw, jl);
#pragma unroll
      for (int m = 0; m < C::R1; ++m)
        out[size_t((H - ky) & (H - 1)) * L + C::LP * m] = make_float2(u[m].x, -u[m].y);
    }
  }
}

// Fresnel rows: S1 rows -> row FFT -> time queue [ky][kx].
template <int L>
__global__ void __launch_bounds__(RowCfg<L>::NT, (L >= 512 ? 4 : 6)) k_strip_rows_fft(SpatialArgs a, uint32_t nrows) {
  using C = RowCfg<L>;
  extern __shared__ __align__(16) unsigned char smem[];
  float2* tw = reinterpret_cast<float2*>(smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, jl = lane % C::LP, sub = lane / C::LP;
  float2* rowp = tw + C::NTW + (warp * C::RPW + sub) * C::RS;
  load_stage_twiddles<C::R1, C::NTW, C::NT>(tw, a.tw_w);
  __syncthreads();
  float2 kept[C::KEEP + 1];
#pragma unroll
  for (int m = 0; m < C::KEEP; ++m) kept[m] = tw[m * C::R1 + jl];
  // H is a multiple of the rows of a warp: its rows are all valid and of one frame
  for (uint32_t r0 = (blockIdx.x * C::NW + warp) * C::RPW; r0 < nrows; r0 += gridDim.x * C::NW * C::RPW) {
    const uint32_t row = r0 + sub, i = row / a.H, ky = row % a.H;
    const float2* in = a.scratch1 + size_t(row) * L + jl;
    float2 v[C::R1];
#pragma unroll
    for (int m = 0; m < C::R1; ++m) v[m] = in[C::LP * m];
    strip_row_fft<L, -1, C::KEEP>(v, rowp, tw, jl, kept);
    float2* out = static_cast<float2*>(a.tq.base) + (((a.tq.slot0 + i) % a.tq.cap) * a.H + ky) * size_t(L) + jl;
#pragma unroll
    for (int m = 0; m < C::R1; ++m) __stcs(&out[C::LP * m], v[m]);
  }
}

// ---------------------------------------------------------------- focus sweep
//
// The sweep needs IFFT2(W H_z) of each hologram for every distance z, W its spectrum. W is
// formed once (column FFT, then the row FFT in place on S1 rows 0 .. H / 2); per
// (distance, hologram) only the inverse row and column FFTs run, and many distances share
// a launch (per distance the forward row FFT was repeated over all H rows: 17.8 + 10.4 us
// a distance for 64 holograms of 256 x 256 in 130 launches; 7.7 + 12.5 now in 34).

// Row FFT of S1 rows in place (a last warp with a row too many repeats the last row).
template <int L>
__global__ void __launch_bounds__(RowCfg<L>::NT, (L >= 512 ? 4 : 6)) k_strip_rows_fwd(SpatialArgs a, uint32_t nrows) {
  using C = RowCfg<L>;
  extern __shared__ __align__(16) unsigned char smem[];
  float2* tw = reinterpret_cast<float2*>(smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, jl = lane % C::LP, sub = lane / C::LP;
  float2* rowp = tw + C::NTW + (warp * C::RPW + sub) * C::RS;
  load_stage_twiddles<C::R1, C::NTW, C::NT>(tw, a.tw_w);
  __syncthreads();
  float2 kept[C::KEEP + 1];
#pragma unroll
  for (int m = 0; m < C::KEEP; ++m) kept[m] = tw[m * C::R1 + jl];
  for (uint32_t r0 = (blockIdx.x * C::NW + warp) * C::RPW; r0 < nrows; r0 += gridDim.x * C::NW * C::RPW) {
    float2* at = a.scratch1 + size_t(r0 + sub < nrows ? r0 + sub : nrows - 1) * L + jl;
    float2 v[C::R1];
#pragma unroll
    for (int m = 0; m < C::R1; ++m) v[m] = at[C::LP * m];
    strip_row_fft<L, -1, C::KEEP>(v, rowp, tw, jl, kept);
#pragma unroll
    for (int m = 0; m < C::R1; ++m) at[C::LP * m] = v[m];
  }
}

// Rows of nz distances: row (z, i, ky) of nz n (H / 2 + 1): W of hologram i times H_z, inverse
// row FFT -> S2 rows ky and H - ky of image z n + i (the mirror as in k_strip_rows_asp).
// h: [nz][H / 2 + 1][W].
template <int L>
__global__ void __launch_bounds__(RowCfg<L>::NT, (L >= 512 ? 3 : 5)) k_strip_rows_inv(SpatialArgs a, const float2* h,
                                                                                     uint32_t nrows) {
  using C = RowCfg<L>;
  extern __shared__ __align__(16) unsigned char smem[];
  float2* tw = reinterpret_cast<float2*>(smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, jl = lane % C::LP, sub = lane / C::LP;
  float2* rowp = tw + C::NTW + (warp * C::RPW + sub) * C::RS;
  load_stage_twiddles<C::R1, C::NTW, C::NT>(tw, a.tw_w);
  __syncthreads();
  const uint32_t H = a.H, HR = H / 2 + 1;
  for (uint32_t r0 = (blockIdx.x * C::NW + warp) * C::RPW; r0 < nrows; r0 += gridDim.x * C::NW * C::RPW) {
    const uint32_t row = r0 + sub < nrows ? r0 + sub : nrows - 1;
    const uint32_t image = row / HR, ky = row % HR, z = image / a.n, i = image % a.n;
    const float2* in = a.scratch1 + (size_t(i) * HR + ky) * L + jl;
    const float2* hz = h + (size_t(z) * HR + ky) * L + jl;
    float2* out = a.scratch2 + size_t(image) * H * L + jl;
    float2 u[C::R1];
#pragma unroll
    for (int m = 0; m < C::R1; ++m) u[m] = cmul(in[C::LP * m], __ldg(&hz[C::LP * m]));
    strip_row_fft<L, +1>(u, rowp, tw, jl);
#pragma unroll
    for (int m = 0; m < C::R1; ++m) out[size_t(ky) * L + C::LP * m] = u[m];
#pragma unroll
    for (int m = 0; m < C::R1; ++m) {
      // both read again (L1 hits) rather than kept across the first inverse FFT
      float2 v, w;
      asm volatile("ld.global.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "l"(&in[C::LP * m]) : "memory");
      asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];\n" : "=f"(w.x), "=f"(w.y) : "l"(&hz[C::LP * m]) : "memory");
      w.y = -w.y;
      u[m] = cmul(v, w);
    }
    strip_row_fft<L, +1>(u, rowp, tw, jl);
#pragma unroll
    for (int m = 0; m < C::R1; ++m)
      out[size_t((H - ky) & (H - 1)) * L + C::LP * m] = make_float2(u[m].x, -u[m].y);
  }
}

// sqrt(q), q >= 0: one Newton step on the product by the approximate inverse root, to the last
// bit (another than the rounded root's once in some ten million), without the rounded root's slow
// path, whose call in the loop spilled more than the 16 to 80 bytes the kernel spills from
// 256 points on (256 images of 256 x 256: 49.9 us, 36.4 now). 0 for 0. The coefficients of 60 sweeps
// of sides 64 .. 1024 are 0.91 to 1.00 times as far off the float64 ones as with the rounded root
// and the transforms before.
__device__ __forceinline__ float root(float q) {
  const float r = rsqrtf(fmaxf(q, 1e-37f)), s = q * r;
  return fmaf(0.5f * r, fmaf(-s, s, q), s);
}

// Column IFFT of strips of S2; sum |u| and sum |u|^2 of image z n + i added to the float64
// pair z of hologram i at tam_acc + i tam_stride + 2 z.
template <int L>
__global__ void __launch_bounds__(ColCfg<L>::NT, ColCfg<L>::CTAS) k_strip_icols_sums(SpatialArgs a, uint32_t nitems,
                                                                                    uint32_t strips) {
  using C = ColCfg<L>;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ float red[2][C::NT / 32];
  float2* buf = reinterpret_cast<float2*>(smem);
  float2* tw = buf + C::ROWS * C::BT;
  load_stage_twiddles<C::R1, C::NTW, C::NT>(tw, a.tw_h);
  const int b = threadIdx.x % C::BT, t = threadIdx.x / C::BT;
  const uint32_t W = a.W;
  for (uint32_t item = blockIdx.x; item < nitems; item += gridDim.x) {
    const uint32_t image = item / strips, s = item % strips;
    const float2* in = a.scratch2 + size_t(image) * L * W + size_t(s) * C::BT + b;
    float2 v[C::I1][C::R1];
#pragma unroll
    for (int it = 0; it < C::I1; ++it)
#pragma unroll
      for (int m = 0; m < C::R1; ++m) v[it][m] = in[size_t(t + C::NJ * it + (L / C::R1) * m) * W];
    col_stage1<L, +1>(v, buf, t, b);
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int it = 0; it < C::I2; ++it) {
      float2 u[C::R2];
      col_butterfly2<L, +1>(u, buf, tw, col_j2<L>(t, it), b);
#pragma unroll
      for (int m = 0; m < C::R2; ++m) {
        const float q = fmaf(u[m].x, u[m].x, u[m].y * u[m].y);
        s0 += root(q);
        s1 += q;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    }
    // the barriers of the next item's first stage come before its sums are written here
    if ((threadIdx.x & 31) == 0) {
      red[0][threadIdx.x >> 5] = s0;
      red[1][threadIdx.x >> 5] = s1;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
      float q = 0.f;
#pragma unroll
      for (int w = 0; w < C::NT / 32; ++w) q += red[threadIdx.x][w];
      atomicAdd(&a.tam_acc[size_t(image % a.n) * a.tam_stride + 2 * (image / a.n) + threadIdx.x], double(q));
    }
  }
}

// Row of SpatialArgs::fit.
enum StripKernel { COLS_ASP, COLS, ICOLS, ROWS_ASP, ROWS_FFT, ROWS_FWD, ROWS_INV, ICOLS_SUMS };
static_assert(ICOLS_SUMS + 1 == kStripKernels, "one row per kernel");

constexpr uint32_t side_index(int L) { return L == 64 ? 0 : 1 + side_index(L / 2); }

// Persistent grid: every CTA that fits at once, no more than the items. How many fit is asked
// once per caller's table (the two queries and the attribute took longer than the launch).
template <class K, class... Args>
cudaError_t launch_resident(const SpatialArgs& a, StripKernel row, int L, K kern, int nt, size_t smem, uint32_t ctas,
                            cudaStream_t s, Args... args) {
  uint32_t* fit = a.fit ? a.fit + row * kStripSides + side_index(L) : nullptr;
  uint32_t most = fit ? *fit : 0;
  if (most == 0) {
    int per_sm = 0, dev = 0, nsm = 0;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nt, smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    most = uint32_t(per_sm > 0 ? per_sm : 1) * uint32_t(nsm);
    if (fit) *fit = most;
  }
  kern<<<ctas < most ? ctas : most, nt, smem, s>>>(args...);
  return cudaGetLastError();
}

template <int L, bool ASP>
cudaError_t cols(const SpatialArgs& a, cudaStream_t s) {
  using C = ColCfg<L>;
  const uint32_t strips = a.W / (ASP ? 2 * C::BT : C::BT), items = strips * a.n;
  return launch_resident(a, ASP ? COLS_ASP : COLS, L, k_strip_cols<L, ASP>, C::NT, C::SMEM, items, s, a, items, strips);
}

template <int L>
cudaError_t icols(const SpatialArgs& a, cudaStream_t s) {
  using C = ColCfg<L>;
  const uint32_t strips = a.W / C::BT, items = strips * a.n;
  return launch_resident(a, ICOLS, L, k_strip_icols<L>, C::NT, C::SMEM, items, s, a, items, strips);
}

template <int L>
cudaError_t rows(const SpatialArgs& a, cudaStream_t s) {
  using C = RowCfg<L>;
  constexpr uint32_t per = C::NW * C::RPW;
  if (a.spatial == HV_SPATIAL_ASP) {
    const uint32_t nrows = a.n * (a.H / 2 + 1);
    return launch_resident(a, ROWS_ASP, L, k_strip_rows_asp<L>, C::NT, C::SMEM, (nrows + per - 1) / per, s, a, nrows);
  }
  const uint32_t nrows = a.n * a.H;
  return launch_resident(a, ROWS_FFT, L, k_strip_rows_fft<L>, C::NT, C::SMEM, (nrows + per - 1) / per, s, a, nrows);
}

#define HV_BY_SIDE(side, fn)             \
  switch (side) {                        \
    case 64: e = fn(64); break;          \
    case 128: e = fn(128); break;        \
    case 256: e = fn(256); break;        \
    case 512: e = fn(512); break;        \
    case 1024: e = fn(1024); break;      \
    default: e = cudaErrorInvalidValue;  \
  }

template <int L>
cudaError_t rows_fwd(const SpatialArgs& a, cudaStream_t s) {
  using C = RowCfg<L>;
  constexpr uint32_t per = C::NW * C::RPW;
  const uint32_t nrows = a.n * (a.H / 2 + 1);
  return launch_resident(a, ROWS_FWD, L, k_strip_rows_fwd<L>, C::NT, C::SMEM, (nrows + per - 1) / per, s, a, nrows);
}

template <int L>
cudaError_t rows_inv(const SpatialArgs& a, const float2* h, uint32_t nz, cudaStream_t s) {
  using C = RowCfg<L>;
  constexpr uint32_t per = C::NW * C::RPW;
  const uint32_t nrows = nz * a.n * (a.H / 2 + 1);
  return launch_resident(a, ROWS_INV, L, k_strip_rows_inv<L>, C::NT, C::SMEM, (nrows + per - 1) / per, s, a, h, nrows);
}

template <int L>
cudaError_t icols_sums(const SpatialArgs& a, uint32_t nz, cudaStream_t s) {
  using C = ColCfg<L>;
  const uint32_t strips = a.W / C::BT, items = strips * a.n * nz;
  return launch_resident(a, ICOLS_SUMS, L, k_strip_icols_sums<L>, C::NT, C::SMEM, items, s, a, items, strips);
}

}  // namespace

bool spatial_strip_supported(const SpatialArgs& a) {
  auto ok = [](uint32_t v) { return v >= 64 && v <= 1024; };
  return ok(a.W) && ok(a.H) &&
         (a.spatial == HV_SPATIAL_FRESNEL || (a.spatial == HV_SPATIAL_ASP && a.asp_h != nullptr));
}

cudaError_t launch_spatial_strip(const SpatialArgs& a, cudaStream_t s, int* launches) {
  if (a.n == 0) return cudaSuccess;
  if (!spatial_strip_supported(a)) return cudaErrorInvalidValue;
  const bool asp = a.spatial == HV_SPATIAL_ASP;
  cudaError_t e;
#define HV_COLS(L) (asp ? cols<L, true>(a, s) : cols<L, false>(a, s))
#define HV_ROWS(L) rows<L>(a, s)
#define HV_ICOLS(L) icols<L>(a, s)
  HV_BY_SIDE(a.H, HV_COLS)
  if (e != cudaSuccess) return e;
  HV_BY_SIDE(a.W, HV_ROWS)
  *launches += 2;
  if (e != cudaSuccess || !asp) return e;
  HV_BY_SIDE(a.H, HV_ICOLS)
  ++*launches;
  return e;
}

cudaError_t launch_strip_spectrum(const SpatialArgs& a, cudaStream_t s) {
  cudaError_t e;
#define HV_COLS_ASP(L) cols<L, true>(a, s)
#define HV_ROWS_FWD(L) rows_fwd<L>(a, s)
  HV_BY_SIDE(a.H, HV_COLS_ASP)
  if (e != cudaSuccess) return e;
  HV_BY_SIDE(a.W, HV_ROWS_FWD)
  return e;
}

cudaError_t launch_strip_sweep(const SpatialArgs& a, const float2* h, uint32_t nz, cudaStream_t s) {
  cudaError_t e;
#define HV_ROWS_INV(L) rows_inv<L>(a, h, nz, s)
#define HV_ICOLS_SUMS(L) icols_sums<L>(a, nz, s)
  HV_BY_SIDE(a.W, HV_ROWS_INV)
  if (e != cudaSuccess) return e;
  HV_BY_SIDE(a.H, HV_ICOLS_SUMS)
  return e;
}

}  // namespace hv

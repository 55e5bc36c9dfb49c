// strip_dev.cuh -- two-stage FFTs of the register-direct spatial passes (k_spatial_strip.cu,
// k_spatial_pp.cu): columns of a strip by a CTA, rows by a part of a warp.
#pragma once
#include "fft_dev.cuh"
#include "hv_internal.h"

namespace hv {

// v * exp(DIR 2 pi i k / 32), k = 0..15 (k a compile-time constant after unrolling), by the
// constants as pairs hi + lo.
template <int DIR>
__device__ __forceinline__ float2 tw32_pair(float2 v, int k) {
  constexpr double A[9] = {1.0, 0.98078528040323044913, 0.92387953251128675613, 0.83146961230254523708,
                           0.70710678118654752440, 0.55557023301960222474, 0.38268343236508977173,
                           0.19509032201612826785, 0.0};
  const double c = k <= 8 ? A[k] : -A[16 - k], s = DIR * (k <= 8 ? A[8 - k] : A[k - 8]);
  const float ch = float(c), sh = float(s), cl = float(c - double(ch)), sl = float(s - double(sh));
  return make_float2(fmaf(v.x, ch, fmaf(-v.y, sh, fmaf(v.x, cl, -(v.y * sl)))),
                     fmaf(v.y, ch, fmaf(v.x, sh, fmaf(v.y, cl, v.x * sl))));
}

// dft<R> of fft_dev.cuh; R = 32 with the constants of its last stage to 48 bits. Rounded
// constants meet every butterfly, mostly downwards: with float32 ones lengths of 512 and 1024
// came out 3.4e-8 and 4.2e-8 short on the mean, where 16 x 16 x 2 and 16 x 16 x 4 points lose
// 2.7e-8, and M0 of 1024 x 1024 (four transforms, squared) was 3.0e-7 off the float64 result instead
// of 1.7e-7. With the pairs 2.4e-8 at both.
template <int R, int DIR>
__device__ __forceinline__ void strip_dft(float2 (&v)[R]) {
  if constexpr (R != 32) {
    dft<R, DIR>(v);
  } else {
    float2 e[16], o[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      e[i] = v[2 * i];
      o[i] = v[2 * i + 1];
    }
    dft<16, DIR>(e);
    dft<16, DIR>(o);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float2 t = k == 0 ? o[0] : (k == 8 ? mul_i<DIR>(o[8]) : tw32_pair<DIR>(o[k], k));
      v[k] = padd(e[k], t);
      v[k + 16] = psub(e[k], t);
    }
  }
}

// Column CTAs: L = R1 x R2, BT lines, NT threads. A thread holds I1 first-stage and I2
// second-stage butterflies of one line. 16 lines are 128-byte runs of a row; 1024 points keep
// 8, where 16 would leave one CTA of 512 threads on an SM (columns and inverse columns of 1024 x
// 1024 ASP, us a frame: 8 lines 1.83 and 3.58, 16 lines 2.03 and 3.90; of 512 x 512, with 128
// threads and 256: 0.363 and 0.880 against 0.341 and 0.772).
template <int L>
struct ColCfg {
  static constexpr int R1 = L >= 512 ? 32 : (L >= 128 ? 16 : 8);
  static constexpr int R2 = L / R1;
  static constexpr int BT = L == 1024 ? 8 : 16;
  static constexpr int NT = L == 64 ? 64 : (L >= 512 ? 256 : 128);
  static constexpr int NJ = NT / BT;          // threads per line
  static constexpr int I1 = (L / R1) / NJ;    // first-stage butterflies per thread
  static constexpr int I2 = (L / R2) / NJ;    // second-stage butterflies per thread
  static constexpr int NTW = (R2 - 1) * R1;   // second-stage twiddles
  static constexpr int PAD = BT == 8 ? 1 : 0; // padding rows per R1 rows of the exchange buffer
  static constexpr int ROWS = L + PAD * R2;
  static constexpr size_t SMEM = (size_t(ROWS) * BT + NTW) * sizeof(float2);
  static constexpr int CTAS = L >= 512 ? 2 : (L == 64 ? 12 : 5);
  static_assert(I1 >= 1 && I2 >= 1 && I2 <= 2 && L / R2 == R1, "two-stage plan");
};

// Second-stage twiddles w_L^{j m} at (m - 1) R1 + j, from the length-L table.
template <int R1, int NTW, int NT>
__device__ __forceinline__ void load_stage_twiddles(float2* tw, const float2* __restrict__ table) {
  for (int e = threadIdx.x; e < NTW; e += NT) tw[e] = __ldg(&table[(e / R1 + 1) * (e % R1)]);
}

// The exchange buffer holds row r at r + PAD (r / R1). With 8 lines a half-warp covers
// two rows: the padding keeps the two of a first-stage store (r and r + R1) in different
// bank halves, at addresses that stay a register plus a constant (an XOR swizzle here
// and in the row FFTs left 32 and more addresses live across the loop, and spilled).

// First stage of a thread's line b (butterflies j = t + NJ it, inputs in v), exchange.
template <int L, int DIR>
__device__ __forceinline__ void col_stage1(float2 (&v)[ColCfg<L>::I1][ColCfg<L>::R1], float2* buf, int t, int b) {
  using C = ColCfg<L>;
#pragma unroll
  for (int it = 0; it < C::I1; ++it) strip_dft<C::R1, DIR>(v[it]);
  __syncthreads();  // the previous item's second stage has read the buffer
#pragma unroll
  for (int it = 0; it < C::I1; ++it)
#pragma unroll
    for (int m = 0; m < C::R1; ++m) buf[((t + C::NJ * it) * (C::R1 + C::PAD) + m) * C::BT + b] = v[it][m];
  __syncthreads();
}

// Butterfly of item `it` of the second stage: with two per thread, t and its mirror
// R1 - t (0 and R1 / 2 for t = 0), so that bins k and L - k of a line meet in a thread.
template <int L>
__device__ __forceinline__ int col_j2(int t, int it) {
  using C = ColCfg<L>;
  if (C::I2 == 1 || it == 0) return t;
  return t == 0 ? C::R1 / 2 : C::R1 - t;
}

// Second stage of butterfly j: its bins j + R1 m end in u[m].
template <int L, int DIR>
__device__ __forceinline__ void col_butterfly2(float2 (&u)[ColCfg<L>::R2], const float2* buf, const float2* tw, int j,
                                               int b) {
  using C = ColCfg<L>;
#pragma unroll
  for (int m = 0; m < C::R2; ++m) {
    u[m] = buf[(j + (C::R1 + C::PAD) * m) * C::BT + b];
    if (m > 0) {
      float2 w = tw[(m - 1) * C::R1 + j];
      if (DIR > 0) w.y = -w.y;
      u[m] = cmul(u[m], w);
    }
  }
  strip_dft<C::R2, DIR>(u);
}

// Second stage: bins j + R1 m of butterfly j = col_j2(t, it) end in u[it][m].
template <int L, int DIR>
__device__ __forceinline__ void col_stage2(float2 (&u)[ColCfg<L>::I2][ColCfg<L>::R2], const float2* buf,
                                           const float2* tw, int t, int b) {
#pragma unroll
  for (int it = 0; it < ColCfg<L>::I2; ++it) col_butterfly2<L, DIR>(u[it], buf, tw, col_j2<L>(t, it), b);
}

// Spectra of the two real columns packed in one line, from Z(k) and Z(L - k):
// A(k) = (Z(k) + conj Z(-k)) / 2, B(k) = (Z(k) - conj Z(-k)) / 2i.
__device__ __forceinline__ float4 unpack_pair(float2 z, float2 w) {
  return make_float4(0.5f * (z.x + w.x), 0.5f * (z.y - w.y), 0.5f * (z.y + w.y), 0.5f * (w.x - z.x));
}

// First-stage inputs of a raw strip's line b: pixels of frame `frame` (its first pixel's
// index). ASP: columns 2 b and 2 b + 1 of strip s as one complex line, read as one word
// where the frames are aligned for it; Fresnel: column b times the chirp.
template <int L, bool ASP>
__device__ __forceinline__ void load_raw_strip(const SpatialArgs& a, size_t frame, uint32_t s, int t, int b,
                                               float2 (&v)[ColCfg<L>::I1][ColCfg<L>::R1]) {
  using C = ColCfg<L>;
  const uint32_t W = a.W;
  const bool u8 = a.in_kind == IN_U8;
  if constexpr (ASP) {
    const size_t x = size_t(s) * (2 * C::BT) + 2 * b;
    const size_t at = frame + x;
    if (u8) {
      const unsigned char* p = static_cast<const unsigned char*>(a.raw.base) + at;
      if ((reinterpret_cast<uintptr_t>(a.raw.base) & 1) == 0) {
#pragma unroll
        for (int it = 0; it < C::I1; ++it)
#pragma unroll
          for (int m = 0; m < C::R1; ++m) {
            const uint32_t q =
                *reinterpret_cast<const uint16_t*>(p + size_t(t + C::NJ * it + (L / C::R1) * m) * W);
            v[it][m] = make_float2(float(q & 0xffu), float(q >> 8));
          }
      } else {
#pragma unroll
        for (int it = 0; it < C::I1; ++it)
#pragma unroll
          for (int m = 0; m < C::R1; ++m) {
            const unsigned char* q = p + size_t(t + C::NJ * it + (L / C::R1) * m) * W;
            v[it][m] = make_float2(float(q[0]), float(q[1]));
          }
      }
    } else {
      const uint16_t* p = static_cast<const uint16_t*>(a.raw.base) + at;
      if ((reinterpret_cast<uintptr_t>(a.raw.base) & 3) == 0) {
#pragma unroll
        for (int it = 0; it < C::I1; ++it)
#pragma unroll
          for (int m = 0; m < C::R1; ++m) {
            const uint32_t q =
                *reinterpret_cast<const uint32_t*>(p + size_t(t + C::NJ * it + (L / C::R1) * m) * W);
            v[it][m] = make_float2(float(q & 0xffffu), float(q >> 16));
          }
      } else {
#pragma unroll
        for (int it = 0; it < C::I1; ++it)
#pragma unroll
          for (int m = 0; m < C::R1; ++m) {
            const uint16_t* q = p + size_t(t + C::NJ * it + (L / C::R1) * m) * W;
            v[it][m] = make_float2(float(q[0]), float(q[1]));
          }
      }
    }
  } else {
    const size_t x = size_t(s) * C::BT + b;
    const float2 cx = __ldg(&a.chirp_x[x]);
    float r[C::I1][C::R1];
    if (u8) {
      const unsigned char* p = static_cast<const unsigned char*>(a.raw.base) + frame + x;
#pragma unroll
      for (int it = 0; it < C::I1; ++it)
#pragma unroll
        for (int m = 0; m < C::R1; ++m) r[it][m] = float(p[size_t(t + C::NJ * it + (L / C::R1) * m) * W]);
    } else {
      const uint16_t* p = static_cast<const uint16_t*>(a.raw.base) + frame + x;
#pragma unroll
      for (int it = 0; it < C::I1; ++it)
#pragma unroll
        for (int m = 0; m < C::R1; ++m) r[it][m] = float(p[size_t(t + C::NJ * it + (L / C::R1) * m) * W]);
    }
#pragma unroll
    for (int it = 0; it < C::I1; ++it)
#pragma unroll
      for (int m = 0; m < C::R1; ++m)
        v[it][m] = cscale(cmul(__ldg(&a.chirp_y[t + C::NJ * it + (L / C::R1) * m]), cx), r[it][m]);
  }
}

// Row FFTs: LP lanes carry a row (lane jl holds elements jl + LP m in v[m]), RPW rows
// per warp, four warps per CTA.
template <int L>
struct RowCfg {
  static constexpr int R1 = ColCfg<L>::R1, R2 = ColCfg<L>::R2;
  static constexpr int LP = L / R1, RPW = 32 / LP, NW = 4, NT = 32 * NW;
  static constexpr int I2 = R1 / LP;
  static constexpr int NTW = (R2 - 1) * R1;
  static constexpr int RS = L + L / R1;  // exchange row: element e at e + e / R1
  static constexpr size_t SMEM = (size_t(NW) * RPW * RS + NTW) * sizeof(float2);
  static constexpr int KEEP = L >= 512 ? 8 : 0;  // twiddles in registers (single-FFT kernels)
  static constexpr bool AGAIN = L >= 512;  // ASP rows: the forward FFT twice
  static constexpr int ASP_CTAS = L >= 512 || L == 64 ? 5 : 4;
};

// L-point FFT of a row through its exchange buffer rowp (padded: the 16 lanes of a
// half-warp always meet 16 different bank pairs, two rows of 8 lanes too). On return
// bin jl + LP m is in v[m]. kept: the first KEEP twiddles of the lane's first butterfly, the same
// for every row, where the kernel has registers to hold them (with all 31 and 32 more values read
// from shared memory in one go, rows of 1024 points waited for its queue: Fresnel passes 6.55 us
// a frame, 5.60 with 8 kept, 5.59 with 16).
template <int L, int DIR, int KEEP = 0>
__device__ __forceinline__ void strip_row_fft(float2 (&v)[RowCfg<L>::R1], float2* rowp, const float2* tw, int jl,
                                              const float2* kept = nullptr) {
  using C = RowCfg<L>;
  strip_dft<C::R1, DIR>(v);
  __syncwarp();
#pragma unroll
  for (int m = 0; m < C::R1; ++m) rowp[(C::R1 + 1) * jl + m] = v[m];
  __syncwarp();
#pragma unroll
  for (int i = 0; i < C::I2; ++i) {
    const int j = jl + C::LP * i;
    float2 u[C::R2];
#pragma unroll
    for (int m = 0; m < C::R2; ++m) {
      u[m] = rowp[(C::R1 + 1) * m + j];
      if (m > 0) {
        float2 w = i == 0 && m <= KEEP ? kept[m - 1] : tw[(m - 1) * C::R1 + j];
        if (DIR > 0) w.y = -w.y;
        u[m] = cmul(u[m], w);
      }
    }
    strip_dft<C::R2, DIR>(u);
#pragma unroll
    for (int m = 0; m < C::R2; ++m) v[i + C::I2 * m] = u[m];
  }
}

}  // namespace hv

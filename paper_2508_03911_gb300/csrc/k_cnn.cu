// k_cnn.cu -- the autofocus network's training and inference kernels.
//
// Network (input 1 x 128 x 128, the binned log-spectrum of a hologram):
//   four 3 x 3 convolutions, stride 2, zero padding 1, channels 1 -> 16 -> 32 ->
//   64 -> 64, each followed by ReLU (outputs 64^2, 32^2, 16^2, 8^2); global average
//   pool; dense 64 -> 32 with ReLU; dense 32 -> 1. The output predicts the
//   normalised distance (z - 0.35) / 0.25; the loss is the batch mean of the
//   squared error.
// Arithmetic: activations and convolution weights in bfloat16, every product
// accumulated in float32 (the forward of layers 2-4 on the tensor cores, in
// k_conv_tc.cu; layer 1 and the backward pass here on the CUDA cores); the dense layers, gradients and the Adam state in
// float32. Layouts: activations [n][c][h][w]; the flat float32 parameter vector
// holds w1 [16][1][3][3], b1, w2 [32][16][3][3], b2, w3, b3, w4, b4, f1w [32][64],
// f1b, f2w [1][32], f2b; a bfloat16 mirror of it feeds the convolutions.
#include <cuda_bf16.h>

#include "cnn_internal.h"

namespace hv {
namespace cnn {

namespace {

constexpr int NT = 256;

__device__ __forceinline__ float bf(const __nv_bfloat16 v) { return __bfloat162float(v); }

// ------------------------------------------------------------------ forward
//
// The 3 x 9 inputs of 4 neighbouring outputs 4 q .. 4 q + 3 of row i of layer 1: columns 8 q
// - 1 .. 8 q + 7 of rows 2 i - 1 .. 2 i + 1 (zero outside). VEC: x 16-byte aligned. The left
// column comes from the neighbouring lane (16 lanes hold a row).
template <bool VEC>
__device__ __forceinline__ void load_inputs1(const __nv_bfloat16* __restrict__ xn, int i, int q, float (&xv)[3][9]) {
  constexpr int HI = 128;
#pragma unroll
  for (int di = 0; di < 3; ++di) {
    const int yy = 2 * i + di - 1;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    __nv_bfloat162* p = reinterpret_cast<__nv_bfloat162*>(&v);
    if (yy >= 0) {
      const __nv_bfloat16* row = xn + yy * HI + 8 * q;
      if (VEC) v = *reinterpret_cast<const uint4*>(row);
      else
        for (int e = 0; e < 4; ++e) p[e] = __nv_bfloat162(row[2 * e], row[2 * e + 1]);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 f = __bfloat1622float2(p[e]);
      xv[di][1 + 2 * e] = f.x;
      xv[di][2 + 2 * e] = f.y;
    }
    const float left = __shfl_up_sync(0xffffffffu, xv[di][8], 1);
    xv[di][0] = q == 0 ? 0.f : left;
  }
}

// Layer 1 (one input channel): y[n][o][i][j] = relu(b[o] + sum_{di,dj} w[o][di][dj]
// x[n][2i+di-1][2j+dj-1]). Bound by its output (67 MB at n = 512). A thread forms 4
// neighbouring pixels of all 16 channels from inputs in registers and broadcast weights
// (staging input rows and weights per 4 channels x 4 pixels took 39 us at n = 512; 23 now).
template <bool VEC>
__global__ void __launch_bounds__(NT) k_conv1(const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ w,
                                              const float* __restrict__ bias, __nv_bfloat16* __restrict__ y) {
  constexpr int HO = 64;
  __shared__ __align__(16) float ws[9][16];
  __shared__ float bs[16];
  const int tid = threadIdx.x, q = tid & 15;
  if (tid < 144) ws[tid % 9][tid / 9] = bf(w[tid]);
  if (tid < 16) bs[tid] = bias[tid];
  __syncthreads();
  const uint32_t row = blockIdx.x * (NT / 16) + tid / 16;  // 16 rows of 64 pixels per CTA
  const uint32_t n = row / HO;
  const int i = int(row % HO);
  float xv[3][9];
  load_inputs1<VEC>(x + size_t(n) * 128 * 128, i, q, xv);
  float acc[16][4];
#pragma unroll
  for (int o = 0; o < 16; ++o)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[o][e] = 0.f;
#pragma unroll
  for (int t = 0; t < 9; ++t)
#pragma unroll
    for (int o = 0; o < 16; o += 4) {
      const float4 wv = *reinterpret_cast<const float4*>(&ws[t][o]);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float v = xv[t / 3][2 * e + t % 3];
        acc[o][e] = fmaf(wv.x, v, acc[o][e]);
        acc[o + 1][e] = fmaf(wv.y, v, acc[o + 1][e]);
        acc[o + 2][e] = fmaf(wv.z, v, acc[o + 2][e]);
        acc[o + 3][e] = fmaf(wv.w, v, acc[o + 3][e]);
      }
    }
#pragma unroll
  for (int o = 0; o < 16; ++o) {
    __align__(8) __nv_bfloat16 v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = __float2bfloat16_rn(fmaxf(acc[o][e] + bs[o], 0.f));
    *reinterpret_cast<uint2*>(y + ((size_t(n) * 16 + o) * HO + i) * HO + 4 * q) = *reinterpret_cast<uint2*>(v);
  }
}

// ------------------------------------------------------------ input gradient
//
// dX[n][c][y][x] = sum_{o,di,dj: y = 2i+di-1, x = 2j+dj-1} w[o][c][di][dj] dZ[n][o][i][j],
// times the ReLU mask of the layer input (its stored activation > 0): the
// result is the previous layer's dZ.
//
// Bound by the FP32 pipe (2.4 GFLOP a layer at n = 256). The four inputs (2i, 2j) ..
// (2i+1, 2j+1) take the 9 taps between them from dZ at (i, j), (i, j+1), (i+1, j) and
// (i+1, j+1), so a thread owns 4 channels x QJ such quads of one row: per output
// channel o, 9 broadcast float4 weights and 2 (QJ + 1) values feed 36 QJ multiply-adds
// (a tile of 4 inputs of one parity class took 4 to 8 loads for 16 to 64). A CTA covers
// 8 rows of quads of one image and 4 CG channels, dZ and weights staged OC output
// channels at a time. n = 256: layers 4, 3, 2 in 129, 195, 198 us before, 52, 81, 83 now.
template <int CI, int CO, int HI>
struct DxCfg {
  static constexpr int HO = HI / 2;
  static constexpr int QJ = HO == 8 ? 2 : 4;             // quads along a row per thread
  static constexpr int GJ = HO / QJ;                     // threads along a row
  static constexpr int CG = CI < 32 ? CI / 4 : 8;        // channel groups of 4 per CTA
  static constexpr int SETS = 8 * GJ / 32;               // warps per channel group
  static constexpr int NTX = CG * SETS * 32;
  static constexpr int OC = 16;
  static constexpr int BANDS = HO / 8, CPARTS = CI / (4 * CG);
  static_assert(SETS >= 1 && HO % 8 == 0 && CO % OC == 0, "tile");
};

template <int CI, int CO, int HI>
__global__ void __launch_bounds__(DxCfg<CI, CO, HI>::NTX, 512 / DxCfg<CI, CO, HI>::NTX)
    k_conv_dx(const float* __restrict__ dz, const __nv_bfloat16* __restrict__ w,
              const __nv_bfloat16* __restrict__ aprev, float* __restrict__ dprev) {
  using D = DxCfg<CI, CO, HI>;
  constexpr int HO = D::HO, QJ = D::QJ, CG = D::CG, OC = D::OC;
  __shared__ __align__(16) float zs[OC][9][HO];       // dZ rows i0 .. i0 + 8
  __shared__ __align__(16) float ws[OC][CG][9][4];
  const int n = blockIdx.x / D::BANDS, i0 = (blockIdx.x % D::BANDS) * 8, cpart = blockIdx.y * CG * 4;
  const int tid = threadIdx.x, cg = tid / (32 * D::SETS), q = tid % (32 * D::SETS);
  const int r = q / D::GJ, j0 = (q % D::GJ) * QJ;
  const bool last = j0 + QJ == HO;  // dZ beyond the last column is zero
  float acc[4][4][QJ];              // channel, 2 py + px, quad
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int x = 0; x < QJ; ++x) acc[c][k][x] = 0.f;
  for (int o0 = 0; o0 < CO; o0 += OC) {
    __syncthreads();
    for (int e = tid; e < OC * 9 * (HO / 4); e += D::NTX) {
      const int c4 = e % (HO / 4), row = (e / (HO / 4)) % 9, o = e / (9 * (HO / 4));
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i0 + row < HO)
        v = *reinterpret_cast<const float4*>(dz + ((size_t(n) * CO + o0 + o) * HO + i0 + row) * HO + 4 * c4);
      *reinterpret_cast<float4*>(&zs[o][row][4 * c4]) = v;
    }
    for (int e = tid; e < OC * CG * 36; e += D::NTX) {
      const int t = e % 9, c = (e / 9) % (4 * CG), o = e / (36 * CG);
      ws[o][c >> 2][t][c & 3] = bf(w[(size_t(o0 + o) * CI + cpart + c) * 9 + t]);
    }
    __syncthreads();
#pragma unroll 1
    for (int o = 0; o < OC; ++o) {
      float z0[QJ + 1], z1[QJ + 1];
#pragma unroll
      for (int x = 0; x < QJ; ++x) {
        z0[x] = zs[o][r][j0 + x];
        z1[x] = zs[o][r + 1][j0 + x];
      }
      // the next value of the row, or (last thread) whatever follows it, unused
      z0[QJ] = last ? 0.f : zs[o][r][(j0 + QJ) & (HO - 1)];
      z1[QJ] = last ? 0.f : zs[o][r + 1][(j0 + QJ) & (HO - 1)];
      auto tap = [&](int t, int k, const float* z) {
        const float4 wv = *reinterpret_cast<const float4*>(&ws[o][cg][t][0]);
#pragma unroll
        for (int x = 0; x < QJ; ++x) {
          acc[0][k][x] = fmaf(wv.x, z[x], acc[0][k][x]);
          acc[1][k][x] = fmaf(wv.y, z[x], acc[1][k][x]);
          acc[2][k][x] = fmaf(wv.z, z[x], acc[2][k][x]);
          acc[3][k][x] = fmaf(wv.w, z[x], acc[3][k][x]);
        }
      };
      // tap 3 di + dj: di = 1 reaches even y, di = 2 odd y from dZ row i, di = 0 from row
      // i + 1; columns alike
      tap(4, 0, z0);
      tap(5, 1, z0);
      tap(3, 1, z0 + 1);
      tap(7, 2, z0);
      tap(1, 2, z1);
      tap(8, 3, z0);
      tap(6, 3, z0 + 1);
      tap(2, 3, z1);
      tap(0, 3, z1 + 1);
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int py = 0; py < 2; ++py) {
      const size_t at = ((size_t(n) * CI + cpart + 4 * cg + c) * HI + 2 * (i0 + r) + py) * HI + 2 * j0;
#pragma unroll
      for (int x = 0; x < QJ; x += 2) {  // inputs 2 (j0 + x) .. + 3
        const uint2 m = *reinterpret_cast<const uint2*>(aprev + at + 2 * x);
        const __nv_bfloat162 lo = *reinterpret_cast<const __nv_bfloat162*>(&m.x);
        const __nv_bfloat162 hi = *reinterpret_cast<const __nv_bfloat162*>(&m.y);
        *reinterpret_cast<float4*>(dprev + at + 2 * x) =
            make_float4(bf(lo.x) > 0.f ? acc[c][2 * py][x] : 0.f, bf(lo.y) > 0.f ? acc[c][2 * py + 1][x] : 0.f,
                        bf(hi.x) > 0.f ? acc[c][2 * py][x + 1] : 0.f,
                        bf(hi.y) > 0.f ? acc[c][2 * py + 1][x + 1] : 0.f);
      }
    }
}

// ----------------------------------------------------------- weight gradient
//
// dW[o][c][t] = sum over pixels (n, i, j) of dZ[n][o][i][j] x[n][c][2i+di-1][2j+dj-1]
// (t = 3 di + dj), db[o] = sum dZ.
//
// Layers 2-4, bound by the FP32 pipe: a thread owns 8 output channels x the 9 taps of one
// input channel and walks output pixels along a row, its 3 x 3 inputs sliding by two
// columns: 2 broadcast float4 of dZ and 6 inputs from shared memory feed 72 multiply-adds
// (a 4 x 4 tile of an im2col product took 2 float4 for 16). A CTA of 256 threads (32
// input channels x 8 groups of outputs, or 16 x 4 x 4 pixel subsets) stages bands of 64
// output pixels and keeps its sums in registers over all of its bands; one partial per
// CTA, summed in CTA order by k_sum_parts, so the result does not depend on scheduling.
// n = 256: layers 4, 3, 2 in 94, 184, 286 us before, 56, 86, 96 now.
template <int CI, int CO, int HI>
struct DwCfg {
  static constexpr int HO = HI / 2;
  static constexpr int CC = CI < 32 ? CI : 32, CPARTS = CI / CC;  // input channels per CTA
  static constexpr int OG = CO / 8;
  static constexpr int SUB = NT / (CC * OG);                      // pixel subsets
  static constexpr int RB = 64 / HO, BANDS = HO / RB;             // output rows of a band, bands per image
  static constexpr int SR = 2 * RB + 1, SC = HI + 1;              // staged input rows, columns -1 .. HI - 1
  static constexpr int ZLD = CO + 4;
  static constexpr int XS = CC * SR * SC;
  static constexpr size_t SMEM = (64 * ZLD + XS) * sizeof(float);
  static constexpr int PART = CO * CC * 9 + CO;                   // floats of a partial: dW, then db
  static_assert(SUB >= 1 && CC * OG * SUB == NT && (SR * SC) % 2 == 1 && 64 % SUB == 0, "tile");
};

template <int CI, int CO, int HI>
__global__ void __launch_bounds__(NT, 2) k_conv_dw(const float* __restrict__ dz, const __nv_bfloat16* __restrict__ x,
                                                   uint32_t nbands, float* __restrict__ part) {
  using D = DwCfg<CI, CO, HI>;
  constexpr int HO = D::HO, PPS = 64 / D::SUB;  // pixels per subset
  extern __shared__ __align__(16) float sm[];
  float* zs = sm;                  // [64 pixels][ZLD]
  float* xs = sm + 64 * D::ZLD;    // [CC][SR][SC]
  const int tid = threadIdx.x, c = tid % D::CC, og = (tid / D::CC) % D::OG, sub = tid / (D::CC * D::OG);
  const int c0 = blockIdx.y * D::CC;
  float acc[8][9], accb = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k)
#pragma unroll
    for (int t = 0; t < 9; ++t) acc[k][t] = 0.f;
  for (uint32_t band = blockIdx.x; band < nbands; band += gridDim.x) {
    const uint32_t n = band / D::BANDS;
    const int i0 = int(band % D::BANDS) * D::RB;
    __syncthreads();
    const float* zsrc = dz + size_t(n) * CO * HO * HO + i0 * HO;
    for (int e = tid; e < CO * 64; e += NT) zs[(e % 64) * D::ZLD + e / 64] = zsrc[size_t(e / 64) * HO * HO + e % 64];
    for (int e = tid; e < D::CC * D::SR * (HI / 2); e += NT) {
      const int q = e % (HI / 2), row = (e / (HI / 2)) % D::SR, ch = e / (D::SR * (HI / 2));
      const int yy = 2 * i0 - 1 + row;
      float2 v = make_float2(0.f, 0.f);
      if (yy >= 0)
        v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(
            x + ((size_t(n) * CI + c0 + ch) * HI + yy) * HI + 2 * q));
      float* d = xs + (ch * D::SR + row) * D::SC + 1 + 2 * q;
      d[0] = v.x;
      d[1] = v.y;
    }
    for (int e = tid; e < D::CC * D::SR; e += NT) xs[e * D::SC] = 0.f;  // column -1
    __syncthreads();
    if (blockIdx.y == 0) {  // bias: pixels tid / CO + k NT / CO of output channel tid % CO
#pragma unroll 4
      for (int p = tid / CO; p < 64; p += NT / CO) accb += zs[p * D::ZLD + tid % CO];
    }
    // a subset's pixels: PPS consecutive ones of the band, whole rows or part of one
    constexpr int ROWS = PPS >= HO ? PPS / HO : 1, COLS = PPS >= HO ? HO : PPS;
#pragma unroll 1
    for (int rr = 0; rr < ROWS; ++rr) {
      const int p0 = sub * PPS + rr * HO, il = p0 / HO, j0 = p0 % HO;
      const float* xr = xs + (c * D::SR + 2 * il) * D::SC + 2 * j0;
      const float* zr = zs + p0 * D::ZLD + 8 * og;
      float xv[3][3];
#pragma unroll
      for (int di = 0; di < 3; ++di) xv[di][2] = xr[di * D::SC];
#pragma unroll 4
      for (int j = 0; j < COLS; ++j) {
#pragma unroll
        for (int di = 0; di < 3; ++di) {
          xv[di][0] = xv[di][2];
          xv[di][1] = xr[di * D::SC + 2 * j + 1];
          xv[di][2] = xr[di * D::SC + 2 * j + 2];
        }
        const float4 za = *reinterpret_cast<const float4*>(zr + j * D::ZLD);
        const float4 zb = *reinterpret_cast<const float4*>(zr + j * D::ZLD + 4);
        const float z[8] = {za.x, za.y, za.z, za.w, zb.x, zb.y, zb.z, zb.w};
#pragma unroll
        for (int k = 0; k < 8; ++k)
#pragma unroll
          for (int t = 0; t < 9; ++t) acc[k][t] = fmaf(z[k], xv[t / 3][t % 3], acc[k][t]);
      }
    }
  }
  // this CTA's partial: [o][c][t] of its input channels, then the bias sums
  float* out = part + (size_t(blockIdx.y) * gridDim.x + blockIdx.x) * D::PART;
  __syncthreads();
  if constexpr (D::SUB > 1) {
    // subsets added in order through shared memory
    for (int s = 0; s < D::SUB; ++s) {
      if (sub == s) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
#pragma unroll
          for (int t = 0; t < 9; ++t) {
            float* d = sm + ((8 * og + k) * D::CC + c) * 9 + t;
            *d = s == 0 ? acc[k][t] : *d + acc[k][t];
          }
      }
      __syncthreads();
    }
    for (int e = tid; e < CO * D::CC * 9; e += NT) out[e] = sm[e];
    __syncthreads();
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
      for (int t = 0; t < 9; ++t) out[((8 * og + k) * D::CC + c) * 9 + t] = acc[k][t];
  }
  if (blockIdx.y == 0) {
    sm[tid] = accb;
    __syncthreads();
    if (tid < CO) {
      float s = 0.f;
      for (int k = 0; k < NT / CO; ++k) s += sm[k * CO + tid];
      out[CO * D::CC * 9 + tid] = s;
    }
  }
}

// Layer 1 (one input channel), bound by reading dZ1 (67 MB at n = 256): a thread takes 4
// neighbouring pixels x 4 output channels, dZ and the 3 x 9 inputs straight from global
// memory, 144 multiply-adds into 36 sums. A warp covers two rows of 64, the CTA 4 rows x
// the 16 channels. 927 us before (the im2col tile staged 32 pixels x 9 scattered bf16
// loads for 16 x 9 products), 19 now.
constexpr int DW1_PART = 16 * 9 + 16;
template <bool VEC>  // x 16-byte aligned
__global__ void __launch_bounds__(NT, 3) k_conv_dw1(const float* __restrict__ dz, const __nv_bfloat16* __restrict__ x,
                                                    uint32_t nquads, float* __restrict__ part) {
  constexpr int HI = 128, HO = 64;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int og = warp & 3, il = 2 * (warp >> 2) + (lane >> 4), j0 = 4 * (lane & 15);
  float acc[4][9], accb[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    accb[k] = 0.f;
#pragma unroll
    for (int t = 0; t < 9; ++t) acc[k][t] = 0.f;
  }
  for (uint32_t quad = blockIdx.x; quad < nquads; quad += gridDim.x) {
    const uint32_t n = quad / (HO / 4);
    const int i = 4 * int(quad % (HO / 4)) + il;
    float xv[3][9];
    load_inputs1<VEC>(x + size_t(n) * HI * HI, i, lane & 15, xv);
    const float* zp = dz + ((size_t(n) * 16 + 4 * og) * HO + i) * HO + j0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 z = *reinterpret_cast<const float4*>(zp + size_t(k) * HO * HO);
      const float zz[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        accb[k] += zz[e];
#pragma unroll
        for (int t = 0; t < 9; ++t) acc[k][t] = fmaf(zz[e], xv[t / 3][2 * e + t % 3], acc[k][t]);
      }
    }
  }
  __shared__ float red[8][40];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int t = 0; t < 10; ++t) {
      float s = t < 9 ? acc[k][t] : accb[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) red[warp][k * 10 + t] = s;
    }
  __syncthreads();
  if (tid < 160) {
    const int o = tid / 10, t = tid % 10;
    const float s = red[o >> 2][(o & 3) * 10 + t] + red[4 + (o >> 2)][(o & 3) * 10 + t];
    part[size_t(blockIdx.x) * DW1_PART + (t < 9 ? o * 9 + t : 144 + o)] = s;
  }
}

// Sums of partials in a fixed order: element e of a layer's parameters over its nparts
// partials. A CTA takes 32 elements; 8 threads each sum every eighth partial, then the 8
// sums in order.
struct SumLayer {
  const float* part;
  uint32_t nparts, stride;  // partials, floats between them
  uint32_t co, ci, cc;      // dW [co][ci][9]; a partial holds cc input channels
  uint32_t off;             // first parameter; dW then db
  uint32_t count;           // co * ci * 9 + co
};
struct SumArgs {
  SumLayer l[4];
  uint32_t first[5];  // first CTA of each layer
};
__global__ void __launch_bounds__(NT) k_sum_parts(SumArgs a, float* __restrict__ grad) {
  int k = 0;
  while (k < 3 && blockIdx.x >= a.first[k + 1]) ++k;
  const SumLayer& l = a.l[k];
  const uint32_t e = (blockIdx.x - a.first[k]) * 32 + (threadIdx.x & 31), g = threadIdx.x >> 5;
  __shared__ float red[8][32];
  float s = 0.f;
  if (e < l.count) {
    const uint32_t nw = l.co * l.ci * 9;
    const float* p;
    if (e < nw) {
      const uint32_t o = e / (l.ci * 9), c = (e / 9) % l.ci, t = e % 9;
      p = l.part + size_t(c / l.cc) * l.nparts * l.stride + (o * l.cc + c % l.cc) * 9 + t;
    } else {
      p = l.part + l.co * l.cc * 9 + (e - nw);
    }
#pragma unroll 4
    for (uint32_t q = g; q < l.nparts; q += 8) s += p[size_t(q) * l.stride];
  }
  red[g][threadIdx.x & 31] = s;
  __syncthreads();
  if (g == 0 && e < l.count) {
#pragma unroll
    for (int q = 1; q < 8; ++q) s += red[q][threadIdx.x];
    grad[l.off + e] = s;
  }
}

// --------------------------------------------------------------------- head
//
// One CTA of 64 threads per image: pool, dense layers, output. With training,
// also the loss term, the gradient of the pooled features and dZ4 (times the
// ReLU mask of a4). Scratch per image: g[64], h[32], dh[32], dy, err.
constexpr int HS = 64 + 32 + 32 + 2;

__global__ void __launch_bounds__(64) k_head(const __nv_bfloat16* __restrict__ a4, const float* __restrict__ prm,
                                            const float* __restrict__ ztarget, uint32_t n, float* __restrict__ zout,
                                            float* __restrict__ scratch, float* __restrict__ dz4) {
  const int t = blockIdx.x, c = threadIdx.x;
  __shared__ float g[64], h[32], dh[32], s_dy;
  // this channel's 64 activations, 8 per load
  const uint4* src = reinterpret_cast<const uint4*>(a4 + (size_t(t) * 64 + c) * 64);
  uint4 q[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) q[e] = src[e];
  auto act = [&](int e) { return bf(reinterpret_cast<const __nv_bfloat16*>(&q[e >> 3])[e & 7]); };
  float s = 0.f;
#pragma unroll
  for (int e = 0; e < 64; ++e) s += act(e);
  g[c] = s * (1.f / 64.f);
  __syncthreads();
  const float* f1w = prm + OFF_F1W;
  const float* f1b = prm + OFF_F1B;
  const float* f2w = prm + OFF_F2W;
  if (c < 32) {
    float v = f1b[c];
#pragma unroll 16
    for (int k = 0; k < 64; ++k) v = fmaf(f1w[c * 64 + k], g[k], v);
    h[c] = fmaxf(v, 0.f);
  }
  __syncthreads();
  if (c == 0) {
    float v = prm[OFF_F2B];
    for (int k = 0; k < 32; ++k) v = fmaf(f2w[k], h[k], v);
    if (zout) zout[t] = 0.35f + 0.25f * v;
    if (ztarget) {
      const float err = v - (ztarget[t] - 0.35f) * 4.0f;  // (z - 0.35) / 0.25
      s_dy = 2.f * err / float(n);
      scratch[size_t(t) * HS + 128] = s_dy;
      scratch[size_t(t) * HS + 129] = err;
    }
  }
  if (!ztarget) return;
  __syncthreads();
  if (c < 32) dh[c] = h[c] > 0.f ? s_dy * f2w[c] : 0.f;
  __syncthreads();
  float dg = 0.f;
#pragma unroll
  for (int k = 0; k < 32; ++k) dg = fmaf(dh[k], f1w[k * 64 + c], dg);
  dg *= 1.f / 64.f;
  float4* d = reinterpret_cast<float4*>(dz4 + (size_t(t) * 64 + c) * 64);
#pragma unroll
  for (int e = 0; e < 16; ++e)
    d[e] = make_float4(act(4 * e) > 0.f ? dg : 0.f, act(4 * e + 1) > 0.f ? dg : 0.f, act(4 * e + 2) > 0.f ? dg : 0.f,
                       act(4 * e + 3) > 0.f ? dg : 0.f);
  float* sc = scratch + size_t(t) * HS;
  sc[c] = g[c];
  if (c < 32) {
    sc[64 + c] = h[c];
    sc[96 + c] = dh[c];
  }
}

// Dense-layer gradients and the loss, summed over the batch in a fixed order: a CTA
// takes 32 of the 2,114 sums, 8 threads each (every eighth image), then the 8 in order
// (one thread per sum walked the batch on 9 CTAs: 13 us at n = 256, all latency).
__global__ void __launch_bounds__(NT) k_head_grads(const float* __restrict__ scratch, uint32_t n,
                                                   float* __restrict__ grad, float* __restrict__ loss) {
  const int e = blockIdx.x * 32 + (threadIdx.x & 31), g = threadIdx.x >> 5;
  // sum = products of two scratch words of each image (one: the sum of the word itself)
  int ia = -1, ib = -1;
  if (e < 2048) {  // f1w[k][c] = sum dh[k] g[c]
    ia = 96 + e / 64;
    ib = e % 64;
  } else if (e < 2080) {  // f1b[k] = sum dh[k]
    ia = 96 + (e - 2048);
  } else if (e < 2112) {  // f2w[k] = sum dy h[k]
    ia = 128;
    ib = 64 + (e - 2080);
  } else if (e == 2112) {  // f2b = sum dy
    ia = 128;
  } else if (e == 2113) {  // loss
    ia = ib = 129;
  }
  float s = 0.f;
  if (ia >= 0) {
#pragma unroll 4
    for (uint32_t t = g; t < n; t += 8) {
      const float a = scratch[t * HS + ia];
      s = ib >= 0 ? fmaf(a, scratch[t * HS + ib], s) : s + a;
    }
  }
  __shared__ float red[8][32];
  red[g][threadIdx.x & 31] = s;
  __syncthreads();
  if (g != 0 || ia < 0) return;
#pragma unroll
  for (int q = 1; q < 8; ++q) s += red[q][threadIdx.x];
  if (e < 2048) grad[OFF_F1W + e] = s;
  else if (e < 2080) grad[OFF_F1B + e - 2048] = s;
  else if (e < 2112) grad[OFF_F2W + e - 2080] = s;
  else if (e == 2112) grad[OFF_F2B] = s;
  else if (loss) *loss = s / float(n);
}

// ---------------------------------------------------------------------- Adam

__global__ void k_adam(float* __restrict__ prm, const float* __restrict__ grad, float* __restrict__ m,
                       float* __restrict__ v, __nv_bfloat16* __restrict__ prm_bf, __nv_bfloat16* __restrict__ wtc,
                       uint32_t count, float lr, float b1, float b2, float eps, float c1, float c2) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const float g = grad[i];
    const float mi = fmaf(b1, m[i], (1.f - b1) * g);
    const float vi = fmaf(b2, v[i], (1.f - b2) * g * g);
    m[i] = mi;
    v[i] = vi;
    const float p = prm[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
    prm[i] = p;
    prm_bf[i] = __float2bfloat16_rn(p);
    const int k = tc_place(int(i));
    if (k >= 0) wtc[k] = prm_bf[i];
  }
}

__global__ void k_to_bf16(const float* __restrict__ prm, __nv_bfloat16* __restrict__ out,
                          __nv_bfloat16* __restrict__ wtc, uint32_t count) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    out[i] = __float2bfloat16_rn(prm[i]);
    const int k = tc_place(int(i));
    if (k >= 0) wtc[k] = out[i];
  }
}

// ------------------------------------------------------------------ launchers

// Partials of the weight gradients: CTAs per layer (about two per SM; layer 4 has 256
// bands at the largest batch of the reference workload and large partials: one per SM).
constexpr uint32_t DW_CTAS[4] = {304, 304, 152, 128};

uint32_t least(uint32_t a, uint32_t b) { return a < b ? a : b; }

// dW and db of a layer as partials at `part` (its end is returned in it), described in l;
// then dprev, the previous layer's dZ.
template <int CI, int CO, int HI>
cudaError_t conv_bwd(const Net& t, int layer, const float* dz, const __nv_bfloat16* x, int off_w, float* dprev,
                     uint32_t n, float*& part, SumLayer& l, cudaStream_t s) {
  using D = DwCfg<CI, CO, HI>;
  using X = DxCfg<CI, CO, HI>;
  const uint32_t nbands = n * D::BANDS, ctas = least(nbands, DW_CTAS[layer]);
  cudaError_t e = cudaFuncSetAttribute(k_conv_dw<CI, CO, HI>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(D::SMEM));
  if (e != cudaSuccess) return e;
  k_conv_dw<CI, CO, HI><<<dim3(ctas, D::CPARTS), NT, D::SMEM, s>>>(dz, x, nbands, part);
  l = SumLayer{part, ctas, uint32_t(D::PART), uint32_t(CO), uint32_t(CI), uint32_t(D::CC), uint32_t(off_w),
               uint32_t(CO * CI * 9 + CO)};
  part += size_t(ctas) * D::CPARTS * D::PART;
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_conv_dx<CI, CO, HI><<<dim3(n * X::BANDS, X::CPARTS), X::NTX, 0, s>>>(dz, t.prm_bf + off_w, x, dprev);
  return cudaGetLastError();
}

}  // namespace

cudaError_t net_forward(const Net& t, const void* x, uint32_t n, const float* ztarget, float* zout, cudaStream_t s) {
  const auto* xi = static_cast<const __nv_bfloat16*>(x);
  const uint32_t rows = n * 64;
  if ((reinterpret_cast<uintptr_t>(x) & 15) == 0)
    k_conv1<true><<<rows / 16, NT, 0, s>>>(xi, t.prm_bf + OFF_W1, t.prm + OFF_B1, t.a1);
  else
    k_conv1<false><<<rows / 16, NT, 0, s>>>(xi, t.prm_bf + OFF_W1, t.prm + OFF_B1, t.a1);
  cudaError_t e = cudaGetLastError();
  // layers 2-4 (K = 144, 288, 576): implicit GEMMs on the tensor cores
  if (e == cudaSuccess) e = conv_tc<16, 32, 64>(t.a1, t.wtc + OFF_TC2, t.prm + OFF_B2, t.a2, n, t.err, s);
  if (e == cudaSuccess) e = conv_tc<32, 64, 32>(t.a2, t.wtc + OFF_TC3, t.prm + OFF_B3, t.a3, n, t.err, s);
  if (e == cudaSuccess) e = conv_tc<64, 64, 16>(t.a3, t.wtc + OFF_TC4, t.prm + OFF_B4, t.a4, n, t.err, s);
  if (e != cudaSuccess) return e;
  k_head<<<n, 64, 0, s>>>(t.a4, t.prm, ztarget, n, zout, t.head, t.dbuf0);
  return cudaGetLastError();
}

cudaError_t net_backward(const Net& t, const void* x, uint32_t n, float* loss, cudaStream_t s) {
  // dZ4 is in dbuf0 (from the head); dZ3 -> dbuf1, dZ2 -> dbuf0, dZ1 -> dbuf1
  k_head_grads<<<(2114 + 31) / 32, NT, 0, s>>>(t.head, n, t.grad, loss);
  cudaError_t e = cudaGetLastError();
  float* part = t.part;
  SumArgs sum{};
  if (e == cudaSuccess) e = conv_bwd<64, 64, 16>(t, 3, t.dbuf0, t.a3, OFF_W4, t.dbuf1, n, part, sum.l[3], s);
  if (e == cudaSuccess) e = conv_bwd<32, 64, 32>(t, 2, t.dbuf1, t.a2, OFF_W3, t.dbuf0, n, part, sum.l[2], s);
  if (e == cudaSuccess) e = conv_bwd<16, 32, 64>(t, 1, t.dbuf0, t.a1, OFF_W2, t.dbuf1, n, part, sum.l[1], s);
  if (e != cudaSuccess) return e;
  const uint32_t quads = n * 16, ctas = least(quads, DW_CTAS[0]);
  const auto* xi = static_cast<const __nv_bfloat16*>(x);
  if ((reinterpret_cast<uintptr_t>(x) & 15) == 0) k_conv_dw1<true><<<ctas, NT, 0, s>>>(t.dbuf1, xi, quads, part);
  else k_conv_dw1<false><<<ctas, NT, 0, s>>>(t.dbuf1, xi, quads, part);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  sum.l[0] = SumLayer{part, ctas, DW1_PART, 16, 1, 1, OFF_W1, 160};
  for (int k = 0; k < 4; ++k) sum.first[k + 1] = sum.first[k] + (sum.l[k].count + 31) / 32;
  k_sum_parts<<<sum.first[4], NT, 0, s>>>(sum, t.grad);
  return cudaGetLastError();
}

cudaError_t net_adam(const Net& t, float lr, float b1, float b2, float eps, float c1, float c2, cudaStream_t s) {
  k_adam<<<(NPARAMS + 255) / 256, 256, 0, s>>>(t.prm, t.grad, t.m, t.v, t.prm_bf, t.wtc, NPARAMS, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

cudaError_t net_sync_bf16(const Net& t, cudaStream_t s) {
  k_to_bf16<<<(NPARAMS + 255) / 256, 256, 0, s>>>(t.prm, t.prm_bf, t.wtc, NPARAMS);
  return cudaGetLastError();
}

size_t dw_part_floats() {
  return size_t(DW_CTAS[0]) * DW1_PART + size_t(DW_CTAS[1]) * DwCfg<16, 32, 64>::PART +
         size_t(DW_CTAS[2]) * DwCfg<32, 64, 32>::PART + size_t(DW_CTAS[3]) * 2 * DwCfg<64, 64, 16>::PART;
}

}  // namespace cnn
}  // namespace hv

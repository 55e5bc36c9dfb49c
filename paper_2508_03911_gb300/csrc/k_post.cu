// k_post.cu -- post-processing of rendered images (Sec. III-B, "post processing and
// image accumulation"): periodic K x K convolution, re-normalisation by the mean,
// moving average over the last A images of each output.
//
// Rendered images of one call are [window][image][H][W]. Each image, after the
// convolution, goes to slot (count + window) mod R of a ring that keeps the last
// R images of every output (R >= A - 1 + windows per call), with its float64 sum
// beside it (kPostSub partial sums, added by the CTAs that write the slot); the
// moving average then reads the slots it needs, so every window of the call is
// averaged in parallel. Without a convolution the STFT epilogue writes the slots
// and their sums itself, and only the average runs here.
#include "pair_dev.cuh"
#include "hv_internal.h"

namespace hv {

namespace {

constexpr int PY = 16;  // rows of a convolution tile; TX = 16, 32 or 64 columns, 4 per thread

// Sums and scales in pairs of float32 (pair_dev.cuh): one conversion to float64 and five
// shuffled additions of it per pixel took most of the kernel's time (see below).

// ring[slot][m][y][x] = sum_{a,b} k[a][b] img[(y + a - c) mod H][(x + b - c) mod W]
// for image m of window w (slot = (count + w) mod R); K = 0 copies. Re-normalising,
// the tile's sum goes into one of the slot image's partial sums.
//
// A thread forms 4 neighbouring outputs of a row: per 4 taps one float4 of the tile and
// one of the weights for 16 multiply-adds (one output per thread took 2 loads per
// multiply-add), and the image sum is carried in float32 pairs. 45 images of 1024 x 512,
// K = 5, re-normalised: 388 us before, 179 now.
template <int TX>
__global__ void __launch_bounds__(TX / 4 * PY) k_post_conv(const float* __restrict__ img, PostArgs a) {
  constexpr int NT = TX / 4 * PY;
  extern __shared__ __align__(16) float sm[];
  const int K = a.K, c = K / 2, KP = (K + 3) & ~3, LD = TX + KP;
  const int rows = PY + (K > 0 ? K - 1 : 0), cols = TX + (K > 0 ? K - 1 : 0);
  float* tile = sm;             // rows x LD
  float* kw = sm + rows * LD;   // K x KP
  const uint32_t tiles_x = a.W / TX;
  const int ty0 = int(blockIdx.x / tiles_x) * PY, tx0 = int(blockIdx.x % tiles_x) * TX;
  const uint32_t im = blockIdx.y;  // w * nout + m
  const uint32_t w = im / a.nout, m = im % a.nout;
  const size_t hw = size_t(a.W) * a.H;
  const float* src = img + size_t(im) * hw;
  for (int e = threadIdx.x; e < K * K; e += NT) kw[e / K * KP + e % K] = a.kern[e];
  for (int r = threadIdx.x / TX; r < rows; r += NT / TX) {
    const float* line = src + size_t((ty0 + r - c) & int(a.H - 1)) * a.W;
    for (int x = threadIdx.x % TX; x < cols; x += TX) tile[r * LD + x] = line[(tx0 + x - c) & int(a.W - 1)];
  }
  __syncthreads();
  const int ly = threadIdx.x / (TX / 4), lx = 4 * (threadIdx.x % (TX / 4));
  float v[4] = {0.f, 0.f, 0.f, 0.f};
  if (K > 0) {
    for (int p = 0; p < K; ++p) {
      const float* t = tile + (ly + p) * LD + lx;
      float4 lo = *reinterpret_cast<const float4*>(t);
      for (int q = 0; q < K; q += 4) {
        const float4 up = *reinterpret_cast<const float4*>(t + q + 4);
        const float4 k4 = *reinterpret_cast<const float4*>(kw + p * KP + q);
        const float x[7] = {lo.x, lo.y, lo.z, lo.w, up.x, up.y, up.z};
        const float kk[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (q + i < K) {  // taps of the padding are not formed: 0 x infinity is not 0
#pragma unroll
            for (int o = 0; o < 4; ++o) v[o] = fmaf(kk[i], x[i + o], v[o]);
          }
        lo = up;
      }
    }
  } else {
#pragma unroll
    for (int o = 0; o < 4; ++o) v[o] = tile[ly * LD + lx + o];
  }
  const uint32_t slot = uint32_t((a.count + w) % a.R);
  *reinterpret_cast<float4*>(a.ring + (size_t(slot) * a.nout + m) * hw + size_t(ty0 + ly) * a.W + tx0 + lx) =
      make_float4(v[0], v[1], v[2], v[3]);
  if (a.renorm) {
    float2 t = pair_add(two_sum(v[0], v[1]), two_sum(v[2], v[3]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      t = pair_add(t, make_float2(__shfl_xor_sync(0xffffffffu, t.x, o), __shfl_xor_sync(0xffffffffu, t.y, o)));
    double d = double(t.x) + double(t.y);
    if (__any_sync(0xffffffffu, !isfinite(d))) {  // an infinity or NaN, or a sum past the largest float
      d = (double(v[0]) + double(v[1])) + (double(v[2]) + double(v[3]));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    }
    __shared__ double red[NT / 32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = d;
    __syncthreads();
    if (threadIdx.x == 0) {
      double u = 0.0;
      for (int i = 0; i < NT / 32; ++i) u += red[i];
      atomicAdd(&a.sums[(size_t(slot) * a.nout + m) * kPostSub + blockIdx.x % kPostSub], u);
    }
  }
}

// float(double(v) * s) for s = hi + lo (s rounded to 48 bits) in float32: the product's
// error by fma. Where that is not exact (s or the product outside the normal range, an
// infinity or NaN) the float64 product.
__device__ __forceinline__ float scaled(float v, float hi, float lo, double s) {
  const float p = __fmul_rn(v, hi);
  if (fabsf(p) > 1e-30f && fabsf(p) < 1e38f) return __fadd_rn(p, fmaf(v, lo, fmaf(v, hi, -p)));
  return v == 0.f && hi != 0.f ? p : float(double(v) * s);
}

// out[w][m][p] = mean over the last min(A, count + w + 1) slots of image m,
// each divided by its mean when re-normalising. Bound by the ring's reads; four pixels
// per thread (VEC: out 16-byte aligned) and the products in float32 pairs (a float64
// product and two conversions per pixel and slot, as above, took 537 us for 45 images
// of 1024 x 512, A = 4; 98 now).
template <bool VEC>
__global__ void __launch_bounds__(256) k_post_avg(float* __restrict__ out, PostArgs a) {
  __shared__ double scale[64];      // hw / sum of each slot read (A <= 64)
  __shared__ float2 pair[64];       // the same as hi + lo
  __shared__ const float* line[64];
  const uint32_t im = blockIdx.y, w = im / a.nout, m = im % a.nout;
  const size_t hw = size_t(a.W) * a.H;
  const uint64_t newest = a.count + w;
  const uint32_t n = uint32_t(newest + 1 < a.A ? newest + 1 : a.A);
  for (uint32_t j = threadIdx.x >> 5; j < n; j += blockDim.x >> 5) {
    const uint32_t slot = uint32_t((newest - j) % a.R);
    double t = a.renorm ? a.sums[(size_t(slot) * a.nout + m) * kPostSub + (threadIdx.x & 31)] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) {
      const double s = t != 0.0 ? double(hw) / t : 0.0;
      const float hi = float(s);
      scale[j] = s;
      // a scale outside the range where hi + lo holds it: all products in float64
      pair[j] = fabsf(hi) > 1e-20f && fabsf(hi) < 1e30f ? make_float2(hi, float(s - double(hi))) : make_float2(0.f, 0.f);
      line[j] = a.ring + (size_t(slot) * a.nout + m) * hw;
    }
  }
  __syncthreads();
  constexpr int V = VEC ? 4 : 1;
  for (size_t p = (blockIdx.x * size_t(blockDim.x) + threadIdx.x) * V; p < hw; p += size_t(gridDim.x) * blockDim.x * V) {
    float acc[V];
#pragma unroll
    for (int e = 0; e < V; ++e) acc[e] = 0.f;
#pragma unroll 4
    for (uint32_t j = 0; j < n; ++j) {
      float v[V];
      if constexpr (VEC) {
        const float4 q = *reinterpret_cast<const float4*>(line[j] + p);
        v[0] = q.x;
        v[1] = q.y;
        v[2] = q.z;
        v[3] = q.w;
      } else {
        v[0] = line[j][p];
      }
#pragma unroll
      for (int e = 0; e < V; ++e) {
        if (a.renorm) v[e] = scaled(v[e], pair[j].x, pair[j].y, scale[j]);
        acc[e] += v[e];
      }
    }
#pragma unroll
    for (int e = 0; e < V; ++e) acc[e] /= float(n);
    float* d = out + size_t(im) * hw + p;
    if constexpr (VEC) *reinterpret_cast<float4*>(d) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    else *d = acc[0];
  }
}

template <int TX>
cudaError_t launch_conv(const float* images, const PostArgs& a, uint32_t nimg, cudaStream_t s) {
  const int KP = (a.K + 3) & ~3, rows = PY + (a.K > 0 ? a.K - 1 : 0);
  const size_t smem = (size_t(rows) * (TX + KP) + size_t(a.K) * KP) * sizeof(float);
  k_post_conv<TX><<<dim3((a.W / TX) * (a.H / PY), nimg), TX / 4 * PY, smem, s>>>(images, a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_post_zero(const PostArgs& a, uint32_t nwin, cudaStream_t s) {
  if (!a.renorm || nwin == 0) return cudaSuccess;
  // the slots (count + w) mod R of the call, w < nwin <= R: one run, or two across the wrap
  const size_t per_slot = size_t(a.nout) * kPostSub * sizeof(double);
  const uint32_t first = uint32_t(a.count % a.R);
  const uint32_t run = nwin < a.R - first ? nwin : a.R - first;
  cudaError_t e = cudaMemsetAsync(a.sums + size_t(first) * a.nout * kPostSub, 0, run * per_slot, s);
  if (e == cudaSuccess && run < nwin) e = cudaMemsetAsync(a.sums, 0, (nwin - run) * per_slot, s);
  return e;
}

cudaError_t launch_post(float* images, uint32_t nwin, const PostArgs& a, cudaStream_t s, int* launches) {
  if (nwin == 0) return cudaSuccess;
  if (nwin > a.R || a.A > 64) return cudaErrorInvalidValue;
  const uint32_t nimg = nwin * a.nout;
  cudaError_t e;
  if (!a.fused) {
    e = launch_post_zero(a, nwin, s);
    if (e != cudaSuccess) return e;
    e = a.W >= 64 ? launch_conv<64>(images, a, nimg, s)
        : a.W == 32 ? launch_conv<32>(images, a, nimg, s)
                    : launch_conv<16>(images, a, nimg, s);
    if (e != cudaSuccess) return e;
    *launches += 1;
  }
  const size_t hw = size_t(a.W) * a.H;
  if ((reinterpret_cast<uintptr_t>(images) & 15) == 0) {
    const unsigned gx = unsigned((hw + 1023) / 1024 < 64 ? (hw + 1023) / 1024 : 64);
    k_post_avg<true><<<dim3(gx, nimg), 256, 0, s>>>(images, a);
  } else {
    const unsigned gx = unsigned((hw + 255) / 256 < 64 ? (hw + 255) / 256 : 64);
    k_post_avg<false><<<dim3(gx, nimg), 256, 0, s>>>(images, a);
  }
  *launches += 1;
  return cudaGetLastError();
}

}  // namespace hv

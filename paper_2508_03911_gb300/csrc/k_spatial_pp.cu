// k_spatial_pp.cu -- the spatial transform (Sec. III-B.1) of 256 x 256 frames as one
// persistent, warp-specialised launch for every pass of every frame of a render (the
// kernel's own comment says how). Its column passes run the block-wide FFT stages of
// pp_dev.cuh on strips of 16 lines staged in shared memory.
#include <cuda.h>

#include "pp_dev.cuh"
#include "hv_internal.h"
#include "../../include/hv.h"

namespace hv {

namespace {

// Two real raw columns as one complex line: line b of the strip is columns 2b
// (real part) and 2b + 1 (imaginary part); 32 columns staged, rows 32 pixels apart.
template <bool U8>
struct PackedRawSrc {
  static constexpr bool kAliasesBuf = true;  // staged inside the FFT buffer: read all before writing
  const unsigned char* raw;
  __device__ __forceinline__ float2 operator()(int t, int b) const {
    if constexpr (U8) {
      const uint16_t p = reinterpret_cast<const uint16_t*>(raw)[t * 16 + b];
      return make_float2(float(p & 0xffu), float(p >> 8));
    } else {
      const uint32_t p = reinterpret_cast<const uint32_t*>(raw)[t * 16 + b];
      return make_float2(float(p & 0xffffu), float(p >> 16));
    }
  }
};

// Bin k of line b to the buffer at buf[k * LD + b] (after every read of it).
template <int LD>
struct SmemOut {
  static constexpr bool kSyncFirst = true;
  static constexpr bool kJFast = false;
  float2* buf;
  __device__ __forceinline__ void operator()(int b, int k, float2 v) const { buf[k * LD + b] = v; }
};

constexpr int RW_L = 256;  // side of the fused transform's frames

__device__ __forceinline__ uint32_t rw_smem(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Bounded wait (about 2^32 clocks) for phase `parity` of an mbarrier.
__device__ __forceinline__ bool rw_wait(uint32_t mbar, uint32_t parity) {
  const long long t0 = clock64();
  while (true) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(mbar), "r"(parity)
        : "memory");
    if (ok) return true;
    if (clock64() - t0 > (1ll << 32)) return false;
  }
}

// ------------------------------------------- fused transform, 256 x 256 frames
//
// Every pass of every frame of a launch in one persistent kernel. As launches of their
// own over a chunk of frames, the passes take their intermediates (S1, S2: up to 512 KB
// per frame) through HBM, once written and once read. Here work items come in a fixed global order from an atomic ticket
// counter: row r of the order holds the column items of frame r and the items of
// each later pass of frame r - (the lags up to that pass). A Fresnel frame takes two passes of 16
// items: 16 chirped (complex) columns per column item, 16 rows per row item,
// the row FFT writing the time queue. ASP takes four passes, using that the
// hologram is real:
//   1. 8 column items of 32 real columns, packed in pairs as the real and
//      imaginary parts of 16 complex lines whose spectra Z are separated after
//      the transform (for real a and b, z = a + i b: A(k) = (Z(k) + conj Z(-k)) / 2,
//      B(k) = (Z(k) - conj Z(-k)) / 2i). Only bins ky = 1 .. 127 are stored, row
//      by row, with the real rows ky = 0 and 128 packed into row 0 as
//      S1(0, x) + i S1(128, x): the other half is their conjugate.
//   2. 8 row items over S1 rows 0 .. 127: the forward row FFT W(ky, .) is kept
//      in the second half of the S1 slot (S3), then x H(ky) and the inverse row
//      FFT give S2 rows 0 .. 127 (row 0 takes W(0) = (Wp(k) + conj Wp(-k)) / 2
//      from the packed row's transform Wp).
//   3. 8 mirror items: the spectrum of row ky in 128 .. 255 is
//      conj W(256 - ky, -kx) (row 128: (Wp(k) - conj Wp(-k)) / 2i), read from S3;
//      x H(ky) and the inverse row FFT give S2 rows 128 .. 255. A frame takes
//      128 forward row FFTs instead of 256.
//   4. 16 column-IFFT items of 16 columns of S2 write the time queue.
// S1 (with S3) and S2 are rings of RING frames that stay in L2. An item may start
// once the counters that make its input complete and its output slot free have
// been published (P1 .. P4 the ASP passes above; each chain of release adds and
// acquire loads orders what it covers, so a condition implied through an
// earlier item's wait is not checked again):
//   P1 of f: the P2 items of f - RING have read S1 slot f mod RING
//   P2 of f: P1 of f wrote S1; the P4 items of f - RING have read S2 (and so the
//            P3 items of f - RING have read S3)
//   P3 of f: P2 of f wrote S3 (and so P4 of f - RING has read S2)
//   P4 of f: P3 of f wrote S2 (and so P2 of f did)
// and for Fresnel: column items of f after the row items of f - RING, row items
// of f after the column items of f.
// A CTA is warp-specialised: one producer thread takes the tickets, waits (bounded
// spin on acquire loads) for each item's counters, stages its input strip into
// one of two buffers with one copy (a TMA tensor copy, or a 1-D bulk copy)
// completing on the buffer's mbarrier, and publishes every finished item, in
// order (release add on its slot counter); eight consumer warps transform the
// staged strip while the next one streams in. The producer readies the following
// item (ticket and counters) while the consumers still hold both buffers, so its
// copy starts as soon as one frees. Every wait is on an item with a smaller
// ticket (RING > 2 LAG), a CTA takes its items in ticket order, and the producer
// publishes finished items from inside each of its waits, so the item with the
// smallest unfinished ticket always completes: the launch ends. Raw frames are read with an evict-first L2
// policy and the propagated frames stored with streaming stores, so that the two
// rings keep their L2 lines.
constexpr int FZ_NT = 256;       // consumer threads (one pass's thread layout)
constexpr int FZ_THREADS = FZ_NT + 32;
// rows of tickets between a frame's passes: at least the tickets in flight (3 per
// CTA: the transformed item, the staged one, the one waiting for its buffer) over
// the items per row, so that an item's inputs are usually published when it is
// staged. A ticket is fetched only when the producer is ready to handle it: every
// ticket held but not worked on delays the frames that wait for it (fetching one
// ahead measured 1.5 % slower, lags of 40 and 56 rows 1-2 % slower)
constexpr int FZ_LAG = 48;
// ASP runs four passes of 8, 8, 8 and 16 items per frame (the row pass split into
// the rows it transforms forward and the rows it takes as mirrors), so 40 items
// per ticket row; FZ_LAG_ASP1 rows from the column pass to the row pass, then
// FZ_LAG_ASP between the later passes. The rings must outlast the two later lags
// (the row pass of frame f + R waits for the column IFFT of f)
constexpr int FZ_LAG_ASP1 = 36;
constexpr int FZ_LAG_ASP = 36;
constexpr int FZ_BAR = 1;        // named barrier of the consumer warps
constexpr size_t FZ_FRAME = size_t(RW_L) * RW_L;  // complex values per frame
constexpr size_t FZ_BUF = size_t(256) * 16;       // complex values per buffer
constexpr size_t FZ_RAW = 256 * 64;               // bytes of a raw strip (32 uint16 columns), in the buffer's tail
// every wait is on a smaller ticket when the rings are longer than the lag; the
// headroom above it keeps column items from waiting for a slot to be freed
static_assert(kFusedRing > FZ_LAG && kFusedRing > FZ_LAG_ASP1 && kFusedRing > 2 * FZ_LAG_ASP,
              "the rings must outlast the lags between passes");
// shared memory: pass twiddles (256), row-FFT stage-2 twiddles (240), Fresnel
// chirp along y (256), two buffers of 16 lines x 256 (the column passes' lines
// fastest with row stride 16, the row tile 16 x 256; a raw strip lands in the
// tail of its buffer and is read whole by the first FFT stage before it writes)
constexpr size_t FZ_SMEM = 1024 + (256 + 240 + 256 + 2 * FZ_BUF) * sizeof(float2);  // + alignment slack
constexpr uint32_t FZ_STOP = 0xffffffffu;

// Bin k of line b to global memory at out[k * stride + b] with a streaming store.
struct GlobalOutCs {
  static constexpr bool kSyncFirst = false;
  static constexpr bool kJFast = false;
  float2* out;
  uint32_t stride;
  __device__ __forceinline__ void operator()(int b, int k, float2 v) const { __stcs(&out[size_t(k) * stride + b], v); }
};

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ bool mbar_test(uint32_t mbar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(mbar), "r"(parity)
      : "memory");
  return ok != 0;
}

struct FzItem {
  uint32_t pass, frame, strip;
};

// 256-point FFT of a row held by 16 lanes (lane jl: elements jl + 16 m in v[m]) as
// 16 x 16: the 16-point DFTs over m, a transpose through the row's shared buffer
// (XOR-swizzled), twiddles, the 16-point DFTs over the lanes' first digits. Bin
// jl + 16 m ends in v[m]. DIR -1 forward, +1 inverse (unscaled).
template <int DIR>
__device__ __forceinline__ void row_fft16x16(float2 (&v)[16], float2* rowp, const float2* tw2, int jl) {
  dft<16, DIR>(v);
  __syncwarp();
#pragma unroll
  for (int m = 0; m < 16; ++m) rowp[16 * jl + (m ^ jl)] = v[m];
  __syncwarp();
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    v[m] = rowp[16 * m + (jl ^ m)];
    if (m > 0) {
      float2 w = tw2[(m - 1) * 16 + jl];
      if (DIR > 0) w.y = -w.y;
      v[m] = cmul(v[m], w);
    }
  }
  dft<16, DIR>(v);
}

__global__ void __launch_bounds__(FZ_THREADS, 3)
    k_spatial_fused(SpatialArgs a, uint32_t nticket, const __grid_constant__ CUtensorMap raw_map,
                    const __grid_constant__ CUtensorMap s2_map) {
  extern __shared__ __align__(16) unsigned char smem[];
  // the two buffers first, 1024-byte aligned (bulk-copy destinations), then the tables
  unsigned char* base = smem + ((1024u - (rw_smem(smem) & 1023u)) & 1023u);
  float2* bufs = reinterpret_cast<float2*>(base);  // buffer b at bufs + b FZ_BUF
  float2* tws = bufs + 2 * FZ_BUF;
  float2* tw2 = tws + 256;
  float2* cys = tw2 + 240;
  // raw strip of buffer b: its last FZ_RAW bytes
  auto raw_of = [&](int b) {
    return reinterpret_cast<unsigned char*>(bufs + (b + 1) * FZ_BUF) - FZ_RAW;
  };
  __shared__ __align__(8) unsigned long long full[2], freed[2];
  __shared__ FzItem desc[2];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool asp = a.spatial == HV_SPATIAL_ASP;
  const bool u8 = a.in_kind == IN_U8;
  // items per ticket row (ASP: 8 + 8 + 8 + 16, Fresnel: 16 + 16), rows between passes
  const uint32_t ipr = asp ? 40u : 32u, R = a.ring;
  for (int e = tid; e < 256; e += FZ_THREADS) {
    tws[e] = __ldg(&a.tw_h[e]);
    cys[e] = asp ? make_float2(1.f, 0.f) : __ldg(&a.chirp_y[e]);
  }
  for (int e = tid; e < 240; e += FZ_THREADS) {
    const int m = e / 16 + 1, j = e % 16;
    tw2[e] = __ldg(&a.tw_w[j * m]);
  }
  if (tid == 0) {
    for (int b = 0; b < 2; ++b) {
      // full: the producer's arrival with the item's byte count, completed by its copy
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(rw_smem(&full[b])) : "memory");
      // freed: one arrival per consumer warp
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(rw_smem(&freed[b])), "n"(FZ_NT / 32) : "memory");
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  float2* const tq = static_cast<float2*>(a.tq.base);
  unsigned* const done = a.fused_ctr + 1;  // done[pass * R + slot]

  if (warp == FZ_NT / 32) {
    // ------------------------------------------------------------ producer (lane 0)
    if (lane != 0) return;
    uint64_t pol_first;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(pol_first));
    const long long limit = 1ll << 31;
    bool stuck = false;  // a wait for the consumers gave up
    // items are staged in order, item k into buffer k & 1; `issued` items were staged,
    // the first `published` of them transformed and counted. The counter of item k
    // sits at done[cnt0] or done[cnt1] (by k & 1) until it is published.
    uint32_t issued = 0, published = 0, cnt0 = 0, cnt1 = 0;
    // publish, in order, the items below `upto` whose transform is done; block: wait
    // for each (false when a wait gave up). Release-add: the consumers' stores, ordered
    // before this thread by the buffer's mbarrier, are visible at GPU scope before the
    // count; nothing waits on a reply.
    auto drain = [&](uint32_t upto, bool block) -> bool {
      const long long t0 = clock64();
      while (published < upto) {
        if (mbar_test(rw_smem(&freed[published & 1]), (published >> 1) & 1)) {
          const uint32_t c = (published & 1) ? cnt1 : cnt0;
          asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(&done[c]) : "memory");
          ++published;
        } else if (!block) {
          return true;
        } else if (clock64() - t0 > limit) {
          return false;
        }
      }
      return true;
    };
    // the next item with its counters satisfied, publishing finished items meanwhile;
    // false when the tickets are used up or a wait gave up
    auto prepare = [&](FzItem& it) -> bool {
      uint32_t pass, f, strip;
      while (true) {
        const uint32_t t = atomicAdd(a.fused_ctr, 1u);
        if (t >= nticket) return false;
        const uint32_t row = t / ipr, kk = t % ipr;
        pass = asp ? (kk < 24u ? kk >> 3 : 3u) : kk >> 4;
        strip = asp ? (kk < 24u ? kk & 7u : kk - 24u) : kk & 15u;
        const uint32_t off = !asp ? pass * FZ_LAG : pass == 0 ? 0u : FZ_LAG_ASP1 + (pass - 1) * FZ_LAG_ASP;
        const long long fl = (long long)row - (long long)off;
        if (fl >= 0 && fl < (long long)a.n) {
          f = uint32_t(fl);
          break;
        }
      }
      const uint32_t slot = f % R, gen = f / R;
      const long long t0 = clock64();
      while (true) {
        bool ready;
        if (!asp) ready = pass == 0 ? ld_acquire_u32(&done[R + slot]) >= 16u * gen
                                    : ld_acquire_u32(&done[slot]) >= 16u * (gen + 1);
        else if (pass == 0) ready = ld_acquire_u32(&done[R + slot]) >= 8u * gen;
        else if (pass == 1) ready = ld_acquire_u32(&done[slot]) >= 8u * (gen + 1) &&
                                    ld_acquire_u32(&done[3 * R + slot]) >= 16u * gen;
        else ready = ld_acquire_u32(&done[(pass - 1) * R + slot]) >= 8u * (gen + 1);
        if (a.stall && pass == 1) ready = false;  // fault injection: a condition nothing sets
        drain(issued, false);
        if (ready) break;
        if ((*reinterpret_cast<const volatile unsigned*>(a.err) & 16u) || clock64() - t0 > limit) {
          atomicOr(a.err, 16u);
          return false;
        }
        __nanosleep(32);
      }
      it = FzItem{pass, f, strip};
      return true;
    };
    // the next item is ready before its buffer frees, so that its copy starts the
    // moment the consumers are done with the item two before it
    FzItem it{0, 0, 0};
    bool more = prepare(it);
    while (more) {
      const uint32_t k = issued, b = k & 1;
      // buffer b is free once item k - 2 is transformed (published here, in order)
      if (k >= 2 && !drain(k - 1, true)) {
        stuck = true;
        atomicOr(a.err, 16u);
        break;
      }
      // one copy per item: the raw strip (256 rows x 16 pixels) and the column-IFFT
      // strip (256 rows x 16 complex) by a TMA tensor copy, the row pass's 16 rows
      // (contiguous) by a 1-D bulk copy. The rings were written by other CTAs'
      // generic stores, fenced for the async proxy before their publication; this
      // thread acquired the counters that published them.
      const uint32_t s0 = it.strip * (it.pass == 0 && asp ? 32u : 16u), slot = it.frame % R;
      const float2* s1 = a.scratch1 + size_t(slot) * FZ_FRAME;
      desc[b] = it;
      const uint32_t fb = rw_smem(&full[b]);
      if (it.pass == 0) {
        const uint32_t bytes = 256u * (asp ? 32u : 16u) * (u8 ? 1u : 2u);
        const uint32_t rslot = uint32_t((a.raw.slot0 + it.frame) % a.raw.cap);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(fb), "r"(bytes) : "memory");
        asm volatile(
            "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint "
            "[%0], [%1, {%2, %3}], [%4], %5;\n" ::"r"(rw_smem(raw_of(b))),
            "l"(reinterpret_cast<uint64_t>(&raw_map)), "r"(int(s0)), "r"(int(rslot * 256u)), "r"(fb),
            "l"(pol_first)
            : "memory");
      } else if (it.pass == 1 || (asp && it.pass == 2)) {
        // 16 rows of S1 (row pass), or (mirror pass) the S3 rows 256 - r of its
        // output rows r = 143 + s0 - b, b = 0 .. 15: rows 113 - s0 .. 128 - s0; the
        // first strip's last row (r = 128) is the packed row S3(0)
        asm volatile("fence.proxy.async.global;\n" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(fb), "r"(32768u) : "memory");
        const float2* src = it.pass == 1 ? s1 + size_t(s0) * 256 : s1 + size_t(128 + 113 - s0) * 256;
        const uint32_t bytes = it.pass == 2 && s0 == 0 ? 15u * 2048u : 32768u;
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                rw_smem(bufs + b * FZ_BUF)),
            "l"(src), "r"(bytes), "r"(fb)
            : "memory");
        if (bytes != 32768u)
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                  rw_smem(bufs + b * FZ_BUF + 15 * 256)),
              "l"(s1 + size_t(128) * 256), "r"(2048u), "r"(fb)
              : "memory");
      } else {
        asm volatile("fence.proxy.async.global;\n" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(fb), "r"(32768u) : "memory");
        asm volatile(
            "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
            "[%4];\n" ::"r"(rw_smem(bufs + b * FZ_BUF)),
            "l"(reinterpret_cast<uint64_t>(&s2_map)), "r"(int(s0)), "r"(int(slot * 256u)), "r"(fb)
            : "memory");
      }
      const uint32_t c = it.pass * R + slot;
      if (b) cnt1 = c;
      else cnt0 = c;
      issued = k + 1;
      more = prepare(it);
    }
    // publish the rest as it finishes, then tell the consumers to stop (item `issued`,
    // whose buffer the last drain freed); if a wait gave up, the consumers' own
    // bounded waits end them
    if (!stuck && drain(issued, true)) {
      const int b = int(issued & 1);
      desc[b] = FzItem{FZ_STOP, 0, 0};
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(rw_smem(&full[b])) : "memory");
    } else {
      atomicOr(a.err, 16u);
    }
    return;
  }

  // ------------------------------------------------------------- consumers
  const int rb = 2 * warp + (lane >> 4), jl = lane & 15;  // row pass: row of the strip, lane in the row
  for (uint32_t k = 0;; ++k) {
    const int b = int(k & 1);
    if (!rw_wait(rw_smem(&full[b]), (k >> 1) & 1)) {
      if (tid == 0) atomicOr(a.err, 16u);
      break;
    }
    const FzItem it = desc[b];
    if (it.pass == FZ_STOP) break;
    const uint32_t pass = it.pass, f = it.frame, s0 = it.strip * (pass == 0 && asp ? 32u : 16u), slot = f % R;
    float2* buf = bufs + b * FZ_BUF;
    float2* s1 = a.scratch1 + size_t(slot) * FZ_FRAME;
    float2* s2 = a.scratch2 + size_t(slot) * FZ_FRAME;
    const size_t tslot = (a.tq.slot0 + f) % a.tq.cap;
    if (pass == 0) {
      const unsigned char* raw = raw_of(b);
      const GlobalOut out{s1 + s0, 256u};
      if (asp) {
        // column FFT of 32 real raw columns, packed in pairs (conversion in the first
        // stage), spectra Z of the 16 lines into the buffer [k][line]; then the two
        // columns' spectra A, B at bins 1 .. 127 -> S1 [ky][x], and at the real bins 0
        // and 128 packed as A(0) + i A(128), B(0) + i B(128) -> S1 row 0
        if (u8) pp_stages<256, 1, -1, PackedRawSrc<true>, SmemOut<16>, 16, FZ_BAR>(PackedRawSrc<true>{raw}, buf,
                                                                                    tws, SmemOut<16>{buf});
        else pp_stages<256, 1, -1, PackedRawSrc<false>, SmemOut<16>, 16, FZ_BAR>(PackedRawSrc<false>{raw}, buf,
                                                                                  tws, SmemOut<16>{buf});
        pp_sync<FZ_BAR, FZ_NT>();
        const int line = tid % 16;
        float4* o = reinterpret_cast<float4*>(s1 + s0 + 2 * line);  // columns 2 line, 2 line + 1
#pragma unroll
        for (int k = tid / 16; k < 128; k += FZ_NT / 16) {
          const float2 z = buf[k * 16 + line];  // Z(k)
          if (k == 0) {
            const float2 h = buf[128 * 16 + line];  // Z(128): A(128) = Re, B(128) = Im
            o[0] = make_float4(z.x, h.x, z.y, h.y);
          } else {
            const float2 w = buf[(256 - k) * 16 + line];                    // Z(-k)
            const float ax = 0.5f * (z.x + w.x), ay = 0.5f * (z.y - w.y);  // A(k) = (Z + conj W) / 2
            const float bx = 0.5f * (z.y + w.y), by = 0.5f * (w.x - z.x);  // B(k) = (Z - conj W) / 2i
            o[size_t(k) * 128] = make_float4(ax, ay, bx, by);
          }
        }
      } else {
        // column FFT of 16 raw columns (conversion and chirp in the first stage) -> S1 [ky][x]
        const float2 cx = __ldg(&a.chirp_x[s0 + (tid % 16)]);
        if (u8) pp_stages<256, 1, -1, RawSrc<true, true, 16, true>, GlobalOut, 16, FZ_BAR>(
                    RawSrc<true, true, 16, true>{raw, cys, cx}, buf, tws, out);
        else pp_stages<256, 1, -1, RawSrc<false, true, 16, true>, GlobalOut, 16, FZ_BAR>(
                 RawSrc<false, true, 16, true>{raw, cys, cx}, buf, tws, out);
      }
    } else if (pass == 3 || (pass == 1 && !asp)) {
      if (asp) {
        // column IFFT of 16 columns x = s0 .. s0 + 15 of S2 -> time queue [y][x]
        asm volatile("discard.global.L2 [%0], 128;\n" ::"l"(s2 + s0 + size_t(tid) * 256) : "memory");
        pp_stages<256, 1, +1, SmemSrc<16>, GlobalOutCs, 16, FZ_BAR>(SmemSrc<16>{buf}, buf, tws,
                                                                    GlobalOutCs{tq + tslot * FZ_FRAME + s0, 256u});
      } else {
        // 16 rows ky = s0 .. s0 + 15 of S1 -> row FFT -> time queue [ky][kx]
        asm volatile("discard.global.L2 [%0], 128;\n" ::"l"(s1 + size_t(s0) * 256 + size_t(tid) * 16) : "memory");
        float2* rowp = buf + rb * 256;
        float2 v[16];
#pragma unroll
        for (int m = 0; m < 16; ++m) v[m] = rowp[jl + 16 * m];
        row_fft16x16<-1>(v, rowp, tw2, jl);
        float2* out = tq + (tslot * 256 + size_t(s0 + rb)) * 256;
#pragma unroll
        for (int m = 0; m < 16; ++m) __stcs(&out[jl + 16 * m], v[m]);
      }
    } else {
      float2* rowp = buf + rb * 256;
      float2 v[16];
      int ky;
      if (pass == 1) {
        // rows ky = s0 .. s0 + 15 of S1 (row 0 packed with row 128): forward row FFT,
        // kept in S3 for the mirror pass; the staged strip of S1 is dead: drop its
        // L2 lines unwritten
        asm volatile("discard.global.L2 [%0], 128;\n" ::"l"(s1 + size_t(s0) * 256 + size_t(tid) * 16) : "memory");
        ky = int(s0) + rb;
#pragma unroll
        for (int m = 0; m < 16; ++m) v[m] = rowp[jl + 16 * m];
        row_fft16x16<-1>(v, rowp, tw2, jl);
        float2* w3 = s1 + size_t(128 + ky) * 256;
#pragma unroll
        for (int m = 0; m < 16; ++m) w3[jl + 16 * m] = v[m];
        if (s0 == 0 && warp == 0) {
          // row 0: W(0, k) = (Wp(k) + conj Wp(-k)) / 2 through the row's buffer
          __syncwarp();
#pragma unroll
          for (int m = 0; m < 16; ++m) rowp[jl + 16 * m] = v[m];
          __syncwarp();
          if (rb == 0) {
#pragma unroll
            for (int m = 0; m < 16; ++m) {
              const float2 w = rowp[(256 - jl - 16 * m) & 255];
              v[m] = make_float2(0.5f * (v[m].x + w.x), 0.5f * (v[m].y - w.y));
            }
          }
        }
      } else {
        // mirror rows ky = 143 + s0 - b of buffer row b, spectrum conj W(256 - ky, -kx);
        // row 128 from the packed row: W(128, k) = (Wp(k) - conj Wp(-k)) / 2i. The
        // staged rows of S3 are dead (16 threads a row; the first strip's last 16
        // threads reach S3 row 0 from 15 rows before it)
        const float2* w3 = s1 + size_t(s0 == 0 && tid >= 240 ? 128 - 15 : 128 + 113 - s0) * 256;
        asm volatile("discard.global.L2 [%0], 128;\n" ::"l"(w3 + size_t(tid) * 16) : "memory");
        ky = 143 + int(s0) - rb;
        if (ky == 128) {
#pragma unroll
          for (int m = 0; m < 16; ++m) {
            const float2 z = rowp[jl + 16 * m], w = rowp[(256 - jl - 16 * m) & 255];
            v[m] = make_float2(0.5f * (z.y + w.y), 0.5f * (w.x - z.x));
          }
        } else {
#pragma unroll
          for (int m = 0; m < 16; ++m) {
            const float2 w = rowp[(256 - jl - 16 * m) & 255];
            v[m] = make_float2(w.x, -w.y);
          }
        }
      }
      // x H(ky), inverse row FFT -> S2 [ky][x]
      const float2* hrow = a.asp_h + size_t(ky) * 256;
#pragma unroll
      for (int m = 0; m < 16; ++m) v[m] = cmul(v[m], __ldg(&hrow[jl + 16 * m]));
      row_fft16x16<+1>(v, rowp, tw2, jl);
      float2* out = s2 + size_t(ky) * 256;
#pragma unroll
      for (int m = 0; m < 16; ++m) out[jl + 16 * m] = v[m];
    }
    // the ring stores are read back by bulk copies (the async proxy) of other CTAs
    if (pass == 0 || (asp && pass < 3)) asm volatile("fence.proxy.async.global;\n" ::: "memory");
    // this warp is done with the buffer and has issued its stores: each warp releases
    // the buffer on its own and goes on to the next staged item (a column pass's
    // named barriers keep the warps in step within an item)
    __syncwarp();
    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(rw_smem(&freed[b])) : "memory");
  }
}

}  // namespace

bool spatial_fused_supported(const SpatialArgs& a) {
  return a.W == RW_L && a.H == RW_L && (a.spatial == HV_SPATIAL_ASP || a.spatial == HV_SPATIAL_FRESNEL) &&
         a.ring >= kFusedRing && a.fused_ctr && a.err && a.scratch1 &&
         (a.spatial == HV_SPATIAL_FRESNEL || (a.scratch2 && a.asp_h));
}

cudaError_t launch_spatial_fused(const SpatialArgs& a, cudaStream_t s, int* launches) {
  if (a.n == 0) return cudaSuccess;
  if (!spatial_fused_supported(a)) return cudaErrorInvalidValue;
  const bool asp = a.spatial == HV_SPATIAL_ASP;
  // ticket rows: one per frame plus the lags of the last pass; items per row
  const uint64_t nt = (uint64_t(a.n) + (asp ? FZ_LAG_ASP1 + 2u * FZ_LAG_ASP : FZ_LAG)) * (asp ? 40u : 32u);
  if (nt >= (1ull << 31)) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(a.fused_ctr, 0, (1 + kFusedPasses * size_t(a.ring)) * sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_spatial_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, int(FZ_SMEM));
  if (e != cudaSuccess) return e;
  int per_sm = 0, dev = 0, nsm = 0;
  // tensor maps: the raw ring (256 x cap 256 pixels, boxes of 32 (ASP) or 16 x 256) and
  // the S2 ring (256 x ring 256 complex, boxes of 16 x 256)
  CUtensorMap raw_map{}, s2_map{};
  const int bpp = a.in_kind == IN_U8 ? 1 : 2;
  if (!encode_map_2d(&raw_map, a.raw.base, bpp, RW_L, uint64_t(a.raw.cap) * RW_L, uint64_t(RW_L) * bpp,
                     a.spatial == HV_SPATIAL_ASP ? 32 : 16, 256))
    return cudaErrorNotSupported;
  if (a.spatial == HV_SPATIAL_ASP &&
      !encode_map_2d(&s2_map, a.scratch2, 8, RW_L, uint64_t(a.ring) * RW_L, uint64_t(RW_L) * 8, 16, 256))
    return cudaErrorNotSupported;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_spatial_fused, FZ_THREADS, FZ_SMEM);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  uint64_t grid = uint64_t(per_sm) * nsm;  // every CTA resident: the items' waits rely on it
  if (grid > nt) grid = nt;
  k_spatial_fused<<<unsigned(grid), FZ_THREADS, FZ_SMEM, s>>>(a, uint32_t(nt), raw_map, s2_map);
  ++*launches;
  return cudaGetLastError();
}

}  // namespace hv

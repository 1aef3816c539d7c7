// Streaming kernels with TMA-staged inputs: fake quantiser (Eq. 1 + Eq. 2) and
// quantise + pack for every group length; the straight-through backward
// (Eqs. 3-5) and the min/max initialisation for groups of at most 256 elements.
//
// These kernels move 2-6 bytes per element and would be bound by HBM bandwidth
// if the instruction stream per element were short enough; at 10-25 executed
// instructions per element it is the issue rate of the SM that decides, so the
// layout is chosen to keep everything that is per group or per access out of
// the per-element count:
//   * the loads are taken out of the compute threads altogether.  Each
//     persistent CTA has one producer thread that streams 16 KB tiles of the
//     input(s) into a shared-memory ring with tensor copies
//     (cp.async.bulk.tensor, completion on an mbarrier) while 8 consumer warps
//     compute; the flattened weight is described to the copy engine as a matrix
//     of 128-byte rows with the 128-byte swizzle;
//   * a consumer lane owns 32 CONSECUTIVE elements (half a row of the tile, four
//     16-byte vectors, always inside one quantisation group), so the group's
//     step size, zero point, reciprocal and clamp bounds are set up once per 32
//     elements, the group sums need one shuffle per doubling of the group
//     beyond 32, and the lane writes 64 contiguous bytes.  The swizzle makes
//     the lanes' 16-byte shared-memory reads conflict-free although they are 64
//     bytes apart.
// Three CTAs fit on an SM (24 consumer warps, up to 190 KB of reads in flight).
//
// Group sums are fixed-order (serial inside a lane, then a shuffle tree), so
// results are run-to-run identical.
#include <cuda.h>

#include "common.cuh"
#include "elementwise.cuh"
#include "gemm.cuh"
#include "ptx.cuh"
#include "quant_math.cuh"
#include "wait.cuh"

namespace eqat {

namespace {

constexpr int kConsumers = 256;
constexpr int kThreadsS = kConsumers + 32;           // + one producer warp
constexpr int kLaneElems = 32;                       // consecutive elements per consumer lane and tile
constexpr int kTileRows = kConsumers / 2;            // 128-byte rows per tile (two lanes per row)
constexpr int kTileElems = kConsumers * kLaneElems;  // 8192
constexpr int kTileBytes = kTileElems * 2;           // 16 KB per input stream
// Ring depth and CTAs per SM.  The stage a consumer works on is released as soon as its vectors are in
// registers, so a few stages are enough to keep the copy engine busy.
#ifndef EQAT_STREAM_CTAS1
#define EQAT_STREAM_CTAS1 3
#define EQAT_STREAM_STAGES1 4
#endif
constexpr int kStages1 = EQAT_STREAM_STAGES1, kCtas1 = EQAT_STREAM_CTAS1;   // kernels with one input stream
constexpr int kStages2 = 2, kCtas2 = 3;                                    // two input streams (32 KB per stage)

template <int NIN, int STAGES>
struct Ring {
  static constexpr int kStages = STAGES;
  static constexpr int kStageBytes = NIN * kTileBytes;
  static constexpr int kSmemBytes = kStages * kStageBytes + 1024 /*alignment slack*/ + 256 /*control block*/;
};

struct RingCtl {
  uint64_t full[8];
  uint64_t empty[8];
  int abort;
};
static_assert(sizeof(RingCtl) <= 256, "ring control block must fit its reservation");

// Runs `body(e0, raw, params)` on every consumer lane for every tile this CTA
// owns: e0 is the index of the lane's first element, raw[i][u] the lane's
// vector u (elements e0 + 8u .. e0 + 8u + 7) of input stream i, and params what
// `fetch(e0)` returned for this tile.  fetch is called one tile ahead, so the
// small per-group loads it makes (step size, zero point) are in flight while
// the previous tile is being computed.  The maps describe each input as
// [n_elem / 64, 64] bf16; rows beyond the end read as zeros, and a lane whose
// e0 is at or beyond n_elem must ignore its vectors.  BACKWARDS: from the end of the weight to its start, for kernels that
// usually run before or after one that reads a matrix of this size from its start: what the one reads last the other
// reads first, out of L2.  Min/max: quantise + pack follows it, itself forwards, because it takes 1 to 3 % longer backwards
// when nothing is in L2 (11008 x 4096, 2 bits 24.5 -> 25.1 us); min/max, quantise + pack and unpacking of that weight 52.8 -> 49.4
// us.  Straight-through backward: the weight gradient has been written just before (fake quantiser, three contractions of
// 256 tokens, backward of 11008 x 4096: 154.8 -> 152.3 us; of 28672 x 8192 with none between 421 -> 414 us, but 288 -> 312 us
// where 320 MB have been written since).
template <int NIN, int STAGES, bool BACKWARDS, typename Params, typename Fetch, typename Body>
__device__ __forceinline__ void stream_tiles(const CUtensorMap* const (&maps)[NIN], size_t n_elem, Fetch&& fetch,
                                             Body&& body) {
  using R = Ring<NIN, STAGES>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = ptx::smem_addr(smem_raw);
  const uint32_t smem_base = (raw_addr + 1023u) & ~1023u;            // stages are 1024-byte aligned (swizzle period)
  RingCtl* ctl = reinterpret_cast<RingCtl*>(smem_raw + (smem_base - raw_addr) + R::kStages * R::kStageBytes);
  volatile int* abort_flag = &ctl->abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t n_tiles = (n_elem + kTileElems - 1) / kTileElems;
  auto place = [&](size_t tile) { return BACKWARDS ? n_tiles - 1 - tile : tile; };

  if (threadIdx.x == 0) {
    for (int s = 0; s < R::kStages; ++s) {
      ptx::mbar_init(ptx::smem_addr(&ctl->full[s]), 1);
      ptx::mbar_init(ptx::smem_addr(&ctl->empty[s]), kConsumers / 32);
    }
    ctl->abort = 0;
    ptx::fence_mbar_init();
#pragma unroll
    for (int i = 0; i < NIN; ++i) ptx::tma_prefetch_desc(maps[i]);
  }
  __syncthreads();
  ptx::grid_dependency_wait();

  if (warp == kConsumers / 32) {
    // ---------------------------------------------------------------- producer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      size_t issued = 0;
      bool ok = true;
      for (size_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        if (!bounded_wait(ptx::smem_addr(&ctl->empty[stage]), phase ^ 1u, abort_flag, WAIT_STREAM_EMPTY, 32)) {
          ok = false;
          break;
        }
        ptx::fence_proxy_async_smem();                             // consumers' reads of this stage before the copy's writes
        const uint32_t full = ptx::smem_addr(&ctl->full[stage]);
        ptx::mbar_expect_tx(full, NIN * kTileBytes);               // rows past the end are zero-filled and counted
#pragma unroll
        for (int i = 0; i < NIN; ++i)
          ptx::tma_load_2d(smem_base + stage * R::kStageBytes + i * kTileBytes, maps[i], 0, (int)(place(tile) * kTileRows), full);
        ++issued;
        if (++stage == R::kStages) { stage = 0; phase ^= 1u; }
      }
      // The next launch may start when this CTA is about to finish: its last tile (with two inputs) or the one before has been
      // handed back.  Let in at once, its CTAs took the slots as they fell free, several of the low-numbered ones, which have
      // a tile more, on one SM: the straight-through backward of 1024 x 8192 took 15.4 us, without overlap 14.8, now 14.2;
      // of 512 x 2048 5.4, 4.9, 4.2 us; the fake quantiser of 1024 x 8192 8.9, 8.9, 8.6 us.
      if (ok && issued > 1) {
        const size_t last = issued - (NIN > 1 ? 1 : 2);
        ok = bounded_wait(ptx::smem_addr(&ctl->empty[last % R::kStages]), (uint32_t)((last / R::kStages) & 1), abort_flag,
                          WAIT_STREAM_EMPTY, 32);
      }
      ptx::grid_dependents_launch();
      if (!ok || *abort_flag) {
        // every copy this thread started must land before the CTA exits
        const size_t first = issued > (size_t)R::kStages ? issued - R::kStages : 0;
        for (size_t i = first; i < issued; ++i) {
          const uint32_t bar = ptx::smem_addr(&ctl->full[i % R::kStages]);
          const uint32_t par = (uint32_t)((i / R::kStages) & 1);
          const uint64_t t0 = ptx::globaltimer_ns();
          while (!ptx::mbar_try_wait(bar, par)) {
            if (ptx::globaltimer_ns() - t0 > 50000000ull) {
              atomicExch(&g_wait_status[1], (int)WAIT_TEARDOWN);
              break;
            }
          }
        }
      }
    }
  } else {
    // ---------------------------------------------------------------- consumers
    // lane t owns half (t & 1) of row (t >> 1): 16-byte chunk c of a row sits at chunk (c ^ (row & 7))
    const uint32_t row = threadIdx.x >> 1;
    const uint32_t row_off = row * 128u, sx = row & 7u, c0 = (threadIdx.x & 1u) * 4u;
    int stage = 0;
    uint32_t phase = 0;
    Params next = fetch(place(blockIdx.x) * kTileElems + (size_t)threadIdx.x * kLaneElems);
    for (size_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
      const Params cur = next;
      if (tile + gridDim.x < n_tiles) next = fetch(place(tile + gridDim.x) * kTileElems + (size_t)threadIdx.x * kLaneElems);
      if (!bounded_wait_warp(ptx::smem_addr(&ctl->full[stage]), phase, abort_flag, WAIT_STREAM_FULL)) break;
      uint4 raw[NIN][4];
      const uint32_t st = smem_base + stage * R::kStageBytes + row_off;
#pragma unroll
      for (int i = 0; i < NIN; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u) raw[i][u] = ptx::lds_128(st + i * kTileBytes + (((c0 + u) ^ sx) << 4));
      // The stage is handed back before the compute.  Its next user is a copy of the asynchronous proxy, which
      // is not ordered after these generic-proxy reads by the barrier alone: without a proxy fence on the way
      // a few lanes read rows of the tile four steps ahead (seen on 8192 x 8192 weights with three CTAs per SM).
      // The readers fence here, and the producer fences again between its wait and the copy.
      ptx::fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&ctl->empty[stage]));   // the stage can be refilled now
      if (++stage == R::kStages) { stage = 0; phase ^= 1u; }
      body(place(tile) * kTileElems + (size_t)threadIdx.x * kLaneElems, raw, cur);
    }
  }
}

// Step size and (already rounded) zero point of the group a lane's elements belong to.
struct GroupParams {
  float s, z;
};

// Group of a lane's elements.  Groups of up to 256 elements are powers of two; a longer one is any multiple of a lane's
// 32 elements, and one 32-bit division per lane and tile finds it (a weight has at most 2^34 elements).
template <bool LONG>
__device__ __forceinline__ size_t group_index(size_t e0, int group) {
  return LONG ? (size_t)((uint32_t)(e0 >> 5) / (uint32_t)group) : e0 >> group;
}

// `group`: log2 of the group length, or (LONG) the length in units of 32 elements.
template <bool LONG = false>
__device__ __forceinline__ GroupParams fetch_group(const float* s, const float* z, size_t e0,
                                                   size_t n_elem, int group) {
  GroupParams p{1.0f, 0.0f};
  if (e0 < n_elem) {
    const size_t g = group_index<LONG>(e0, group);
    p.s = ptx::ld_global(s + g);
    p.z = ptx::ld_global(z + g);
  }
  return p;
}

// A lane's 64 output bytes: two 32-byte stores where the tensor allows it, four 16-byte stores otherwise.
__device__ __forceinline__ void store_lane(eqat_bf16* dst, const uint4 (&o)[4], bool wide) {
  if (wide) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + 16 * h), "r"(o[2 * h].x),
                   "r"(o[2 * h].y), "r"(o[2 * h].z), "r"(o[2 * h].w), "r"(o[2 * h + 1].x), "r"(o[2 * h + 1].y),
                   "r"(o[2 * h + 1].z), "r"(o[2 * h + 1].w) : "memory");
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) reinterpret_cast<uint4*>(dst)[u] = o[u];
  }
}

// ------------------------------------------------------------------ 2-bit codes by comparison
// For s > 0 the code of Eq. 1, clamp(round(w / s) + zr, 0, 3), does not fall as w grows, so a group has three bf16 numbers
// T1 <= T2 <= T3 with code(w) = (w >= T1) + (w >= T2) + (w >= T3), and the packed comparison of bf16 pairs decides two
// elements at once.  The boundary of "round(w / s) >= m" is at (m - 0.5) s, which fp32 gives to half a unit in its last
// place; the bf16 numbers beside its nearest one v are at least a quarter of a bf16 unit away, 2^14 of those units, subnormal
// or not.  So they are decided, and v itself is put through the defining sequence.  About 25 instructions per threshold and
// lane and 3 per element, where the arithmetic on each element takes 9 and redoes the elements near a rounding boundary.  NaN compares false, i.e. code 0, like fmaxf and fminf.
// Groups of 64: fake quantiser of 28672 x 8192 175.6 -> 168.9 us, of 4096 x 4096 14.4 -> 13.7; quantise + pack on the min/max
// grid, whose quotients hit rounding boundaries, 109.8 -> 92.8 and 13.0 -> 11.6 us, with trained step sizes, which hardly do,
// 103.4 -> 93.1 and 12.2 -> 11.6 us.  (The thresholds from the residual of v instead of a division, or made before the wait for
// the tile, were 3 % slower: the ALU pipe sets the pace, and the divisions run on another.)
struct Thresholds2 {
  uint32_t t[3];                                        // bf16 pairs, both halves the same
  __device__ __forceinline__ Thresholds2(float s, float zr) {
#pragma unroll
    for (int k = 1; k <= 3; ++k) {
      const float m = (float)k - zr;                    // exact, |zr| <= 16
      uint32_t v = pack_bf16x2((m - 0.5f) * s, 0.0f) & 0xFFFFu;
      if (!(rintf(__fdiv_rn(__uint_as_float(v << 16), s)) >= m))
        v = (v & 0x8000u) != 0u ? (v == 0x8000u ? 1u : v - 1u) : v + 1u;      // the next greater number
      t[k - 1] = v * 0x10001u;
    }
  }
  // All-ones halves where w >= T(k + 1).
  __device__ __forceinline__ uint32_t at_least(int k, uint32_t w) const {
    return __hge2_mask(*reinterpret_cast<const __nv_bfloat162*>(&w), *reinterpret_cast<const __nv_bfloat162*>(&t[k]));
  }
  // The comparisons stand for the definition where the reciprocal path does (group_rcp) and s is positive.
  __device__ __forceinline__ static bool apply(float s, float rs) { return s > 0.0f && rs == rs; }
};

// ------------------------------------------------------------------ Eq. 1 + Eq. 2
// (clamp(r + z, 0, Q) - z) * s == clamp(r, -z, Q - z) * s for integer r and z.
template <bool LONG, bool TWO_BITS>
__global__ void __launch_bounds__(kThreadsS, kCtas1)
fakequant_stream_kernel(const __grid_constant__ CUtensorMap map_w, const float* s,
                        const float* z, eqat_bf16* __restrict__ What, size_t n_elem, int group,
                        float Q, int wide) {
  const CUtensorMap* const maps[1] = {&map_w};
  stream_tiles<1, kStages1, false, GroupParams>(maps, n_elem,
      [&](size_t e0) { return fetch_group<LONG>(s, z, e0, n_elem, group); },
      [&](size_t e0, const uint4 (&raw)[1][4], const GroupParams& gp) {
    if (e0 >= n_elem) return;
    const float sv = gp.s;
    const float zr = rintf(gp.z);
    const float rs = group_rcp(sv, zr);
    const float lo = -zr, hi = Q - zr;
    uint4 o[4];
    if (TWO_BITS && Thresholds2::apply(sv, rs)) {
      const Thresholds2 th(sv, zr);
      uint32_t value[4];                                  // the four values of the group, as bf16 pairs
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float v = fmaf((float)k - zr, sv, 0.0f);    // (a zero is +0, as Eq. 2 gives it)
        value[k] = pack_bf16x2(v, v);
      }
      auto pick = [&](uint32_t w) {
        uint32_t v = value[0];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const uint32_t m = th.at_least(k, w);
          v = (value[k + 1] & m) | (v & ~m);
        }
        return v;
      };
#pragma unroll
      for (int u = 0; u < 4; ++u) o[u] = make_uint4(pick(raw[0][u].x), pick(raw[0][u].y), pick(raw[0][u].z), pick(raw[0][u].w));
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float w[8], r[8], rt[8];
        unpack8(raw[0][u], w);
        quotient_round8(w, sv, rs, r, rt);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float c = fminf(fmaxf(r[i], lo), hi);
          w[i] = LONG ? fmaf(c, sv, 0.0f) : c * sv;         // (LONG: a zero is always +0; else -0 where r or the clamp is)
        }
        o[u] = pack8(w);
      }
    }
    store_lane(What + e0, o, wide != 0);
  });
}

// ------------------------------------------------------------------ Eqs. 3-5 + group sums
// With lo = -z, hi = Q - z and c = clamp(r, lo, hi): the element is in range iff
// c == r, and on the clamped branches Eq. 3's value (-z or Q - z) is c itself.
// Eq. 4 is a constant per group times the sum of the gradient over the clamped
// elements.  LPG = lanes per group (group / 32).
template <int LPG>
__global__ void __launch_bounds__(kThreadsS, kCtas2)
ste_bwd_stream_kernel(const __grid_constant__ CUtensorMap map_g, const __grid_constant__ CUtensorMap map_w,
                      const float* s, const float* z, eqat_bf16* __restrict__ dW,
                      float* __restrict__ ds, float* __restrict__ dz, size_t n_elem, float Q, int dz_literal, int wide) {
  const CUtensorMap* const maps[2] = {&map_g, &map_w};
  constexpr int group_shift = LPG == 1 ? 5 : LPG == 2 ? 6 : LPG == 4 ? 7 : 8;
  stream_tiles<2, kStages2, true, GroupParams>(maps, n_elem,
      [&](size_t e0) { return fetch_group(s, z, e0, n_elem, group_shift); },
      [&](size_t e0, const uint4 (&raw)[2][4], const GroupParams& gp) {
    const bool live = e0 < n_elem;                      // uniform over the lanes of a group
    float acc_s = 0.0f, acc_g = 0.0f;
    const float sv = gp.s;
    if (live) {
      const float zr = rintf(gp.z);
      const float rs = group_rcp(sv, zr);
      const float lo = -zr, hi = Q - zr;
      uint4 o[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float gr[8], w[8], r[8], rt[8];
        unpack8(raw[0][u], gr);
        unpack8(raw[1][u], w);
        quotient_round8(w, sv, rs, r, rt);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float c = fminf(fmaxf(r[i], lo), hi);
          const bool inside = (c == r[i]);
          acc_s = fmaf(gr[i], inside ? rt[i] : c, acc_s);     // Eq. 3
          acc_g += inside ? 0.0f : gr[i];                      // Eq. 4
          w[i] = inside ? gr[i] : 0.0f;                        // Eq. 5
        }
        o[u] = pack8(w);
      }
      store_lane(dW + e0, o, wide != 0);
    }
#pragma unroll
    for (int d = LPG / 2; d >= 1; d >>= 1) {
      acc_s += __shfl_xor_sync(0xFFFFFFFFu, acc_s, d);
      acc_g += __shfl_xor_sync(0xFFFFFFFFu, acc_g, d);
    }
    if (live && (threadIdx.x % LPG) == 0) {
      const size_t g = e0 >> group_shift;
      ds[g] = acc_s;
      if (dz != nullptr) dz[g] = (dz_literal ? -1.0f : -sv) * acc_g;
    }
  });
}

// ------------------------------------------------------------------ min/max initialisation
struct NoParams {};

__device__ __forceinline__ uint32_t bf162_max(uint32_t a, uint32_t b) {
  const __nv_bfloat162 r = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
  return *reinterpret_cast<const uint32_t*>(&r);
}
__device__ __forceinline__ uint32_t bf162_min(uint32_t a, uint32_t b) {
  const __nv_bfloat162 r = __hmin2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
  return *reinterpret_cast<const uint32_t*>(&r);
}

template <int LPG>
__global__ void __launch_bounds__(kThreadsS, kCtas1)
minmax_stream_kernel(const __grid_constant__ CUtensorMap map_w, float* __restrict__ s, float* __restrict__ z,
                     size_t n_elem, float Q) {
  const CUtensorMap* const maps[1] = {&map_w};
  constexpr int group_shift = LPG == 1 ? 5 : LPG == 2 ? 6 : LPG == 4 ? 7 : 8;
  stream_tiles<1, kStages1, true, NoParams>(maps, n_elem, [](size_t) { return NoParams{}; },
      [&](size_t e0, const uint4 (&raw)[1][4], const NoParams&) {
    // extrema on packed bf16 pairs (exact: comparisons only), widened to fp32 at the end
    uint32_t mx2 = 0xFF80FF80u, mn2 = 0x7F807F80u;      // (-inf, -inf) and (+inf, +inf) as bf16 pairs
    const bool live = e0 < n_elem;                      // uniform over the lanes of a group
    if (live) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint4 r4 = raw[0][u];
        mx2 = bf162_max(mx2, bf162_max(bf162_max(r4.x, r4.y), bf162_max(r4.z, r4.w)));
        mn2 = bf162_min(mn2, bf162_min(bf162_min(r4.x, r4.y), bf162_min(r4.z, r4.w)));
      }
    }
#pragma unroll
    for (int d = LPG / 2; d >= 1; d >>= 1) {
      mx2 = bf162_max(mx2, __shfl_xor_sync(0xFFFFFFFFu, mx2, d));
      mn2 = bf162_min(mn2, __shfl_xor_sync(0xFFFFFFFFu, mn2, d));
    }
    if (live && (threadIdx.x % LPG) == 0) {
      const float mx = fmaxf(__uint_as_float(mx2 << 16), __uint_as_float(mx2 & 0xFFFF0000u));
      const float mn = fminf(__uint_as_float(mn2 << 16), __uint_as_float(mn2 & 0xFFFF0000u));
      // s = max((max - min) / Q, 2^-14), z = clamp(-round(min / s), 0, Q), all in binary32
      float sv = __fdiv_rn(mx - mn, Q);
      sv = fmaxf(sv, 6.103515625e-05f);
      float zv = -rintf(__fdiv_rn(mn, sv));
      zv = fminf(fmaxf(zv, 0.0f), Q) + 0.0f;
      s[e0 >> group_shift] = sv;
      z[e0 >> group_shift] = zv;
    }
  });
}

// ------------------------------------------------------------------ quantise + pack (hand-off)
// A lane turns its 32 weights into 32 codes = BITS consecutive 32-bit words of the
// little-endian stream (code j of the lane at bits [BITS*j, BITS*j + BITS)).
//
// Only the clamped code is wanted here, not r or r - w/s, which allows a shorter
// exact evaluation of Eq. 1 than quotient_round8.  With cz = 2^23 + zr (an
// integer) t = fma(w, rs, cz) rounds w*rs + zr to an integer held in the low
// mantissa bits of t whenever the sum is in [0, 2^23), and lands below 2^23
// (code 0 after the clamp) when it is negative.  The code is DEFINED through
// y0 = rn(w / s).  Take the two reciprocals rs_lo = rs (1 - 2^-16) and
// rs_hi = rs (1 + 2^-16), rs good to 1 ulp: the exact products w*rs_lo and
// w*rs_hi enclose y0 with a margin of 2^-17 |y0| on either side, and rounding is
// monotone, so when t_lo == t_hi every value between the products, y0 among
// them, rounds to the same integer; y0 itself cannot be an exact tie then, since
// a tie strictly inside the interval would separate t_lo from t_hi.  (The
// integer added before rounding changes which neighbour a tie goes to, but a tie
// never reaches this branch.)  When they differ (the quotient is within about
// 2^-16 |y0| of a rounding boundary: a few elements per thousand) the element
// is redone with the defining sequence.  Two multiply-adds and one logic
// operation per element, and the clamped t feeds the bit packing directly: its
// low bits ARE the code.
template <int BITS, bool LONG>
__global__ void __launch_bounds__(kThreadsS, kCtas1)
quantize_pack_stream_kernel(const __grid_constant__ CUtensorMap map_w, const float* s,
                            const float* z, uint8_t* __restrict__ packed, uint8_t* __restrict__ z8,
                            eqat_fp16* __restrict__ s16, size_t n_elem, int group) {
  const CUtensorMap* const maps[1] = {&map_w};
  constexpr float Q = (float)((1 << BITS) - 1);
  constexpr float kTwo23 = 8388608.0f;
  // sum over the 8 codes of a vector of the bit pattern of 2^23 shifted to the code's place (mod 2^32)
  constexpr uint32_t kBias = (uint32_t)(0x4B000000ull * (((1ull << (8 * BITS)) - 1ull) / ((1ull << BITS) - 1ull)));
  stream_tiles<1, kStages1, false, GroupParams>(maps, n_elem,
      [&](size_t e0) { return fetch_group<LONG>(s, z, e0, n_elem, group); },
      [&](size_t e0, const uint4 (&raw)[1][4], const GroupParams& gp) {
    if (e0 >= n_elem) return;
    const float sv = gp.s;
    const float zr = rintf(gp.z);
    const float rs = group_rcp(sv, zr);                 // NaN: the whole group takes the defining sequence
    uint32_t* dst = reinterpret_cast<uint32_t*>(packed) + (e0 >> 5) * BITS;
    // Zero point and step size, by the group's first lane: before the comparisons (28672 x 8192, groups of 64: 92.8 against 96.7
    // us with it after them), after everything else (3 bits 111.8 against 114.5 us, 4 bits 120.8 against 124.0 us).
    auto hand_over = [&] {
      const size_t g = group_index<LONG>(e0, group);
      if (e0 == (LONG ? g * (size_t)group << 5 : g << group)) {
        z8[g] = (uint8_t)(__float_as_uint(fminf(fmaxf(zr, 0.0f), Q) + 8388608.0f) & 0xFFu);
        s16[g] = __half_as_ushort(__float2half_rn(sv));
      }
    };
    constexpr bool kFirst = BITS == 2 && !LONG;
    if constexpr (kFirst) hand_over();
    if constexpr (BITS == 2) {
      if (Thresholds2::apply(sv, rs)) {
        // Codes j and j + 8 of a word are decided as a pair.  With c and d their codes, the three masks, each -1 in a half
        // where it holds, add up to -(c + 2^16 (d - c)) as 32-bit numbers; so do the sums over all j, shifted by 2 j.  The lower
        // half, the first eight codes, is missing in the upper one, and is added by the last multiplication.  (Selecting and
        // masking bits took three logic operations per pair, this takes one addition and one shifted one, which the FMA pipe
        // can do, and the ALU pipe sets the pace: 28672 x 8192, groups of 64, 106.5 -> 93.2 us, 11008 x 4096 24.8 -> 22.5 us.)
        const Thresholds2 th(sv, zr);
        const uint32_t w[16] = {raw[0][0].x, raw[0][0].y, raw[0][0].z, raw[0][0].w, raw[0][1].x, raw[0][1].y, raw[0][1].z, raw[0][1].w,
                                raw[0][2].x, raw[0][2].y, raw[0][2].z, raw[0][2].w, raw[0][3].x, raw[0][3].y, raw[0][3].z, raw[0][3].w};
        uint32_t word[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t acc = 0u;
#pragma unroll
          for (int j = 7; j >= 0; --j) {
            const uint32_t pair = __byte_perm(w[8 * h + (j >> 1)], w[8 * h + 4 + (j >> 1)], (j & 1) ? 0x7632 : 0x5410);
            acc = 4u * acc + (th.at_least(0, pair) + th.at_least(1, pair) + th.at_least(2, pair));
          }
          word[h] = 0u - acc * 0x10001u;
        }
        if constexpr (!kFirst) hand_over();
        *reinterpret_cast<uint2*>(dst) = make_uint2(word[0], word[1]);
        return;
      }
    }
    const bool exact_only = !(fabsf(rs) >= 2.5e-38f);   // (also when rs_lo would lose bits to underflow)
    const float rs_lo = rs * 0.9999847412109375f, rs_hi = rs * 1.0000152587890625f;
    const float cz = kTwo23 + zr;
    uint32_t piece[4];                                  // vector u's 8 codes, code i at bits [BITS*i, BITS*i + BITS)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float w[8], t[8];
      unpack8(raw[0][u], w);
      uint32_t differ[2] = {exact_only ? 1u : 0u, exact_only ? 1u : 0u};   // elements 0..3 and 4..7
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        t[i] = fmaf(w[i], rs_lo, cz);
        differ[i >> 2] |= __float_as_uint(t[i]) ^ __float_as_uint(fmaf(w[i], rs_hi, cz));
      }
      if ((differ[0] | differ[1]) != 0u) {
        // the whole warp walks what one lane walks, so the walk goes by halves of the vector (see quotient_round8)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (differ[h] != 0u) {
#pragma unroll
            for (int i = 4 * h; i < 4 * h + 4; ++i) {
              if (exact_only || !(t[i] == fmaf(w[i], rs_hi, cz))) {
                const float r = rintf(__fdiv_rn(w[i], sv));
                t[i] = (r + zr) + kTwo23;
              }
            }
          }
        }
      }
      uint32_t acc = 0u;
#pragma unroll
      for (int i = 7; i >= 0; --i)
        acc = (acc << BITS) + __float_as_uint(fminf(fmaxf(t[i], kTwo23), kTwo23 + Q));
      piece[u] = acc - kBias;
    }
    if constexpr (!kFirst) hand_over();
    if constexpr (BITS == 2) {
      *reinterpret_cast<uint2*>(dst) = make_uint2(piece[0] | (piece[1] << 16), piece[2] | (piece[3] << 16));
    } else if constexpr (BITS == 3) {
      dst[0] = piece[0] | (piece[1] << 24);
      dst[1] = (piece[1] >> 8) | (piece[2] << 16);
      dst[2] = (piece[2] >> 16) | (piece[3] << 8);
    } else {
      *reinterpret_cast<uint4*>(dst) = make_uint4(piece[0], piece[1], piece[2], piece[3]);
    }
  });
}

// The flattened [out, in] weight as rows of 64 elements, one tile of kTileRows rows per copy.
inline bool weight_map(CUtensorMap* tm, const eqat_bf16* p, size_t n_elem) {
  return make_tmap_bf16(tm, p, 64, n_elem / 64, kTileRows);
}

inline bool aligned32(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 31u) == 0; }

// Persistent grid: every CTA resident at once, never more CTAs than tiles.  The kernel is a template
// argument so that each kernel has its own per-device state: the shared-memory opt-in and the number of
// CTAs that fit on an SM (both asked of the runtime once per device).
template <auto kernel, typename... Args>
int launch_stream(int smem_bytes, size_t n_elem, cudaStream_t st, Args... args) {
  static SmemOptIn opt_in;
  static std::atomic<int> ctas_per_sm[kMaxCachedDevices];
  if (!opt_in.ensure(kernel, smem_bytes)) return EQAT_ERR_CUDA;
  const int dev = current_device(), sms = sm_count();
  if (dev < 0 || sms <= 0) return EQAT_ERR_CUDA;
  int per_sm = dev < kMaxCachedDevices ? ctas_per_sm[dev].load(std::memory_order_relaxed) : 0;
  if (per_sm <= 0) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kThreadsS, smem_bytes) != cudaSuccess ||
        per_sm <= 0) {
      (void)cudaGetLastError();
      return EQAT_ERR_CUDA;
    }
    if (dev < kMaxCachedDevices) ctas_per_sm[dev].store(per_sm, std::memory_order_relaxed);
  }
  const size_t tiles = (n_elem + kTileElems - 1) / kTileElems;
  const size_t resident = (size_t)sms * per_sm;
  const unsigned grid = (unsigned)(tiles < resident ? tiles : resident);
  return launch_overlapped(kernel, dim3(grid), dim3(kThreadsS), (size_t)smem_bytes, st, args...);
}

inline int group_shift_of(int group) {
  int sh = 5;
  while ((1 << sh) < group) ++sh;
  return sh;
}

}  // namespace

int launch_fakequant(const eqat_desc& d, const eqat_bf16* W, const float* s, const float* z, eqat_bf16* What,
                            cudaStream_t st) {
  const size_t n_elem = (size_t)d.out_features * d.in_features;
  const float Q = (float)((1 << d.bits) - 1);
  CUtensorMap mw;
  if (!weight_map(&mw, W, n_elem)) return EQAT_ERR_CUDA;
  constexpr int smem = Ring<1, kStages1>::kSmemBytes;
  const int wide = (int)aligned32(What);
  const int group = d.group > 256 ? d.group / 32 : group_shift_of(d.group);
  switch ((d.group > 256 ? 2 : 0) + (d.bits == 2 ? 1 : 0)) {
    case 0:  return launch_stream<fakequant_stream_kernel<false, false>>(smem, n_elem, st, mw, s, z, What, n_elem, group, Q, wide);
    case 1:  return launch_stream<fakequant_stream_kernel<false, true>>(smem, n_elem, st, mw, s, z, What, n_elem, group, Q, wide);
    case 2:  return launch_stream<fakequant_stream_kernel<true, false>>(smem, n_elem, st, mw, s, z, What, n_elem, group, Q, wide);
    default: return launch_stream<fakequant_stream_kernel<true, true>>(smem, n_elem, st, mw, s, z, What, n_elem, group, Q, wide);
  }
}

int launch_ste_bwd_stream(const eqat_desc& d, const eqat_bf16* dWhat, const eqat_bf16* W, const float* s,
                          const float* z, eqat_bf16* dW, float* ds, float* dz, cudaStream_t st) {
  const size_t n_elem = (size_t)d.out_features * d.in_features;
  const float Q = (float)((1 << d.bits) - 1);
  const int lit = d.dz_mode == 1, wide = (int)aligned32(dW);
  CUtensorMap mg, mw;
  if (!weight_map(&mg, dWhat, n_elem) || !weight_map(&mw, W, n_elem)) return EQAT_ERR_CUDA;
  constexpr int smem = Ring<2, kStages2>::kSmemBytes;
  switch (d.group) {
    case 32:  return launch_stream<ste_bwd_stream_kernel<1>>(smem, n_elem, st, mg, mw, s, z, dW, ds, dz, n_elem, Q, lit, wide);
    case 64:  return launch_stream<ste_bwd_stream_kernel<2>>(smem, n_elem, st, mg, mw, s, z, dW, ds, dz, n_elem, Q, lit, wide);
    case 128: return launch_stream<ste_bwd_stream_kernel<4>>(smem, n_elem, st, mg, mw, s, z, dW, ds, dz, n_elem, Q, lit, wide);
    default:  return launch_stream<ste_bwd_stream_kernel<8>>(smem, n_elem, st, mg, mw, s, z, dW, ds, dz, n_elem, Q, lit, wide);
  }
}

int launch_minmax_stream(const eqat_desc& d, const eqat_bf16* W, float* s, float* z, cudaStream_t st) {
  const size_t n_elem = (size_t)d.out_features * d.in_features;
  const float Q = (float)((1 << d.bits) - 1);
  CUtensorMap mw;
  if (!weight_map(&mw, W, n_elem)) return EQAT_ERR_CUDA;
  constexpr int smem = Ring<1, kStages1>::kSmemBytes;
  switch (d.group) {
    case 32:  return launch_stream<minmax_stream_kernel<1>>(smem, n_elem, st, mw, s, z, n_elem, Q);
    case 64:  return launch_stream<minmax_stream_kernel<2>>(smem, n_elem, st, mw, s, z, n_elem, Q);
    case 128: return launch_stream<minmax_stream_kernel<4>>(smem, n_elem, st, mw, s, z, n_elem, Q);
    default:  return launch_stream<minmax_stream_kernel<8>>(smem, n_elem, st, mw, s, z, n_elem, Q);
  }
}

int launch_quantize_pack(const eqat_desc& d, const eqat_bf16* W, const float* s, const float* z,
                                uint8_t* packed, uint8_t* z8, eqat_fp16* s16, cudaStream_t st) {
  const size_t n_elem = (size_t)d.out_features * d.in_features;
  const bool longer = d.group > 256;
  const int group = longer ? d.group / 32 : group_shift_of(d.group);
  CUtensorMap mw;
  if (!weight_map(&mw, W, n_elem)) return EQAT_ERR_CUDA;
  constexpr int smem = Ring<1, kStages1>::kSmemBytes;
  switch (d.bits * 2 + (longer ? 1 : 0)) {
    case 4:  return launch_stream<quantize_pack_stream_kernel<2, false>>(smem, n_elem, st, mw, s, z, packed, z8, s16, n_elem, group);
    case 5:  return launch_stream<quantize_pack_stream_kernel<2, true>>(smem, n_elem, st, mw, s, z, packed, z8, s16, n_elem, group);
    case 6:  return launch_stream<quantize_pack_stream_kernel<3, false>>(smem, n_elem, st, mw, s, z, packed, z8, s16, n_elem, group);
    case 7:  return launch_stream<quantize_pack_stream_kernel<3, true>>(smem, n_elem, st, mw, s, z, packed, z8, s16, n_elem, group);
    case 8:  return launch_stream<quantize_pack_stream_kernel<4, false>>(smem, n_elem, st, mw, s, z, packed, z8, s16, n_elem, group);
    default: return launch_stream<quantize_pack_stream_kernel<4, true>>(smem, n_elem, st, mw, s, z, packed, z8, s16, n_elem, group);
  }
}

int launch_wait_expiry_stream(cudaStream_t st) { return launch_wait_expiry(st); }
int read_stream_status(int* status, int* detail) { return read_wait_status(status, detail); }

}  // namespace eqat

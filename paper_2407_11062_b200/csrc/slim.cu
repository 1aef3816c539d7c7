// Packed-weight forward for a few tokens,
//     Y[T,out] = X[T,in] * dequant(Wq)^T,
// on tiles of 128 WEIGHT rows: the weight is the M side of the tensor-core tile (its rows fill the 128 tensor-memory
// lanes whatever the number of tokens) and the tokens are the narrow N side.
//
// Every code is expanded once per token tile, to the exact small integer q - z (or q, see below) as bf16, and the
// step sizes multiply fp32 accumulators afterwards: a group's products are accumulated in tensor memory by itself,
// read back and added to the row's running sums as s * D.  Nothing is rounded between the codes and the sums.
//
// The rows of the A operand live in TENSOR MEMORY (tcgen05.mma with A in TMEM): lane = weight row, so the thread that
// owns a row reads its codes, expands them in registers and writes them with one tcgen05.st per 64 codes; the same
// thread later reads the row's accumulators back, so the group's step size never leaves its registers.
//
// 32 lanes on 32 rows make every global load 32 L1 lookups, so nothing is fetched that way: codes and activations arrive
// by TMA, 256 columns per stage, and the step sizes and zero points of the CTA's whole K slice are laid out in shared
// memory once, read along the rows.
//
// K is split over the CTAs of a cluster (and over the groups of row threads of a CTA), which is what fills the chip: a
// 4096-row weight has only 32 row tiles.  The partial sums meet in the shared memory of the CTA that owns a token column
// and are added there in a fixed order, so results are run-to-run identical and no scratch memory is needed.
//
// Roles: warp 0 TMA producer, warp 1 MMA issuer and TMEM owner, then two groups (three, for more than 32 token columns)
// of 128 row threads.  A run = 128 codes of a row.  Group g takes the runs g, g + groups, ... of the CTA's K slice:
// add up the accumulators of the group's run before, expand the run into the group's TMEM buffer, signal.  While one
// group's MMAs run, the other group and the other CTA of the SM expand.
//
// What bounds it: at a few row tiles per SM the chain of hand-offs outside the runs (about 4 us: barriers and TMEM, the
// parameters, the exchange); on large weights the issue slots and the hand-offs of the runs, about 700 cycles per run and
// SM where the eight MMAs of a run take 340 (an MMA of 16 columns costs its A operand's 4 KB).
#include <cuda.h>

#include <type_traits>

#include "common.cuh"
#include "expand.cuh"
#include "gemm.cuh"
#include "gemv.cuh"
#include "ptx.cuh"
#include "slim.cuh"
#include "wait.cuh"

namespace eqat {
namespace {

constexpr int kRows = 128;             // weight rows per tile = TMEM lanes
constexpr int kRun = 128;              // codes of a row per run
constexpr int kSlimMaxTokens = 64;
constexpr int kMaxSplit = 8;           // CTAs of a cluster (portable limit)
constexpr int kMaxSmem = 232448;

struct SlimParams : PackedWeight {
  eqat_bf16* Y;                        // [T, out]
  int T;
  int split, split_log2, runs;         // runs = in_features / 128
};

// A stage of the ring: the codes of two runs, a box of 128 rows of 64, 96 or 128 bytes, and their activations.
constexpr int kBoxRuns = 2;
__host__ __device__ constexpr int box_bytes(int bits) { return kBoxRuns * 16 * bits; }

// A CTA's K slice: whole boxes, as even as they go.
__device__ inline void slice_of(int runs, int split_log2, int rank, int& run0, int& nruns) {
  const int boxes = (runs + kBoxRuns - 1) / kBoxRuns;
  const int b0 = (boxes * rank) >> split_log2, b1 = (boxes * (rank + 1)) >> split_log2;
  run0 = b0 * kBoxRuns;
  nruns = (b1 * kBoxRuns < runs ? b1 * kBoxRuns : runs) - run0;
}
// Groups of a row that a slice touches, and the first of them.
__device__ inline int slice_groups(int run0, int nruns, int group_shift, int& first) {
  first = (run0 * kRun) >> group_shift;
  return (((run0 + nruns) * kRun - 1) >> group_shift) - first + 1;
}
constexpr int kParamPitch = kRows + 1;   // words per group: a word = one row's step size and zero point

struct SlimCtl {
  uint64_t full[4], empty[4];
  uint64_t a_full[3], d_ready[3];      // per group
  uint32_t tmem_base;
  int abort;
  int past127;                         // some zero point byte of the slice is past 127
};

// Shared memory and tensor memory of a CTA for token tiles of 16*NT columns and ND accumulators per run.
template <int BITS, int NT, int ND>
struct Slim {
  static constexpr int kTn = 16 * NT;
  static constexpr int kGroups = NT <= 2 ? 2 : 3;                        // groups of 128 row threads
  static constexpr int kRowWarps = 4 * kGroups;
  static constexpr int kThreads = (2 + kRowWarps) * 32;
  static constexpr int kCodes = kRows * box_bytes(BITS);
  static constexpr int kBlock = kTn * 128;                               // activations of one K block (64 columns)
  static constexpr int kStage = kCodes + 2 * kBoxRuns * kBlock;
  static constexpr int kStages = NT == 1 ? (BITS == 2 ? 4 : 3) : (NT == 3 ? 3 : 2);
  static constexpr int kOnesOff = kStages * kStage;
  static constexpr int kOnes = 16384;                                    // constant A operand of the column sums
  static constexpr int kPart = kGroups * kTn * kRows * 4;                // partial sums received from the cluster
  static constexpr int kTmemA = kGroups * 64;
  static constexpr int kTmemD = kGroups * ND * kTn;
  __host__ __device__ static constexpr int tmem_cols(bool zf) { return kTmemA + kTmemD * (zf ? 2 : 1) <= 256 ? 256 : 512; }
  __host__ __device__ static constexpr int part_off(bool zf) { return kOnesOff + (zf ? kOnes : 0); }
  // `groups`: the most quantisation groups of a row that a CTA's slice touches
  static constexpr int smem_bytes(bool zf, int groups) {
    const int need = part_off(zf) + kPart + groups * kParamPitch * 4 + (int)sizeof(SlimCtl) + 1024;
    // Tensor memory is what must never be waited for (a CTA of a cluster that waits for columns held by another
    // cluster could close a circle): with 256 columns at most two CTAs may share an SM, with 512 only one, and shared
    // memory is what enforces it, against CTAs of the other variants too.
    const int least = tmem_cols(zf) == 256 ? 78 * 1024 : 156 * 1024;
    return need > least ? need : least;
  }
};

__device__ __forceinline__ uint32_t add_bf16x2(uint32_t a, uint32_t b) {
  const __nv_bfloat162 r = __hadd2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
  return *reinterpret_cast<const uint32_t*>(&r);
}
// (t & MASK) | magic with the mask as an immediate of the instruction and the magic in a register (given two
// compile-time constants the compiler re-creates one of them with a move in front of every use).
template <uint32_t MASK>
__device__ __forceinline__ uint32_t and_imm_or(uint32_t t, uint32_t magic) {
  uint32_t r;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(t), "n"(MASK), "r"(magic));
  return r;
}

// The bf16 pairs (128, 128) and (8, 8), built from a value that is zero at run time only.
struct Magics {
  uint32_t m128, m8;
  __device__ __forceinline__ explicit Magics(uint32_t zero) : m128(0x43004300u | zero), m8(0x41004100u | zero) {}
};

// Negated offsets of a group: -(bias + z) for the biases 128 and 8 that the expansion leaves on a code, as bf16 pairs.
// z is an integer of at most 7 bits here, so every one of them, and every difference below, is exact in bf16; a zero
// point byte past 127, which no hand-off produces, comes off in a second addition (q - z has at most eight bits then).
struct Offsets {
  uint32_t n128, n8;
  __device__ __forceinline__ explicit Offsets(float z)
      : n128(pack_bf16x2(-128.0f - z, -128.0f - z)), n8(pack_bf16x2(-8.0f - z, -8.0f - z)) {}
};

// 32 consecutive codes -> 16 registers of bf16 pairs (q - z of codes 2i, 2i + 1), in the order of the stream, which is
// the order of the activations.  A code at the bottom of a 16-bit half with 0x4300 above it is the bf16 number
// 128 + q; at bit 4 with 0x4100, 8 + q.  `y` holds a run of codes in its low half and the same run, one code later, in
// its high half (a shift and a byte permute): a pair then is one logic operation, and the offset comes off in one
// packed addition.
template <int BITS>
__device__ __forceinline__ void expand32(const uint32_t* w, const Offsets& f, const Magics& k, uint32_t* r) {
  if constexpr (BITS == 2) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {                        // codes 8h .. 8h+7 of the word
        const uint32_t y = h == 0 ? __byte_perm(w[i], w[i] << 14, 0x7610) : __byte_perm(w[i], w[i] >> 2, 0x7632);
        const uint32_t y8 = y >> 8;
        uint32_t* o = r + 8 * i + 4 * h;
        o[0] = add_bf16x2(and_imm_or<0x00030003u>(y, k.m128), f.n128);
        o[1] = add_bf16x2(and_imm_or<0x00300030u>(y, k.m8), f.n8);
        o[2] = add_bf16x2(and_imm_or<0x00030003u>(y8, k.m128), f.n128);
        o[3] = add_bf16x2(and_imm_or<0x00300030u>(y8, k.m8), f.n8);
      }
    }
  } else if constexpr (BITS == 4) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {                        // codes 4h .. 4h+3 of the word
        const uint32_t y = h == 0 ? __byte_perm(w[i], w[i] << 12, 0x7610) : __byte_perm(w[i], w[i] >> 4, 0x7632);
        uint32_t* o = r + 4 * i + 2 * h;
        o[0] = add_bf16x2(and_imm_or<0x000F000Fu>(y, k.m128), f.n128);
        o[1] = add_bf16x2(and_imm_or<0x000F000Fu>(y >> 8, k.m128), f.n128);
      }
    }
  } else {
#pragma unroll
    for (int m = 0; m < 8; ++m) {                          // codes 4m .. 4m+3: bits 12m .. 12m+11 of the 96
      const int start = 12 * m, word = start >> 5, sh = start & 31;
      const uint32_t lo = sh == 0 ? w[word] : (sh <= 16 ? w[word] >> sh : __funnelshift_r(w[word], w[word + 1 < 3 ? word + 1 : 2], sh));
      const uint32_t y = __byte_perm(lo, lo << 13, 0x7610);
      r[2 * m] = add_bf16x2(and_imm_or<0x00070007u>(y, k.m128), f.n128);
      r[2 * m + 1] = add_bf16x2(and_imm_or<0x00070007u>(y >> 6, k.m128), f.n128);
    }
  }
}

// The 128 codes of run j of a box, of box row `row`: 4*BITS words.  16-byte piece c of row r sits at piece c ^ (r & 7)
// of 128-byte rows, c ^ ((r >> 1) & 3) of 64-byte rows (the copy engine's swizzles); 96-byte rows are not swizzled.
template <int BITS>
__device__ __forceinline__ void load_run(uint32_t box, int row, int j, uint32_t (&w)[4 * BITS]) {
  const uint32_t sx = BITS == 4 ? (uint32_t)(row & 7) : (BITS == 2 ? (uint32_t)((row >> 1) & 3) : 0u);
#pragma unroll
  for (int i = 0; i < BITS; ++i) {
    const uint4 t = ptx::lds_128(box + (uint32_t)(row * box_bytes(BITS)) + (((uint32_t)(j * BITS + i) ^ sx) << 4));
    w[4 * i] = t.x; w[4 * i + 1] = t.y; w[4 * i + 2] = t.z; w[4 * i + 3] = t.w;
  }
}

// NT: token columns / 16.  ND: accumulators per run, one per quantisation group (1: groups of 128 and longer; 2: 64;
// 4: 32).
template <int BITS, int NT, int ND>
__global__ void __launch_bounds__(Slim<BITS, NT, ND>::kThreads, NT <= 2 ? 2 : 1)
slim_fwd_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, const SlimParams p) {
  using C = Slim<BITS, NT, ND>;
  constexpr int kGroups = C::kGroups, kThreads = C::kThreads;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = ptx::smem_addr(smem_raw);
  const uint32_t ring_addr = (raw_addr + 1023u) & ~1023u;
  uint8_t* ring = smem_raw + (ring_addr - raw_addr);
  const bool zf = p.z_fp16 != 0;
  constexpr uint32_t ones_off = C::kOnesOff;
  const uint32_t part_off = (uint32_t)C::part_off(zf);
  SlimCtl* ctl = reinterpret_cast<SlimCtl*>(ring + part_off + C::kPart);
  const uint32_t param_off = part_off + C::kPart + (uint32_t)sizeof(SlimCtl);
  volatile int* abort_flag = &ctl->abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // grid: row tiles x CTAs of a cluster x token tiles
  const int rank = (int)blockIdx.y;
  const int t0 = (int)blockIdx.z * C::kTn, m0 = (int)blockIdx.x * kRows;
  int run0, nruns, group0;
  slice_of(p.runs, p.split_log2, rank, run0, nruns);
  const int ngroups = slice_groups(run0, nruns, p.group_shift, group0);

  // The codes, step sizes and zero points of this CTA's slice are asked into L2 before the wait for the launches before
  // this one: a prefetch changes nothing that can be observed, and it takes the DRAM latency out of the loop below.
  if (warp == 0 && ptx::elect_one()) {
    for (int r = 0; r < nruns; r += kBoxRuns) ptx::tma_prefetch_2d(&map_w, (run0 + r) * (16 * BITS), m0);
  }
  if (threadIdx.x >= kRows && threadIdx.x < 2 * kRows && m0 + (int)threadIdx.x - kRows < p.out_features) {
    const size_t g0 = (size_t)(m0 + threadIdx.x - kRows) * p.groups_per_row + group0;
    const char* sp = reinterpret_cast<const char*>(p.s16 + g0);
    const char* zp = static_cast<const char*>(p.zq) + g0 * (zf ? 2 : 1);
    const int sb = 2 * ngroups, zb = zf ? sb : ngroups;
    for (int o = 0; o < sb; o += 128) ptx::prefetch_l2_line(sp + o);
    for (int o = 0; o < zb; o += 128) ptx::prefetch_l2_line(zp + o);
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kStages; ++s) {
      ptx::mbar_init(ptx::smem_addr(&ctl->full[s]), 1);
      ptx::mbar_init(ptx::smem_addr(&ctl->empty[s]), 4 * kBoxRuns + 1);   // the row warps of its runs, and the MMAs
    }
    for (int g = 0; g < kGroups; ++g) {
      ptx::mbar_init(ptx::smem_addr(&ctl->a_full[g]), 4);
      ptx::mbar_init(ptx::smem_addr(&ctl->d_ready[g]), 1);
    }
    ctl->abort = 0;
    ctl->past127 = 0;
    ptx::fence_mbar_init();
    ptx::tma_prefetch_desc(&map_x);
    ptx::tma_prefetch_desc(&map_w);
  }
  const uint32_t tmem_cols = (uint32_t)C::tmem_cols(zf);
  if (warp == 1) {
    ptx::tmem_alloc(ptx::smem_addr(&ctl->tmem_base), tmem_cols);
    ptx::tmem_relinquish();
  }
  if (zf) {
    for (int i = (int)threadIdx.x; i < C::kOnes / 16; i += kThreads)
      ptx::sts_128(ring_addr + ones_off + i * 16, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
    ptx::fence_proxy_async_smem();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = ctl->tmem_base;
  ptx::grid_dependents_launch();                           // once the columns are taken (see gemm.cu)
  ptx::cluster_arrive_relaxed();                           // waited for before the first store to another CTA
  ptx::grid_dependency_wait();

  float tot[C::kTn];
#pragma unroll
  for (int n = 0; n < C::kTn; ++n) tot[n] = 0.0f;

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (ptx::elect_one()) {
      const int nboxes = (nruns + kBoxRuns - 1) / kBoxRuns;
      int st = 0;
      uint32_t ph = 1u;
      for (int b = 0; b < nboxes; ++b) {
        if (!bounded_wait(ptx::smem_addr(&ctl->empty[st]), ph, abort_flag, WAIT_PRODUCER_EMPTY, 32)) break;
        ptx::fence_proxy_async_smem();                     // the row threads' reads of this stage before the copies' writes
        const uint32_t full = ptx::smem_addr(&ctl->full[st]), dst = ring_addr + st * C::kStage;
        const int run = run0 + b * kBoxRuns;
        ptx::mbar_expect_tx(full, C::kStage);              // what lies past the matrices is zero-filled and counted
        ptx::tma_load_2d(dst, &map_w, run * (16 * BITS), m0, full);
        ptx::tma_load_3d(dst + C::kCodes, &map_x, 0, t0, run * 2, full);
        if (++st == C::kStages) { st = 0; ph ^= 1u; }
      }
      if (*abort_flag) {                                   // outwait the copies in flight (microseconds)
        const uint64_t w0 = ptx::globaltimer_ns();
        while (ptx::globaltimer_ns() - w0 < 2000000ull) __nanosleep(1000);
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(C::kTn >> 3) << 17) | ((uint32_t)(kRows >> 4) << 24);
    int st = 0, g = 0;
    uint32_t ph = 0, aph = 0;
    for (int r = 0; r < nruns; ++r) {
      const int in_box = r & (kBoxRuns - 1);
      bool got = in_box != 0 || bounded_wait(ptx::smem_addr(&ctl->full[st]), ph, abort_flag, WAIT_MMA_FULL);
      if (got) got = bounded_wait(ptx::smem_addr(&ctl->a_full[g]), aph, abort_flag, WAIT_MMA_FULL);
      ptx::tc_fence_after();
      // With three groups of row threads the issue does not look at `got` either (2 % of 3-bit codes at 40 tokens: 13824 x 5120
      // 24.9 -> 24.5 us): after a wait that ran out it multiplies what is there, once, and nothing of it is stored.
      if (ptx::elect_one() && (kGroups > 2 || got)) {
        const uint32_t a = tmem + (uint32_t)(g * 64);
        const uint32_t d = tmem + (uint32_t)(C::kTmemA + g * ND * C::kTn);
        const uint64_t b = ptx::smem_desc(ring_addr + st * C::kStage + C::kCodes + in_box * 2 * C::kBlock);
        constexpr int kPer = 8 / ND;                       // instructions (16 columns each) per accumulator
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint32_t acc = (kk % kPer) != 0 ? 1u : 0u;
          const uint64_t bk = b + (uint64_t)((kk >> 2) * (C::kBlock >> 4) + (kk & 3) * 2);
          ptx::mma_bf16_ts(d + (uint32_t)((kk / kPer) * C::kTn), a + kk * 8, bk, idesc, acc);
          if (zf)                                          // rows of ones: the sums of the activations, in every lane
            ptx::mma_bf16_ss(d + (uint32_t)(C::kTmemD + (kk / kPer) * C::kTn), ptx::smem_desc(ring_addr + ones_off), bk, idesc, acc);
        }
        ptx::mma_commit(ptx::smem_addr(&ctl->d_ready[g]));
        if (in_box == kBoxRuns - 1) ptx::mma_commit(ptx::smem_addr(&ctl->empty[st]));
      }
      if (!__all_sync(0xFFFFFFFFu, got)) break;            // the warp gives up as a whole; off the path of the issue
      if (++g == kGroups) { g = 0; aph ^= 1u; }
      if (in_box == kBoxRuns - 1 && ++st == C::kStages) { st = 0; ph ^= 1u; }
    }
  } else {
    // ---------------------------------------------------------------- row threads
    const int g = (warp - 2) >> 2, quad = warp & 3;
    const int box_row = quad * 32 + lane;                  // the thread's row of the tile
    const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
    const uint32_t t_a = tmem + lane_base + (uint32_t)(g * 64);
    const uint32_t t_d = tmem + lane_base + (uint32_t)(C::kTmemA + g * ND * C::kTn);
    const Magics magics((uint32_t)p.split >> 30);          // split is at most kMaxSplit
    // Step sizes and zero points of the slice: word [group][row] = step size (fp16) | zero point << 16.  A warp reads
    // along the rows, a power of two of groups at a time; rows past the matrix are zeros, their sums are not stored.
    uint32_t* params = reinterpret_cast<uint32_t*>(ring + param_off);
    {
      // pairs of groups where the rows keep the alignment (always for groups of 32 and 64), single groups otherwise
      const bool pairs = ((ngroups | p.groups_per_row | group0) & 1) == 0;
      const int items = pairs ? ngroups >> 1 : ngroups;    // per row
      int k = 0;
      while (k < 5 && (1 << k) < items) ++k;
      const int rstep = 32 >> k, rows_live = min(kRows, p.out_features - m0);
      const int steps = ((kRows / rstep) + C::kRowWarps - 1) / C::kRowWarps;
      constexpr int kBatch = 8;                            // items in flight per lane
      uint32_t all_z = 0u;
      for (int c = lane & ((1 << k) - 1); c < items; c += 32) {
        for (int i0 = 0; i0 < steps; i0 += kBatch) {
          uint32_t vs[kBatch], vz[kBatch];
#pragma unroll
          for (int i = 0; i < kBatch; ++i) {
            const int rr = ((i0 + i) * C::kRowWarps + warp - 2) * rstep + (lane >> k);
            vs[i] = vz[i] = 0u;
            if (rr < rows_live) {
              const size_t gi = (size_t)(m0 + rr) * p.groups_per_row + group0 + (pairs ? 2 * c : c);
              const eqat_fp16* z16 = static_cast<const eqat_fp16*>(p.zq) + gi;
              const uint8_t* z8 = static_cast<const uint8_t*>(p.zq) + gi;
              if (pairs) {
                vs[i] = ptx::ld_global(reinterpret_cast<const uint32_t*>(p.s16 + gi));
                vz[i] = zf ? ptx::ld_global(reinterpret_cast<const uint32_t*>(z16)) : (uint32_t)ptx::ld_global(reinterpret_cast<const unsigned short*>(z8));
              } else {
                vs[i] = (uint32_t)ptx::ld_global(p.s16 + gi);
                vz[i] = zf ? (uint32_t)ptx::ld_global(z16) : (uint32_t)ptx::ld_global(z8);
              }
            }
          }
#pragma unroll
          for (int i = 0; i < kBatch; ++i) {
            const int rr = ((i0 + i) * C::kRowWarps + warp - 2) * rstep + (lane >> k);
            all_z |= vz[i];
            if (rr < kRows) {
              if (pairs) {
                const uint32_t z0 = zf ? vz[i] & 0xFFFFu : vz[i] & 0xFFu, z1 = zf ? vz[i] >> 16 : vz[i] >> 8;
                params[(2 * c) * kParamPitch + rr] = (vs[i] & 0xFFFFu) | (z0 << 16);
                params[(2 * c + 1) * kParamPitch + rr] = (vs[i] >> 16) | (z1 << 16);
              } else {
                params[c * kParamPitch + rr] = vs[i] | (vz[i] << 16);
              }
            }
          }
        }
      }
      if (!zf && (all_z & 0x8080u) != 0u) ctl->past127 = 1;
      __syncwarp();
      asm volatile("bar.sync 1, %0;" ::"n"(C::kRowWarps * 32) : "memory");
    }
    uint32_t ph = 0;
    float s_run[ND], sz_run[ND];                           // step sizes of the run in flight (and -s z, fp16 zero points)
    auto collect = [&]() -> bool {                         // adds the accumulators of the run in flight
      if (!bounded_wait_warp(ptx::smem_addr(&ctl->d_ready[g]), ph, abort_flag, WAIT_EPI_ACC_FULL)) return false;
      ph ^= 1u;
      ptx::tc_fence_after();
#pragma unroll
      for (int i = 0; i < ND; ++i) {
#pragma unroll
        for (int c = 0; c < NT; ++c) {
          uint32_t d[16];
          ptx::tmem_ld_32x16(t_d + (uint32_t)(i * C::kTn + c * 16), d);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int n = 0; n < 16; ++n) tot[c * 16 + n] = fmaf(s_run[i], __uint_as_float(d[n]), tot[c * 16 + n]);
          if (zf) {
            ptx::tmem_ld_32x16(t_d + (uint32_t)(C::kTmemD + i * C::kTn + c * 16), d);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int n = 0; n < 16; ++n) tot[c * 16 + n] = fmaf(sz_run[i], __uint_as_float(d[n]), tot[c * 16 + n]);
          }
        }
      }
      return true;
    };
    auto word_zero_point = [&](uint32_t v) {
      return zf ? __half2float(__ushort_as_half((unsigned short)(v >> 16))) : (float)(v >> 16);
    };
    // A run into the group's buffer.  PAST127: the zero point takes an addition of its own.
    auto expand_run = [&](const uint32_t (&w)[4 * BITS], const uint32_t (&gp)[ND], auto PAST127) {
      uint32_t a[32];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {                      // 32 codes: always inside one group
          const float z = zf ? 0.0f : word_zero_point(gp[(2 * h + q) * ND / 4]);
          const Offsets f(PAST127.value ? 0.0f : z);
          expand32<BITS>(w + (2 * h + q) * BITS, f, magics, a + 16 * q);
          if constexpr (PAST127.value) {
            const uint32_t nz = pack_bf16x2(-z, -z);
#pragma unroll
            for (int i = 0; i < 16; ++i) a[16 * q + i] = add_bf16x2(a[16 * q + i], nz);
          }
        }
        ptx::tmem_st_32x32(t_a + (uint32_t)(32 * h), a);
      }
    };
    const bool past127 = ctl->past127 != 0;
    bool ok = true;
    for (int r = g; r < nruns; r += kGroups) {
      const int box = r / kBoxRuns, st = box % C::kStages;
      // A wait by parity tells a phase from the one before it only.  With two groups every group has waited for every box.
      // With three a group skips boxes, and the box that used the stage last may be one of them: the group's run before is
      // collected first, since its MMAs come after those of that box.
      if (kGroups > 2 && r != g && !(ok = collect())) break;
      if (!bounded_wait_warp(ptx::smem_addr(&ctl->full[st]), (uint32_t)(box / C::kStages) & 1u, abort_flag, WAIT_STREAM_FULL)) {
        ok = false;
        break;
      }
      uint32_t w[4 * BITS], gp[ND];                        // codes of the run, parameters of its groups
      load_run<BITS>(ring_addr + st * C::kStage, box_row, r & (kBoxRuns - 1), w);
      const uint32_t* pw = params + ((((run0 + r) * kRun) >> p.group_shift) - group0) * kParamPitch + box_row;
#pragma unroll
      for (int i = 0; i < ND; ++i) gp[i] = pw[i * kParamPitch];
      ptx::fence_proxy_async_smem();                       // the codes are in registers
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&ctl->empty[st]));
      if (kGroups <= 2 && r != g && !(ok = collect())) break;   // the accumulators of the run before
      if (!past127) expand_run(w, gp, std::false_type{});
      else expand_run(w, gp, std::true_type{});
#pragma unroll
      for (int i = 0; i < ND; ++i) {
        s_run[i] = __half2float(__ushort_as_half((unsigned short)(gp[i] & 0xFFFFu)));
        sz_run[i] = -s_run[i] * word_zero_point(gp[i]);
      }
      ptx::tmem_st_wait();
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&ctl->a_full[g]));
    }
    if (ok && g < nruns) collect();
  }

  // ------------------------------------------------------------------ partial sums to the owners of the columns
  // CTA k of the cluster owns token columns [k, k + 1) * kTn / split of the tile.
  __syncwarp();
  ptx::cluster_wait();                                     // every CTA of the cluster has started
  const int slice = C::kTn >> p.split_log2;
  if (warp >= 2) {
    const int g = (warp - 2) >> 2, quad = warp & 3;
    const int src = rank * kGroups + g;                    // order of the final addition
    const uint32_t dst0 = ring_addr + part_off + (uint32_t)((src * slice * kRows + quad * 32 + lane) * 4);
    const int live = min(C::kTn, p.T - t0);
    int owner = 0, col = 0;
    uint32_t dst = ptx::map_to_cta(dst0, 0);
#pragma unroll
    for (int n = 0; n < C::kTn; ++n) {
      if (n < live) ptx::st_cluster_f32(dst + (uint32_t)(col * kRows * 4), tot[n]);
      if (++col == slice && n + 1 < C::kTn) { col = 0; ++owner; dst = ptx::map_to_cta(dst0, (uint32_t)owner); }
    }
  }
  __syncwarp();
  ptx::tc_fence_before();
  ptx::cluster_arrive();
  ptx::cluster_wait();
  if (!*abort_flag) {
    const int cols = min(slice, p.T - t0 - rank * slice), srcs = p.split * kGroups;
    const float4* part = reinterpret_cast<const float4*>(ring + part_off);
    for (int c = warp; c < cols; c += kThreads / 32) {
      float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      for (int s0 = 0; s0 < srcs; s0 += 2 * kGroups) {     // fixed order: deterministic
        float4 u[2 * kGroups];
#pragma unroll
        for (int i = 0; i < 2 * kGroups; ++i) {
          u[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          if (s0 + i < srcs) u[i] = part[((s0 + i) * slice + c) * 32 + lane];
        }
#pragma unroll
        for (int i = 0; i < 2 * kGroups; ++i) { v.x += u[i].x; v.y += u[i].y; v.z += u[i].z; v.w += u[i].w; }
      }
      if (m0 + 4 * lane < p.out_features)
        *reinterpret_cast<uint2*>(p.Y + (size_t)(t0 + rank * slice + c) * p.out_features + m0 + 4 * lane) =
            make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
    }
  }
  if (warp == 1) {
    if (*abort_flag) {                                     // outwait the MMAs in flight (microseconds)
      const uint64_t w0 = ptx::globaltimer_ns();
      while (ptx::globaltimer_ns() - w0 < 2000000ull) __nanosleep(1000);
    }
    __syncwarp();
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, tmem_cols);
  }
}

template <int BITS, int NT, int ND>
int launch_one(const SlimParams& p, const eqat_bf16* X, dim3 ctas, int groups, cudaStream_t st) {
  using C = Slim<BITS, NT, ND>;
  auto kern = slim_fwd_kernel<BITS, NT, ND>;
  static SmemOptIn opt_in;
  const bool zf = p.z_fp16 != 0;
  const int smem = C::smem_bytes(zf, groups);
  if (smem > kMaxSmem) return EQAT_ERR_UNSUPPORTED;        // not reached for a problem slim_fwd_applies() accepted
  if (!opt_in.ensure(kern, kMaxSmem)) return EQAT_ERR_CUDA;
  CUtensorMap mx, mw;
  if (!make_tmap_blocks_bf16(&mx, X, (uint64_t)p.in_features, (uint64_t)p.T, C::kTn, 2 * kBoxRuns)) return EQAT_ERR_CUDA;
  const uint64_t row_bytes = (uint64_t)p.in_features * BITS / 8;
  if (!make_tmap_u8(&mw, p.Wq, row_bytes, (uint64_t)p.out_features, box_bytes(BITS), kRows, BITS == 3 ? 0 : box_bytes(BITS)))
    return EQAT_ERR_CUDA;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = ctas;
  cfg.blockDim = dim3(C::kThreads, 1, 1);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  // Programmatic stream serialisation: the start-up of a launch overlaps the tail of the one before (see gemv.cu).
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = (unsigned)p.split;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, kern, mx, mw, p) != cudaSuccess) {
    (void)cudaGetLastError();
    return EQAT_ERR_CUDA;
  }
  return launch_status();
}

template <int BITS>
int smem_for(int nt, int nd, bool zf, int groups) {
  switch (nd * 8 + nt) {
    case 4 * 8 + 1: return Slim<BITS, 1, 4>::smem_bytes(zf, groups);
    case 2 * 8 + 1: return Slim<BITS, 1, 2>::smem_bytes(zf, groups);
    case 2 * 8 + 2: return Slim<BITS, 2, 2>::smem_bytes(zf, groups);
    case 2 * 8 + 3: return Slim<BITS, 3, 2>::smem_bytes(zf, groups);
    case 1 * 8 + 1: return Slim<BITS, 1, 1>::smem_bytes(zf, groups);
    case 1 * 8 + 2: return Slim<BITS, 2, 1>::smem_bytes(zf, groups);
    case 1 * 8 + 3: return Slim<BITS, 3, 1>::smem_bytes(zf, groups);
    default: return Slim<BITS, 4, 1>::smem_bytes(zf, groups);
  }
}

// The split of K (CTAs per cluster) with the least expected time.  The terms are fits to timings of every split on the
// 7B, 13B and 70B shapes, 2 to 4 bits (within 15 %): a CTA costs about 4 us
// outside its runs (start, exchange) and 0.06 us per group of parameters, a run 0.38 us alone on its SM and 0.34 us per
// SM where two CTAs share it (a quarter more with more than 16 token columns); behind the first two, a CTA's fixed part
// is mostly hidden by its neighbour's runs, and clusters of eight leave SMs of a GPC empty.
SlimPlan slim_plan(const eqat_desc& d, int sms) {
  SlimPlan best{};
  const bool zf = d.zero_point_format == EQAT_ZP_FP16;
  const int T = (int)d.tokens;
  if (sms <= 0) return best;
  const int nd = d.group == 32 ? 4 : (d.group == 64 ? 2 : 1);
  // 16-column accumulators that fit tensor memory beside the A operand (fp16 zero points need the column sums as well)
  const int cap = nd == 4 ? 1 : (nd == 2 ? (zf ? 2 : 3) : (zf ? 3 : 4));
  const int runs = d.in_features / kRun;
  const int boxes = (runs + kBoxRuns - 1) / kBoxRuns, shift = d.group <= 256 ? log2_exact(d.group) : 31;
  // The fewest token tiles that fit: a tile's parameters and partial sums share a CTA's shared memory, and on very long rows
  // (49152 columns, 3-bit codes, groups of 64, 40 tokens: 235 KB) only narrower tiles leave room for them.
  for (int token_tiles = (T + 16 * cap - 1) / (16 * cap); best.us == 0.0 && token_tiles <= (T + 15) / 16; ++token_tiles) {
    const int nt = ((T + token_tiles - 1) / token_tiles + 15) / 16;
    const int tiles = ((d.out_features + kRows - 1) / kRows) * token_tiles;
    for (int lg = 0; (1 << lg) <= kMaxSplit && (1 << lg) <= boxes; ++lg) {
      const int split = 1 << lg;
      // the longest slice, and the groups it touches (it starts at a multiple of 256 columns)
      const int most = min(runs, ((boxes + split - 1) >> lg) * kBoxRuns);
      const int groups = ((most * kRun - 1) >> shift) + 1;
      const int smem = d.bits == 2   ? smem_for<2>(nt, nd, zf, groups)
                       : d.bits == 3 ? smem_for<3>(nt, nd, zf, groups)
                                     : smem_for<4>(nt, nd, zf, groups);
      if (smem > kMaxSmem) continue;
      const bool two = nt <= 2 && smem <= 113 * 1024;
      const int n = (tiles * split + sms - 1) / sms;         // CTAs of the busiest SM
      const double wide = nt == 1 ? 1.0 : 1.25, fixed = 4.0 + 0.06 * groups;
      double us = two ? fixed + n * most * (n == 1 ? 0.38 : 0.34) * wide + (n > 2 ? (n - 2) * 0.7 : 0.0)
                      : n * (fixed + most * 0.36 * wide);
      // Two CTAs share an SM, so the last of an odd number runs by itself: a fixed part more where most SMs have it (three on
      // 136 of 148 SMs, 13824 x 5120: estimated 15.5 without it, 19.8 with it, measured 21.5 us).  Where few have it the
      // next launch fills in (12288 x 6144, 88 SMs: 17.7 us without, measured 19.5 us).
      const int last = (tiles * split) % sms;
      if (two && n > 2 && (n & 1) != 0 && 5 * last > 3 * sms) us += fixed * last / sms;
      if (split == 8 && n > 2) us *= 1.15;
      if (best.us == 0.0 || us < best.us) best = SlimPlan{nt, nd, token_tiles, split, groups, us};
    }
  }
  return best;
}

template <int BITS>
int launch_bits(const SlimPlan& pl, const SlimParams& p, const eqat_bf16* X, dim3 ctas, cudaStream_t st) {
  switch (pl.nd * 8 + pl.nt) {
    case 4 * 8 + 1: return launch_one<BITS, 1, 4>(p, X, ctas, pl.groups, st);
    case 2 * 8 + 1: return launch_one<BITS, 1, 2>(p, X, ctas, pl.groups, st);
    case 2 * 8 + 2: return launch_one<BITS, 2, 2>(p, X, ctas, pl.groups, st);
    case 2 * 8 + 3: return launch_one<BITS, 3, 2>(p, X, ctas, pl.groups, st);
    case 1 * 8 + 1: return launch_one<BITS, 1, 1>(p, X, ctas, pl.groups, st);
    case 1 * 8 + 2: return launch_one<BITS, 2, 1>(p, X, ctas, pl.groups, st);
    case 1 * 8 + 3: return launch_one<BITS, 3, 1>(p, X, ctas, pl.groups, st);
    default: return launch_one<BITS, 4, 1>(p, X, ctas, pl.groups, st);
  }
}

}  // namespace

// Which kernel takes few tokens.  The matrix-vector kernel streams the weight with less start-up (5.1 against 6.8 us for
// one token of 4096 x 4096, 2-bit codes) but pays for every token and holds at most eight; this one costs the same for
// any number up to 16 (7.1 us against 10.0 us at 8 tokens, 19.8 us in two launches at 16).  Two estimates are compared,
// so this one has to be a quarter better (11008 x 4096, 4-bit codes, 8 tokens: estimated 13.3 against 15.0 us, measured
// 14.8 against 15.1 us).  Small weights keep the matrix-vector kernel for the sake of their bits (packed_gemv_keeps_bits).
bool slim_fwd_applies(const eqat_desc& d, int sms, SlimPlan& pl) {
  if (d.tokens > kSlimMaxTokens) return false;
  const FewTokenPlan gemv = packed_gemv_plan(d);
  if (gemv.launches == 1 && d.tokens <= 2) return false;   // the matrix-vector kernel on every shape measured
  if (packed_gemv_keeps_bits(d)) return false;
  pl = slim_plan(d, sms);
  if (pl.us == 0.0) return false;
  if (!packed_gemv_applies(d)) return true;
  return gemv.launches > 1 || pl.us * 1.25 < gemv.us;
}

int launch_slim_fwd(const eqat_desc& d, const eqat_bf16* X, const uint8_t* Wq, const eqat_fp16* s16, const void* zq,
                    eqat_bf16* Y, const SlimPlan& pl, cudaStream_t st) {
  SlimParams p{};
  set_weight(p, d, Wq, s16, zq);
  p.Y = Y;
  p.T = (int)d.tokens;
  p.split = pl.split;
  p.split_log2 = log2_exact(pl.split);
  p.runs = d.in_features / kRun;
  const dim3 ctas((unsigned)((d.out_features + kRows - 1) / kRows), (unsigned)pl.split, (unsigned)pl.token_tiles);
  switch (d.bits) {
    case 2: return launch_bits<2>(pl, p, X, ctas, st);
    case 3: return launch_bits<3>(pl, p, X, ctas, st);
    default: return launch_bits<4>(pl, p, X, ctas, st);
  }
}

int launch_wait_expiry_slim(cudaStream_t st) { return launch_wait_expiry(st); }
int read_slim_status(int* status, int* detail) { return read_wait_status(status, detail); }

}  // namespace eqat

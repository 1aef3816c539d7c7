// Packed-weight forward for more than a few tokens (prompts, large decoding batches),
//     Y[T,out] = X[T,in] * dequant(Wq)^T,
// on tiles of 256 WEIGHT rows x up to 256 tokens, computed by a pair of CTAs that share one MMA (tcgen05 cta_group::2).
//
// As in slim.cu the weight is the M side and its rows live in TENSOR MEMORY: lane = weight row, the thread that owns a
// row expands its codes in registers ((q - z) * s, rounded once to bf16) and writes them with tcgen05.st; no expanded
// operand passes through shared memory.  Here the accumulators stay in tensor memory over the whole of K.  Each CTA of
// a pair holds its own 128 rows and half of the tokens' activations; the tensor cores exchange the halves, so a tile
// costs half the activation traffic of two single CTAs, which L2 could not deliver.
//
// K is split over the pairs of a cluster where the tiles alone do not fill the chip; the partial sums meet in the shared
// memory of the CTA that owns a token column and are added in a fixed order (run-to-run identical, no scratch memory).
//
// Roles (18 warps, one CTA per SM): warp 0 TMA producer, warp 1 MMA issuer (first CTA of the pair) and TMEM owner, four
// groups of 128 row threads.  A run = 128 codes of a row; group g takes the runs g, g + 4, ... of the CTA's K slice.
#include <cuda.h>

#include "common.cuh"
#include "expand.cuh"
#include "gemm.cuh"
#include "ptx.cuh"
#include "wide.cuh"
#include "wait.cuh"

namespace eqat {
namespace {

constexpr int kRows = 128;             // weight rows per CTA = TMEM lanes
constexpr int kRun = 128;              // codes of a row per run
constexpr int kGroups = 4;             // groups of 128 row threads
constexpr int kThreads = (2 + 4 * kGroups) * 32;
constexpr int kMaxTn = 256;
constexpr int kTmemA = kGroups * 64;   // columns of the A operand; the accumulators follow
constexpr int kMaxSmem = 232448;

struct WideParams : PackedWeight {
  eqat_bf16* Y;                        // [T, out]
  int T, tn;                           // tokens, tokens per tile (a multiple of 32)
  int split, split_log2, runs;         // runs = in_features / 128
  int stages;
  int tile0;                           // first row tile of the launch (an even number)
};

struct WideCtl {
  uint64_t full_x[8];                  // activations of a run landed                (pair: first CTA's)
  uint64_t full_c[8];                  // its codes landed                           (each CTA its own)
  uint64_t empty[8];                   // codes read and MMAs done: stage and, with it, the run's TMEM buffer free (each CTA its own)
  uint64_t a_full[kGroups];            // a run's rows are in tensor memory          (pair: first CTA's)
  uint64_t acc_full;                   //                                            (each CTA its own)
  uint32_t tmem_base;
  int abort;
};

__host__ __device__ constexpr int code_bytes(int bits) { return 16 * bits; }             // of a row per run
__host__ __device__ inline int stage_bytes(int bits, int tn) { return kRows * code_bytes(bits) + tn * 128; }

// The 128 codes of box row `row`: rows of 32, 48 or 64 bytes; 16-byte piece c of row r sits at piece c ^ ((r >> 2) & 1)
// of 32-byte rows, c ^ ((r >> 1) & 3) of 64-byte rows (the copy engine's swizzles); 48-byte rows need none.
template <int BITS>
__device__ __forceinline__ void load_run(uint32_t box, int row, uint32_t (&w)[4 * BITS]) {
  const uint32_t sx = BITS == 4 ? (uint32_t)((row >> 1) & 3) : (BITS == 2 ? (uint32_t)((row >> 2) & 1) : 0u);
#pragma unroll
  for (int i = 0; i < BITS; ++i) {
    const uint4 t = ptx::lds_128(box + (uint32_t)(row * code_bytes(BITS)) + (((uint32_t)i ^ sx) << 4));
    w[4 * i] = t.x; w[4 * i + 1] = t.y; w[4 * i + 2] = t.z; w[4 * i + 3] = t.w;
  }
}

template <int BITS>
__global__ void __launch_bounds__(kThreads, 1)
wide_fwd_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, const WideParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = ptx::smem_addr(smem_raw);
  const uint32_t ring_addr = (raw_addr + 1023u) & ~1023u;
  uint8_t* ring = smem_raw + (ring_addr - raw_addr);
  const int stage_size = stage_bytes(BITS, p.tn), stages = p.stages;
  constexpr int kCodes = kRows * code_bytes(BITS);
  WideCtl* ctl = reinterpret_cast<WideCtl*>(ring + stages * stage_size);
  volatile int* abort_flag = &ctl->abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // grid: row tiles (an even number) x pairs of a cluster x token tiles; cluster = 2 row tiles x split
  const int half = (int)(blockIdx.x & 1u), ks = (int)blockIdx.y;
  const int m0 = (p.tile0 + (int)blockIdx.x) * kRows, t0 = (int)blockIdx.z * p.tn;
  const int run0 = (p.runs * ks) >> p.split_log2, nruns = ((p.runs * (ks + 1)) >> p.split_log2) - run0;
  // barriers that both CTAs of a pair signal live in its first CTA
  auto lead = [&](const void* bar) { return ptx::map_to_cta(ptx::smem_addr(bar), (uint32_t)(2 * ks)); };

  if (warp == 0 && m0 < p.out_features && ptx::elect_one()) {   // into L2 before the wait for the launches before this one
    for (int r = 0; r < nruns; ++r) ptx::tma_prefetch_2d(&map_w, (run0 + r) * code_bytes(BITS), m0);
  }
  if (threadIdx.x == 64) {
    for (int s = 0; s < stages; ++s) {
      ptx::mbar_init(ptx::smem_addr(&ctl->full_x[s]), 2);
      ptx::mbar_init(ptx::smem_addr(&ctl->full_c[s]), 1);
      ptx::mbar_init(ptx::smem_addr(&ctl->empty[s]), 4 + 1);
    }
    for (int g = 0; g < kGroups; ++g) ptx::mbar_init(ptx::smem_addr(&ctl->a_full[g]), 8);
    ptx::mbar_init(ptx::smem_addr(&ctl->acc_full), 1);
    ctl->abort = 0;
    ptx::fence_mbar_init();
    ptx::tma_prefetch_desc(&map_x);
  }
  __syncthreads();
  ptx::cluster_arrive();
  ptx::grid_dependency_wait();
  ptx::cluster_wait();                                     // the other CTAs run, and their barriers exist, from here on
  // an operation of the pair: not before the other CTA is known to run
  if (warp == 1) {
    ptx::tmem_alloc_pair(ptx::smem_addr(&ctl->tmem_base), 512);
    ptx::tmem_relinquish_pair();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = ctl->tmem_base;
  ptx::grid_dependents_launch();                           // once the columns are taken (see gemm.cu)

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (ptx::elect_one()) {
      int st = 0;
      uint32_t ph = 1u;
      for (int r = 0; r < nruns; ++r) {
        if (!bounded_wait(ptx::smem_addr(&ctl->empty[st]), ph, abort_flag, WAIT_PRODUCER_EMPTY, 32)) break;
        ptx::fence_proxy_async_smem();                     // the row threads' reads of this stage before the copies' writes
        const uint32_t dst = ring_addr + st * stage_size, full_c = ptx::smem_addr(&ctl->full_c[st]);
        const uint32_t full_x = lead(&ctl->full_x[st]);
        ptx::mbar_expect_tx(full_c, kCodes);               // what lies past the matrices is zero-filled and counted
        ptx::tma_load_2d(dst + p.tn * 128, &map_w, (run0 + r) * code_bytes(BITS), m0, full_c);
        ptx::mbar_expect_tx_cluster(full_x, (uint32_t)p.tn * 128);
        ptx::tma_load_3d_pair(dst, &map_x, 0, t0 + half * (p.tn >> 1), (run0 + r) * 2, full_x);
        if (++st == stages) { st = 0; ph ^= 1u; }
      }
      if (*abort_flag) {                                   // outwait the copies in flight (microseconds)
        const uint64_t w0 = ptx::globaltimer_ns();
        while (ptx::globaltimer_ns() - w0 < 2000000ull) __nanosleep(1000);
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (half == 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.tn >> 3) << 17) | ((uint32_t)((2 * kRows) >> 4) << 24);
      const uint16_t both = (uint16_t)(3u << (2 * ks));    // the pair's CTAs of the cluster
      int st = 0, g = 0;
      uint32_t ph = 0, aph = 0;
      bool ok = true;
      for (int r = 0; r < nruns; ++r) {
        bool got = bounded_wait(ptx::smem_addr(&ctl->full_x[st]), ph, abort_flag, WAIT_MMA_FULL);
        if (got) got = bounded_wait(ptx::smem_addr(&ctl->a_full[g]), aph, abort_flag, WAIT_MMA_FULL);
        ptx::tc_fence_after();
        if (ptx::elect_one() && got) {
          const uint32_t a = tmem + (uint32_t)(g * 64);
          const uint64_t b = ptx::smem_desc(ring_addr + st * stage_size);
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)                   // a K block's activations of this CTA: tn/2 rows of 128 bytes
            ptx::mma_bf16_ts_pair(tmem + kTmemA, a + kk * 8, b + (uint64_t)((kk >> 2) * (p.tn * 4) + (kk & 3) * 2), idesc,
                                  (r | kk) != 0 ? 1u : 0u);
          ptx::mma_commit_pair_mask(ptx::smem_addr(&ctl->empty[st]), both);
        }
        ok = __all_sync(0xFFFFFFFFu, got);                 // the warp gives up as a whole; off the path of the issue
        if (!ok) break;
        if (++g == kGroups) { g = 0; aph ^= 1u; }
        if (++st == stages) { st = 0; ph ^= 1u; }
      }
      if (ok && ptx::elect_one()) ptx::mma_commit_pair_mask(ptx::smem_addr(&ctl->acc_full), both);
      __syncwarp();
    }
  } else {
    // ---------------------------------------------------------------- row threads
    const int g = (warp - 2) >> 2, quad = warp & 3;
    const int box_row = quad * 32 + lane, row = m0 + box_row;
    const bool valid = row < p.out_features;               // uniform over a warp: out_features is a multiple of 64
    const uint32_t t_a = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(g * 64);
    const size_t g_row = (size_t)(valid ? row : 0) * p.groups_per_row;
    const int g_count = max(1, kRun >> min(p.group_shift, 30));       // 1, 2 or 4
    const uint32_t a_full = lead(&ctl->a_full[g]);
    GroupParamsRaw gp;
    gp.s = gp.z = make_uint2(0u, 0u);
    auto fetch = [&](int r) { load_group_params(p, g_row + (size_t)(((run0 + r) * kRun) >> p.group_shift), g_count, gp); };
    if (g < nruns) fetch(g);
    for (int r = g; r < nruns; r += kGroups) {
      // First the group's run before has to have left its TMEM buffer, i.e. its stage is empty: its MMAs, and with them those
      // of every run before it, are done.  The order matters for the wait after it too.  A wait by parity tells a phase
      // from the one before it only: the run that used stage `st` last belongs to another group, and if its codes were
      // still on their way the wait for this run's would pass at once.  There are at least as many stages as groups, so
      // that run is not after the group's run before, whose MMAs are done.
      if (r != g) {
        const int before = r - kGroups;
        if (!bounded_wait_warp(ptx::smem_addr(&ctl->empty[before % stages]), (uint32_t)(before / stages) & 1u, abort_flag,
                               WAIT_DEQ_OPERAND_EMPTY))
          break;
        ptx::tc_fence_after();
      }
      const int st = r % stages;
      if (!bounded_wait_warp(ptx::smem_addr(&ctl->full_c[st]), (uint32_t)(r / stages) & 1u, abort_flag, WAIT_STREAM_FULL)) break;
      uint32_t w[4 * BITS];
      load_run<BITS>(ring_addr + st * stage_size + p.tn * 128, box_row, w);
      ptx::fence_proxy_async_smem();                       // the codes are in registers
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&ctl->empty[st]));
      GroupValues<BITS> gv[4];                             // of the run's four runs of 32 codes
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = g_count == 4 ? q : (g_count == 2 ? q >> 1 : 0);
        if (q == 0 || g_count == 4 || (g_count == 2 && q == 2))
          gv[q] = GroupValues<BITS>(step_size_at(gp, i), zero_point_at(gp, i, p.z_fp16));
        else
          gv[q] = gv[q - 1];
      }
      if (r + kGroups < nruns) fetch(r + kGroups);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t a[32];
        values32<BITS>(w + (2 * h) * BITS, gv[2 * h], a);
        values32<BITS>(w + (2 * h + 1) * BITS, gv[2 * h + 1], a + 16);
        ptx::tmem_st_32x32(t_a + (uint32_t)(32 * h), a);
      }
      ptx::tmem_st_wait();
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive_cluster(a_full);
    }
  }

  // ------------------------------------------------------------------ partial sums to the owners of the columns
  // CTA ks of a row tile owns token columns [ks, ks + 1) * tn / split of the tile.  The ring is free once every CTA's
  // MMAs are done: the sums go over it, [source][column / 4][row][column % 4] fp32.
  __syncwarp();
  const bool all_done = bounded_wait_warp(ptx::smem_addr(&ctl->acc_full), 0u, abort_flag, WAIT_EPI_ACC_FULL, 64);
  ptx::tc_fence_after();
  ptx::cluster_arrive();
  ptx::cluster_wait();
  const int slice = p.tn >> p.split_log2;
  if (warp >= 2 && all_done) {
    const int g = (warp - 2) >> 2, quad = warp & 3;
    const uint32_t t_d = tmem + ((uint32_t)(quad * 32) << 16) + kTmemA;
    const int c_end = (g + 1) * (p.tn / kGroups);
    for (int c = g * (p.tn / kGroups); c < c_end && t0 + c < p.T; c += 8) {      // slice is a multiple of 8
      uint32_t d[8];
      ptx::tmem_ld_32x8(t_d + (uint32_t)c, d);
      int owner = 0, col = c;
      while (col >= slice) { col -= slice; ++owner; }
      const uint32_t local = ring_addr + (uint32_t)(((ks * slice + col) * kRows + (quad * 32 + lane) * 4) * 4);
      ptx::tmem_ld_wait();
      if (owner == ks) {
#pragma unroll
        for (int j = 0; j < 2; ++j) ptx::sts_128(local + (uint32_t)(j * kRows * 16), d[4 * j], d[4 * j + 1], d[4 * j + 2], d[4 * j + 3]);
      } else {
        const uint32_t dst = ptx::map_to_cta(local, (uint32_t)(2 * owner + half));
#pragma unroll
        for (int j = 0; j < 2; ++j) ptx::st_cluster_128(dst + (uint32_t)(j * kRows * 16), d[4 * j], d[4 * j + 1], d[4 * j + 2], d[4 * j + 3]);
      }
    }
  }
  __syncwarp();
  ptx::tc_fence_before();
  ptx::cluster_arrive();
  ptx::cluster_wait();
  // Tensor memory goes back here, where both CTAs of a pair stand, and no CTA leaves before all have given theirs back (the
  // wait at the end): the release is an operation of the pair, and an SM whose CTA is gone may already hold a CTA of the
  // next cluster or launch, with columns of its own.
  if (warp == 1) {
    if (*abort_flag) {                                     // outwait the MMAs in flight (microseconds)
      const uint64_t w0 = ptx::globaltimer_ns();
      while (ptx::globaltimer_ns() - w0 < 2000000ull) __nanosleep(1000);
    }
    __syncwarp();
    ptx::tc_fence_after();
    ptx::tmem_dealloc_pair(tmem, 512);
  }
  __syncwarp();
  ptx::cluster_arrive_relaxed();
  if (!*abort_flag) {
    // a lane sums four columns of two neighbouring rows; a warp stores 128 bytes of each column
    const int cols = min(slice, p.T - t0 - ks * slice);
    const float4* part = reinterpret_cast<const float4*>(ring);
    for (int i = warp; i < (slice >> 2) * 2; i += kThreads / 32) {
      const int cg = i >> 1, row2 = (i & 1) * 64 + 2 * lane;
      if (4 * cg >= cols) break;
      float4 v[2] = {part[cg * kRows + row2], part[cg * kRows + row2 + 1]};
      for (int s = 1; s < p.split; ++s) {                  // fixed order: deterministic
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float4 u = part[(s * (slice >> 2) + cg) * kRows + row2 + j];
          v[j].x += u.x; v[j].y += u.y; v[j].z += u.z; v[j].w += u.w;
        }
      }
      if (m0 + row2 < p.out_features) {
        const uint32_t o[4] = {pack_bf16x2(v[0].x, v[1].x), pack_bf16x2(v[0].y, v[1].y), pack_bf16x2(v[0].z, v[1].z),
                               pack_bf16x2(v[0].w, v[1].w)};
        eqat_bf16* y = p.Y + (size_t)(t0 + ks * slice + 4 * cg) * p.out_features + m0 + row2;
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (4 * cg + c < cols) *reinterpret_cast<uint32_t*>(y + (size_t)c * p.out_features) = o[c];
      }
    }
  }
  __syncwarp();
  ptx::cluster_wait();
}

int stages_that_fit(int bits, int tn) {                    // at least five (256 tokens, 4-bit codes)
  int s = (kMaxSmem - 1024 - (int)sizeof(WideCtl)) / stage_bytes(bits, tn);
  return s < 8 ? s : 8;
}

constexpr int kMaxSplit = 4;           // pairs per cluster: eight CTAs, the portable limit
// Clusters of two, four and eight CTAs that a B200 of 148 SMs kept resident, for plans made without a device.
constexpr int kResidentOf148[3] = {74, 32, 13};

template <int BITS>
bool opted_in() {
  static SmemOptIn opt_in;
  return opt_in.ensure(wide_fwd_kernel<BITS>, kMaxSmem);
}

void set_launch(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[2], dim3 ctas, int split, cudaStream_t st) {
  cfg.gridDim = ctas;
  cfg.blockDim = dim3(kThreads, 1, 1);
  // All of tensor memory and, so that no other kernel of this library that wants some shares the SM, all of shared
  // memory: a CTA never waits for columns (see slim.cu).
  cfg.dynamicSmemBytes = kMaxSmem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = (unsigned)split;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
}

// Clusters of 2 << lg CTAs that are resident at a time (asked of the runtime once per device; SMs of a GPC that do not
// make up a whole cluster stay empty).  0 on error.
int max_clusters(int bits, int lg) {
  static std::atomic<int> cache[kMaxCachedDevices][3];
  const int dev = current_device();
  if (dev < 0) return 0;
  if (dev < kMaxCachedDevices) {
    const int c = cache[dev][lg].load(std::memory_order_relaxed);
    if (c > 0) return c;
  }
  if (!(bits == 2 ? opted_in<2>() : (bits == 3 ? opted_in<3>() : opted_in<4>()))) return 0;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[2];
  set_launch(cfg, attr, dim3(2u, 1u << lg, 1u), 1 << lg, nullptr);
  cfg.numAttrs = 1;
  int n = 0;
  const cudaError_t e = bits == 2   ? cudaOccupancyMaxActiveClusters(&n, wide_fwd_kernel<2>, &cfg)
                        : bits == 3 ? cudaOccupancyMaxActiveClusters(&n, wide_fwd_kernel<3>, &cfg)
                                    : cudaOccupancyMaxActiveClusters(&n, wide_fwd_kernel<4>, &cfg);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  if (dev < kMaxCachedDevices) cache[dev][lg].store(n, std::memory_order_relaxed);
  return n;
}

template <int BITS>
int launch_bits(const WideParams& p, const eqat_bf16* X, dim3 ctas, cudaStream_t st) {
  auto kern = wide_fwd_kernel<BITS>;
  if (!opted_in<BITS>()) return EQAT_ERR_CUDA;
  CUtensorMap mx, mw;
  if (!make_tmap_blocks_bf16(&mx, X, (uint64_t)p.in_features, (uint64_t)p.T, (uint32_t)p.tn / 2, 2)) return EQAT_ERR_CUDA;
  if (!make_tmap_u8(&mw, p.Wq, (uint64_t)p.in_features * BITS / 8, (uint64_t)p.out_features, code_bytes(BITS), kRows,
                    BITS == 3 ? 0 : code_bytes(BITS)))
    return EQAT_ERR_CUDA;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[2];
  set_launch(cfg, attr, ctas, p.split, st);
  if (cudaLaunchKernelEx(&cfg, kern, mx, mw, p) != cudaSuccess) {
    (void)cudaGetLastError();
    return EQAT_ERR_CUDA;
  }
  return launch_status();
}

int launch_rows(WideParams& p, int bits, const eqat_bf16* X, int pairs, int split, int token_tiles, cudaStream_t st) {
  p.split = split;
  p.split_log2 = log2_exact(split);
  const dim3 ctas((unsigned)pairs * 2u, (unsigned)split, (unsigned)token_tiles);
  switch (bits) {
    case 2: return launch_bits<2>(p, X, ctas, st);
    case 3: return launch_bits<3>(p, X, ctas, st);
    default: return launch_bits<4>(p, X, ctas, st);
  }
}

}  // namespace

// Whether this kernel is expected to beat the tiled kernel of gemm.cu (512 or 256 TOKENS x 256 weight rows per tile, or 128 x
// 128 where all of those fit the chip at once), and with which token tiles and split of K.  The terms are fits to timings on
// the 7B, 13B and 70B shapes from 65 to 2048 tokens (within 15 %).  Here: a CTA costs 5 us plus 0.018 us per token column
// outside its runs, a run 0.41 / 0.62 / 0.41 us (2 / 3 / 4-bit codes: its expansion) or 0.0021 us per token column (its MMAs),
// a quarter more when most SMs are loading.  There: 8 us and 0.65 / 0.72 / 0.67 us per tile and 64 input columns, a tenth more
// with most SMs at work, or, for at most 256 tokens, 0.88 / 1.13 / 1.15 us on one CTA.  4096 x 4096, 2 bits: 128 tokens 64.2 ->
// 13.2 us, 333 tokens 49.4 -> 16.2 us, 1024 tokens 49.8 -> 29 us; at 2048 tokens the tiled kernel is ahead (51 against 58 us).
// Tiles of 128 x 128 take 3.6 us and 0.42 / 0.49 / 0.47 us per 64 input columns; the line that picks the faster kernel is a
// little above that, because the estimate here is 10 to 15 % high for problems of that size.  Over 1024 of them (65 to 4096
// tokens, 128 to 16384 columns) the kernel picked takes 0.13 % more than the faster one; by the price of 256-column tiles,
// 2.7 % (1022 tokens of 64 x 128, 3 bits: 5.8 against 3.8 us; 1536 of 1536 x 512, 2 bits: 9.0 against 8.0 us).
bool wide_fwd_applies(const eqat_desc& d, int given_sms, WidePlan& best) {
  best = WidePlan{};
  const int sms = given_sms > 0 ? given_sms : sm_count();
  if (d.tokens > 4096 || sms < 2) return false;
  const int T = (int)d.tokens, runs = d.in_features / kRun, pairs = (d.out_features + 2 * kRows - 1) / (2 * kRows);
  const int least = (T + kMaxTn - 1) / kMaxTn;
  auto resident = [&](int lg) { return given_sms > 0 ? sms * kResidentOf148[lg] / 148 : max_clusters(d.bits, lg); };
  auto columns = [&](int tt) { return ((T + tt - 1) / tt + 31) / 32 * 32; };                // of each of tt token tiles
  auto round_us = [&](int tn, int lg, int clusters) {        // of clusters that are resident together
    const double expand = d.bits == 3 ? 0.62 : 0.41, mma = 0.0021 * tn;
    const double load = (clusters << lg) * 2 > 100 ? 1.25 : 1.0;
    return 5.0 + 0.018 * tn + ((runs + (1 << lg) - 1) >> lg) * (expand > mma ? expand : mma) * load;
  };
  const int splits = runs >= kMaxSplit ? 3 : (runs >= 2 ? 2 : 1);
  static_assert(kMaxSplit == 4, "splits of 1, 2 and 4");
  for (int tt = least; tt <= least + 3; ++tt) {
    const int tn = columns(tt);
    for (int lg = 0; lg < splits; ++lg) {
      const int clusters = pairs * tt, fit = resident(lg);
      if (fit <= 0) continue;
      const double us = (clusters + fit - 1) / fit * round_us(tn, lg, clusters);
      if (best.us == 0.0 || us < best.us) best = WidePlan{tn, (T + tn - 1) / tn, 1 << lg, pairs, 1, us};
    }
  }
  if (best.us == 0.0) return false;
  // The whole rounds as they are, and what is left over split finer: 11008 x 4096, 2 bits, 333 tokens has 86 clusters of
  // which 74 are resident, 50.0 us in two rounds (or tiled), 38.5 us with the last twelve split four ways; 28672 x 8192,
  // 4 bits, 333 tokens 174.2 -> 157.1 us, 4096 x 11008, 4 bits, 1531 tokens 122.2 -> 112.0 us.  Not on narrower token tiles
  // than one launch would take: more tiles expand the weight more often, which costs more than the estimate says (22976 x
  // 25216, 4 bits, 949 tokens: 969 us in one launch on four token tiles, 1082 us in two on five).  Of 2045 problems of 65 to
  // 4096 tokens 37 take more than 3 % longer than by a rule that knows one launch only, with the narrower tiles 76; all of
  // them together take 0.886 of the time.
  for (int tt = least, least_tn = best.tn; tt <= least + 3; ++tt) {
    const int tn = columns(tt);
    if (tn < least_tn) break;
    for (int lg = 0; lg < splits; ++lg) {
      const int clusters = pairs * tt, fit = resident(lg);
      if (fit <= 0) continue;
      const int whole = clusters / fit * fit / tt;           // pairs of row tiles, with all their token tiles
      for (int lg2 = lg + 1; whole > 0 && whole < pairs && lg2 < splits; ++lg2) {
        const int rest = (pairs - whole) * tt, fit2 = resident(lg2);
        if (fit2 <= 0) continue;
        const double two = clusters / fit * round_us(tn, lg, clusters) + (rest + fit2 - 1) / fit2 * round_us(tn, lg2, rest);
        if (two < best.us) best = WidePlan{tn, (T + tn - 1) / tn, 1 << lg, whole, 1 << lg2, two};
      }
    }
  }
  const int cols = (d.out_features + 255) / 256, kb = d.in_features / 64;
  double tiled;
  if (packed_shape(T, d.out_features, sms).bn == 128)
    return best.us < 5.0 + kb * (d.bits == 2 ? 0.48 : (d.bits == 3 ? 0.58 : 0.52));
  if (T <= 256) {
    tiled = 8.0 + ((cols + sms - 1) / sms) * kb * (d.bits == 2 ? 0.88 : (d.bits == 3 ? 1.13 : 1.15));
  } else {
    const int tiles = cols * ((T + 511) / 512), slots = sms / 2;
    tiled = 8.0 + ((tiles + slots - 1) / slots) * kb * (d.bits == 2 ? 0.65 : (d.bits == 3 ? 0.72 : 0.67)) *
                      (tiles * 5 > slots * 4 ? 1.1 : 1.0);
  }
  // With 4-bit codes this kernel takes 15 % more than its estimate on average, the tiled one 2 %, over 300 calls of 300 to
  // 4096 tokens (8192 x 28672, 2048 tokens: estimated 616 against 668 us, measured 910 against 760 us).
  return best.us * (d.bits == 4 ? 1.08 : 1.0) < 0.95 * tiled;
}

int launch_wide_fwd(const eqat_desc& d, const eqat_bf16* X, const uint8_t* Wq, const eqat_fp16* s16, const void* zq,
                    eqat_bf16* Y, const WidePlan& pl, cudaStream_t st) {
  WideParams p{};
  set_weight(p, d, Wq, s16, zq);
  p.Y = Y;
  p.T = (int)d.tokens;
  p.tn = pl.tn;
  p.runs = d.in_features / kRun;
  p.stages = stages_that_fit(d.bits, pl.tn);
  const int pairs = (d.out_features + 2 * kRows - 1) / (2 * kRows);
  int rc = launch_rows(p, d.bits, X, pl.first_pairs, pl.split, pl.token_tiles, st);
  if (rc == EQAT_OK && pl.first_pairs < pairs) {
    p.tile0 = 2 * pl.first_pairs;
    rc = launch_rows(p, d.bits, X, pairs - pl.first_pairs, pl.rest_split, pl.token_tiles, st);
  }
  return rc;
}

int launch_wait_expiry_wide(cudaStream_t st) { return launch_wait_expiry(st); }
int read_wide_status(int* status, int* detail) { return read_wait_status(status, detail); }

}  // namespace eqat

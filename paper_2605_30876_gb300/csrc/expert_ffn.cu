// Expert execution of the MoE layer: grouped SwiGLU FFN over the unique experts of one
// forward (plus the shared expert), on tcgen05 tensor cores.
//
// Both GEMMs are "swap-AB": the expert weights are the MMA's M operand (streamed by TMA with
// the 128-byte swizzle), the tokens routed to an expert are the N operand, K is the reduction
// dimension, and the fp32 accumulator lives in TMEM. Two CTAs on neighbouring SMs (a cluster
// of two) share every MMA (cta_group::2, M = 256): each brings its own 128 weight rows and
// half of the token rows, so that a 128 x 256 x 64 step of one SM takes 32 KB from L2 instead
// of 48 KB. What one SM can pull from L2 bounds this launch once an expert has many tokens.
//
//   gather_kernel       x rows in dispatch order -> xperm [T*k, d]; clears the tile counters
//   moe_experts_kernel  one persistent launch with two kinds of unit:
//     gate/up unit      (group, 128 rows of I, token tile): each CTA's A tile holds 64 rows of
//                       W_gate and the same 64 rows of W_up, 16 rows of each in turn, so one
//                       MMA chain leaves gate and up of a row in one warp's TMEM lanes (l and
//                       l + 16); the two lanes swap half of their columns by shuffles, write
//                       h = silu(gate) * up as bf16 H and then publish the tile (h_ready
//                       counter)
//     down unit         (group, 256 rows of d, token tile): D = W_down * H^T; the epilogue
//                       stores the rows per (token, slot) as bf16 (half the bytes of fp32
//                       through HBM twice; the combine adds them in fp32)
//   combine_kernel      y_t = sum over slots (slot order) of g_tj * row + shared -> bf16
//
// A group is one unique expert (dispatch order) or the shared expert (all T tokens). The
// expert kernel is warp-specialised: warp 0 issues the TMA loads of the weights, warp 10 those
// of the token rows, warp 1 of the cluster's first CTA the MMAs, warp 11 hands out the units
// and watches for their token rows, warps 2-9 run the epilogue. The unit list is derived on
// the device from the dispatch output, so no host round-trip is needed. Consecutive
// kernels are chained with programmatic dependent launch: each kernel's set-up (barriers,
// TMEM, tensor-map prefetch) overlaps the previous kernel, and griddepcontrol.wait orders
// the reads of its outputs.
//
// What bounds it, measured (d = 2048, I = 512, E = 256, k = 8, bias 0.5): at 2048 tokens with
// block top-k the gate/up units run at 1.8 PFLOP/s while the MMAs alone, with no loads at
// all, run at 1.85 (a 256 x 256 x 16 pair MMA every 86 ns; cuBLAS peaks at 1.92); with token
// routing the gate/up phase streams weights at 6.5 TB/s (a copy: 6.7).
#include <math.h>

#include <algorithm>
#include <mutex>

#include "dmoe_internal.cuh"
#include "silu.cuh"
#include "sm100_ptx.cuh"
#include "trace_log.cuh"

namespace dmoe {
namespace {

constexpr int kThreads = 384;                      // 12 warps
constexpr int kEpiThreads = 256;                   // warps 2-9: the epilogue
constexpr int kRowWarp = 10;                       // the producer of the token rows
constexpr int kPlanWarp = 11;                      // decodes the units, watches for their H tiles
constexpr int kCluster = 2;                        // CTAs that share an MMA
constexpr int kGateRows = 16;                      // rows of W_gate, then of W_up, in an A tile
constexpr int kATileBytes = kTileM * 128;          // 16 KB: 128 rows x 64 K
constexpr int kLevels = 3;                         // heights of the token row boxes
constexpr int kMaxGroups = kMaxExperts + 1;
constexpr uint64_t kWaitTimeoutNs = 1000000000ull;  // 1 s
constexpr int kMaxStages = 12;                     // ring slots of the weights, at most
constexpr int kRowStages = 5;                      // ring slots of the token rows
constexpr int kProgress = 64;                      // steps (K = 128) whose completion is remembered
constexpr int kQueue = 4;                          // units handed out and not yet taken up by every role
constexpr int kSpecBlocks = 64;                    // blocks of a block top-k forward, at most

struct GemmParams {
  const int32_t* n_unique;
  const int32_t* unique_ids;
  const int32_t* offsets;
  __nv_bfloat16* h;       // [T*k, I]
  __nv_bfloat16* hs;      // [T, Is]
  __nv_bfloat16* yslot;   // [T*k, d] bf16 (the combine sums them in fp32)
  __nv_bfloat16* yshared; // [T, d] bf16
  int32_t* h_ready;       // [(E+1) * ntiles]: gate/up tiles done per (group, token tile)
  int32_t* next_unit;     // units handed out beyond every cluster's first
  DevErrRecord* err;
  const void* ws_gate; const void* ws_up; const void* ws_down;  // shared, prefetched if set
  int T, d, E, k, I, Is;
  int n_max;              // token tile, at most; a multiple of `unit`
  int unit;               // rows that every tile is a multiple of (expert_tile_unit(blk) or 32)
  int box[kLevels];       // rows of the token row boxes: n_max / 2 (a CTA's half), and smaller
  int ntiles;             // token tiles per group at most
  int a_stages, b_stages; // ring slots: 128 weight rows x K = 64, and box[0] x K = 64 of token rows
                          // (a shorter box leaves room for more of K in a slot)
  int n_acc;              // accumulator buffers in TMEM
  uint32_t acc_cols;      // ... columns apart
  uint32_t tmem_cols;
  int has_shared;
  int gu_box, sgu_box;    // gate and up rows come in one box (Maps::gu / sgu): 1: gate first,
                          // 2: up first; 0 (both): a box per 16 rows (routed, shared expert)
  // Block top-k (spec_words != nullptr): the groups come from the coresets that the block
  // routing launch publishes (n_blocks blocks of blk rows). The unique experts are their
  // union, ascending; an expert's token rows are its blocks' rows in block order, which is
  // the dispatch's order. Each token tile is whole blocks, read from x block by block (a box
  // of blk rows each), so the rows are not copied into dispatch order first; and this launch
  // writes the dispatch's outputs n_unique, unique_ids and pos (the row of every (token,
  // slot), from topk_idx).
  const uint32_t* spec_words;
  int n_blocks, blk;      // (a block of 256 rows counts as two, which share its coreset:
  int halves;             // halves = 1)
  const int32_t* topk_idx;
  int32_t* pos_out;
  int32_t* n_unique_out;
  int32_t* unique_ids_out;
};

// Weights and the shared expert's rows: [rows, K] in boxes of 64 columns (K). Routed token rows:
// [rows, K] seen as [K / 64][rows][64], so that one box brings several K steps of few rows.
struct Maps {
  CUtensorMap wg, wu, sg, su;   // gate/up weights apart: [rows / 8][K / 64][8][64], 16 rows and
                                // K = 128 in one box (routed [E*I,d], shared [Is,d])
  CUtensorMap gu, sgu;          // both at once: [rows / 16][2][16][d], 64 rows of each in one box
  CUtensorMap wd, sd;           // down weights, 128-row boxes (routed [E*d,I], shared [d,Is])
  CUtensorMap x, hs;            // shared expert's token rows: x [T,d], Hs [T,Is]
  CUtensorMap xp[kLevels];      // gate/up token rows xperm [T*k,d] by box height
  CUtensorMap h[kLevels];       // down token rows H [T*k,I] by box height
  CUtensorMap xb;               // block top-k: x in boxes of one block
};

using ptx::fence_proxy_async_global;
using ptx::ld_acquire;
using ptx::named_bar_sync;
using ptx::pair_rows;
using ptx::red_release_add;

// A store that asks L2 to keep the line (the slot rows are read back by the combine right
// after this launch, while the weights stream through L2 with evict-first)
__device__ __forceinline__ void st_u32_keep(void* p, uint32_t v, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.b32 [%0], %1, %2;" ::"l"(p), "r"(v), "l"(pol) : "memory");
}

// AND of `v` over the kEpiThreads epilogue threads (named barrier 1), so that they take the
// warp-collective TMEM loads, or leave the unit loop, together
__device__ __forceinline__ bool epi_all_threads(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v), "n"(kEpiThreads)
      : "memory");
  return r != 0;
}

// Debug builds (-DDMOE_TRACE) record a per-CTA timeline of the expert kernel: slot 0 entry,
// 1 after the unit list, 62 exit; for the i-th unit of the CTA from
// DMOE_TRACE_UNIT0 on (i < 8), at 2 + 6i: unit id,
// weight producer start, last weight load issued, H ready (down units), last MMA commit,
// epilogue done; at 50 + i: the epilogue's first TMEM read of that unit.
#ifndef DMOE_TRACE_UNIT0
#define DMOE_TRACE_UNIT0 0   // the first unit of a CTA that is recorded
#endif
#define TRU(i) ((unsigned)((i) - DMOE_TRACE_UNIT0))
#ifdef DMOE_TRACE
__device__ uint64_t g_trace[kMaxPersistentCtas * 64];
#define DMOE_TRACE_AT(slot) (g_trace[blockIdx.x * 64 + (slot)] = ptx::globaltimer_ns())
#define DMOE_TRACE_SET(slot, v) (g_trace[blockIdx.x * 64 + (slot)] = (uint64_t)(v))
#else
#define DMOE_TRACE_AT(slot) ((void)0)
#define DMOE_TRACE_SET(slot, v) ((void)0)
#endif

// The expert FFN of one forward in one persistent launch. Units: first every gate/up tile
// (group, 128 rows of I, token tile), then every down tile (group, 256 rows of d, token
// tile); the shared expert's group comes first in both lists. A cluster's first unit is its
// number; it takes every further one from a global counter when it begins to load the one
// before (units differ in cost, and a fixed share left the last cluster 12-20 us behind the
// first at 256 to 2048 tokens). A cluster's unit numbers ascend, so its gate/up units precede
// its down units and a gate/up unit never waits on another unit. The weights of a down unit are
// loaded as ring slots free; only its token rows wait (bounded) for the gate/up tiles of those
// rows to be published (h_ready), so weight streaming of both phases overlaps. kSpec: the block
// top-k form (GemmParams::spec_words), compiled separately so that the other form carries none
// of its code. kFar: W_gate and W_up too far apart for one map (2^40 bytes or more: allocations
// in two address ranges; or the same tensor), 16 rows of each over K = 128 in a box of their own,
// filling two slots, issued by eight lanes. Token routing, 128 experts of I = 384, 256 / 128 / 2048
// tokens: 112.5 / 106.3 / 182.8 us with one map, 118.9 / 112.7 / 187.3 so, 125.1 / 119.0 / 190.5
// with all boxes from one lane; 16 rows over K = 64 a box are slower still (2 KB copies).
template <bool kSpec, bool kFar>
__global__ void __launch_bounds__(kThreads, 1)
moe_experts_kernel(const __grid_constant__ Maps tm, const GemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = ptx::smem_addr(smem_raw);
  uint8_t* smem = smem_raw + ((1024u - (raw_addr & 1023u)) & 1023u);  // 1024-B aligned

  const int a_stages = p.a_stages, b_stages = p.b_stages;
  const uint32_t b_slot = (uint32_t)p.box[0] * 128u;
  const uint32_t off_a = 0;
  const uint32_t off_b = off_a + (uint32_t)a_stages * kATileBytes;
  const uint32_t off_bar = off_b + (uint32_t)b_stages * b_slot;
  uint64_t* a_full = reinterpret_cast<uint64_t*>(smem + off_bar);
  uint64_t* b_full = a_full + a_stages;
  uint64_t* progress = b_full + b_stages;          // step t done: phase t / kProgress of entry
                                                   // t % kProgress
  uint64_t* acc_full = progress + kProgress;
  uint64_t* acc_empty = acc_full + 4;
  uint64_t* drain = acc_empty + 4;
  uint64_t* q_full = drain + 1;                    // the queue of units: entry i written
  uint64_t* q_empty = q_full + kQueue;             // ... and read by both CTAs (first CTA's)
  uint64_t* d_full = q_empty + kQueue;             // the same units decoded: entry written
  uint64_t* d_empty = d_full + kQueue;             // ... and read by every role of the CTA
  int2* s_desc = reinterpret_cast<int2*>(d_empty + kQueue);   // [kQueue]
  int* misc = reinterpret_cast<int*>(s_desc + kQueue);
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(misc + 0);
  volatile int* s_abort = misc + 1;
  int* s_rows_ok = misc + 2;                       // units whose token rows are there
  volatile int* s_queue = misc + 8;                // [kQueue]
  int* s_sched = misc + 4;                         // G, U, gu_units, dn_units
  int* gu_prefix = misc + 12;                      // [kMaxGroups + 1], by slot
  int* dn_prefix = gu_prefix + (kMaxGroups + 1);   // [kMaxGroups + 1], by slot
  int* g_row0 = dn_prefix + (kMaxGroups + 1);      // by group
  int* g_cnt = g_row0 + kMaxGroups;
  int* g_e = g_cnt + kMaxGroups;
  // block top-k planning: blocks per expert (bit b of s_bmask[2e + b / 32]) and the blocks of
  // the groups before its own
  uint32_t* s_bmask = reinterpret_cast<uint32_t*>(g_e + kMaxGroups);   // [2 * kMaxExperts]
  int16_t* s_bpos = reinterpret_cast<int16_t*>(s_bmask + 2 * kMaxExperts);   // [kMaxExperts]

  constexpr bool spec = kSpec;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = (int)ptx::cluster_ctarank();
  const int cl = (int)blockIdx.x / kCluster, ncl = (int)gridDim.x / kCluster;
  if (tid == 0) DMOE_TRACE_AT(0);
  KLOG(DMOE_KERNEL_EXPERTS, 0);

  if (tid == 0) {
    for (int s = 0; s < a_stages; ++s) ptx::mbar_init(&a_full[s], 1);
    for (int s = 0; s < b_stages; ++s) ptx::mbar_init(&b_full[s], 1);
    for (int s = 0; s < kProgress; ++s) ptx::mbar_init(&progress[s], 1);
    for (int a = 0; a < 4; ++a) {
      ptx::mbar_init(&acc_full[a], 1);
      ptx::mbar_init(&acc_empty[a], kCluster * kEpiThreads / 32);   // every epilogue warp
    }
    ptx::mbar_init(drain, 1);
    for (int i = 0; i < kQueue; ++i) {
      ptx::mbar_init(&q_full[i], 1);
      ptx::mbar_init(&q_empty[i], kCluster);
      ptx::mbar_init(&d_full[i], 1);
      // the two producers, the epilogue warps and, in the first CTA, the MMA issuer
      ptx::mbar_init(&d_empty[i], 2 + kEpiThreads / 32 + (rank == 0 ? 1 : 0));
      ptx::mbar_arrive_expect_tx(&q_full[i], 4);   // the entry's first unit
    }
    *s_rows_ok = 0;
    ptx::fence_mbarrier_init();
    *s_abort = 0;
    ptx::prefetch_tensormap(kFar ? &tm.wg : &tm.gu);
    ptx::prefetch_tensormap(&tm.wd);
    ptx::prefetch_tensormap(spec ? &tm.xb : &tm.xp[0]);
    ptx::prefetch_tensormap(&tm.h[0]);
  }
  if (warp == 1) {
    ptx::tmem_alloc2(s_tmem, p.tmem_cols);
    ptx::tmem_relinquish2();
  }
  ptx::cluster_arrive();   // the barriers of both CTAs are set up
  ptx::cluster_wait();
  // No dependency wait here. The launch before this one released it once the unique list and
  // the offsets were written and visible (the dispatch placement), or after its own wait for the
  // launch that wrote them (the gather); what it writes besides (the rows in dispatch order, the
  // zeroed counters) is used by the row producer, the plan warp's polls and the unit counter,
  // which wait first. The weights of the first unit are on their way by then.

  // Enters the cluster's unit i >= 1 into the queue of both CTAs (one thread of the first CTA;
  // the entry's last unit must have been read by both).
  auto enter_unit = [&](int i, int u) {
    const int e = (i - 1) % kQueue;
#pragma unroll
    for (int r = 0; r < kCluster; ++r)
      ptx::st_async_u32(ptx::peer_smem(const_cast<const int*>(s_queue) + e, r), (uint32_t)u,
                        ptx::peer_smem(&q_full[e], r));
  };

  // ---------------- groups and unit lists (slot 0 = the shared expert when present)
  if (warp == 0) {
    int U;
    if (spec) {
      // Block top-k: poll every block's published coreset words until all are nonzero (a
      // nonzero word is complete), recording each block's members and, per expert, the
      // blocks that use it
      const int nw = spec_words(p.k), total = (p.n_blocks >> p.halves) * nw;
      for (int i = lane; i < 2 * kMaxExperts; i += 32) s_bmask[i] = 0u;
      __syncwarp();
      bool bad = false;
      const uint64_t t0 = ptx::globaltimer_ns();
      for (;;) {
        bool all = true;
        for (int i = lane; i < total; i += 32) {
          const uint32_t w = ptx::ld_relaxed_u32(p.spec_words + i);
          if (w == 0u) {
            all = false;
            continue;
          }
          const int b = (i / nw) << p.halves, r0 = 3 * (i % nw);
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            if (r0 + j >= p.k) break;
            const int e = (int)((w >> (8 * j)) & 0xffu);
            if (e >= p.E) {
              bad = true;
            } else {
              atomicOr(&s_bmask[2 * e + (b >> 5)], (1u | (uint32_t)p.halves << 1) << (b & 31));
            }
          }
        }
        if (__all_sync(0xffffffffu, all)) break;
        if (ptx::globaltimer_ns() - t0 > kWaitTimeoutNs) {   // the coresets did not come
          if (lane == 0) record_error(p.err, kErrTimeout, kAtGateUp, -1);
          bad = true;
          break;
        }
      }
      bad = __any_sync(0xffffffffu, bad);
      __syncwarp();
      // the unique experts ascending (lane l: experts 8l .. 8l + 7): group u's rows are its
      // blocks' rows, so it starts at blk * (blocks of the groups before it)
      int nbq[8], cu = 0, cb = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int e = 8 * lane + q;
        nbq[q] = e < p.E ? __popc(s_bmask[2 * e]) + __popc(s_bmask[2 * e + 1]) : 0;
        cu += nbq[q] > 0 ? 1 : 0;
        cb += nbq[q];
      }
      int iu = cu, ib = cb;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, iu, o);
        const int c = __shfl_up_sync(0xffffffffu, ib, o);
        if (lane >= o) { iu += a; ib += c; }
      }
      int u = iu - cu, bp = ib - cb;
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (nbq[q] > 0) {
          const int e = 8 * lane + q;
          s_bpos[e] = (int16_t)bp;
          g_e[u] = e;
          g_row0[u] = p.blk * bp;
          g_cnt[u] = p.blk * nbq[q];
          ++u;
          bp += nbq[q];
        }
      U = bad ? 0 : __shfl_sync(0xffffffffu, iu, 31);
      if (bad && lane == 0) record_error(p.err, kErrBadDispatch, kAtGateUp, -1);
      if (lane == 0 && p.has_shared) {
        g_row0[U] = 0;
        g_cnt[U] = p.T;
        g_e[U] = -1;
      }
      __syncwarp();
    } else {
      U = __ldcg(p.n_unique);
      if (U < 0 || U > p.E) {
        if (lane == 0) record_error(p.err, kErrBadDispatch, kAtGateUp, U);
        U = 0;
      }
    }
    const int G = U + (p.has_shared ? 1 : 0);
    int carry_gu = 0, carry_dn = 0;
    for (int base = 0; base < G; base += 32) {
      const int slot = base + lane;
      int gu = 0, dn = 0;
      if (slot < G) {
        const int g = p.has_shared ? (slot == 0 ? U : slot - 1) : slot;
        int cnt, row0, e, Ig;
        if (spec) {
          cnt = g_cnt[g];
          row0 = g_row0[g];
          e = g_e[g];
          Ig = g < U ? p.I : p.Is;
        } else if (g < U) {
          row0 = __ldcg(p.offsets + g);
          cnt = __ldcg(p.offsets + g + 1) - row0;
          e = __ldcg(p.unique_ids + g);
          Ig = p.I;
          if (e < 0 || e >= p.E || cnt < 0 || cnt > p.T || row0 < 0 ||
              row0 + cnt > p.T * p.k) {
            record_error(p.err, kErrBadDispatch, kAtGateUp, g);
            cnt = 0;
            e = 0;
            row0 = 0;
          }
        } else {
          row0 = 0;
          cnt = p.T;
          e = -1;
          Ig = p.Is;
        }
        g_row0[g] = row0;
        g_cnt[g] = cnt;
        g_e[g] = e;
        const int nt = (cnt + p.n_max - 1) / p.n_max;
        gu = nt * (Ig / 128);
        dn = nt * ((p.d + 255) / 256);
      }
      int igu = gu, idn = dn;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, igu, o);
        const int b = __shfl_up_sync(0xffffffffu, idn, o);
        if (lane >= o) { igu += a; idn += b; }
      }
      if (slot < G) {
        gu_prefix[slot + 1] = carry_gu + igu;
        dn_prefix[slot + 1] = carry_dn + idn;
      }
      carry_gu += __shfl_sync(0xffffffffu, igu, 31);
      carry_dn += __shfl_sync(0xffffffffu, idn, 31);
    }
    if (lane == 0) {
      gu_prefix[0] = 0;
      dn_prefix[0] = 0;
      s_sched[0] = G;
      s_sched[1] = U;
      s_sched[2] = carry_gu;
      s_sched[3] = carry_dn;
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *s_tmem;
  const int G = s_sched[0], U = s_sched[1], n_gu = s_sched[2], n_dn = s_sched[3];
  const int units = n_gu + n_dn;
  if (tid == 0) DMOE_TRACE_AT(1);
  // (No L2 prefetch of the routed weights: the units' own loads keep HBM busy, and W_down pulled
  // into L2 at this point competed with the gate/up stream that the down units wait for
  // anyway: 256 tokens 51.1 us a layer without it, 55.4 with it; 5 x 60 tokens 65.4 and 70.7.)
  if (tid == 64 && p.ws_gate != nullptr) {
    L2Prefetch sp;
    sp.ptr[0] = p.ws_gate;
    sp.ptr[1] = p.ws_up;
    sp.ptr[2] = p.ws_down;
    sp.bytes = (int64_t)p.d * p.Is * 2;
    const int sper = (int)((sp.bytes + kPrefetchChunk - 1) / kPrefetchChunk);
    for (int c = blockIdx.x; c < 3 * sper; c += gridDim.x) l2_prefetch_chunk(sp, nullptr, 1, c);
  }

  // A unit: phase, group, m tile, n tile, rows of the token tile. The plan warp finds it from
  // its number and passes it on packed in two words (a search and a division of about 0.7 us
  // per unit, which the tensor pipe would wait for in the issuing thread).
  struct Unit {
    bool end, gu, shared;
    int g, m, n, rows, col0;   // col0: the tile's first row within the group
  };
  auto find_unit = [&](int u) -> int2 {
    if (u >= units) return make_int2(-1, 0);
    const bool gu = u < n_gu;
    const int* pre = gu ? gu_prefix : dn_prefix;
    const int v = gu ? u : u - n_gu;
    int lo = 0, hi = G - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (pre[mid] <= v) lo = mid; else hi = mid - 1;
    }
    const int g = p.has_shared ? (lo == 0 ? U : lo - 1) : lo;
    if (g_cnt[g] <= p.n_max)   // one token tile
      return make_int2((gu ? 1 : 0) | (g >= U ? 2 : 0) | g_cnt[g] << 2 | (v - pre[lo]) << 12, g);
    // token tile innermost: the clusters that take a weight tile's token tiles take them at
    // the same time, so that the tile comes from HBM once and from L2 for the others
    const int nt = (g_cnt[g] + p.n_max - 1) / p.n_max;
    const int local = v - pre[lo], m = local / nt, n = local - m * nt;
    // the group's tiles are of one size (300 rows: 160 + 140, not 256 + 44)
    const int step = nt * p.unit, tile = (g_cnt[g] + step - 1) / step * p.unit;
    const int rows = min(tile, g_cnt[g] - n * tile);
    return make_int2((gu ? 1 : 0) | (g >= U ? 2 : 0) | rows << 2 | m << 12 | n << 20,
                     g | (n * tile) << 16);
  };
  auto unpack = [&](int2 d) -> Unit {
    Unit r;
    r.end = d.x < 0;
    r.gu = d.x & 1;
    r.shared = d.x & 2;
    r.rows = (d.x >> 2) & 0x3ff;
    r.m = (d.x >> 12) & 0xff;
    r.n = (d.x >> 20) & 0x3f;
    r.g = d.y & 0xffff;
    r.col0 = d.y >> 16;
    return r;
  };
  // token rows per CTA of a unit's MMA (N is twice that, a multiple of 32): half of the tile's
  // rows, in whole blocks where the rows come from x block by block
  auto half_of = [&](const Unit& un) -> int {
    if (spec && un.gu && !un.shared) return (un.rows + p.unit - 1) / p.unit * (p.unit / 2);
    return (un.rows + 31) / 32 * 16;
  };
  // rows of one K step in a slot of token rows: whole blocks, or the smallest box that holds
  // the half; the slot holds box[0] / rows K steps
  auto slot_rows = [&](const Unit& un, int half, int* level) -> int {
    *level = 0;
    if (un.shared) return p.box[0];
    if (spec && un.gu) return half;
    int lv = 0;
#pragma unroll
    for (int l = 1; l < kLevels; ++l)
      if (p.box[l] >= half) lv = l;
    *level = lv;
    return lv == 0 ? p.box[0] : (lv == 1 ? p.box[1] : p.box[2]);
  };
  auto wait_on = [&](auto try_wait, int value) -> bool {
    if (try_wait()) return true;
    const uint64_t t0 = ptx::globaltimer_ns();
    for (uint32_t i = 1;; ++i) {
      if (try_wait()) return true;
      if ((i & 63u) == 0u) {
        if (*s_abort) return false;
        if (ptx::globaltimer_ns() - t0 > kWaitTimeoutNs) {
          record_error(p.err, kErrTimeout, kAtGateUp, value);
          *s_abort = 1;
          return false;
        }
      }
    }
  };
  auto wait = [&](uint64_t* bar, uint32_t parity, int value) -> bool {
    return wait_on([&] { return ptx::mbar_try_wait(bar, parity); }, value);
  };

  // The cluster's i-th unit for a role of this CTA: a thread, or (warp_wide) a warp, all lanes
  // of which read it. The entry is free again once all roles have read it. A wait that failed gives
  // an end, and the entry stays taken: another role may still have to read what it held before.
  auto unit_at = [&](int i, bool warp_wide) -> Unit {
    const int e = i % kQueue;
    bool got = wait(&d_full[e], (uint32_t)(i / kQueue) & 1u, i);
    if (warp_wide) got = __all_sync(0xffffffffu, got);
    const Unit un = unpack(got ? s_desc[e] : make_int2(-1, 0));
    if (warp_wide) __syncwarp();
    if (got && (!warp_wide || lane == 0)) ptx::mbar_arrive(&d_empty[e]);
    return un;
  };
  // Steps (K = 128) are counted over all units of the cluster; one commit per step reports to
  // both CTAs that its MMAs are done, and with them the slots that they read: a commit costs
  // the issuing thread about 0.1 us, as much as two MMAs. A producer is never kProgress steps
  // behind a step it waits for (the MMAs run on what it has loaded), so the parity is that of
  // step t or of no later one.
  auto step_done = [&](int t, int value) -> bool {
    return wait(&progress[t % kProgress], (uint32_t)(t / kProgress) & 1u, value);
  };
  // A producer leaves only once the MMAs of its last step are done, which its copies came before;
  // if they do not come to be done, the abort flag is set and the CTA stays a while (see the end).
  auto landed = [&](int steps) {
    if (steps > 0) step_done(steps - 1, -1);
  };

  if (warp == 0) {
    // ================= TMA producer of the weights: waits for ring slots only, so the weights
    // of the next unit follow those of the last without a gap. The bytes of both CTAs
    // complete on the first CTA's barriers, where its producers expect them.
    // kFar: the whole warp, lane j issues the j-th of a step's eight boxes.
    if (kFar || lane == 0) {
      // a wait's result for every lane that takes part
      auto agreed = [&](bool v) { return kFar ? __all_sync(0xffffffffu, v) != 0 : v; };
      const uint64_t pol_first = ptx::policy_evict_first();   // weights read by one tile
      const uint64_t pol_norm = ptx::policy_evict_normal();   // ... or by several
      const uint32_t full0 = ptx::peer_smem(a_full, 0);
      int stage = 0, chunk = 0;
      bool ok = true;
      for (int i = 0; ok; ++i) {
        const Unit un = unit_at(i, kFar);
        if (un.end) break;
        const bool shared = un.shared;
        const uint64_t pol_w = g_cnt[un.g] > p.n_max ? pol_norm : pol_first;
        if (TRU(i) < 8) { DMOE_TRACE_SET(2 + 6 * TRU(i), un.gu); DMOE_TRACE_AT(3 + 6 * TRU(i)); }
        // the next unit: the first CTA asks for it now and enters it for both CTAs once half
        // of this unit's loads are issued
        int next = units;
        if (rank == 0 && lane == 0 && i > 0) next = ncl + atomicAdd(p.next_unit, 1);
        const int kc = (un.gu ? p.d : (shared ? p.Is : p.I)) / kTileK;
        // (d % 256 = 128: the last down unit's second half reads the rows that follow and
        // stores nothing)
        const int arow = un.gu ? (shared ? 0 : g_e[un.g] * p.I) + un.m * 128 + rank * 64
                               : (shared ? 0 : g_e[un.g] * p.d) + un.m * 256 + rank * kTileM;
        const CUtensorMap* m0 = un.gu ? (shared ? &tm.sg : &tm.wg) : (shared ? &tm.sd : &tm.wd);
        const CUtensorMap* m1 = shared ? &tm.su : &tm.wu;
        const CUtensorMap* m01 = shared ? &tm.sgu : &tm.gu;
        for (int c = 0; c < kc; ++c, ++chunk) {
          // the slot's last K step was chunk - a_stages
          if (chunk >= a_stages && !agreed(step_done((chunk - a_stages) >> 1, i))) {
            ok = false;
            break;
          }
          if (rank == 0 && lane == 0)
            ptx::mbar_arrive_expect_tx(&a_full[stage], kCluster * kATileBytes);
          uint8_t* dst = smem + off_a + stage * kATileBytes;
          const uint32_t bar = full0 + 8u * (uint32_t)stage;
          if (!un.gu) {
            if (lane == 0) ptx::tma_load_2d_pair(dst, m0, bar, c * kTileK, arow, pol_w);
          } else if (!kFar) {
            ptx::tma_load_4d_pair(dst, m01, bar, c * kTileK, 0, 0, arow / kGateRows, pol_w);
          } else if ((c & 1) == 0 && lane < 8) {   // two slots at once (their number is even)
            ptx::tma_load_4d_pair(dst + lane * 2 * kGateRows * 128, (lane & 1) ? m1 : m0,
                                  bar + 8u * (uint32_t)(lane / 4), 0, 0, c,
                                  arow / 8 + (lane >> 1) * (kGateRows / 8), pol_w);
          }
          if (++stage == a_stages) stage = 0;
          if (rank == 0 && c == kc / 2) {
            if (i == 0) {
              if (!spec) pdl_wait();   // the counter is zero from here on
              if (lane == 0) next = ncl + atomicAdd(p.next_unit, 1);
            }
            if (i >= kQueue && !agreed(wait(&q_empty[i % kQueue], ((i / kQueue) & 1) ^ 1, i))) {
              ok = false;
              break;
            }
            if (lane == 0) enter_unit(i + 1, next);
          }
        }
        if (TRU(i) < 8) DMOE_TRACE_AT(4 + 6 * TRU(i));
      }
      landed(chunk >> 1);
      // the issuer's last commit arrives on this CTA's barrier as well (waited for here, while the
      // last tile is stored: after the pair's last barrier it took 0.6 us of 2048 tokens' 142)
      if (rank != 0) wait(drain, 0, -1);
    }
  } else if (warp == kRowWarp) {
    // ================= TMA producer of the token rows (x or H; lane i issues the i-th box of a
    // slot): at the start of a down unit it waits until every gate/up tile of its token tile
    // is published
    const uint64_t pol_x = ptx::policy_evict_last();    // activations: re-read by tiles
    const uint32_t full0 = ptx::peer_smem(b_full, 0);
    int stage = 0, issued = 0;
    int step0 = 0;          // the unit's first step
    if (!spec) pdl_wait();   // the rows in dispatch order are complete from here on
    int last = 0;           // lane s: the last step that reads what slot s holds
    bool ok = true;
    for (int i = 0; ok; ++i) {
      const Unit un = unit_at(i, true);
      if (!__all_sync(0xffffffffu, !un.end)) break;
      const bool shared = un.shared;
      const int half = half_of(un);
      const int Kg = un.gu ? p.d : (shared ? p.Is : p.I);
      int lv;
      const int rows = slot_rows(un, half, &lv);    // per K step
      const int kpb = p.box[0] / rows;              // K steps per slot
      int nbox = 1;                                 // boxes per K step
      int y = (shared ? 0 : g_row0[un.g]) + un.col0 + rank * half;
      const CUtensorMap* mb = un.gu ? (shared ? &tm.x : &tm.xp[lv]) : (shared ? &tm.hs : &tm.h[lv]);
      if (spec && un.gu && !shared) {
        // this CTA's blocks of the tile, from the group's blocks in ascending order (past the
        // last one any block: its columns are not used)
        nbox = half / p.blk;
        mb = &tm.xb;
        const uint32_t* bm = s_bmask + 2 * g_e[un.g];
        uint64_t m = (uint64_t)bm[0] | ((uint64_t)bm[1] << 32);
        for (int b = un.col0 / p.blk + rank * nbox + lane % nbox; b > 0 && (m & (m - 1)); --b)
          m &= m - 1;
        y = (__ffsll((long long)m) - 1) * p.blk;
      }
      if (!un.gu) {
        // (the plan warp has seen them; its acquire carries over)
        ok = wait_on(
            [&] {
              if (ptx::ld_acquire_cta(s_rows_ok) > i) return true;
              __nanosleep(32);
              return false;
            },
            i);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        fence_proxy_async_global();   // generic stores of the rows before these loads
        if (lane == 0 && TRU(i) < 8) DMOE_TRACE_AT(5 + 6 * TRU(i));
      }
      const uint32_t box_bytes = (uint32_t)(rows / nbox) * 128u;
      const int kc = Kg / kTileK;
      const bool by_block = spec && un.gu && !shared;
      for (int c = 0; c < kc; c += kpb) {
        if (issued >= b_stages) {
          ok = __all_sync(0xffffffffu, step_done(__shfl_sync(0xffffffffu, last, stage), i));
          if (!ok) break;
        }
        uint8_t* dst = smem + off_b + stage * b_slot;
        const uint32_t bar = full0 + 8u * (uint32_t)stage;
        if (by_block) {
          const int n = min(kpb, kc - c) * nbox;      // boxes of this slot (at most 16)
          if (lane == 0 && rank == 0)
            ptx::mbar_arrive_expect_tx(&b_full[stage], kCluster * (uint32_t)n * box_bytes);
          if (lane < n)
            ptx::tma_load_2d_pair(dst + lane * box_bytes, mb, bar, (c + lane / nbox) * kTileK, y,
                                  pol_x);
        } else if (lane == 0) {
          // (kpb K steps in one box; steps past the end of K read as zeros)
          if (rank == 0)
            ptx::mbar_arrive_expect_tx(&b_full[stage], kCluster * (uint32_t)kpb * box_bytes);
          if (shared)
            ptx::tma_load_2d_pair(dst, mb, bar, c * kTileK, y, pol_x);
          else
            ptx::tma_load_3d_pair(dst, mb, bar, 0, y, c, pol_x);
        }
        if (lane == stage) last = step0 + (min(c + kpb, kc) - 1) / 2;
        ++issued;
        if (++stage == b_stages) stage = 0;
      }
      step0 += kc / 2;
    }
    if (lane == 0) landed(step0);
  } else if (warp == kPlanWarp) {
    // ================= the units, decoded one or more ahead of their use, and the readiness of
    // their token rows (a poll is an L2 round trip, 1 us or more while weights stream)
    if (lane == 0) {
      const uint32_t q_empty0 = ptx::peer_smem(q_empty, 0);
      // diagnostic (normally 0): every down unit waits for this many more gate/up tiles than its
      // group has, so that its bounded wait runs out (read once the first unit is handed on: at
      // the start of the kernel it held every launch up by 0.6 to 1.1 us)
      int hold = 0;
      for (int i = 0;; ++i) {
        int u = cl;
        if (i > 0) {
          const int q = (i - 1) % kQueue;
          // (a wait that failed: the other roles leave by the abort flag)
          if (!wait(&q_full[q], (uint32_t)((i - 1) / kQueue) & 1u, i)) break;
          u = s_queue[q];
          ptx::mbar_arrive_expect_tx(&q_full[q], 4);   // the entry's next unit
          ptx::mbar_arrive_pair(q_empty0 + 8u * (uint32_t)q);
        }
        const int2 d = find_unit(u);
        const int e = i % kQueue;
        if (i >= kQueue && !wait(&d_empty[e], ((uint32_t)(i / kQueue) & 1u) ^ 1u, i)) break;
        s_desc[e] = d;
        ptx::mbar_arrive(&d_full[e]);
        if (i == 0) hold = *reinterpret_cast<volatile int32_t*>(&p.err->hold);
        const Unit un = unpack(d);
        if (un.end) break;
        if (!un.gu) {
          if (!spec) pdl_wait();   // the counters are zeroed from here on
          const int32_t* flag = p.h_ready + un.g * p.ntiles + un.n;
          const int need = (un.shared ? p.Is : p.I) / 64 + hold;
          bool ok = true;
          if (ld_acquire(flag) < need) {
            const uint64_t t0 = ptx::globaltimer_ns();
            while (ok && ld_acquire(flag) < need) {
              __nanosleep(64);
              if (*s_abort) ok = false;
              if (ptx::globaltimer_ns() - t0 > kWaitTimeoutNs) {
                record_error(p.err, kErrTimeout, kAtDown, u);
                *s_abort = 1;
              }
            }
          }
          if (!ok) break;
        }
        ptx::st_release_cta(s_rows_ok, i + 1);
      }
    }
  } else if (warp == 1) {
    // ================= MMA issuer: the first CTA's, for both. The tensor pipe queues one or two
    // MMAs, so this thread's pauses are the pipe's: the next slots are tested while MMAs are
    // queued.
    if (rank == 0 && lane == 0) {
      int sa = 0, sb = 0, acc = 0, step = 0;
      bool a_in = false, b_in = false;      // the next slots were seen full
      uint32_t pa = 0, pb = 0, acc_phase = 0;
      bool ok = true;
      for (int i = 0; ok; ++i) {
        const Unit un = unit_at(i, false);
        if (un.end) break;
        const int steps = (un.gu ? p.d : (un.shared ? p.Is : p.I)) / (2 * kTileK);
        const int half = half_of(un);
        const uint32_t idesc = ptx::idesc_bf16(kCluster * kTileM, (uint32_t)(2 * half));
        int lv;
        const uint32_t step_bytes = (uint32_t)slot_rows(un, half, &lv) * 128u;
        const int kpb = (int)(b_slot / step_bytes);
        {
          ok = wait(&acc_empty[acc], acc_phase ^ 1u, i);
          ptx::tc_fence_after();
          const uint32_t d0 = tmem_base + (uint32_t)acc * p.acc_cols;
          const uint32_t a0 = ptx::smem_addr(smem + off_a), b0 = ptx::smem_addr(smem + off_b);
          int kb = kpb - 1;           // K box within the slot of token rows
          uint32_t bs = 0;
          for (int c = 0; ok && c < steps; ++c, ++step) {
#pragma unroll
            for (int k2 = 0; k2 < 2; ++k2) {
              ok = ok && (a_in || wait(&a_full[sa], pa, i));
              uint32_t as = a0 + (uint32_t)sa * kATileBytes;
              uint32_t sbo = 1024u;
              if (kFar && un.gu) {    // two slots hold the step: rows of 8 over both K boxes
                if (k2 == 0) ok = ok && wait(&a_full[sa + 1], pa, i);
                as = a0 + (uint32_t)(sa - k2) * kATileBytes + (uint32_t)k2 * 1024u;
                sbo = 2048u;
              }
              if (++sa == a_stages) { sa = 0; pa ^= 1u; }
              bs += step_bytes;
              if (++kb == kpb) {      // the next slot
                ok = ok && (b_in || wait(&b_full[sb], pb, i));
                bs = b0 + (uint32_t)sb * b_slot;
                kb = 0;
                if (++sb == b_stages) { sb = 0; pb ^= 1u; }
              }
              if (!ok) break;
              ptx::tc_fence_after();
#pragma unroll
              for (int kk = 0; kk < kTileK / 16; ++kk) {
                ptx::mma_bf16_pair(d0, ptx::sdesc_k_sw128(as + kk * 32, sbo),
                                   ptx::sdesc_k_sw128(bs + kk * 32), idesc,
                                   (c > 0 || k2 > 0 || kk > 0) ? 1u : 0u);
                if (kk == 1) {
                  a_in = ptx::mbar_test_wait(&a_full[sa], pa);
                  b_in = ptx::mbar_test_wait(&b_full[sb], pb);
                }
              }
            }
            if (!ok) break;
            ptx::mma_commit_pair(&progress[step % kProgress]);
          }
          if (ok) ptx::mma_commit_pair(&acc_full[acc]);
          if (TRU(i) < 8) DMOE_TRACE_AT(6 + 6 * TRU(i));
        }
        if (++acc == p.n_acc) { acc = 0; acc_phase ^= 1u; }
      }
      // make sure no MMA is still running when TMEM is released
      ptx::mma_commit_pair(drain);
      const uint64_t t0 = ptx::globaltimer_ns();
      while (!ptx::mbar_try_wait(drain, 0) && ptx::globaltimer_ns() - t0 < kWaitTimeoutNs) {
      }
    }
  } else {
    // ================= epilogue: warps 2..9, TMEM lanes 32*(warp%4) ..; two column groups
    // (warps 2-5 and 6-9) take alternate 16-column slices of the accumulator (the epilogue math
    // is latency-bound: two groups finish a tile in about half the time)
    if (spec && warp == 2) {
      // the dispatch's outputs: the row of every (token, slot) of this CTA's share of the
      // tokens (expert e = topk_idx[t, j] of block b: the group's rows start at
      // blk * s_bpos[e], block b is its rank-th block), once the routing launch has ended
      pdl_wait();
      const int per = (p.T + (int)gridDim.x - 1) / (int)gridDim.x;
      const int t_begin = (int)blockIdx.x * per;
      const int t_end = min(p.T, t_begin + per);
      for (int i = t_begin * p.k + lane; i < t_end * p.k; i += 32) {
        const int t = i / p.k, b = t / p.blk;
        const int e = __ldcg(p.topk_idx + i);
        int r = -1;
        if (U > 0 && e >= 0 && e < p.E && b < p.n_blocks) {
          const uint32_t lo = s_bmask[2 * e], hi = s_bmask[2 * e + 1];
          const bool in = b < 32 ? ((lo >> b) & 1u) != 0u : ((hi >> (b - 32)) & 1u) != 0u;
          const int rank = b < 32 ? __popc(lo & ((1u << b) - 1u))
                                  : __popc(lo) + __popc(hi & ((1u << (b - 32)) - 1u));
          if (in) r = p.blk * (s_bpos[e] + rank) + (t - b * p.blk);
        }
        if (r < 0) {
          record_error(p.err, kErrBadDispatch, kAtDown, i);
          r = 0;
        }
        p.pos_out[i] = r;
      }
      if (blockIdx.x == 0) {
        if (lane == 0) *p.n_unique_out = U;
        for (int u = lane; u < p.E; u += 32) p.unique_ids_out[u] = u < U ? g_e[u] : -1;
      }
      // visible before this launch releases the combine (at its end): the combine reads
      // pos before its dependency wait
      __threadfence();
    }
    const int q = warp & 3;
    const int cg = (warp - 2) >> 2;                 // column group
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;
    const int odd = lane & 1;
    const uint64_t pol_keep = ptx::policy_evict_last();   // the slot rows, for the combine
    const uint32_t acc_empty0 = ptx::peer_smem(acc_empty, 0);
    int acc = 0;
    uint32_t acc_phase = 0;
    for (int i = 0;; ++i) {
      const Unit un = unit_at(i, true);
      const bool shared = un.shared;
      const int nvalid = un.rows;
      // (a warp whose wait failed leaves with the others)
      if (!epi_all_threads(!un.end && wait(&acc_full[acc], acc_phase, i))) break;
      ptx::tc_fence_after();
      if (tid == 64 && TRU(i) < 8) DMOE_TRACE_AT(50 + TRU(i));
      const uint32_t tbase = tmem_base + lane_off + (uint32_t)acc * p.acc_cols;
      const int col0 = un.col0;                     // first token column of the tile
      if (un.gu) {
        // lanes 0-15 of a quadrant: gate rows, lanes 16-31: up rows of the same 16 intermediate
        // units (or the other way round). Per 16-token slice a gate lane gives its last 8
        // columns to the lane that holds its row's up values and takes that one's first 8: each
        // then has gate and up of one row for 8 tokens. Two slices at a time (32 columns apart):
        // their latencies overlap
        const int Ig = shared ? p.Is : p.I;
        const int row = un.m * 128 + rank * 64 + q * kGateRows + (lane & 15);
        __nv_bfloat16* hout = (shared ? p.hs : p.h) +
                              (size_t)((shared ? 0 : g_row0[un.g]) + col0) * Ig + (row & ~1);
        const bool is_gate = (lane < 16) == ((shared ? p.sgu_box : p.gu_box) != 2);
        for (int c0 = 16 * cg; c0 < nvalid; c0 += 64) {
          // (past the last slice the first one again, and nothing is stored)
          const int c1 = c0 + 32 < nvalid ? c0 + 32 : c0;
          float v[2][16];
          ptx::tmem_ld16(tbase + c0, v[0]);
          ptx::tmem_ld16(tbase + c1, v[1]);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int j = 0; j < 16; ++j) asm volatile("" : "+f"(v[s][j]));   // only after the wait
          float h[16], up[16];
#pragma unroll
          for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float other =
                  __shfl_xor_sync(0xffffffffu, is_gate ? v[s][8 + j] : v[s][j], kGateRows);
              h[8 * s + j] = is_gate ? v[s][j] : other;
              up[8 * s + j] = is_gate ? other : v[s][8 + j];
            }
          silu_all(h);
#pragma unroll
          for (int j = 0; j < 16; ++j) h[j] *= up[j];
#pragma unroll
          for (int s = 0; s < 2; ++s) {
            float hs[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) hs[j] = h[8 * s + j];
            uint32_t w[4];
            pair_rows(hs, w);
            const int t0 = (s == 0 ? c0 : c0 + 32) + (is_gate ? 0 : 8) + 4 * odd;
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (t0 + j < nvalid)
                *reinterpret_cast<uint32_t*>(hout + (size_t)(t0 + j) * Ig) = w[j];
          }
        }
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive_pair(acc_empty0 + 8u * (uint32_t)acc);
        // publish the tile: the barrier orders every epilogue thread's H stores before one
        // release add; a reader acquires the counter, then fences the async proxy
        named_bar_sync(4, kEpiThreads);
        if (tid == 64) red_release_add(p.h_ready + un.g * p.ntiles + un.n, 1);
      } else {
        const int drow = un.m * 256 + rank * kTileM + q * 32 + lane;
        __nv_bfloat16* out = (shared ? p.yshared + (size_t)col0 * p.d
                                     : p.yslot + (size_t)(g_row0[un.g] + col0) * p.d) + (drow & ~1);
        if (drow < p.d) {   // the same for the whole CTA (d is a multiple of 128)
          for (int c0 = 16 * cg; c0 < nvalid; c0 += 64) {
            const int c1 = c0 + 32 < nvalid ? c0 + 32 : c0;
            float v[2][16];
            ptx::tmem_ld16(tbase + c0, v[0]);
            ptx::tmem_ld16(tbase + c1, v[1]);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
              for (int j = 0; j < 16; ++j) asm volatile("" : "+f"(v[s][j]));
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              float h[8];
#pragma unroll
              for (int j = 0; j < 8; ++j) h[j] = v[g >> 1][8 * (g & 1) + j];
              uint32_t w[4];
              pair_rows(h, w);
              const int t0 = c0 + 32 * (g >> 1) + 8 * (g & 1) + 4 * odd;
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (t0 + j < nvalid) st_u32_keep(out + (size_t)(t0 + j) * p.d, w[j], pol_keep);
            }
          }
        }
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive_pair(acc_empty0 + 8u * (uint32_t)acc);
      }
      if (tid == 64 && TRU(i) < 8) DMOE_TRACE_AT(7 + 6 * TRU(i));
      if (++acc == p.n_acc) { acc = 0; acc_phase ^= 1u; }
    }
  }

  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  // the combine may start now (launched earlier, its waiting CTAs would share the SMs with this
  // launch and slow it down); it reads the placement's output before its own wait
  pdl_wait();
  pdl_launch_dependents();
  if (tid == 0) DMOE_TRACE_AT(62);
  KLOG(DMOE_KERNEL_EXPERTS, 1);
  // neither CTA leaves while the other may still signal its barriers or read its tiles
  ptx::cluster_arrive();
  ptx::cluster_wait();
  if (warp == 1) {
    __syncwarp();
    ptx::tmem_dealloc2(tmem_base, p.tmem_cols);
  }
  // After a wait that failed, copies into this CTA's shared memory and stores and arrivals from the
  // other CTA may not have been waited for. Nothing new is issued any more (the barrier above): the
  // CTA stays until they have long landed (they take microseconds).
  if (*s_abort) {
    const uint64_t t0 = ptx::globaltimer_ns();
    while (ptx::globaltimer_ns() - t0 < kWaitTimeoutNs / 10) __nanosleep(1000);
  }
}

// xperm[r, :] = x[rows[r] / k, :]; block 0 also clears the gate/up tile counters. After a fault that
// the dispatch recorded (a bad id, an expert twice in a token) entries of `rows` are whatever the
// caller's buffer held: they are kept in range.
__global__ void __launch_bounds__(256)
gather_kernel(const __nv_bfloat16* __restrict__ x, const int32_t* __restrict__ rows,
              __nv_bfloat16* __restrict__ xperm, int32_t* __restrict__ h_ready, int n_ready,
              int pairs, int k, int d) {
  pdl_wait();
  pdl_launch_dependents();   // after the wait: a waiting dependent would share the SMs
  KLOG(DMOE_KERNEL_GATHER, 0);
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < n_ready; i += blockDim.x) h_ready[i] = 0;
  const int vec = d / 8;  // uint4 per row
  for (int r = blockIdx.x; r < pairs; r += gridDim.x) {
    const int t = (int)min((uint32_t)rows[r], (uint32_t)pairs - 1u) / k;
    const uint4* src = reinterpret_cast<const uint4*>(x + (size_t)t * d);
    uint4* dst = reinterpret_cast<uint4*>(xperm + (size_t)r * d);
    for (int i = threadIdx.x; i < vec; i += blockDim.x) dst[i] = src[i];
  }
  KLOG(DMOE_KERNEL_GATHER, 1);
}

// kCombineCols consecutive row values: the raw 16-byte pieces (one for 8 bf16, two for 8
// fp32), loaded first and converted to fp32 as they are used (registers bound the CTAs per
// SM, and with them the loads in flight).
constexpr int kCombineCols = 8;
template <typename Row> struct Raw8;
template <> struct Raw8<__nv_bfloat16> {
  uint4 a;
  __device__ __forceinline__ void load(const __nv_bfloat16* src) {
    a = *reinterpret_cast<const uint4*>(src);
  }
  __device__ __forceinline__ void unpack(float (&v)[8]) const {
    const uint32_t w[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[i]));
      v[2 * i] = f.x;
      v[2 * i + 1] = f.y;
    }
  }
};
template <> struct Raw8<float> {
  float4 a, b;
  __device__ __forceinline__ void load(const float* src) {
    a = *reinterpret_cast<const float4*>(src);
    b = *reinterpret_cast<const float4*>(src + 4);
  }
  __device__ __forceinline__ void unpack(float (&v)[8]) const {
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  }
};

// y[t, :] = bf16( sum_j g[t,j] * yslot[pos[t*k + j], :] (slot order) + yshared[t, :] );
// block (0, 0) also clears `zero[0 .. n_zero)` and `zero2[0 .. n_zero2)` (counters and
// flags of the launches before, now done). With meta_early the slot indices and gates are
// read before the dependency wait: the caller guarantees that they were complete before the
// launch before this one could let this one start (the decode-size expert launch releases
// it only at its end, after its own wait for the routing launch that wrote them).
template <typename Row>
__global__ void __launch_bounds__(256, sizeof(Row) == 2 ? 3 : 1)   // bf16 rows: three CTAs per SM
combine_kernel(const Row* __restrict__ yslot, const Row* __restrict__ yshared,
               const int32_t* __restrict__ pos, const float* __restrict__ gate,
               __nv_bfloat16* __restrict__ y, int k, int d, int has_shared, int32_t* zero,
               int n_zero, uint32_t* zero2, int n_zero2, int meta_early) {
  pdl_launch_dependents();
  const int t = blockIdx.y;
  const int c = (blockIdx.x * blockDim.x + threadIdx.x) * kCombineCols;
  // the slot indices and gates, eight slots at a time
  int r[8];
  float gj[8];
  auto load_meta = [&](int j0) {
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j0 + j < k) {
        r[j] = __ldcg(pos + t * k + j0 + j);
        gj[j] = __ldcg(gate + t * k + j0 + j);
      }
  };
  if (meta_early) load_meta(0);
  pdl_wait();
  KLOG(DMOE_KERNEL_COMBINE, 0);
  if (blockIdx.x == 0 && blockIdx.y == 0) {
    for (int i = threadIdx.x; i < n_zero; i += blockDim.x) zero[i] = 0;
    for (int i = threadIdx.x; i < n_zero2; i += blockDim.x) zero2[i] = 0u;
  }
  if (c >= d) return;
  // eight slots at a time: their row loads (and the shared row's) are issued before the
  // first product; the sum keeps the slot order
  float acc[kCombineCols];
#pragma unroll
  for (int i = 0; i < kCombineCols; ++i) acc[i] = 0.f;
  Raw8<Row> raw_s;
  if (has_shared) raw_s.load(yshared + (size_t)t * d + c);
  for (int j0 = 0; j0 < k; j0 += 8) {
    if (!meta_early || j0 > 0) load_meta(j0);
    Raw8<Row> raw[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j0 + j < k) raw[j].load(yslot + (size_t)r[j] * d + c);
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j0 + j < k) {
        float v[kCombineCols];
        raw[j].unpack(v);
#pragma unroll
        for (int i = 0; i < kCombineCols; ++i) acc[i] = fmaf(gj[j], v[i], acc[i]);
      }
  }
  if (has_shared) {
    float vs[kCombineCols];
    raw_s.unpack(vs);
#pragma unroll
    for (int i = 0; i < kCombineCols; ++i) acc[i] += vs[i];
  }
  uint32_t out[kCombineCols / 2];
#pragma unroll
  for (int i = 0; i < kCombineCols / 2; ++i) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(acc[2 * i], acc[2 * i + 1]);
    out[i] = *reinterpret_cast<const uint32_t*>(&h);
  }
  *reinterpret_cast<uint4*>(y + (size_t)t * d + c) = make_uint4(out[0], out[1], out[2], out[3]);
  KLOG(DMOE_KERNEL_COMBINE, 1);
}

// ------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000,
                                         cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  });
  return fn;
}

// bf16 matrix [rows, cols] row-major, box = 64 columns (128 B) x box_rows rows, 128-B swizzle.
bool make_map(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  EncodeTiledFn enc = encode_fn();
  if (enc == nullptr) return false;
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {cols * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kTileK, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The same matrix as [cols / 64][rows][64]: a box of `ksteps` 64-column steps of box_rows rows.
bool make_map_k(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows,
                uint32_t ksteps) {
  EncodeTiledFn enc = encode_fn();
  if (enc == nullptr) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)kTileK, rows, cols / kTileK};
  const cuuint64_t strides[2] = {cols * 2, (cuuint64_t)kTileK * 2};
  const cuuint32_t box[3] = {(cuuint32_t)kTileK, box_rows, ksteps};
  const cuuint32_t estr[3] = {1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Two matrices [rows, cols] of one shape as [rows / 16][2][16][cols], the one at the lower
// address first: one box brings 64 rows of both, 16 of each in turn (a copy costs the SM's copy
// engine about 100 cycles besides its rows). Their distance is a stride of the map: a multiple
// of 16 bytes below 2^40. Returns 1 (a first), 2 (b first) or 0: the distance is no such stride,
// no map is made.
int make_map_two(CUtensorMap* m, const void* a, const void* b, uint64_t rows, uint64_t cols) {
  EncodeTiledFn enc = encode_fn();
  const uintptr_t pa = reinterpret_cast<uintptr_t>(a), pb = reinterpret_cast<uintptr_t>(b);
  const uint64_t dist = pa < pb ? pb - pa : pa - pb;
  if (enc == nullptr || dist == 0 || dist % 16 != 0 || dist >= ((uint64_t)1 << 40)) return 0;
  const cuuint64_t dims[4] = {cols, kGateRows, 2, rows / kGateRows};
  const cuuint64_t strides[3] = {cols * 2, dist, cols * 2 * kGateRows};
  const cuuint32_t box[4] = {(cuuint32_t)kTileK, kGateRows, 2, 64 / kGateRows};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  if (enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(pa < pb ? a : b), dims, strides,
          box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return 0;
  return pa < pb ? 1 : 2;
}

// One matrix as [rows / 8][cols / 64][8][64]: a box of 16 rows and K = 128, each 8 rows over both
// K boxes (4 KB a copy, where 2 KB over one K box leave the copy engine short of the HBM rate).
bool make_map_far(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols) {
  EncodeTiledFn enc = encode_fn();
  if (enc == nullptr) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)kTileK, 8, cols / kTileK, rows / 8};
  const cuuint64_t strides[3] = {cols * 2, (cuuint64_t)kTileK * 2, cols * 16};
  const cuuint32_t box[4] = {(cuuint32_t)kTileK, 8, 2, kGateRows / 8};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

uint32_t pow2_cols(uint32_t c) {
  uint32_t r = 32;
  while (r < c) r <<= 1;
  return r;
}

size_t experts_fixed_smem() {
  // alignment slack + barriers + misc/group arrays + block top-k planning
  return 1024 + 8 * (kMaxStages + kRowStages + kProgress + 9 + 5 * kQueue) + sizeof(int) * (12 + 5 * (kMaxGroups + 1)) +
         64 + 4 * 2 * kMaxExperts + 2 * kMaxExperts;
}

int max_smem_optin() {
  int dev = 0, v = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return v;
}

// The pairs of CTAs of the expert launch that the current device runs at once; on the first call per
// device it also raises the kernels' limit of dynamic shared memory to `smem`, which is set per
// device.
cudaError_t resident_pairs(int smem, int* pairs) {
  static std::atomic<int> known[32];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  *pairs = dev < 32 ? known[dev].load(std::memory_order_acquire) : 0;
  if (*pairs > 0) return cudaSuccess;
  for (auto* kernel : {moe_experts_kernel<false, false>, moe_experts_kernel<true, false>,
                       moe_experts_kernel<false, true>, moe_experts_kernel<true, true>})
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = kCluster;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kCluster);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveClusters(pairs, moe_experts_kernel<false, false>, &cfg);
  if (e == cudaSuccess && dev < 32) known[dev].store(*pairs, std::memory_order_release);
  return e;
}

}  // namespace

#ifdef DMOE_TRACE
extern "C" int dmoe_debug_trace(void* host, size_t bytes) {
  if (bytes > sizeof(g_trace)) bytes = sizeof(g_trace);
  return (int)cudaMemcpyFromSymbol(host, g_trace, bytes);
}
extern "C" int dmoe_debug_trace_clear() {
  static uint64_t zeros[kMaxPersistentCtas * 64] = {};
  return (int)cudaMemcpyToSymbol(g_trace, zeros, sizeof(zeros));
}
DMOE_KLOG_EXPORT(dmoe_debug_klog_experts)
#endif

int experts_ready_counters(int T, int E, int n_max) {
  return (E + 1) * ((T + n_max - 1) / n_max) + 1;   // and the counter of units
}

bool experts_spec_ok(const dmoe_layer_desc& d, int n_max) {
  // blocks (or their halves) that fill a CTA's half of a token tile whole (expert_tile_unit), at
  // most kSpecBlocks of them (a 64-bit block mask per expert)
  const int part = expert_tile_part(d.block_size);
  return d.mode == DMOE_ROUTE_BLOCK && d.top_p <= 0.f && mask_top_k(d) == d.top_k && part > 0 &&
         d.n_blocks >= 1 && d.n_blocks * (d.block_size / part) <= kSpecBlocks &&
         n_max % expert_tile_unit(part) == 0 && d.n_experts <= kMaxExperts;
}

cudaError_t launch_experts(const ExpertArgs& a, cudaStream_t s) {
  const int pairs = a.T * a.k;
  const bool has_shared = a.Is > 0;
  const int n_ready = experts_ready_counters(a.T, a.E, a.n_max);
  const bool spec = a.spec_words != nullptr;
  // 1. gather x in dispatch order; clear the gate/up tile counters (unless the dispatch
  //    placement of the fused layer call has done both, or, for block top-k, the block
  //    routing launch has cleared them and the token rows are read from x by block)
  if (!a.gathered && !spec) {
    const int grid = pairs < 1024 ? pairs : 1024;
    static std::atomic<uint32_t> carveout;
    cudaError_t e = max_shared_carveout(gather_kernel, carveout);
    if (e != cudaSuccess) return e;
    prof_begin(DMOE_KERNEL_GATHER, s);
    e = launch_ex(gather_kernel, dim3(grid), dim3(256), 0, s, true, a.x, a.rows,
                              a.xperm, a.h_ready, n_ready, pairs, a.k, a.d);
    prof_end(DMOE_KERNEL_GATHER, s);
    if (e != cudaSuccess) return e;
  }
  GemmParams gp{};
  gp.n_unique = a.n_unique;
  gp.unique_ids = a.unique_ids;
  gp.offsets = a.offsets;
  gp.h = a.h;
  gp.hs = a.hs;
  gp.yslot = static_cast<__nv_bfloat16*>(a.yslot);
  gp.yshared = static_cast<__nv_bfloat16*>(a.yshared);
  gp.h_ready = a.h_ready;
  gp.next_unit = a.h_ready + n_ready - 1;
  gp.err = a.err;
  if (has_shared && a.prefetch_shared) {
    gp.ws_gate = a.ws_gate;
    gp.ws_up = a.ws_up;
    gp.ws_down = a.ws_down;
  }
  gp.T = a.T; gp.d = a.d; gp.E = a.E; gp.k = a.k; gp.I = a.I; gp.Is = a.Is;
  gp.n_max = a.n_max;
  gp.unit = 32;
  gp.box[0] = a.n_max / 2;
  for (int i = 1; i < kLevels; ++i) gp.box[i] = ((gp.box[i - 1] / 2) + 7) & ~7;
  gp.ntiles = (a.T + a.n_max - 1) / a.n_max;
  gp.has_shared = has_shared ? 1 : 0;
  if (spec) {
    gp.spec_words = a.spec_words;
    gp.blk = expert_tile_part(a.T / a.spec_blocks);
    gp.n_blocks = a.T / gp.blk;
    gp.halves = gp.n_blocks > a.spec_blocks ? 1 : 0;
    gp.unit = expert_tile_unit(gp.blk);   // whole blocks
    gp.topk_idx = a.topk_idx;
    gp.pos_out = a.pos_out;
    gp.n_unique_out = a.n_unique_out;
    gp.unique_ids_out = a.unique_ids_out;
  }

  // 2. gate/up + SwiGLU and down projection in one persistent launch
  // (only the maps that this call uses: each costs the host time)
  Maps m{};
  const uint64_t gu_rows = (uint64_t)a.E * a.I;
  bool ok = make_map(&m.wd, a.w_down, (uint64_t)a.E * a.d, a.I, kTileM);
  gp.gu_box = make_map_two(&m.gu, a.w_gate, a.w_up, gu_rows, a.d);
  if (spec) ok = ok && make_map(&m.xb, a.x, (uint64_t)a.T, a.d, (uint32_t)gp.blk);
  for (int i = 0; i < kLevels; ++i) {
    const uint32_t rows = (uint32_t)gp.box[i], ksteps = (uint32_t)(gp.box[0] / gp.box[i]);
    if (!spec) ok = ok && make_map_k(&m.xp[i], a.xperm, (uint64_t)pairs, a.d, rows, ksteps);
    ok = ok && make_map_k(&m.h[i], a.h, (uint64_t)pairs, a.I, rows, ksteps);
  }
  if (has_shared) {
    ok = ok && make_map(&m.sd, a.ws_down, (uint64_t)a.d, a.Is, kTileM) &&
         make_map(&m.x, a.x, (uint64_t)a.T, a.d, (uint32_t)gp.box[0]) &&
         make_map(&m.hs, a.hs, (uint64_t)a.T, a.Is, (uint32_t)gp.box[0]);
    gp.sgu_box = make_map_two(&m.sgu, a.ws_gate, a.ws_up, (uint64_t)a.Is, a.d);
  }
  // tensors too far apart for one map (the form with a box per 16 rows then loads all of them)
  const bool far = gp.gu_box == 0 || (has_shared && gp.sgu_box == 0);
  if (far) {
    gp.gu_box = gp.sgu_box = 0;
    ok = ok && make_map_far(&m.wg, a.w_gate, gu_rows, a.d) &&
         make_map_far(&m.wu, a.w_up, gu_rows, a.d);
    if (has_shared)
      ok = ok && make_map_far(&m.sg, a.ws_gate, (uint64_t)a.Is, a.d) &&
           make_map_far(&m.su, a.ws_up, (uint64_t)a.Is, a.d);
  }
  if (!ok) return cudaErrorInvalidValue;

  // ring slots: five of token rows, the rest of the shared memory for the weights (what is in
  // flight of them sets the rate they come from HBM at). Four / five / six, us per layer: 256
  // tokens 51.8 / 50.6 / 50.1 (block top-k) and 79.9 / 79.0 / 79.8 (p = 0.6), 1024 tokens with
  // p = 0.6 136 / 134 / 136, 2048 tokens with token routing 320 / 315 / 324
  const size_t fixed = experts_fixed_smem(), row_slot = (size_t)gp.box[0] * 128;
  const int limit = max_smem_optin();
  gp.b_stages = kRowStages;
  const long left = (long)limit - (long)fixed - (long)(gp.b_stages * row_slot);
  gp.a_stages = left < 0 ? 0 : (int)(left / kATileBytes);
  // (block top-k: room for a CTA of the block routing launch beside this launch's, which
  // start while it runs)
  const int most = spec ? kMaxStages - 4 : kMaxStages;
  if (gp.a_stages > most) gp.a_stages = most;
  if (far) gp.a_stages &= ~1;
  if (gp.a_stages < 2) return cudaErrorInvalidConfiguration;
  gp.acc_cols = pow2_cols((uint32_t)a.n_max);
  gp.n_acc = 512 / (int)gp.acc_cols;
  if (gp.n_acc > 4) gp.n_acc = 4;
  gp.tmem_cols = (uint32_t)gp.n_acc * gp.acc_cols;
  const size_t smem = fixed + (size_t)gp.a_stages * kATileBytes + gp.b_stages * row_slot;
  int pairs_max = 0;
  cudaError_t e = resident_pairs(limit, &pairs_max);
  if (e != cudaSuccess) return e;
  // (every pair owns its first unit, which other pairs' down units may wait for: no more pairs than
  // can run at once)
  int grid = std::min(device_sm_count() / kCluster, pairs_max) * kCluster;
  if (grid > kMaxPersistentCtas) grid = kMaxPersistentCtas;
  if (grid < kCluster) return cudaErrorInvalidConfiguration;
  prof_begin(DMOE_KERNEL_EXPERTS, s);
  e = launch_cluster(
      far ? (spec ? moe_experts_kernel<true, true> : moe_experts_kernel<false, true>)
          : (spec ? moe_experts_kernel<true, false> : moe_experts_kernel<false, false>),
      dim3(grid), dim3(kThreads), smem, s, kCluster, !prof_serial(DMOE_KERNEL_EXPERTS), m, gp);
  prof_end(DMOE_KERNEL_EXPERTS, s);
  if (e != cudaSuccess) return e;

  // 3. gate-weighted combine of the bf16 rows (the slot rows and gates were complete before
  //    this launch released it: the combine may read them before its dependency wait)
  return launch_combine(a, s, nullptr, 0, nullptr, 0, true, true);
}

cudaError_t launch_combine(const ExpertArgs& a, cudaStream_t s, int32_t* zero, int n_zero,
                           uint32_t* zero2, int n_zero2, bool meta_early, bool rows_bf16) {
  // CTAs of 256 threads; fewer (down to 32) while that leaves fewer than 128 CTAs, so
  // that a decode-sized forward spreads its rows over most SMs
  int thr = 256;
  while (thr > 32 && (a.d / kCombineCols + thr - 1) / thr * a.T < 128) thr >>= 1;
  dim3 cgrid((a.d / kCombineCols + thr - 1) / thr, a.T);
  prof_begin(DMOE_KERNEL_COMBINE, s);
  cudaError_t e =
      rows_bf16
          ? launch_ex(combine_kernel<__nv_bfloat16>, cgrid, dim3(thr), 0, s, true,
                      static_cast<const __nv_bfloat16*>(a.yslot),
                      static_cast<const __nv_bfloat16*>(a.yshared), a.pos, a.topk_gate,
                      a.y, a.k, a.d, a.Is > 0 ? 1 : 0, zero, n_zero, zero2, n_zero2,
                      meta_early ? 1 : 0)
          : launch_ex(combine_kernel<float>, cgrid, dim3(thr), 0, s, true,
                      static_cast<const float*>(a.yslot), static_cast<const float*>(a.yshared),
                      a.pos, a.topk_gate, a.y, a.k, a.d, a.Is > 0 ? 1 : 0, zero, n_zero,
                      zero2, n_zero2, meta_early ? 1 : 0);
  prof_end(DMOE_KERNEL_COMBINE, s);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace dmoe

// branch_attn_tc.cu -- the branch-attention step on 5th-generation tensor
// cores: shared prefix and private suffixes in one persistent kernel.
//
// What it computes (Sec. 3.3, "Dynamic Branch Forking and Efficient Context
// Isolation"; Sec. 3.4 for the m P-MTP queries): all query rows of a page's
// branches that read KV head g are stacked (row r <-> token
// branch_cu[d]*m + r/G, query head g*G + r%G).  Each row attends to
//   - the page's shared prefix keys [0, P_b), P_b its branch's fork-position
//     prefix length (P_d when none is given), and
//   - its own branch's private keys j <= L_b - m + i (i = the row's query).
// The page's prefix is read once per 128 stacked rows instead of once per
// branch: that is the shared-prefix KV reuse the method relies on.
//
// Key blocks: a unit walks 128-key blocks of two kinds,
//   prefix blocks  128 consecutive prefix keys: one 3-D TMA box per 64
//                  columns from the contiguous prefix, or, with a paged
//                  prefix, 8 pool pages of 16 keys from the page's prefix
//                  page table (Algorithm 1: forks share the parent's pages),
//   suffix blocks  8 pages of 16 keys, packed from the private caches of the
//                  unit's branches in branch order.
// A paged block whose 8 pages are consecutive pool pages loads as one 8-page
// box, else as one box per page, issued by 8 lanes at once (one 4 KB box per
// page instead of one per 64 columns, in a loop, took the batch with scattered
// prefix pages from 67.3 to 57.9 us per call).
// For every row and block the visible columns form one interval [lo, hi):
// a prefix block's keys below the row's limit, or the row's own branch's
// pages up to its causal bound.  Rows of other branches see nothing of a
// suffix page, so their probabilities are zero there.
//
// Work units: (row tile of 128 stacked rows, KV head, split), a split being
// an even share of the tile's blocks.  One CTA per SM takes units from an
// atomic counter, and its roles run one unit apart so that nothing drains
// between units:
//   warp 10     scheduler: takes the next unit and prepares its metadata
//               (page, rows, private lengths, fork limits, packed page ids)
//               in one of two shared-memory slots while the other is in use.
//   warps 0, 11 TMA producers: warp 0 the unit's Q tile and then its K
//               blocks, warp 11 its V blocks, each into a three-stage ring
//               (128-byte swizzle); a K stage is refilled as soon as its Q
//               K^T (or Q copy) is done, whatever the V ring waits for.
//   warps 1, 12 MMA issuers (warp 1 owns TMEM).  Warp 1 copies each unit's
//               Q tile from its K stage into TMEM (tcgen05.cp, double
//               buffered by unit) and issues
//                 S = Q K^T   Q read from TMEM, K from shared memory; S into
//                             TMEM (fp32, double buffered by block)
//               and warp 12
//                 O += P V    P read from TMEM (bf16, written over S), V from
//                             shared memory; O accumulated in TMEM
//               With both A operands in TMEM, shared memory serves only K,
//               V and their TMA writes.  (TWO: P in two bf16 parts, its
//               rounding and what that left, and two MMAs for each; see
//               launch_branch_attn_tc.)  Each warp's waits and bookkeeping
//               pass while the other's MMAs run.
//   warps 2..9  softmax: two warpgroups, each owning half of every block's
//               128 key columns and half of O's columns; thread t of warp w
//               owns TMEM lane 32*(w%4)+t, i.e. one query row.  The two
//               halves of a row exchange their partial max through shared
//               memory only in the first block that some row of the warp
//               sees keys of: that maximum is the row's base, and later
//               blocks take their exponentials against it without waiting
//               for anything.  Should a score exceed its base by more than
//               2^64, or O come out not finite, the unit runs once more with
//               running maxima in every block (O then rescaled in TMEM when
//               one grows by more than 2^8).  Which units do so is a matter of
//               their own scores and values alone, so that a call's bits do
//               not depend on which CTA took which unit.
// One split: the unit writes the final bf16 output and lse.  Several splits:
// it writes its normalised fp32 partial and lse for merge.cu.
// Code size: every CTA fetches the kernel's instructions anew, at some 150
// cycles a 128-byte line on a cold path, and the roles' hot loops share one
// instruction cache.  Code off the softmax's inner loop therefore exists
// once and keeps its loops (producers, page look-ups), and divides by
// multiplying: 124 KB of instructions became 64 KB, which took one call of
// c3's shape from 41.4 to 37.6 us, of a scattered paged batch from 75.8 to
// 68.3 us, and the attention of c5's shape from 133.3 to 129.7 us.  (77 KB
// now, with the softmax loop of its own that fully visible blocks have.)
// What bounds it: per S buffer the chain softmax, P V, S free, Q K^T, of
// 1,400-1,575 cycles a block against 1,024 of MMA, and whole units: one call
// of 152 units of 64 blocks, one for each SM, takes 61.3 us (70.6 with 2,100
// cycles a block), 256 units of the same length 110.5 us (127.1).
// All waits are bounded; a timeout sets HPD_DEVERR_TIMEOUT, every role
// leaves its loop, and the CTA drains its in-flight copies and MMAs, frees
// its TMEM and exits.  No role waits on a hardware barrier (bar.sync) inside
// its loop, so a role that leaves early cannot strand another.
#include <algorithm>
#include <atomic>

#include "tc_common.cuh"

namespace hpd {
namespace {

using namespace sm100;
using tc::kBlk;
using tc::kRows;

constexpr uint32_t kTmemCols = 512;
constexpr int kMaxUnitBranches = kRows + 1;  // branches touching 128 stacked rows
constexpr int kPageCap = 2048;               // suffix page ids kept in shared memory
constexpr int kPagesPerBlock = kBlk / kPage;
constexpr int kSoftmaxWarps = 8;
constexpr int kSchedWarp = 2 + kSoftmaxWarps;
constexpr int kVWarp = kSchedWarp + 1;
constexpr int kPvWarp = kVWarp + 1;
constexpr int kThreads = 32 * (kPvWarp + 1);
// consumers of a metadata slot: two producers, two MMA issuers, softmax warps
constexpr uint32_t kMetaConsumers = 4 + kSoftmaxWarps;
constexpr int kMaxRing = 3;  // largest K / V ring
constexpr int kStageInts = 2560;  // offsets and lengths staged in shared memory
constexpr uint64_t kBlockLimitNs = 10000;  // of a unit's time: a block takes some 0.7 us

// Metadata of one unit, written by the scheduler warp.
struct UnitMeta {
  int valid;     // 0: no units left
  int g;         // KV head
  int split;     // split index
  int tok0;      // first query token of the tile
  int nrows;     // stacked rows (ntok * G)
  int b_lo;      // first branch
  int nbc;       // branches of the rows
  int nP;        // prefix blocks
  int pc0;       // first prefix token of the page
  int blk_lo;    // first block of the split
  int n_blocks;  // blocks of the split (> 0)
  int doc;       // page (document) of the tile
  int pp_last;   // paged prefix: last prefix page any row of the tile sees
  int exact;     // every block's base is the running maximum
  int page_start[kMaxUnitBranches + 1];  // packed page offset of each branch
  int blen[kMaxUnitBranches];            // private length L_b (clamped)
  int fork[kMaxUnitBranches];            // prefix keys visible to the branch
  int page_tab[kPageCap];                // packed suffix page ids
};

template <int D>
struct TcLayout {
  static constexpr int kChunks = D / 64;                // 64-column (128-byte) boxes
  static constexpr uint32_t kChunkBytes = kRows * 128;  // 128 rows x 128 bytes
  static constexpr uint32_t kTileBytes = kChunks * kChunkBytes;
  // paged blocks: 8-key groups of kChunks x 1024 bytes instead of whole chunks
  static constexpr uint32_t kGroupBytes = kChunks * 1024, kPageBytes = 2 * kGroupBytes;
  static constexpr int kKStages = 3, kVStages = 3;
  static_assert(kKStages == kVStages, "one producer code for both rings");
  static constexpr uint32_t kK = 0;
  static constexpr uint32_t kV = kK + kKStages * kTileBytes;
  static constexpr uint32_t kMeta = kV + kVStages * kTileBytes;  // 2 UnitMeta slots
  static constexpr uint32_t kStage = kMeta + 2 * sizeof(UnitMeta);
  static constexpr uint32_t kBytes = kStage + kStageInts * sizeof(int);
  static constexpr uint32_t kDynSmem = kBytes + 1024;   // slack to align to 1024
  // TMEM columns: S of block buffer i at col_s(i), O at kColO, the Q rows of
  // unit slot u at col_q(u) (D / 2 columns: two bf16 per column)
  static constexpr uint32_t kColO = 256;
  static __device__ __forceinline__ uint32_t col_s(int i) { return i ? 128u : 0u; }
  static __device__ __forceinline__ uint32_t col_q(int u) { return u ? 448u : 384u; }
};

struct __align__(8) TcShared {
  uint64_t stage_full;
  uint64_t meta_full[2], tab_full[2], meta_empty[2];  // tab: the packed page ids
  uint64_t k_full[kMaxRing], v_full[kMaxRing];
  uint64_t k_empty[kMaxRing], v_empty[kMaxRing];
  // per S buffer: scores written; P written; P V done (the buffer is free and
  // O holds the block)
  uint64_t s_full[2], p_full[2], s_free[2];
  uint64_t o_full, o_empty;
  uint64_t mma_done[2];
  uint32_t tmem_base;
  int abort;
  // the two column halves of a row exchange their partial row max (double
  // buffered by block parity) and, at the end of a unit, their partial sums;
  // seq counters publish each value ([half][TMEM lane quadrant])
  float xmax[2][2][kRows];  // [half][block parity][row]
  float xsum[2][2][kRows];  // [unit parity][half][row]
  int xseq[2][2][4];        // [max | sum][half][quadrant]
  // units (by number in this CTA, modulo 32) whose scores left the window of
  // their base, or whose O is not finite, and that run once more, with running
  // maxima
  unsigned redo;
  int units_done;    // softmax warps that finished a unit's epilogue
  int unit_id[32];   // the last units issued
};

__device__ __forceinline__ void set_abort(TcShared &sh, uint32_t *err) {
  atomicExch(&sh.abort, 1);
  flag_error(err, HPD_DEVERR_TIMEOUT);
}
__device__ __forceinline__ bool aborted(const TcShared &sh) {
  return *reinterpret_cast<const volatile int *>(&sh.abort) != 0;
}

// Publish `seq` at *flag after this warp's earlier shared-memory writes
// (release store by lane 0 once the warp's lanes are ordered by __syncwarp).
__device__ __forceinline__ void publish_seq(int *flag, int seq) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0)
    asm volatile("st.release.cta.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(flag)), "r"(seq)
                 : "memory");
}
__device__ __forceinline__ int load_seq(const int *flag) {
  int v;
  asm volatile("ld.acquire.cta.shared::cta.b32 %0, [%1];" : "=r"(v) : "r"(smem_u32(flag)) : "memory");
  return v;
}
// Slow path of await_seq, out of line so that the clock read stays off the
// fast path.
__device__ __noinline__ bool await_seq_slow(const int *flag, int seq, const int *abort) {
  const uint64_t t0 = globaltimer();
  for (uint32_t i = 1; load_seq(flag) < seq; ++i)
    if ((i & 63u) == 0 &&
        (*reinterpret_cast<const volatile int *>(abort) || globaltimer() - t0 > kWaitLimitNs))
      return false;
  return true;
}
// Wait (bounded) until *flag >= seq, with acquire ordering; false on timeout
// or abort.
__device__ __forceinline__ bool await_seq(const int *flag, int seq, const TcShared &sh) {
  return load_seq(flag) >= seq || await_seq_slow(flag, seq, &sh.abort);
}

// Natural log of 2^m * l.
template <bool EXACT>
__device__ __forceinline__ float lse_of(float m, float l) {
  if constexpr (!EXACT) return (m + __log2f(l)) * kLn2;
  // one rounding at the result's size: the log of l's mantissa and m first
  const int e = static_cast<int>(__float_as_uint(l) >> 23) - 127;
  const float f = __uint_as_float((__float_as_uint(l) & 0x007fffffu) | 0x3f800000u);
  return fmaf(static_cast<float>(e), kLn2, fmaf(m, kLn2, logf(f)));
}

template <int D, bool TWO>
__global__ void __launch_bounds__(kThreads, 1)
    branch_attn_tc_kernel(const __grid_constant__ CUtensorMap tm_k,
                          const __grid_constant__ CUtensorMap tm_v,
                          const __grid_constant__ CUtensorMap tm_kc,
                          const __grid_constant__ CUtensorMap tm_vc,
                          const __grid_constant__ CUtensorMap tm_k8,
                          const __grid_constant__ CUtensorMap tm_v8,
                          const __grid_constant__ CUtensorMap tm_q, const AttnParams p) {
  using L = TcLayout<D>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ TcShared sh;
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t *sgen = smem_raw + (sbase - smem_u32(smem_raw));
  UnitMeta *meta = reinterpret_cast<UnitMeta *>(sgen + L::kMeta);
  // The step's offsets and lengths, when they fit: the softmax warps fetch
  // them all at once while the roles start, instead of the scheduler fetching
  // them one dependent load after another.
  int *stage = reinterpret_cast<int *>(sgen + L::kStage);
  const int n_cu = p.n_docs + 1, n_stage = 2 * n_cu + p.B * (p.branch_prefix_len ? 2 : 1);
  const bool staged = p.n_docs < kStageInts && p.B < kStageInts && n_stage <= kStageInts;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = p.G, m = p.m;
  const int TT = kRows / G;  // tokens per 128-row tile
  const float NEG_INF = -__int_as_float(0x7f800000);
  auto bar = [](uint64_t &b) { return smem_u32(&b); };
  // bounded wait on an mbarrier phase, warp-uniform outcome; false on abort
  auto wait_bar = [&](uint64_t &b, int parity) {
    return __all_sync(0xffffffffu, mbar_wait(bar(b), parity, &sh.abort));
  };

  // ------------------------------------------------------ once per CTA --
  if (tid == 0) {
    sh.abort = 0;
    sh.redo = 0u;
    sh.units_done = 0;
    for (int s = 0; s < kMaxRing; ++s) {
      mbar_init(bar(sh.k_full[s]), 1);
      mbar_init(bar(sh.v_full[s]), 1);
      mbar_init(bar(sh.k_empty[s]), 1);
      mbar_init(bar(sh.v_empty[s]), 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(bar(sh.meta_full[s]), 1);
      mbar_init(bar(sh.tab_full[s]), 1);
      mbar_init(bar(sh.meta_empty[s]), kMetaConsumers);
      mbar_init(bar(sh.s_full[s]), 1);
      mbar_init(bar(sh.p_full[s]), kSoftmaxWarps);
      mbar_init(bar(sh.s_free[s]), 1);
    }
    mbar_init(bar(sh.stage_full), 32 * kSoftmaxWarps);
    mbar_init(bar(sh.o_full), 1);
    mbar_init(bar(sh.o_empty), kSoftmaxWarps);
    mbar_init(bar(sh.mma_done[0]), 1);
    mbar_init(bar(sh.mma_done[1]), 1);
    fence_mbar_init();
  }
  if (tid < 16) (&sh.xseq[0][0][0])[tid] = 0;
  if (warp == 1) {
    tmem_alloc(smem_u32(&sh.tmem_base), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem_base;
  pdl_wait();     // the unit order (and everything before it) is complete
  pdl_trigger();  // the merge of the splits may launch; it waits for this grid

  if (warp == kSchedWarp) {
    // ------------------------------------------------------- scheduler --
    // Fills slot k & 1 with the k-th unit of this CTA that has keys; units
    // without any get their output written here and are skipped.
    const int *const branch_cu = staged ? stage : p.branch_cu;
    const int *const prefix_cu = staged ? stage + n_cu : p.prefix_cu;
    const int *const branch_len = staged ? stage + 2 * n_cu : p.branch_len;
    const int *const fork_len =
        staged && p.branch_prefix_len ? stage + 2 * n_cu + p.B : p.branch_prefix_len;
    bool fetched = !staged;
    unsigned redo = 0;  // units to run once more
    int nb_last = 0, nb_before = 0;  // blocks of the last two units
    // (The softmax warps write the words read here meanwhile: one lane reads
    // for all, so that the warp never takes two ways at once.)
    auto take_redo = [&] {
      unsigned r = 0;
      if (lane == 0 && *static_cast<volatile unsigned *>(&sh.redo)) r = atomicExch(&sh.redo, 0u);
      return __shfl_sync(0xffffffffu, r, 0);
    };
    for (int k = 0;; ++k) {
      const int slot = k & 1;
      if (k >= 2 && !wait_bar(sh.meta_empty[slot], ((k >> 1) - 1) & 1)) {
        if (lane == 0) set_abort(sh, p.err);
        break;
      }
      UnitMeta &M = meta[slot];
      bool have = false;
      for (;;) {
        int u = 0;
        if (!redo) redo = take_redo();
        const bool again = redo != 0;
        if (again) {
          u = sh.unit_id[__ffs(redo) - 1];
          redo &= redo - 1;
        } else {
          if (lane == 0) u = atomicAdd(p.unit_ctr, 1);
          u = __shfl_sync(0xffffffffu, u, 0);
          if (__any_sync(0xffffffffu, aborted(sh))) break;
          if (u >= p.n_units) {
            // none left, once the units still running (the last two) need no
            // second pass; who gives up here has set the abort word and the error
            const uint64_t limit =
                kWaitLimitNs + (static_cast<uint64_t>(nb_last) + nb_before) * kBlockLimitNs;
            if (!__all_sync(0xffffffffu,
                            await_count(smem_u32(&sh.units_done), kSoftmaxWarps * k, &sh.abort,
                                        p.err, HPD_DEVERR_TIMEOUT, limit)))
              break;
            redo = take_redo();
            if (!redo) break;
            continue;
          }
          if (p.unit_order) u = p.unit_order[u];  // longest units first
        }
        const int u_id = u;
        if (!fetched) {
          if (!wait_bar(sh.stage_full, 0)) {
            if (lane == 0) set_abort(sh, p.err);
            break;
          }
          fetched = true;
        }
        const int us = p.div_S(u), split = u - us * p.S_p;
        const int tile = p.div_Hkv(us), g = us - tile * p.H_kv;
        // the page owning the tile: page d has ceil(#branches(d) * m / TT) tiles
        int d = -1, lt = 0, b0 = 0, b1 = 0;
#pragma unroll 1
        for (int d0 = 0, base = 0; d0 < p.n_docs && base <= tile; d0 += 32) {
          const int dd = d0 + lane;
          int tiles = 0, c0 = 0, c1 = 0;
          if (dd < p.n_docs) {
            c0 = min(max(branch_cu[dd], 0), p.B);
            c1 = min(max(branch_cu[dd + 1], 0), p.B);
            if (c1 < c0) {
              flag_error(p.err, HPD_DEVERR_BRANCH_CU);
              c1 = c0;
            }
            tiles = p.div_tile((c1 - c0) * m + TT - 1);
          }
          int incl = tiles;
#pragma unroll 1
          for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
          }
          const int excl = incl - tiles;
          const unsigned hit =
              __ballot_sync(0xffffffffu, tiles > 0 && tile >= base + excl && tile < base + incl);
          if (hit) {
            const int src = __ffs(hit) - 1;
            d = __shfl_sync(0xffffffffu, dd, src);
            lt = __shfl_sync(0xffffffffu, tile - base - excl, src);
            b0 = __shfl_sync(0xffffffffu, c0, src);
            b1 = __shfl_sync(0xffffffffu, c1, src);
            break;
          }
          base += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (d < 0) continue;
        int pc0, P_d;
        bool bad_prefix;
        page_prefix(p, prefix_cu, d, pc0, P_d, bad_prefix);
        if (lane == 0 && bad_prefix) flag_error(p.err, HPD_DEVERR_PREFIX_CU);
        const int tok0 = b0 * m + lt * TT;
        const int ntok = min(TT, (b1 - b0) * m - lt * TT);
        const int b_lo = p.div_m(tok0);
        const int nbc = p.div_m(tok0 + ntok - 1) - b_lo + 1;
        // private lengths, packed page offsets and fork limits of the branches
        int base = 0, kmax = 0;
#pragma unroll 1
        for (int c0 = 0; c0 < nbc; c0 += 32) {
          const int bl = c0 + lane;
          int np = 0;
          if (bl < nbc) {
            int Lb = branch_len[b_lo + bl];
            const int cap = p.max_pages * kPage;
            if (Lb < 0 || Lb > cap) {
              flag_error(p.err, HPD_DEVERR_BRANCH_LEN);
              Lb = min(max(Lb, 0), cap);
            }
            int f = P_d;
            if (fork_len) {
              f = fork_len[b_lo + bl];
              if (f < 0 || f > P_d) {
                flag_error(p.err, HPD_DEVERR_FORK_LEN);
                f = min(max(f, 0), P_d);
              }
            }
            M.blen[bl] = Lb;
            M.fork[bl] = f;
            kmax = max(kmax, f);
            np = ceil_div_i(Lb, kPage);
          }
          int incl = np;
#pragma unroll 1
          for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
          }
          if (bl < nbc) M.page_start[bl] = base + incl - np;
          base += __shfl_sync(0xffffffffu, incl, 31);
        }
        kmax = __reduce_max_sync(0xffffffffu, kmax);
        const int P_s = base;
        if (lane == 0) M.page_start[nbc] = P_s;
        __syncwarp();
        const int N = ceil_div_i(kmax, kBlk) + ceil_div_i(P_s, kPagesPerBlock);
        // (a unit has fewer than 2^27 blocks and at most 8 splits)
        const int blk_lo = p.div_S(split * N), blk_hi = p.div_S((split + 1) * N);
        const int nrows = ntok * G;
        if (blk_hi <= blk_lo) {
          // no key in this split: zero output (one split) or an empty partial
#pragma unroll 1
          for (int r = lane; r < nrows; r += 32) {
            const int rt = p.div_G(r);
            const size_t pair = static_cast<size_t>(tok0 + rt) * p.H_q + g * G + r - rt * G;
            if (p.S_p == 1) {
              uint4 *o = reinterpret_cast<uint4 *>(p.out + pair * D);
#pragma unroll 1
              for (int c = 0; c < D / 8; ++c) o[c] = make_uint4(0u, 0u, 0u, 0u);
              if (p.lse) p.lse[pair] = NEG_INF;
            } else {
              p.l_part[static_cast<size_t>(split) * p.rows_total * p.H_q + pair] = NEG_INF;
            }
          }
          continue;
        }
        if (lane == 0) {
          M.valid = 1;
          M.g = g;
          M.split = split;
          M.tok0 = tok0;
          M.nrows = nrows;
          M.b_lo = b_lo;
          M.nbc = nbc;
          M.nP = ceil_div_i(kmax, kBlk);
          M.pc0 = pc0;
          M.doc = d;
          M.pp_last = max(kmax - 1, 0) / kPage;
          M.blk_lo = blk_lo;
          M.n_blocks = blk_hi - blk_lo;
          M.exact = again;
          sh.unit_id[k & 31] = u_id;
        }
        nb_before = nb_last;
        nb_last = blk_hi - blk_lo;
        // published without the page ids, which only suffix blocks need
        __syncwarp();
        __threadfence_block();
        if (lane == 0) mbar_arrive(bar(sh.meta_full[slot]));
        // packed suffix page ids: every lookup in flight, then the valid ones kept
        const int n_tab = min(P_s, kPageCap);
#pragma unroll 1
        for (int gp = lane; gp < n_tab; gp += 32) {
          int lo = 0, hi = nbc;  // largest bl with page_start[bl] <= gp
          while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (M.page_start[mid] <= gp) lo = mid; else hi = mid;
          }
          cp_async4(smem_u32(&M.page_tab[gp]),
                    p.page_table + static_cast<size_t>(b_lo + lo) * p.max_pages +
                        (gp - M.page_start[lo]));
        }
        cp_async_commit();
        cp_async_wait<0>();
#pragma unroll 1
        for (int gp = lane; gp < n_tab; gp += 32)
          if (static_cast<unsigned>(M.page_tab[gp]) >= static_cast<unsigned>(p.num_pages)) {
            flag_error(p.err, HPD_DEVERR_PAGE_ID);
            M.page_tab[gp] = 0;
          }
        have = true;
        break;
      }
      if (!have && lane == 0) M.valid = 0;
      __syncwarp();
      __threadfence_block();
      if (lane == 0) mbar_arrive(have ? bar(sh.tab_full[slot]) : bar(sh.meta_full[slot]));
      if (!have) break;
    }
  } else if (warp == 0 || warp == kVWarp) {
    // ------------------------------------------------------- producers --
    // The whole warp runs this loop with warp-uniform values; one elected
    // lane issues each copy.  Warp 0: Q and K; warp kVWarp: V.  The K ring
    // carries each unit's Q tile ahead of its K blocks, as one more entry.
    const bool is_k = warp == 0;
    if (lane == 0) {
      prefetch_tmap(&tm_q);
      prefetch_tmap(&tm_k);
      prefetch_tmap(&tm_v);
      prefetch_tmap(&tm_kc);
      prefetch_tmap(&tm_vc);
      prefetch_tmap(&tm_k8);
      prefetch_tmap(&tm_v8);
    }
    __syncwarp();
    // (one copy of this code, loops left as loops: a CTA of a small step runs
    // it once or twice, and is bound by fetching its instructions)
    uint64_t *const full = is_k ? sh.k_full : sh.v_full, *const empty = is_k ? sh.k_empty : sh.v_empty;
    const CUtensorMap *const prefix_map = is_k ? &tm_k : &tm_v;
    const CUtensorMap *const page_map = is_k ? &tm_kc : &tm_vc;
    const CUtensorMap *const run_map = is_k ? &tm_k8 : &tm_v8;
    const uint32_t ring = sbase + (is_k ? L::kK : L::kV);
    const bool paged_prefix = p.prefix_page_table != nullptr;
    int issued = 0;  // ring entries
    bool ok = true;
    for (int k = 0; ok; ++k) {
      const int slot = k & 1;
      if (!(ok = wait_bar(sh.meta_full[slot], (k >> 1) & 1))) break;
      const UnitMeta &M = meta[slot];
      if (!M.valid) break;
      const int g = M.g, nP = M.nP, pc0 = M.pc0, blk_lo = M.blk_lo, nb = M.n_blocks;
      const int P_s = M.page_start[M.nbc];
      bool tab = false;  // the packed page ids are complete
      // entry -1 of the K ring: the unit's Q tile, tokens [tok0, tok0 + TT),
      // heads of KV head g
#pragma unroll 1
      for (int j = is_k ? -1 : 0; j < nb; ++j) {
        const int jb = blk_lo + j;
        const bool contiguous = j < 0 || (jb < nP && !paged_prefix);
        // A paged block is 8 pages (lane i < 8 holds page i, looked up before
        // waiting for the ring slot); pages past the last one any row sees
        // repeat it (finite values, never visible).
        int pg = 0;
        if (!contiguous && jb >= nP && !tab) {
          if (!(ok = wait_bar(sh.tab_full[slot], (k >> 1) & 1))) break;
          tab = true;
        }
        if (!contiguous && lane < kPagesPerBlock) {
          if (jb < nP) {
            pg = prefix_page(p, M.doc, min(jb * kPagesPerBlock + lane, M.pp_last));
          } else {
            const int gp = min((jb - nP) * kPagesPerBlock + lane, P_s - 1);
            if (gp < kPageCap) {
              pg = M.page_tab[gp];
            } else {  // past the shared-memory table: looked up again
              int lo = 0, hi = M.nbc;
              while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (M.page_start[mid] <= gp) lo = mid; else hi = mid;
              }
              pg = p.page_table[static_cast<size_t>(M.b_lo + lo) * p.max_pages +
                                (gp - M.page_start[lo])];
              if (pg < 0 || pg >= p.num_pages) {
                flag_error(p.err, HPD_DEVERR_PAGE_ID);
                pg = 0;
              }
            }
          }
        }
        const int e = issued, s = e % L::kKStages;
        if (e >= L::kKStages && !(ok = wait_bar(empty[s], ((e / L::kKStages) - 1) & 1))) break;
        ++issued;
        const uint32_t dst = ring + s * L::kTileBytes, b = bar(full[s]);
        mbar_arrive_expect_tx_elect(b, j < 0 ? L::kChunks * TT * G * 128 : L::kTileBytes);
        if (contiguous) {
#pragma unroll 1
          for (int c = 0; c < L::kChunks; ++c)
            tma_load_3d_elect(dst + c * L::kChunkBytes, j < 0 ? &tm_q : prefix_map, b, c * 64,
                              j < 0 ? g * G : g, j < 0 ? M.tok0 : pc0 + jb * kBlk);
          continue;
        }
        // consecutive pool pages load as one 8-page box, else one box per page
        const int next = __shfl_down_sync(0xffffffffu, pg, 1);
        const unsigned run =
            __ballot_sync(0xffffffffu, lane < kPagesPerBlock - 1 && next == pg + 1);
        const bool one = p.num_pages >= kPagesPerBlock && (run & 0x7fu) == 0x7fu;
        if (lane < (one ? 1 : kPagesPerBlock))  // each lane its page
          tma_load_5d(dst + lane * L::kPageBytes, one ? run_map : page_map, b, 0, 0, 0, 2 * pg, g);
        __syncwarp();
      }
      if (ok && !tab) ok = wait_bar(sh.tab_full[slot], (k >> 1) & 1);  // written before reuse
      if (!ok) break;
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(sh.meta_empty[slot]));
    }
    if (!ok && lane == 0) set_abort(sh, p.err);
    // Do not exit while a copy into this CTA's shared memory is in flight:
    // wait for the most recent phase of every barrier a copy may complete.
    for (int e = max(0, issued - L::kKStages); e < issued; ++e)
      mbar_wait(bar(full[e % L::kKStages]), (e / L::kKStages) & 1);
  } else if (warp == 1) {
    // ---------------------------------------------------- Q K^T issuer --
    // The whole warp runs this loop with warp-uniform values; one elected
    // lane issues each group of MMAs and its commits (see sm100.cuh).  Stages
    // and phases advance by counting: the warp's own instructions between the
    // MMAs are time the tensor cores may idle.
    constexpr uint32_t idesc_qk = idesc_bf16_f32(kRows, kBlk, false);
    // Shared-memory descriptors: a stage / k-step offset only adds (offset >>
    // 4) to the start-address field (bits 0-13), which cannot carry: every
    // address stays below 256 KB.
    const uint64_t dk0 = smem_desc_sw128(sbase + L::kK, 16, 1024);
    const uint64_t dk0_paged = smem_desc_sw128(sbase + L::kK, 16, L::kGroupBytes);
    const bool issuer = elect_one();
    uint32_t sk = 0, pk = 0;  // K ring: stage, phase
    int jg = 0;               // blocks issued
    bool ok = true;
    for (int k = 0; ok; ++k) {
      const int slot = k & 1;
      if (!(ok = wait_bar(sh.meta_full[slot], (k >> 1) & 1))) break;
      const bool valid = meta[slot].valid != 0;
      const int nb = meta[slot].n_blocks;
      // first paged block of the unit
      const int j_paged = p.prefix_page_table ? 0 : meta[slot].nP - meta[slot].blk_lo;
      __syncwarp();
      if (!valid) break;
      if (lane == 0) mbar_arrive(bar(sh.meta_empty[slot]));
      // entry -1 of the unit: its Q, copied into TMEM slot k & 1 (in order
      // with the MMAs: unit k - 2's Q K^T are done with the slot)
      for (int j = -1; j < nb; ++j) {
        if (!(ok = wait_bar(sh.k_full[sk], pk))) break;
        // the S buffer is free once P V of the block before last has read P
        if (j >= 0 && jg >= 2 && !(ok = wait_bar(sh.s_free[jg & 1], ((jg >> 1) - 1) & 1))) break;
        tc_fence_after();
        if (issuer) {
          const bool paged = j >= 0 && j >= j_paged;
          const uint64_t kd = (paged ? dk0_paged : dk0) + ((sk * L::kTileBytes) >> 4);
          const uint32_t chunk = paged ? 1024 : L::kChunkBytes;
          if (j < 0) {
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk)
              tmem_cp_128x256b(tmem + L::col_q(slot) + kk * 8,
                               kd + (((kk >> 2) * L::kChunkBytes + (kk & 3) * 32) >> 4));
          } else {  // (kk >> 2: the 64-column chunk)
            // A from TMEM, 16 dimensions (8 columns) per MMA; K is K-major
            const uint32_t col = tmem + L::col_s(jg & 1);
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk)
              mma_ts_one(col, tmem + L::col_q(slot) + kk * 8,
                         kd + (((kk >> 2) * chunk + (kk & 3) * 32) >> 4), idesc_qk, kk > 0);
            mma_commit_one(bar(sh.s_full[jg & 1]));
          }
          mma_commit_one(bar(sh.k_empty[sk]));
        }
        __syncwarp();
        if (++sk == L::kKStages) {
          sk = 0;
          pk ^= 1u;
        }
        jg += j >= 0;
      }
    }
    if (!ok && lane == 0) set_abort(sh, p.err);
  } else if (warp == kPvWarp) {
    // ------------------------------------------------------ P V issuer --
    constexpr uint32_t idesc_pv = idesc_bf16_f32(kRows, D, true);
    // V is MN-major (D contiguous): 64-column swizzle atoms kChunkBytes apart
    // along N (leading byte offset), 8-key groups 1024 bytes apart along K
    // (stride byte offset).
    const uint64_t dv0 = smem_desc_sw128(sbase + L::kV, L::kChunkBytes, 1024);
    const uint64_t dv0_paged = smem_desc_sw128(sbase + L::kV, 1024, L::kGroupBytes);
    const bool issuer = elect_one();
    uint32_t sv = 0, pv = 0;  // V ring: stage, phase
    int jg = 0;               // blocks issued
    bool ok = true;
    for (int k = 0; ok; ++k) {
      const int slot = k & 1;
      if (!(ok = wait_bar(sh.meta_full[slot], (k >> 1) & 1))) break;
      const bool valid = meta[slot].valid != 0;
      const int nb = meta[slot].n_blocks;
      const int j_paged = p.prefix_page_table ? 0 : meta[slot].nP - meta[slot].blk_lo;
      __syncwarp();
      if (!valid) break;
      if (lane == 0) mbar_arrive(bar(sh.meta_empty[slot]));
      // O last held the unit before, whose epilogue must have read it
      if (k >= 1 && !(ok = wait_bar(sh.o_empty, (k - 1) & 1))) break;
      for (int j = 0; j < nb; ++j) {
        if (!(ok = wait_bar(sh.v_full[sv], pv))) break;
        if (!(ok = wait_bar(sh.p_full[jg & 1], (jg >> 1) & 1))) break;
        tc_fence_after();
        if (issuer) {
          // O (+)= P V: 16 keys per MMA, P in the S buffer (half h of the keys
          // at column 64 h)
          const uint64_t vd = (j >= j_paged ? dv0_paged : dv0) + ((sv * L::kTileBytes) >> 4);
          const uint32_t step = (j >= j_paged ? 2 * L::kGroupBytes : 2048u) >> 4;  // 16 keys
          const uint32_t col = tmem + L::col_s(jg & 1);
#pragma unroll
          for (int kk = 0; kk < kBlk / 16; ++kk)
            mma_ts_one(tmem + L::kColO, col + kk * 8 + (kk >= 4 ? 32 : 0),
                       vd + kk * step, idesc_pv, (j > 0 || kk > 0) ? 1u : 0u);
          if constexpr (TWO) {
#pragma unroll
            for (int kk = 0; kk < kBlk / 16; ++kk)
              mma_ts_one(tmem + L::kColO, col + 32 + kk * 8 + (kk >= 4 ? 32 : 0), vd + kk * step,
                         idesc_pv, 1u);
          }
          mma_commit_one(bar(sh.s_free[jg & 1]));
          mma_commit_one(bar(sh.v_empty[sv]));
          if (j == nb - 1) mma_commit_one(bar(sh.o_full));
        }
        __syncwarp();
        if (++sv == L::kVStages) {
          sv = 0;
          pv ^= 1u;
        }
        ++jg;
      }
    }
    if (!ok && lane == 0) set_abort(sh, p.err);
  } else {
    // --------------------------------------------------------- softmax --
    // Warpgroup half h owns key columns [64 h, 64 h + 64) of every block and
    // output columns [64 h, 64 h + 64).
    const int h = (warp - 2) >> 2;        // column half
    if (staged) {
#pragma unroll 1
      for (int i = tid - 64; i < n_stage; i += 32 * kSoftmaxWarps) {
        const int *src = i < n_cu              ? p.branch_cu + i
                         : i < 2 * n_cu        ? p.prefix_cu + (i - n_cu)
                         : i < 2 * n_cu + p.B  ? p.branch_len + (i - 2 * n_cu)
                                               : p.branch_prefix_len + (i - 2 * n_cu - p.B);
        cp_async4(smem_u32(stage + i), src);
      }
    }
    cp_async_mbar_arrive(bar(sh.stage_full));
    const int quad = warp & 3;            // TMEM lane quadrant this warp may access
    const int r_in = quad * 32 + lane;    // row within the tile
    const uint32_t t_lane = tmem + (static_cast<uint32_t>(quad * 32) << 16);
    const float sl2 = p.scale_log2;
    // This thread's row of a unit: where it reads Q and writes the output,
    // and its visible keys (prefix below lim_p; own branch's private keys
    // j <= last, which start at packed page ps).
    struct Row {
      bool unit;  // false: no unit left
      bool valid, exact;
      int g, split, nb, blk_lo, nP, lim_p, ps, last;
      int n_plain;  // leading prefix blocks of which every row of the warp sees all keys
      size_t pair;
    };
    // Reads unit k's metadata (slot k & 1) and releases the slot (the unit's
    // Q reaches TMEM through the K ring and the MMA warp); false on timeout /
    // abort.
    auto begin_unit = [&](int k, Row &R) -> bool {
      const int slot = k & 1;
      if (!wait_bar(sh.meta_full[slot], (k >> 1) & 1)) return false;
      const UnitMeta &M = meta[slot];
      R.unit = M.valid != 0;
      if (R.unit) {
        R.g = M.g;
        R.split = M.split;
        R.nb = M.n_blocks;
        R.blk_lo = M.blk_lo;
        R.nP = M.nP;
        R.valid = r_in < M.nrows;
        R.exact = M.exact != 0;
        const int rt = p.div_G(r_in), token = M.tok0 + rt;
        const int bl = R.valid ? p.div_m(token) - M.b_lo : 0;
        // (rows that are no query count as seeing the whole prefix, so that
        // their warp needs no masks there; their results are not stored)
        R.lim_p = R.valid ? M.fork[bl] : R.nP * kBlk;
        R.n_plain = sl2 > 0.f ? __reduce_min_sync(0xffffffffu, R.lim_p) / kBlk : 0;
        R.ps = R.valid ? M.page_start[bl] : 0;
        R.last = R.valid ? M.blen[bl] - m + (token - (M.b_lo + bl) * m) : -1;
        R.pair = static_cast<size_t>(token) * p.H_q + R.g * G + r_in - rt * G;
      }
      __syncwarp();
      if (R.unit && lane == 0) mbar_arrive(bar(sh.meta_empty[slot]));
      return true;
    };
    const uint32_t o_col = L::kColO + h * (D / 2);
    int jbase = 0;
    Row cur{};
    bool ok = true;
    for (int k = 0; ok; ++k) {
      if (!(ok = begin_unit(k, cur)) || !cur.unit) break;
      float m_run = NEG_INF, l_half = 0.f;
      bool inside = true;  // the scores stay in the window of their base
      // A row's base is the maximum of the first block it sees keys of; both
      // halves come to the same answer when that is, and take that block's
      // maximum together (exact: every block's).
      bool based = false;  // every row of the warp has its base
      // the scores of half a block are ready; its P is
      auto await_s = [&](int jg) {
        if (!wait_bar(sh.s_full[jg & 1], (jg >> 1) & 1)) return false;
        tc_fence_after();
        return true;
      };
      auto signal_p = [&](int jg) {
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(sh.p_full[jg & 1]));
      };
      for (int j = 0; j < cur.nb; ++j) {
        // blocks that every row of the warp sees all of, once the bases are
        // there: nothing to decide
        if (based && !cur.exact) {
          const int j_plain = min(cur.nb, cur.n_plain - cur.blk_lo);
          for (; j < j_plain; ++j) {
            const int jg = jbase + j;
            if (!(ok = await_s(jg))) break;
            inside &= tc::softmax_half_based<TWO>(t_lane + L::col_s(jg & 1) + h * 64, true, 0, kBlk, sl2,
                                             m_run, l_half);
            signal_p(jg);
          }
          if (!ok || j >= cur.nb) break;
        }
        const int jg = jbase + j;
        const int si = jg & 1;
        const int jb = cur.blk_lo + j;
        int lo = 0, hi;
        if (jb < cur.nP) {
          hi = min(cur.lim_p - jb * kBlk, kBlk);
        } else {
          const int off = (cur.ps - (jb - cur.nP) * kPagesPerBlock) * kPage;  // column of own key 0
          lo = max(0, off);
          hi = min(kBlk, off + cur.last + 1);
        }
        const bool find_max =
            cur.exact ||
            (!based && __any_sync(0xffffffffu, cur.valid && m_run == NEG_INF && hi > lo));
        // warp-uniform outcome: the tcgen05.ld / st below are warp-collective
        if (!(ok = await_s(jg))) break;
        const uint32_t s_addr = t_lane + L::col_s(si) + h * 64;
        bool rescale = false;
        float alpha = 1.f;
        if (!find_max) {
          inside &= tc::softmax_half_based<TWO>(s_addr, false, lo - h * 64, hi - h * 64, sl2, m_run, l_half);
        } else {
          const int par = jg & 1;
          bool xok = true;
          auto xchg = [&](float mx) {
            sh.xmax[h][par][r_in] = mx;
            publish_seq(&sh.xseq[0][h][quad], jg + 1);
            xok = await_seq(&sh.xseq[0][h ^ 1][quad], jg + 1, sh);
            return fmaxf(mx, sh.xmax[h ^ 1][par][r_in]);
          };
          alpha = tc::softmax_half_max<TWO>(s_addr, lo - h * 64, hi - h * 64, sl2, m_run, l_half, xchg);
          if (!(ok = __all_sync(0xffffffffu, xok))) break;
          rescale = __any_sync(0xffffffffu, j > 0 && alpha != 1.f);
          based = __all_sync(0xffffffffu, !cur.valid || m_run != NEG_INF);
        }
        // Before O may be rescaled, the P V MMA of block jg-1 must have
        // landed: a warp that rescales waits for it.  The test is exact: P V
        // (jg + 1) of the same buffer needs this block's P V first.
        if (rescale) {
          if (!(ok = wait_bar(sh.s_free[si ^ 1], ((jg - 1) >> 1) & 1))) break;
          tc_fence_after();
#pragma unroll 1
          for (int c = 0; c < D / 2; c += 32) {
            uint32_t o[32];
            tmem_ld32(t_lane + o_col + c, o);
            tmem_ld_wait32(o);
#pragma unroll
            for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
            tmem_st32(t_lane + o_col + c, o);
          }
        }
        signal_p(jg);
      }
      if (!ok) break;
      // ---------------------------------------------------- epilogue --
      // row sum over both halves
      // (Two buffers in turn: a half may be a unit of one or two blocks, of
      // which its rows see nothing, ahead of the other, which exchange nothing
      // and need no P of the other's; not two units, as it awaits the other's
      // sum of the first.)
      sh.xsum[k & 1][h][r_in] = l_half;
      publish_seq(&sh.xseq[1][h][quad], k + 1);
      if (!(ok = __all_sync(0xffffffffu, await_seq(&sh.xseq[1][h ^ 1][quad], k + 1, sh)))) break;
      const float l_run = l_half + sh.xsum[k & 1][h ^ 1][r_in];
      if (!(ok = wait_bar(sh.o_full, k & 1))) break;
      tc_fence_after();
      const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
      const float lse = l_run > 0.f ? lse_of<TWO>(m_run, l_run) : NEG_INF;
      const bool final_out = p.S_p == 1;
      const size_t slot_pair = static_cast<size_t>(cur.split) * p.rows_total * p.H_q + cur.pair;
      float2 finite = make_float2(0.f, 0.f);  // NaN once an infinity or NaN is added
#pragma unroll 1
      for (int c = 0; c < D / 2; c += 32) {
        uint32_t o[32];
        tmem_ld32(t_lane + o_col + c, o);
        tmem_ld_wait32(o);
        if (!cur.valid) continue;
#pragma unroll
        for (int e = 0; e < 32; e += 2)
          finite = __ffma2_rn(make_float2(__uint_as_float(o[e]), __uint_as_float(o[e + 1])),
                              make_float2(0.f, 0.f), finite);
        const int dc = h * (D / 2) + c;  // output column
        // 32-byte stores: each fills a whole sector of its row
        if (final_out) {
          uint32_t w[16];
#pragma unroll
          for (int e = 0; e < 16; ++e)
            w[e] = pack_bf16x2(__uint_as_float(o[2 * e]) * inv, __uint_as_float(o[2 * e + 1]) * inv);
          __nv_bfloat16 *dst = p.out + cur.pair * D + dc;
          if (p.out_align32) {
            st_global_v8(dst, w);
            st_global_v8(dst + 16, w + 8);
          } else {
#pragma unroll
            for (int e = 0; e < 16; e += 4)
              reinterpret_cast<uint4 *>(dst)[e / 4] = make_uint4(w[e], w[e + 1], w[e + 2], w[e + 3]);
          }
        } else {
          float *dst = p.o_part + slot_pair * D + dc;
#pragma unroll
          for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * inv);
#pragma unroll
          for (int e = 0; e < 32; e += 8) st_global_v8(dst + e, o + e);
        }
      }
      if (cur.valid && h == 0) {
        if (final_out) {
          if (p.lse) p.lse[cur.pair] = lse;
        } else {
          p.l_part[slot_pair] = lse;
        }
      }
      // Scores out of the window, or an O that may have overflowed (weights of
      // up to 2^64 times values beyond 2^63): the unit runs once more.
      const bool again =
          !cur.exact && cur.valid && (!inside || !(finite.x == 0.f && finite.y == 0.f));
      const bool redo = __any_sync(0xffffffffu, again);
      // O may be overwritten by the next unit once every warp has read it
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(bar(sh.o_empty));
        if (redo) atomicOr(&sh.redo, 1u << (k & 31));
        __threadfence_block();
        atomicAdd(&sh.units_done, 1);
      }
      jbase += cur.nb;
    }
    if (!ok && lane == 0) set_abort(sh, p.err);
    // Do not exit while a staged copy or its arrival is in flight: only a
    // scheduler that gets a unit waits for them.
    mbar_wait(bar(sh.stage_full), 0);
  }

  // ------------------------------------------------------------ teardown --
  // every MMA issued by this CTA has finished before TMEM is released
  if (warp == 1 || warp == kPvWarp) {
    uint64_t &done = sh.mma_done[warp == 1 ? 0 : 1];
    mma_commit(bar(done));
    mbar_wait(bar(done), 0);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
  // the last CTA to finish resets the unit counters for the next call
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(p.unit_ctr + 1, 1) == static_cast<int>(gridDim.x) - 1) {
      atomicExch(p.unit_ctr, 0);
      atomicExch(p.unit_ctr + 1, 0);
    }
  }
}

template <int D, bool TWO>
cudaError_t launch_tc(const AttnParams &p, bool overlap, cudaStream_t s) {
  using L = TcLayout<D>;
  static_assert(L::kDynSmem + sizeof(TcShared) <= 227 * 1024, "shared memory");
  CUtensorMap tk, tv, tkc, tvc, tk8, tv8, tq;
  cudaError_t e = tc::make_prefix_maps(p, &tk, &tv);
  if (e == cudaSuccess) e = tc::make_q_map(p, &tq);
  if (e == cudaSuccess) e = tc::make_page_map(&tkc, p.k_cache, D, p.H_kv, p.num_pages);
  if (e == cudaSuccess) e = tc::make_page_map(&tvc, p.v_cache, D, p.H_kv, p.num_pages);
  const int run = std::min(kPagesPerBlock, p.num_pages);  // box never longer than the pool
  if (e == cudaSuccess) e = tc::make_page_map(&tk8, p.k_cache, D, p.H_kv, p.num_pages, run);
  if (e == cudaSuccess) e = tc::make_page_map(&tv8, p.v_cache, D, p.H_kv, p.num_pages, run);
  if (e != cudaSuccess) return e;
  static std::atomic<uint64_t> configured{0};
  int dev = 0;
  e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = 1ull << (dev & 63);
  if (!(configured.load(std::memory_order_acquire) & bit)) {
    e = cudaFuncSetAttribute(branch_attn_tc_kernel<D, TWO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(L::kDynSmem));
    if (e != cudaSuccess) return e;
    configured.fetch_or(bit, std::memory_order_acq_rel);
  }
  static int sms[64] = {0};
  if (sms[dev & 63] == 0) {
    int n = 0;
    e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    sms[dev & 63] = n;
  }
  const dim3 grid(static_cast<unsigned>(std::min(p.n_units, sms[dev & 63])), 1, 1);
  return launch_kernel(overlap, branch_attn_tc_kernel<D, TWO>, grid, dim3(kThreads), L::kDynSmem, s,
                       tk, tv, tkc, tvc, tk8, tv8, tq, p);
}

}  // namespace

cudaError_t launch_branch_attn_tc(const AttnParams &p, const Plan &plan, bool overlap,
                                  cudaStream_t s) {
  if (plan.tiles_max <= 0 || p.n_units <= 0) return cudaSuccess;
  // Head ratios that do not divide 128 have their weights in two bf16 parts.
  // Their calls came to this kernel from the warp-MMA stages, whose running
  // maxima and merged splits left smaller errors than one rounding against a
  // fixed base: against 64 bits, over 68 random calls, the outputs were off by
  // 1.010 of what they had been and the lse by 1.18; with two parts, and a log of
  // one rounding, by 0.71 and 0.57.  It costs the second half of P V: 77
  // branches of m = 3 on 3 pages, 40 / 8 heads, 30.2 -> 38.6 us (warp MMA 88).
  if (kRows % p.G != 0)
    return p.D == 64 ? launch_tc<64, true>(p, overlap, s) : launch_tc<128, true>(p, overlap, s);
  return p.D == 64 ? launch_tc<64, false>(p, overlap, s) : launch_tc<128, false>(p, overlap, s);
}

}  // namespace hpd

// ttc_kernels.cu -- the hot path of the adaptive TT cross on sm_103a.
//
// One sweep (all bonds at once, Sec. 3.2.3) is three phases:
//   screen : every CTA takes superblock tiles of every bond (the paper's
//            subtensors of Alg. 3 become CTA tiles), generates the entries,
//            forms E = A - T R with the FP64 FMA chain of the arithmetic
//            contract (or the FP32 / float-float forms), and keeps the tile's
//            max |E| (ties: lowest column-major linear index);
//   decide : one CTA per instance merges the tile candidates (the Allgather
//            of Alg. 3), applies the stop test and appends the pivots:
//            nested index sets (eq. nestedpivots) and pivot history;
//   update : every CTA applies eq. aca_approx_T_sub to the old rows of T,
//            replays the pivot history on rows that entered the superblock
//            (Alg. 4), borders P^{-1} (Sherman-Morrison, Sec. 3.1.1), and
//            generates the new rows / columns of R; or, when an instance has
//            converged at its threshold, the sampled error of Sec. 5 is
//            evaluated.
// The phases run either in one persistent cooperative launch separated by
// grid barriers (every wait bounded in time) or as separate launches.
#include <algorithm>
#include <cfloat>
#include <climits>
#include <memory>
#include <vector>

#include "ttc_gen.cuh"
#include "ttc_internal.cuh"
#include "ttc_launch.h"

namespace ttc {

constexpr int NT = 256;  // threads per CTA
constexpr int KC = 32;   // depth of the T / R chunks staged in shared memory


// a Maxwellian tile's entries, per row and per column (fresh tiles; d <= MX_D):
// the operands' shared memory is free once the contraction is done
constexpr int MX_D = 8;
struct MxTile {
  double r[MX_D][BM], c[MX_D][BN];  // x, v form: mx_uv of the row's / column's modes
  double q[BM], coef[BM], nh[BM];   // the row's leading terms of |v - u|^2; its x tables
  int32_t rcombo[BM], ccombo[BN];   // parts of the x combination
};
struct XvTile {
  double rs[BM], bm[BM], bp[BM], h[BM];  // the row's sums; 1 / (2 T) of a position whose
                                         // velocity is the column's first mode
  double dm[BN], dp[BN];                 // that velocity's (v - a_u)^2, (v + a_u)^2
  double c[MX_D / 2][BN], tm[MX_D / 2][BN], tp[MX_D / 2][BN];  // the column's own pairs
};

struct ScreenSmem {
  union {
    struct {
      double Ts[KC][BM];
      double Rs[KC][BN];
    } d;
    struct {
      float Th[KC][BM], Tl[KC][BM];
      float Rh[KC][BN], Rl[KC][BN];
    } f;
    MxTile mx;
    XvTile xv;
  } op;
  int32_t srow[BM], scol[BN];
  int64_t lrow[BM], lcol[BN];
  int32_t ridx[BM][TTC_MAXD];
  int32_t cidx[BN][TTC_MAXD];
  float rowS[BM], colR[BN];
  uint64_t sk[NT / 32];
  int64_t sl[NT / 32];
  int32_t sr[NT / 32], sc[NT / 32];
  float fred[NT / 32];
  const double *acache;  // user generator: the tile's first entry in the cache
  int64_t acache_ld;
};

constexpr int TOPK_MAX = 16;
// stored-residual form: items of a fresh tile that goes out in quarters
constexpr int STORED_SLOTS = 4;

constexpr int DEC_US = 32;  // pivot steps up to this rank stage U in shared memory
struct DecideSmem {
  double ua[RCAP], bu[RCAP], brow[RCAP];
  double hcs[RCAP], hps[RCAP];  // R(:, c*) and T(a*, :) of the pivot step
  double us[DEC_US * DEC_US];   // U before the step (z <= DEC_US)
  int64_t q_nt;                 // control words of the decide item
  int32_t q_nf, q_r, q_maxr, q_prow, q_pcol;
  double q_tau, q_xrms;
  double apiv;                  // A(a*, c*)
  int32_t sel[TOPK_MAX];
  uint64_t skey[TOPK_MAX];
  int64_t slin[TOPK_MAX];
  int32_t srow[TOPK_MAX], scol[TOPK_MAX];
  int32_t cnt;
  double red[NT / 32];
  uint64_t rk[NT / 32];
  int64_t rl[NT / 32];
  int32_t rr[NT / 32], rc[NT / 32];
  int32_t flag;
  // the eight warps' top candidates of the mixed stored decide
  uint64_t wk[NT / 32 * 8];
  int64_t wl[NT / 32 * 8];
  int32_t wr[NT / 32 * 8], wc[NT / 32 * 8];
  // keys and indices of up to 2 NT slots ranked at once (stored decide)
  uint64_t tk[2 * NT];
  int64_t tl[2 * NT];
  int32_t last;  // this CTA finishes the bond's decide
};

constexpr int SPREAD_MAXSM = 1024;
struct SpreadSmem {
  int32_t cnt[SPREAD_MAXSM];  // CTAs per SM id
  int32_t k, place, bad, nsm, not2;
};

// replays (Alg. 4): per replay warp (the first RB_WARPS of a CTA) the rows T(a, :)
// it rebuilds, their entries at the pivot columns, delta, and the history rows
// of RB_STAGES steps in flight (replay_group's layout); after the block
// reductions' words, which the CTA's other warps may be using meanwhile
constexpr int RB_WARPS = 2, RB_STAGES = 3;
constexpr int RB_SMALL = 64;  // pivots up to which a warp rebuilds eight rows
constexpr int RB_BUF = 2 * RCAP + RCAP + 2 * RB_STAGES * RCAP;
constexpr int RB_BUF_SMALL = 2 * 8 * (RB_SMALL + 1) + RB_SMALL + 2 * RB_STAGES * RB_SMALL;
static_assert(RB_BUF >= RB_BUF_SMALL, "replay buffer");
struct ReplaySmem {
  double red_pad[NT / 32];
  double buf[RB_WARPS][RB_BUF];
};

// the error's samples when the tables meet: a warp's 32 samples' table rows
// (up to 16 entries, rows padded to 17 against bank conflicts); after the
// block reduction's words
struct SampleSmem {
  double red_pad[NT / 32];
  double rows[NT / 32][32 * 17];
};

union __align__(16) PhaseSmem {
  ScreenSmem s;
  DecideSmem d;
  SpreadSmem sp;
  ReplaySmem rp;
  SampleSmem sw;
  double red[NT / 32];
};

// The descriptor of instance 0, copied into shared memory when a kernel
// starts: every phase reads its fields all the time, and from global memory
// each one is a dependent load at L2 latency.  It does not change during a
// launch (the host writes it before launching).
__shared__ InstDev s_inst0;

// This CTA's place in the SM-spread order of the grid (the CTAs sorted by
// their slot on their SM, then by SM): work dealt to places 0, 1, 2, ...
// lands on distinct SMs before any SM gets a second share.  Latency-bound
// items (pivot steps, replays) then do not queue for the FP64 pipe, which
// is shared by the whole SM.  blockIdx.x until the order is known.
__shared__ int32_t s_place;
// S when the grid holds exactly two CTAs on each of S SMs (then places p and
// p + S share an SM), else 0 (not known, or another layout)
__shared__ int32_t s_sm2;
// grid barriers this CTA has passed in the running launch
__shared__ uint32_t s_bar_epoch;

__device__ void cache_inst0(const RunArgs &ra) {
  static_assert(sizeof(InstDev) % 8 == 0, "InstDev copies as 8-byte words");
  if (threadIdx.x == 0) {
    s_place = blockIdx.x;
    s_sm2 = 0;
    s_bar_epoch = 0u;
  }
  const unsigned long long *src = reinterpret_cast<const unsigned long long *>(ra.insts[0]);
  unsigned long long *dst = reinterpret_cast<unsigned long long *>(&s_inst0);
  for (int i = threadIdx.x; i < (int)(sizeof(InstDev) / 8); i += blockDim.x) dst[i] = src[i];
  __syncthreads();
}

__device__ __forceinline__ const InstDev &inst(const RunArgs &ra, int ii) {
  return ii == 0 ? s_inst0 : *ra.insts[ii];
}

// sampled screen's decide item (defined with its refinement phases below)
__device__ void decide_bond_sampled(const InstDev &in, Ctrl &cr, int b, DecideSmem &sm);

// sampled-error split (defined with the error evaluation below)
__device__ void choose_split(const InstDev &in, const int32_t *r, int &pL, int &pR);
__device__ double split_cost(const InstDev &in, const int32_t *r, int pL, int pR);
__device__ int64_t error_fmas(const InstDev &in, const int32_t *r);

// ---------------------------------------------------------------------------
// reductions

struct KeyBest {
  uint64_t key;
  int64_t lin;
  int32_t row, col;
};

// a before b: key, then linear index, then superblock coordinates.  (The same
// multi-index stands twice in a superblock only where a pivot set holds one
// twice, which takes pivots of rounding noise; then the first in row-major
// order counts, whatever the order of the candidates.)
__device__ __forceinline__ bool kb_better(const KeyBest &a, const KeyBest &b) {
  if (a.key != b.key) return a.key > b.key;
  if (a.lin != b.lin) return a.lin < b.lin;
  return a.row < b.row || (a.row == b.row && a.col < b.col);
}
__device__ __forceinline__ void kb_take(KeyBest &a, const KeyBest &b) {
  if (b.row >= 0 && (a.row < 0 || key_better(b.key, b.lin, a.key, a.lin))) a = b;
}
// for candidates in no fixed order (the stored forms' lists)
__device__ __forceinline__ void kb_take_any(KeyBest &a, const KeyBest &b) {
  if (b.row >= 0 && (a.row < 0 || kb_better(b, a))) a = b;
}

// block-wide max by key; result valid in thread 0 (ANY: of candidates in no
// fixed order)
template <bool ANY = false>
__device__ KeyBest block_best(KeyBest v, uint64_t *sk, int64_t *sl, int32_t *sr, int32_t *sc) {
  for (int off = 16; off > 0; off >>= 1) {
    KeyBest o;
    o.key = __shfl_down_sync(0xffffffffu, v.key, off);
    o.lin = __shfl_down_sync(0xffffffffu, v.lin, off);
    o.row = __shfl_down_sync(0xffffffffu, v.row, off);
    o.col = __shfl_down_sync(0xffffffffu, v.col, off);
    ANY ? kb_take_any(v, o) : kb_take(v, o);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) { sk[w] = v.key; sl[w] = v.lin; sr[w] = v.row; sc[w] = v.col; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < NT / 32; ++i) {
      KeyBest o{sk[i], sl[i], sr[i], sc[i]};
      ANY ? kb_take_any(v, o) : kb_take(v, o);
    }
  }
  return v;
}

// deterministic block sum (fixed shuffle tree, warps summed in order)
__device__ double block_sum(double v, double *red) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < NT / 32; ++i) s += red[i];
  return s;
}

// ---------------------------------------------------------------------------
// grid barrier for the persistent form: arrive, then wait for the generation
// to change; every wait gives up after wait_ns and raises the abort flag.
// Grid barrier of the persistent kernel.  The arrival counter only rises
// (the host clears it before each launch): the k-th barrier completes when
// it reaches k G, so a CTA arrives with one atomic and polls the same word.
// There is no reset or generation flip by the last arrival, whose extra
// round trips to L2 were on every barrier's critical path.  Every wait is
// bounded by wait_ns; on expiry the CTA records where, raises abort (which
// every poller checks) and returns false.
__device__ bool grid_barrier(const RunArgs &ra, int where) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    Barrier *bar = ra.bar;
    volatile unsigned int *vcount = &bar->count;
    volatile int32_t *vabort = &bar->abort;
    const unsigned int target = (s_bar_epoch + 1u) * gridDim.x;
    s_bar_epoch += 1u;
    __threadfence();  // this CTA's writes before its arrival
    const unsigned int arrived = atomicAdd(&bar->count, 1u) + 1u;
    if (arrived < target) {
      const uint64_t t0 = globaltimer_ns();
      while (*vcount < target) {
        if (*vabort) {
          ok = 0;
          break;
        }
        if (globaltimer_ns() - t0 > (uint64_t)ra.wait_ns) {
          atomicCAS(&bar->where, 0, where);
          atomicExch(&bar->abort, 1);
          ok = 0;
          break;
        }
      }
    }
    __threadfence();  // the other CTAs' writes after the barrier
    if (*vabort) ok = 0;
  }
  __syncthreads();
  return ok != 0;
}

// ---------------------------------------------------------------------------
// tiles of the superblock of bond b.  Without a subtensor grid the rows
// (columns) are cut into BM (BN) chunks; with one, mode b (b+1) is split into
// grid[b] (grid[b+1]) balanced pieces and no tile crosses a piece.

// Balanced split of n indices into C pieces: the first rem = n mod C pieces
// hold q + 1 = n / C + 1 indices, the others q.  Tiles never cross a piece.
struct Pieces {
  int32_t q, rem, tq1, tq0, tpb;  // tiles per piece of size q+1 / q, tiles per block
};

__host__ __device__ __forceinline__ Pieces make_pieces(int32_t n, int32_t C, int32_t te) {
  Pieces P;
  P.q = n / C;
  P.rem = n - P.q * C;
  P.tq1 = (P.q + 1 + te - 1) / te;
  P.tq0 = (P.q + te - 1) / te;
  P.tpb = P.rem * P.tq1 + (C - P.rem) * P.tq0;
  return P;
}

// tile t of one block: start within the block and length
__host__ __device__ __forceinline__ void piece_tile(const Pieces &P, int32_t t, int32_t te,
                                                    int32_t &start, int32_t &len) {
  int32_t k, tin, size;
  if (t < P.rem * P.tq1) {
    k = t / P.tq1;
    tin = t - k * P.tq1;
    size = P.q + 1;
  } else {
    const int32_t u = t - P.rem * P.tq1;
    const int32_t kk = u / P.tq0;
    k = P.rem + kk;
    tin = u - kk * P.tq0;
    size = P.q;
  }
  start = k * P.q + min(k, P.rem) + tin * te;
  len = min(te, size - tin * te);
}

// Tile geometry of bond b for edge te, from the ranks r (no subtensor grid:
// rows / columns cut into te-chunks; grid: pieces of mode b / b+1 per block)
struct TileGeo {
  int32_t nrt, nct;        // row tiles, column tiles
  int32_t rows, cols;
  int32_t te;
  int32_t pr, pc;          // pieces (0 = none)
  Pieces P, Q;             // row / column pieces
};

__host__ __device__ TileGeo tile_geo_e(const InstDev &in, const Ctrl &cr, const int32_t *r, int b,
                                       int te) {
  TileGeo g;
  g.te = te;
  g.rows = (int32_t)rows_of(in, r, b);
  g.cols = (int32_t)cols_of(in, r, b);
  g.pr = cr.grid[b];
  g.pc = cr.grid[b + 1];
  const int32_t nrb = b == 0 ? 1 : r[b - 1];
  const int32_t ncb = b == in.nb - 1 ? 1 : r[b + 1];
  if (g.pr > 0) {
    g.P = make_pieces((int32_t)in.n[b], g.pr, te);
    g.nrt = nrb * g.P.tpb;
  } else {
    g.nrt = (g.rows + te - 1) / te;
  }
  if (g.pc > 0) {
    g.Q = make_pieces((int32_t)in.n[b + 1], g.pc, te);
    g.nct = ncb * g.Q.tpb;
  } else {
    g.nct = (g.cols + te - 1) / te;
  }
  return g;
}

// Tile autotuner (in write_plan_warp): 64 x 64 tiles, unless the instance's
// superblocks give under a quarter wave of them on this grid while the
// contraction is deep (rank >= 24): then 32 x 32 tiles put four times the
// CTAs to work.  At small ranks the per-tile overhead dominates and 64 x 64
// stays faster (measured on the 6D Hilbert workloads).  Entries from TT cores
// cost hundreds of FMAs each: 32 x 32 tiles below four waves of 64 x 64.
// Whether the carried tiles of a screen at ranks r wait for their steps ("lazy
// carried tiles" below).
__device__ bool lazy_at(const InstDev &in, const int32_t *r) {
  if (!in.lazy) return false;
  float e = 0.f;
  for (int b = 0; b < in.nb; ++b) e += (float)rows_of(in, r, b) * (float)cols_of(in, r, b);
  return 8.f * e >= LAZY_BYTES;
}

// the tile plan of the next screen at ranks r, computed by one warp of the
// owner CTA (lane b handles bond b).  The stored forms keep the edge of the
// run's first plan: their tile states and candidate lists are numbered by it,
// and the update phase reads it beside this writer (planned_cut).
__device__ void write_plan_warp(const InstDev &in, Ctrl &cr, const int32_t *r, int grid) {
  const int lane = threadIdx.x & 31;
  const bool act = lane < in.nb;
  if (lane == 0) cr.lazy = lazy_at(in, r);
  const int32_t kept = in.stored ? ld_cg(cr.plan_te) : 0;  // (zero before the first plan)
  if (kept) {
    if (act) {
      const TileGeo g = tile_geo_e(in, cr, r, lane, kept);
      cr.plan_rows[lane] = g.rows;
      cr.plan_cols[lane] = g.cols;
      cr.plan_nrt[lane] = g.nrt;
      cr.plan_nct[lane] = g.nct;
    }
    return;
  }
  TileGeo g64;
  int64_t t64 = 0;
  int kmax = 0;
  if (act) {
    g64 = tile_geo_e(in, cr, r, lane, 64);
    t64 = (int64_t)g64.nrt * g64.nct;
    kmax = r[lane];
  }
  for (int off = 16; off > 0; off >>= 1) {
    t64 += __shfl_xor_sync(0xffffffffu, t64, off);
    kmax = max(kmax, __shfl_xor_sync(0xffffffffu, kmax, off));
  }
  // pieces of the subtensor grid at most 32 wide on every bond: a 64-wide
  // tile would hold one piece and compute three quarters padding; 32 x 32
  // tiles give the same tiles without it (FP64 forms)
  int small = 1;
  if (act) {
    const int64_t pr = cr.grid[lane], pc = cr.grid[lane + 1];
    const int64_t sr = pr > 0 ? (in.n[lane] + pr - 1) / pr : 64;
    const int64_t sc = pc > 0 ? (in.n[lane + 1] + pc - 1) / pc : 64;
    small = sr <= 32 && sc <= 32;
  }
  const bool pieces32 = __all_sync(0xffffffffu, small) && (in.prec == P_FP64 || in.stored);
  int te = 64;
  TileGeo g = g64;
  // a tile edge set for this run (the FP64 and stored forms; the mixed
  // recompute forms keep 64-wide tiles); 32-wide tiles when the candidate
  // slots of every bond allow them
  const int fte = (in.prec == P_FP64 || in.stored) ? cr.force_te : 0;
  int fok = fte == 32 || fte == 64;
  if (fte == 32) {
    TileGeo g32;
    int ok = 1;
    if (act) {
      // (the stored forms', at the run's rank caps: an edge for the whole run)
      const TileGeo gc = tile_geo_e(in, cr, in.stored ? cr.maxr : r, lane, 32);
      g32 = tile_geo_e(in, cr, r, lane, 32);
      ok = (int64_t)gc.nrt * gc.nct <= in.bond[lane].cand_cap;
    }
    fok = __all_sync(0xffffffffu, ok);
    if (fok) {
      te = 32;
      g = g32;
    }
  }
  if (fok) {
    // the edge set for the run
  } else if (pieces32) {
    te = 32;
    if (act) g = tile_geo_e(in, cr, r, lane, 32);
  } else if (!in.stored && in.prec == P_FP64 &&
             ((4 * t64 < (int64_t)grid && kmax >= 24) || (in.gen == 1 && t64 < 4 * (int64_t)grid))) {
    // 32 x 32 tiles when the candidate slots of every bond allow them
    int ok = 1;
    if (act) {
      g = tile_geo_e(in, cr, r, lane, 32);
      ok = (int64_t)g.nrt * g.nct <= in.bond[lane].cand_cap;
    }
    if (__all_sync(0xffffffffu, ok)) {
      te = 32;
    } else {
      g = g64;
    }
  }
  if (act) {
    cr.plan_rows[lane] = g.rows;
    cr.plan_cols[lane] = g.cols;
    cr.plan_nrt[lane] = g.nrt;
    cr.plan_nct[lane] = g.nct;
  }
  if (lane == 0) cr.plan_te = te;
}

// how the planned tiles of bond b cut its blocks: the edge and the pieces, none
// of which a stored form's later plans change (rows, columns and counts stay
// unset)
__device__ __forceinline__ TileGeo planned_cut(const InstDev &in, const Ctrl &cr, int b) {
  TileGeo g = {};
  g.te = ld_cg(cr.plan_te);
  g.pr = cr.grid[b];
  g.pc = cr.grid[b + 1];
  if (g.pr > 0) g.P = make_pieces((int32_t)in.n[b], g.pr, g.te);
  if (g.pc > 0) g.Q = make_pieces((int32_t)in.n[b + 1], g.pc, g.te);
  return g;
}
// geometry of bond b as planned (cheap: no tile counting)
__device__ __forceinline__ TileGeo planned_geo(const InstDev &in, const Ctrl &cr, int b) {
  const int32_t rows = ld_cg(cr.plan_rows[b]), cols = ld_cg(cr.plan_cols[b]);
  const int32_t nrt = ld_cg(cr.plan_nrt[b]), nct = ld_cg(cr.plan_nct[b]);
  TileGeo g = planned_cut(in, cr, b);
  g.rows = rows;
  g.cols = cols;
  g.nrt = nrt;
  g.nct = nct;
  return g;
}

__host__ __device__ __forceinline__ void tile_rows(const InstDev &in, const TileGeo &g, int b,
                                                   int32_t t, int64_t &r0, int &nr) {
  if (g.pr > 0) {
    const int32_t p = t / g.P.tpb;
    int32_t st, len;
    piece_tile(g.P, t - p * g.P.tpb, g.te, st, len);
    r0 = (int64_t)p * in.n[b] + st;
    nr = len;
  } else {
    r0 = (int64_t)t * g.te;
    nr = min(g.te, g.rows - t * g.te);
  }
}

__host__ __device__ __forceinline__ void tile_cols(const InstDev &in, const TileGeo &g, int b,
                                                   int32_t t, int64_t &c0, int &nc) {
  if (g.pc > 0) {
    const int32_t q = t / g.Q.tpb;
    int32_t st, len;
    piece_tile(g.Q, t - q * g.Q.tpb, g.te, st, len);
    c0 = (int64_t)q * in.n[b + 1] + st;
    nc = len;
  } else {
    c0 = (int64_t)t * g.te;
    nc = min(g.te, g.cols - t * g.te);
  }
}

// the tile of one block that holds index i (the inverse of piece_tile)
__device__ __forceinline__ int32_t piece_of(const Pieces &P, int32_t i, int32_t te) {
  const int32_t big = P.rem * (P.q + 1);
  if (i < big) return i / (P.q + 1) * P.tq1 + i % (P.q + 1) / te;
  return P.rem * P.tq1 + (i - big) / P.q * P.tq0 + (i - big) % P.q / te;
}
__device__ __forceinline__ int32_t row_tile_of(const InstDev &in, const TileGeo &g, int b, int32_t a) {
  if (g.pr == 0) return a / g.te;
  const int32_t n = (int32_t)in.n[b], p = a / n;
  return p * g.P.tpb + piece_of(g.P, a - p * n, g.te);
}
__device__ __forceinline__ int32_t col_tile_of(const InstDev &in, const TileGeo &g, int b, int32_t c) {
  if (g.pc == 0) return c / g.te;
  const int32_t n = (int32_t)in.n[b + 1], q = c / n;
  return q * g.Q.tpb + piece_of(g.Q, c - q * n, g.te);
}

// ---------------------------------------------------------------------------
// screen of one tile in FP64: A - chain(T(a,:), R(:,c)) for a 64 x 64 tile,
// 4 x 4 entries per thread, T / R staged through shared memory in 32-deep
// chunks; the accumulation order over t is the contract's serial chain.
// per-row / per-column data of a tile: linear-index parts, index sums
// (Hilbert) or the multi-indices (other generators)
__device__ void stage_meta(const InstDev &in, int b, int64_t r0, int nr, int64_t c0, int nc,
                           ScreenSmem &sm) {
  const SetDev &L = left_set(in, b);
  const SetDev &Rset = right_set(in, b);
  const int tid = threadIdx.x;
  const int64_t nb0 = in.n[b], nb1 = in.n[b + 1];
  const bool hil = in.gen == 0;
  const int wl = b, wr = in.d - b - 2;
  if (tid == 0 && in.gen == 4) {
    sm.acache = in.bond[b].A + r0 * in.bond[b].ldR + c0;
    sm.acache_ld = in.bond[b].ldR;
  }
  for (int x = tid; x < BM; x += NT) {
    if (x < nr) {
      const uint32_t a = (uint32_t)(r0 + x), p = a / (uint32_t)nb0, i = a - p * (uint32_t)nb0;
      sm.lrow[x] = L.lin[p] + i * in.stride[b];
      if (hil) {
        sm.srow[x] = L.sum[p] + (int)i;
      } else {
        for (int m = 0; m < wl; ++m) sm.ridx[x][m] = L.idx[p * wl + m];
        sm.ridx[x][wl] = (int32_t)i;
      }
    }
  }
  for (int x = tid; x < BN; x += NT) {
    if (x < nc) {
      const uint32_t c = (uint32_t)(c0 + x), q = c / (uint32_t)nb1, j = c - q * (uint32_t)nb1;
      sm.lcol[x] = j * in.stride[b + 1] + Rset.lin[q];
      if (hil) {
        sm.scol[x] = (int)j + Rset.sum[q];
      } else {
        sm.cidx[x][0] = (int32_t)j;
        for (int m = 0; m < wr; ++m) sm.cidx[x][1 + m] = Rset.idx[q * wr + m];
      }
    }
  }
}

// TT cores of small ranks: the product of the slices of modes 0..b is the same
// for every entry of a row, so the tile forms it once per row (four threads a
// row), in the operands' shared memory (the tile's contraction is done).  The
// entries then run modes b + 1..d - 1 only: the operations and their order per
// entry are gen_tt's.  (A product per entry from mode 0 on, its vectors in
// local memory, took 4.0 of 5.3 ms of a 5D n = 48 cross of ranks 8.)
__device__ __noinline__ void tt_prefix_rows(const InstDev &in, int b, int nr, ScreenSmem &sm) {
  static_assert(2 * BM * (TT_SMALL + 1) * sizeof(double) <= sizeof(sm.op), "prefix rows");
  double *buf = &sm.op.d.Ts[0][0];
  const int row = threadIdx.x >> 2, s = threadIdx.x & 3;
  __syncthreads();  // the operands are read
  for (int m = 0; m <= b; ++m) {
    // ping-pong, the last mode's vectors in the first half
    double *dst = buf + ((b - m) & 1) * BM * (TT_SMALL + 1);
    const double *src = buf + ((b - m + 1) & 1) * BM * (TT_SMALL + 1);
    if (row < nr) {
      const int ra = in.rho[m], rb = in.rho[m + 1];
      const double *G = in.tt + in.core_off[m] + (int64_t)sm.ridx[row][m] * rb;
      for (int q = s; q < rb; q += 4)
        dst[row * (TT_SMALL + 1) + q] =
            m == 0 ? G[q] : chain(src + row * (TT_SMALL + 1), 1, G + q, in.n[m] * rb, ra);
    }
    __syncthreads();
  }
}

// an entry of a tile whose rows' prefix vectors are formed
__device__ double tt_tail_entry(const InstDev &in, const ScreenSmem &sm, int wl, int wr, int rr,
                                int cc) {
  double v[TT_SMALL], w[TT_SMALL];
  const double *x = &sm.op.d.Ts[0][0] + rr * (TT_SMALL + 1);
  for (int j = 0; j <= wr; ++j) {
    const int m = wl + 1 + j, ra = in.rho[m], rb = in.rho[m + 1];
    const double *G = in.tt + in.core_off[m] + (int64_t)sm.cidx[cc][j] * rb;
    if (j == wr) return chain(x, 1, G, in.n[m], ra);  // (rb = 1)
    contract4(x, ra, G, 1, in.n[m] * rb, w, rb);
    for (int q = 0; q < rb; ++q) v[q] = w[q];
    x = v;
  }
  return x[0];
}

// The Maxwellians: what an entry's exponents and factors take from its row or
// its column alone is formed once per tile; an entry keeps its exps and a few
// operations (the same ones in the same order: leading sums of the row, then
// the mode pair split between row and column, then the column's).  Formed per
// entry from local index arrays they cost as much FP64 time as the exps: 53 of
// 56 ms of the 2d2v cross at n = 1000 went to its 4.2e8 fresh entries.
__device__ __noinline__ void mx_tile(const InstDev &in, int b, int nr, int nc, ScreenSmem &sm) {
  const int x = threadIdx.x & 63, side = threadIdx.x >> 6;  // 64 rows, then 64 columns
  const int d = in.d;
  __syncthreads();  // the operands are read
  if (in.gen == 3) {
    XvTile &o = sm.op.xv;
    const int full = (b + 1) / 2;        // pairs whole in the row
    const bool split = (b & 1) == 0;     // pair `full`: position in the row, velocity in the column
    if (side == 0 && x < nr) {
      double rs = 0.0, bm = 0.0, bp = 0.0;
      for (int q = 0; q < full; ++q) {
        const int64_t ox = in.mx_off[2 * q] + sm.ridx[x][2 * q];
        const double h = in.mx_nh[ox];
        const double v = in.mx_coef[in.mx_off[2 * q + 1] + sm.ridx[x][2 * q + 1]];
        const double dm = __dsub_rn(v, in.a_u), dp = __dadd_rn(v, in.a_u);
        rs = __dadd_rn(rs, in.mx_coef[ox]);
        bm = __dadd_rn(bm, __dmul_rn(__dmul_rn(dm, dm), h));
        bp = __dadd_rn(bp, __dmul_rn(__dmul_rn(dp, dp), h));
      }
      if (split) {
        const int64_t ox = in.mx_off[b] + sm.ridx[x][b];
        rs = __dadd_rn(rs, in.mx_coef[ox]);
        o.h[x] = in.mx_nh[ox];
      }
      o.rs[x] = rs;
      o.bm[x] = bm;
      o.bp[x] = bp;
    } else if (side == 1 && x < nc) {
      if (split) {
        const double v = in.mx_coef[in.mx_off[b + 1] + sm.cidx[x][0]];
        const double dm = __dsub_rn(v, in.a_u), dp = __dadd_rn(v, in.a_u);
        o.dm[x] = __dmul_rn(dm, dm);
        o.dp[x] = __dmul_rn(dp, dp);
      }
      for (int q = full + split, k = 0; q < d / 2; ++q, ++k) {
        const int64_t ox = in.mx_off[2 * q] + sm.cidx[x][2 * q - b - 1];
        const double h = in.mx_nh[ox];
        const double v = in.mx_coef[in.mx_off[2 * q + 1] + sm.cidx[x][2 * q - b]];
        const double dm = __dsub_rn(v, in.a_u), dp = __dadd_rn(v, in.a_u);
        o.c[k][x] = in.mx_coef[ox];
        o.tm[k][x] = __dmul_rn(__dmul_rn(dm, dm), h);
        o.tp[k][x] = __dmul_rn(__dmul_rn(dp, dp), h);
      }
    }
  } else {
    MxTile &o = sm.op.mx;
    const int dx = in.dx, lead = max(0, b - dx + 1);  // velocities in the row (then so is x)
    if (side == 0 && x < nr) {
      int32_t combo = 0;
      for (int m = 0; m <= b; ++m) {
        o.r[m][x] = in.mx_uv[in.mx_off[m] + sm.ridx[x][m]];
        if (m < dx) combo += sm.ridx[x][m] * (int32_t)in.mx_stride[m];
      }
      o.rcombo[x] = combo;
      double q = 0.0;
      for (int j = 0; j < lead; ++j) {
        const double dvu = __dsub_rn(o.r[dx + j][x], o.r[(j + 1) % dx][x]);
        q = __fma_rn(dvu, dvu, q);
      }
      o.q[x] = q;
      if (b >= dx - 1) {
        o.coef[x] = in.mx_coef[combo];
        o.nh[x] = in.mx_nh[combo];
      }
    } else if (side == 1 && x < nc) {
      int32_t combo = 0;
      for (int m = b + 1; m < d; ++m) {
        o.c[m][x] = in.mx_uv[in.mx_off[m] + sm.cidx[x][m - b - 1]];
        if (m < dx) combo += sm.cidx[x][m - b - 1] * (int32_t)in.mx_stride[m];
      }
      o.ccombo[x] = combo;
    }
  }
  __syncthreads();
}

__device__ __forceinline__ double mx_tile_entry(const InstDev &in, const ScreenSmem &sm, int b,
                                                int rr, int cc) {
  if (in.gen == 3) {
    const XvTile &o = sm.op.xv;
    const int full = (b + 1) / 2;
    const bool split = (b & 1) == 0;
    double rs = o.rs[rr], bm = o.bm[rr], bp = o.bp[rr];
    if (split) {
      const double h = o.h[rr];
      const double tm = __dmul_rn(o.dm[cc], h), tp = __dmul_rn(o.dp[cc], h);
      bm = full ? __dadd_rn(bm, tm) : tm;  // (0 + t is t: t is not negative)
      bp = full ? __dadd_rn(bp, tp) : tp;
    }
    for (int q = full + split, k = 0; q < in.d / 2; ++q, ++k) {
      rs = __dadd_rn(rs, o.c[k][cc]);
      bm = __dadd_rn(bm, o.tm[k][cc]);
      bp = __dadd_rn(bp, o.tp[k][cc]);
    }
    return __dmul_rn(rs, __dadd_rn(exp(-bm), exp(-bp)));
  }
  const MxTile &o = sm.op.mx;
  const int dx = in.dx;
  double q = o.q[rr];
  for (int j = max(0, b - dx + 1); j < in.dv; ++j) {
    const int m = dx + j, mu = (j + 1) % dx;
    const double v = m <= b ? o.r[m][rr] : o.c[m][cc];
    const double dvu = __dsub_rn(v, mu <= b ? o.r[mu][rr] : o.c[mu][cc]);
    q = __fma_rn(dvu, dvu, q);
  }
  double coef, nh;
  if (b >= dx - 1) {
    coef = o.coef[rr];
    nh = o.nh[rr];
  } else {
    const int32_t combo = o.rcombo[rr] + o.ccombo[cc];
    coef = in.mx_coef[combo];
    nh = in.mx_nh[combo];
  }
  return __dmul_rn(coef, exp(__dmul_rn(q, nh)));
}

// what a tile's entries need beyond its metadata, once its contraction is done
__device__ __forceinline__ void begin_entries(const InstDev &in, int b, int nr, int nc,
                                              ScreenSmem &sm) {
  if (in.gen == 1 && in.tt_small) tt_prefix_rows(in, b, nr, sm);
  if ((in.gen == 2 || in.gen == 3) && in.d <= MX_D) mx_tile(in, b, nr, nc, sm);
}

__device__ __noinline__ double tile_entry(const InstDev &in, const ScreenSmem &sm, int wl, int wr,
                                             int rr, int cc) {
  if (in.gen == 0) return in.hilb[sm.srow[rr] + sm.scol[cc]];
  if (in.gen == 4) return sm.acache[rr * sm.acache_ld + cc];
  if ((in.gen == 2 || in.gen == 3) && in.d <= MX_D) return mx_tile_entry(in, sm, wl, rr, cc);
  if (in.gen == 1 && in.tt_small) return tt_tail_entry(in, sm, wl, wr, rr, cc);
  int32_t idx[TTC_MAXD];
  for (int m = 0; m <= wl; ++m) idx[m] = sm.ridx[rr][m];
  for (int m = 0; m <= wr; ++m) idx[wl + 1 + m] = sm.cidx[cc][m];
  return gen_full(in, idx);
}

// acc[u][v] = chain(T(r0 + ty + 16u, :), R(:, c0 + tx + 16v)) over t < K, the
// contract's serial FMA order, T / R staged through shared memory in 32-deep
// chunks (the first chunk's barrier also publishes the tile metadata)
template <int TE>
__device__ __forceinline__ void tile_chain_fp64(const BondDev &B, int K, int64_t r0, int nr,
                                                int64_t c0, int nc, double (&acc)[TE / 16][TE / 16],
                                                ScreenSmem &sm) {
  constexpr int U = TE / 16;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) acc[u][v] = 0.0;
  // a chunk's staging issues all its loads before the first store (one round
  // trip to L2 instead of one per loop pass)
  constexpr int PER = KC * TE / NT;
  static_assert(KC * TE % NT == 0, "staging passes");
  for (int t0 = 0; t0 < K; t0 += KC) {
    const int kc = min(KC, K - t0);
    double tl[PER], rl[PER];
#pragma unroll
    for (int m = 0; m < PER; ++m) {
      const int x = tid + NT * m, tt = x / TE, ee = x - tt * TE;
      tl[m] = (tt < kc && ee < nr) ? B.T[(int64_t)(t0 + tt) * B.ldT + r0 + ee] : 0.0;
      rl[m] = (tt < kc && ee < nc) ? B.R[(int64_t)(t0 + tt) * B.ldR + c0 + ee] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < PER; ++m) {
      const int x = tid + NT * m, tt = x / TE, ee = x - tt * TE;
      if (tt < kc) {
        sm.op.d.Ts[tt][ee] = tl[m];
        sm.op.d.Rs[tt][ee] = rl[m];
      }
    }
    __syncthreads();
    for (int tt = 0; tt < kc; ++tt) {
      double tv[U], rv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) tv[u] = sm.op.d.Ts[tt][ty + 16 * u];
#pragma unroll
      for (int v = 0; v < U; ++v) rv[v] = sm.op.d.Rs[tt][tx + 16 * v];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < U; ++v) acc[u][v] = __fma_rn(tv[u], rv[v], acc[u][v]);
    }
  }
}

// acc[u][v] ~ T(r0 + ty + 16u, :) R(:, c0 + tx + 16v) over t < K on the FP32
// pipe, from the (hi, lo) FP32 shadows of T and R (mixed forms of the stored
// screen).  SPLIT: float-float, th rh = p + pe exactly (pe by FMA), the cross
// terms th rl + tl rh and pe join the low word, the high word is summed by
// TwoSum and the pair renormalised every term, so the result carries about
// 44 bits; else plain FP32 products and sums (sl = 0).  The result is the
// pair (sh, sl).
template <int TE, bool SPLIT>
__device__ __forceinline__ void tile_chain_ff(const BondDev &B, int K, int64_t r0, int nr,
                                              int64_t c0, int nc, float (&sh)[TE / 16][TE / 16],
                                              float (&sl)[TE / 16][TE / 16], ScreenSmem &sm) {
  constexpr int U = TE / 16;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) {
      sh[u][v] = 0.f;
      sl[u][v] = 0.f;
    }
  constexpr int PER = KC * TE / NT;
  static_assert(KC * TE % NT == 0, "staging passes");
  for (int t0 = 0; t0 < K; t0 += KC) {
    const int kc = min(KC, K - t0);
    float th[PER], tl[PER], rh[PER], rl[PER];
#pragma unroll
    for (int m = 0; m < PER; ++m) {
      const int x = tid + NT * m, tt = x / TE, ee = x - tt * TE;
      const bool tv = tt < kc && ee < nr, rv = tt < kc && ee < nc;
      const int64_t ot = (int64_t)(t0 + tt) * B.ldT + r0 + ee;
      const int64_t orr = (int64_t)(t0 + tt) * B.ldR + c0 + ee;
      th[m] = tv ? B.Thi[ot] : 0.f;
      rh[m] = rv ? B.Rhi[orr] : 0.f;
      tl[m] = (SPLIT && tv) ? B.Tlo[ot] : 0.f;
      rl[m] = (SPLIT && rv) ? B.Rlo[orr] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < PER; ++m) {
      const int x = tid + NT * m, tt = x / TE, ee = x - tt * TE;
      if (tt < kc) {
        sm.op.f.Th[tt][ee] = th[m];
        sm.op.f.Rh[tt][ee] = rh[m];
        if (SPLIT) {
          sm.op.f.Tl[tt][ee] = tl[m];
          sm.op.f.Rl[tt][ee] = rl[m];
        }
      }
    }
    __syncthreads();
    for (int tt = 0; tt < kc; ++tt) {
      float a[U], al[U], b[U], bl[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        a[u] = sm.op.f.Th[tt][ty + 16 * u];
        al[u] = SPLIT ? sm.op.f.Tl[tt][ty + 16 * u] : 0.f;
      }
#pragma unroll
      for (int v = 0; v < U; ++v) {
        b[v] = sm.op.f.Rh[tt][tx + 16 * v];
        bl[v] = SPLIT ? sm.op.f.Rl[tt][tx + 16 * v] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < U; ++v) {
          if (SPLIT) {
            const float p = __fmul_rn(a[u], b[v]);
            const float pe = __fmaf_rn(a[u], b[v], -p);
            const float cross = __fmaf_rn(al[u], b[v], __fmaf_rn(a[u], bl[v], pe));
            const float s1 = __fadd_rn(sh[u][v], p);
            const float bb = __fsub_rn(s1, sh[u][v]);
            const float e = __fadd_rn(__fsub_rn(sh[u][v], __fsub_rn(s1, bb)), __fsub_rn(p, bb));
            const float lo = __fadd_rn(sl[u][v], __fadd_rn(e, cross));
            const float s2 = __fadd_rn(s1, lo);
            sl[u][v] = __fsub_rn(lo, __fsub_rn(s2, s1));
            sh[u][v] = s2;
          } else {
            sh[u][v] = __fmaf_rn(a[u], b[v], sh[u][v]);
          }
        }
    }
  }
}

// (ah + al) - (bh + bl) as a normalised float-float pair: TwoSum of the high
// words, the low words' difference joins the rounding error, one fast
// renormalisation (11 FP32 operations, no FP64 pipe).  The error is a few
// units of 2^-48 (|a| + |b|), below the chain's own.
__device__ __forceinline__ float2 ff_sub(float ah, float al, float bh, float bl) {
  const float s = __fsub_rn(ah, bh);
  const float v = __fsub_rn(s, ah);
  const float e = __fsub_rn(__fsub_rn(ah, __fsub_rn(s, v)), __fadd_rn(bh, v));
  const float t = __fadd_rn(e, __fsub_rn(al, bl));
  const float hi = __fadd_rn(s, t);
  return make_float2(hi, __fsub_rn(t, __fsub_rn(hi, s)));
}

template <bool HIL, int TE>
__device__ __noinline__ void screen_tile_fp64_t(const InstDev &in, int b, int K, int64_t r0, int nr,
                                                int64_t c0, int nc, Cand *out, ScreenSmem &sm) {
  constexpr int U = TE / 16;  // entries per thread and dimension
  const BondDev &B = in.bond[b];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int wl = b, wr = in.d - b - 2;
  __syncthreads();
  stage_meta(in, b, r0, nr, c0, nc, sm);
  double acc[U][U];
  tile_chain_fp64<TE>(B, K, r0, nr, c0, nc, acc, sm);
  if (!HIL) begin_entries(in, b, nr, nc, sm);
  KeyBest best{0ull, LLONG_MAX, -1, -1};
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int rr = ty + 16 * u;
    if (rr >= nr) continue;
#pragma unroll
    for (int v = 0; v < U; ++v) {
      const int cc = tx + 16 * v;
      if (cc >= nc) continue;
      const double A = HIL ? in.hilb[sm.srow[rr] + sm.scol[cc]] : tile_entry(in, sm, wl, wr, rr, cc);
      const double e = __dsub_rn(A, acc[u][v]);
      const uint64_t k = abs_key(e);
      if (best.row < 0 || k >= best.key) {
        const int64_t l = sm.lrow[rr] + sm.lcol[cc];
        if (best.row < 0 || k > best.key || l < best.lin) {
          best.key = k;
          best.lin = l;
          best.row = (int32_t)(r0 + rr);
          best.col = (int32_t)(c0 + cc);
        }
      }
    }
  }
  best = block_best(best, sm.sk, sm.sl, sm.sr, sm.sc);
  if (tid == 0) {
    out->key = best.key;
    out->lin = best.lin;
    out->row = best.row;
    out->col = best.col;
  }
}

__device__ __forceinline__ void screen_tile_fp64(const InstDev &in, int b, int K, int64_t r0,
                                                 int nr, int64_t c0, int nc, int te, Cand *out,
                                                 ScreenSmem &sm) {
  if (te == 32) {
    if (in.gen == 0)
      screen_tile_fp64_t<true, 32>(in, b, K, r0, nr, c0, nc, out, sm);
    else
      screen_tile_fp64_t<false, 32>(in, b, K, r0, nr, c0, nc, out, sm);
  } else {
    if (in.gen == 0)
      screen_tile_fp64_t<true, 64>(in, b, K, r0, nr, c0, nc, out, sm);
    else
      screen_tile_fp64_t<false, 64>(in, b, K, r0, nr, c0, nc, out, sm);
  }
}

// ---------------------------------------------------------------------------
// Stored residual values.  The FP64 form keeps E, the rank-one step's column
// ew and row erow as doubles and carries E by the FP64 FMA of the stored-form
// contract.  The mixed forms keep them as float-float pairs (hi, lo) in the
// same 8 bytes and carry E on the FP32 pipe (about 44 bits; a carried entry
// then costs no FP64 instruction); their screen keys are |hi|.
template <int MIX>
struct SV;
template <>
struct SV<0> {
  using T = double;
  static __device__ __forceinline__ T load(const double *E, int64_t i) { return E[i]; }
  static __device__ __forceinline__ void store(double *E, int64_t i, T v) { E[i] = v; }
  static __device__ __forceinline__ T zero() { return 0.0; }
  static __device__ __forceinline__ T step(T w, T e, T a) { return __fma_rn(w, e, a); }
  static __device__ __forceinline__ T from(double x) { return x; }
  static __device__ __forceinline__ uint64_t key(T v) { return abs_key(v); }
};
struct SVff {
  using T = float2;
  static __device__ __forceinline__ T load(const double *E, int64_t i) {
    return reinterpret_cast<const float2 *>(E)[i];
  }
  static __device__ __forceinline__ void store(double *E, int64_t i, T v) {
    reinterpret_cast<float2 *>(E)[i] = v;
  }
  static __device__ __forceinline__ T zero() { return make_float2(0.f, 0.f); }
  // a + w e: w.x e.x = p + pe exactly, the cross terms and pe join the low
  // word, TwoSum of the high words, renormalised (12 FP32 operations)
  static __device__ __forceinline__ T step(T w, T e, T a) {
    const float p = __fmul_rn(w.x, e.x);
    const float pe = __fmaf_rn(w.x, e.x, -p);
    const float cr = __fmaf_rn(w.x, e.y, __fmaf_rn(w.y, e.x, pe));
    const float s1 = __fadd_rn(a.x, p);
    const float bb = __fsub_rn(s1, a.x);
    const float er = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s1, bb)), __fsub_rn(p, bb));
    const float lo = __fadd_rn(a.y, __fadd_rn(er, cr));
    const float s2 = __fadd_rn(s1, lo);
    return make_float2(s2, __fsub_rn(lo, __fsub_rn(s2, s1)));
  }
  static __device__ __forceinline__ T from(double x) {
    const float h = __double2float_rn(x);
    return make_float2(h, __double2float_rn(__dsub_rn(x, (double)h)));
  }
  static __device__ __forceinline__ uint64_t key(T v) {
    return (uint64_t)(__float_as_uint(v.x) & 0x7FFFFFFFu);
  }
};
template <>
struct SV<1> : SVff {};
template <>
struct SV<2> : SVff {};

// |x| as a float, rounded up
__device__ __forceinline__ float abs_up(double x) { return __double2float_ru(fabs(x)); }

// a double into stored form (update phase)
__device__ __forceinline__ void sv_put(const InstDev &in, double *E, int64_t i, double x) {
  if (in.prec == P_FP64)
    E[i] = x;
  else
    SVff::store(E, i, SVff::from(x));
}

// stored-residual screen of one tile that reaches beyond the carried tiles (eq.
// aca_approx_E).  Its entries inside the stored extent (row < sr and column <
// sc) are read from E and, when the bond appended a pivot in the last sweep
// (pend), carried through its rank-one step E(a,c) = E(a,c) + ew[a] erow[c]
// with ew[a] = -(E(a,c*) / E(a*,c*)) and erow = E(a*, :).  Entries outside it
// have just entered the superblock and get A - chain(T(a,:), R(:,c)) with the
// current factors (MIX 0: FP64 chain of the contract; 1 / 2: FP32 /
// float-float chain).  Both are written back to E; the tile's best |E| is kept
// as in the FP64 screen.
template <bool HIL, int TE, int MIX>
__device__ __noinline__ void screen_tile_stored_t(const InstDev &in, int b, int K, int64_t r0,
                                                  int nr, int64_t c0, int nc, int32_t sr,
                                                  int32_t sc, int pend, Cand *out,
                                                  ScreenSmem &sm) {
  using V = SV<MIX>;
  using VT = typename V::T;
  constexpr int U = TE / 16;
  const BondDev &B = in.bond[b];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int wl = b, wr = in.d - b - 2;
  const int64_t ld = B.ldR;
  __syncthreads();
  stage_meta(in, b, r0, nr, c0, nc, sm);
  const double *const ew = B.ew + (int64_t)(K - 1) * B.ldw;      // the newest step (pend)
  const double *const erow = B.erow + (int64_t)(K - 1) * B.lde;
  VT ev[U][U];
  {
    // FP64: acc; mixed: the float-float pair (fh, fl), and E = A - T R is
    // formed in float-float too, so the mixed path leaves the FP64 pipe alone
    double acc[MIX == 0 ? U : 1][MIX == 0 ? U : 1];
    float fh[MIX == 0 ? 1 : U][MIX == 0 ? 1 : U], fl[MIX == 0 ? 1 : U][MIX == 0 ? 1 : U];
    if constexpr (MIX == 0)
      tile_chain_fp64<TE>(B, K, r0, nr, c0, nc, acc, sm);
    else
      tile_chain_ff<TE, MIX == 2>(B, K, r0, nr, c0, nc, fh, fl, sm);
    if (!HIL) begin_entries(in, b, nr, nc, sm);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int rr = ty + 16 * u;
      const int64_t a = r0 + rr;
      const bool arow = rr < nr && a < sr;
      const VT wa = (pend && arow) ? V::load(ew, a) : V::zero();
#pragma unroll
      for (int v = 0; v < U; ++v) {
        const int cc = tx + 16 * v;
        const int64_t c = c0 + cc;
        if (rr >= nr || cc >= nc) {
          ev[u][v] = V::zero();
          continue;
        }
        VT e;
        if (arow && c < sc) {
          e = V::load(B.E, a * ld + c);
          if (pend) e = V::step(wa, V::load(erow, c), e);
        } else if constexpr (MIX == 0) {
          const double A =
              HIL ? in.hilb[sm.srow[rr] + sm.scol[cc]] : tile_entry(in, sm, wl, wr, rr, cc);
          e = __dsub_rn(A, acc[u][v]);
        } else {
          float ah, al;
          if (HIL) {
            ah = in.hilb_hi[sm.srow[rr] + sm.scol[cc]];
            al = in.hilb_lo[sm.srow[rr] + sm.scol[cc]];
          } else {
            split2(tile_entry(in, sm, wl, wr, rr, cc), ah, al);
          }
          e = ff_sub(ah, al, fh[u][v], fl[u][v]);
        }
        V::store(B.E, a * ld + c, e);
        ev[u][v] = e;
      }
    }
  }
  KeyBest best{0ull, LLONG_MAX, -1, -1};
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int rr = ty + 16 * u;
    if (rr >= nr) continue;
#pragma unroll
    for (int v = 0; v < U; ++v) {
      const int cc = tx + 16 * v;
      if (cc >= nc) continue;
      const uint64_t k = V::key(ev[u][v]);
      if (best.row < 0 || k >= best.key) {
        const int64_t l = sm.lrow[rr] + sm.lcol[cc];
        if (best.row < 0 || k > best.key || l < best.lin) {
          best.key = k;
          best.lin = l;
          best.row = (int32_t)(r0 + rr);
          best.col = (int32_t)(c0 + cc);
        }
      }
    }
  }
  best = block_best(best, sm.sk, sm.sl, sm.sr, sm.sc);
  if (tid == 0) {
    out->key = best.key;
    out->lin = best.lin;
    out->row = best.row;
    out->col = best.col;
  }
}

template <int MIX>
__device__ __forceinline__ void screen_tile_stored_m(const InstDev &in, int b, int K, int64_t r0,
                                                     int nr, int64_t c0, int nc, int te,
                                                     int32_t sr, int32_t sc, int pend, Cand *out,
                                                     ScreenSmem &sm) {
  if (te == 32) {
    if (in.gen == 0)
      screen_tile_stored_t<true, 32, MIX>(in, b, K, r0, nr, c0, nc, sr, sc, pend, out, sm);
    else
      screen_tile_stored_t<false, 32, MIX>(in, b, K, r0, nr, c0, nc, sr, sc, pend, out, sm);
  } else {
    if (in.gen == 0)
      screen_tile_stored_t<true, 64, MIX>(in, b, K, r0, nr, c0, nc, sr, sc, pend, out, sm);
    else
      screen_tile_stored_t<false, 64, MIX>(in, b, K, r0, nr, c0, nc, sr, sc, pend, out, sm);
  }
}

// the stored screen of one tile; the mixed forms form the entries new to the
// superblock on the FP32 pipe (FP32 or float-float products), the carried
// ones stay FP64
__device__ __forceinline__ void screen_tile_stored(const InstDev &in, int b, int K, int64_t r0,
                                                   int nr, int64_t c0, int nc, int te, int32_t sr,
                                                   int32_t sc, int pend, Cand *out,
                                                   ScreenSmem &sm) {
  if (in.prec == P_FP64)
    screen_tile_stored_m<0>(in, b, K, r0, nr, c0, nc, te, sr, sc, pend, out, sm);
  else if (in.prec == P_FP32)
    screen_tile_stored_m<1>(in, b, K, r0, nr, c0, nc, te, sr, sc, pend, out, sm);
  else
    screen_tile_stored_m<2>(in, b, K, r0, nr, c0, nc, te, sr, sc, pend, out, sm);
}

// ---------------------------------------------------------------------------
// screen of one tile in FP32 (SPLIT = false) or float-float (SPLIT = true)
// from the (hi, lo) shadows of T and R.  Besides the tile's best |E| it
// bounds the FP64 residual of every entry (MCand), so that the merge can
// prove which tiles cannot hold the FP64 argmax.
//   float-float product: T R = (Th + Tl)(Rh + Rl) ~ Th Rh (exact as p + pl)
//   + (Th Rl + Tl Rh); sums (sh, sl) by TwoSum, renormalised every step.
//   bound, with S = max_a sum_t |T(a,t)|, Rm = max |R(t,c)|, A = max |A|:
//     FP32 : 2 (K + 3) u (A + S Rm),  u = 2^-24
//     split: 4 (3K + 8) u^2 (A + S Rm)
//   plus 4u |E| for the last roundings.
template <bool SPLIT, bool HIL, int TE>
__device__ __noinline__ void screen_tile_mixed_t(const InstDev &in, int b, int K, int64_t r0,
                                                 int nr, int64_t c0, int nc, MCand *out,
                                                 ScreenSmem &sm) {
  constexpr int U = TE / 16;  // entries per thread and dimension
  const BondDev &B = in.bond[b];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int wl = b, wr = in.d - b - 2;
  __syncthreads();
  stage_meta(in, b, r0, nr, c0, nc, sm);
  for (int x = tid; x < BM; x += NT) sm.rowS[x] = 0.f;
  for (int x = tid; x < BN; x += NT) sm.colR[x] = 0.f;
  float sh[U][U], sl[U][U];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) {
      sh[u][v] = 0.f;
      sl[u][v] = 0.f;
    }
  for (int t0 = 0; t0 < K; t0 += KC) {
    const int kc = min(KC, K - t0);
    __syncthreads();
    for (int x = tid; x < kc * TE; x += NT) {
      const int tt = x / TE, rr = x - tt * TE;
      const int64_t o = (int64_t)(t0 + tt) * B.ldT + r0 + rr;
      sm.op.f.Th[tt][rr] = rr < nr ? B.Thi[o] : 0.f;
      if (SPLIT) sm.op.f.Tl[tt][rr] = rr < nr ? B.Tlo[o] : 0.f;
    }
    for (int x = tid; x < kc * TE; x += NT) {
      const int tt = x / TE, cc = x - tt * TE;
      const int64_t o = (int64_t)(t0 + tt) * B.ldR + c0 + cc;
      sm.op.f.Rh[tt][cc] = cc < nc ? B.Rhi[o] : 0.f;
      if (SPLIT) sm.op.f.Rl[tt][cc] = cc < nc ? B.Rlo[o] : 0.f;
    }
    __syncthreads();
    if (tid < BM) {
      float acc = sm.rowS[tid];
      for (int tt = 0; tt < kc; ++tt) acc += fabsf(sm.op.f.Th[tt][tid]);
      sm.rowS[tid] = acc;
    } else if (tid < BM + BN) {
      const int c = tid - BM;
      float m = sm.colR[c];
      for (int tt = 0; tt < kc; ++tt) m = fmaxf(m, fabsf(sm.op.f.Rh[tt][c]));
      sm.colR[c] = m;
    }
    for (int tt = 0; tt < kc; ++tt) {
      float th[U], tl[U], rh[U], rl[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        th[u] = sm.op.f.Th[tt][ty + 16 * u];
        tl[u] = SPLIT ? sm.op.f.Tl[tt][ty + 16 * u] : 0.f;
      }
#pragma unroll
      for (int v = 0; v < U; ++v) {
        rh[v] = sm.op.f.Rh[tt][tx + 16 * v];
        rl[v] = SPLIT ? sm.op.f.Rl[tt][tx + 16 * v] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < U; ++v) {
          if (SPLIT) {
            // th rh = p + pl exactly; the cross terms join pl by FMA
            const float p = __fmul_rn(th[u], rh[v]);
            const float pc = __fmaf_rn(tl[u], rh[v], __fmaf_rn(th[u], rl[v], __fmaf_rn(th[u], rh[v], -p)));
            const float s1 = __fadd_rn(sh[u][v], p);
            const float bb = __fsub_rn(s1, sh[u][v]);
            const float e = __fadd_rn(__fsub_rn(sh[u][v], __fsub_rn(s1, bb)), __fsub_rn(p, bb));
            const float lo = __fadd_rn(sl[u][v], __fadd_rn(e, pc));
            const float s2 = __fadd_rn(s1, lo);
            sl[u][v] = __fsub_rn(lo, __fsub_rn(s2, s1));
            sh[u][v] = s2;
          } else {
            sh[u][v] = __fmaf_rn(th[u], rh[v], sh[u][v]);
          }
        }
    }
  }
  if (!HIL) begin_entries(in, b, nr, nc, sm);
  float bv = -1.f, v2 = 0.f, amax = 0.f;
  int64_t bl = LLONG_MAX;
  int32_t brow = -1, bcol = -1;
  bool bad = false;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int rr = ty + 16 * u;
    if (rr >= nr) continue;
#pragma unroll
    for (int v = 0; v < U; ++v) {
      const int cc = tx + 16 * v;
      if (cc >= nc) continue;
      float ah, al;
      if (HIL) {
        ah = in.hilb_hi[sm.srow[rr] + sm.scol[cc]];
        al = in.hilb_lo[sm.srow[rr] + sm.scol[cc]];
      } else {
        split2(tile_entry(in, sm, wl, wr, rr, cc), ah, al);
      }
      const float e = __fadd_rn(__fsub_rn(ah, sh[u][v]), __fsub_rn(al, sl[u][v]));
      const float ae = fabsf(e);
      amax = fmaxf(amax, fabsf(ah));
      if (!(ae <= FLT_MAX)) bad = true;
      const int64_t l = sm.lrow[rr] + sm.lcol[cc];
      if (ae > bv || (ae == bv && l < bl)) {
        v2 = fmaxf(v2, bv);
        bv = ae;
        bl = l;
        brow = (int32_t)(r0 + rr);
        bcol = (int32_t)(c0 + cc);
      } else {
        v2 = fmaxf(v2, ae);
      }
    }
  }
  KeyBest best{brow >= 0 ? (uint64_t)__float_as_uint(bv) : 0ull, bl, brow, bcol};
  best = block_best(best, sm.sk, sm.sl, sm.sr, sm.sc);
  __shared__ int32_t wrow, wcol;
  __shared__ float wval;
  __shared__ int wbad;
  if (tid == 0) {
    wrow = best.row;
    wcol = best.col;
    wval = __uint_as_float((unsigned)best.key);
    wbad = 0;
  }
  __syncthreads();
  if (bad) wbad = 1;
  // the tile's best among the others: every thread's second value, and the
  // thread bests that lost to the winner
  float rest = (brow == wrow && bcol == wcol) ? v2 : fmaxf(fmaxf(bv, 0.f), v2);
  float Smax = 0.f, Rmax = 0.f;
  for (int x = tid; x < nr; x += NT) Smax = fmaxf(Smax, sm.rowS[x]);
  for (int x = tid; x < nc; x += NT) Rmax = fmaxf(Rmax, sm.colR[x]);
  for (int off = 16; off > 0; off >>= 1) {
    rest = fmaxf(rest, __shfl_down_sync(0xffffffffu, rest, off));
    amax = fmaxf(amax, __shfl_down_sync(0xffffffffu, amax, off));
    Smax = fmaxf(Smax, __shfl_down_sync(0xffffffffu, Smax, off));
    Rmax = fmaxf(Rmax, __shfl_down_sync(0xffffffffu, Rmax, off));
  }
  __shared__ float wr4[NT / 32][4];
  const int w = tid >> 5;
  if ((tid & 31) == 0) {
    wr4[w][0] = rest;
    wr4[w][1] = amax;
    wr4[w][2] = Smax;
    wr4[w][3] = Rmax;
  }
  __syncthreads();
  if (tid == 0) {
    for (int i = 1; i < NT / 32; ++i) {
      rest = fmaxf(rest, wr4[i][0]);
      amax = fmaxf(amax, wr4[i][1]);
      Smax = fmaxf(Smax, wr4[i][2]);
      Rmax = fmaxf(Rmax, wr4[i][3]);
    }
    const double u = 5.9604644775390625e-8;  // 2^-24
    const double scale = (double)amax + (double)Smax * (double)Rmax;
    const double eabs = SPLIT ? 4.0 * (3.0 * K + 8.0) * u * u * scale
                              : 2.0 * (K + 3.0) * u * scale;
    out->v = wbad ? INFINITY : wval;
    out->rest = wbad ? INFINITY : rest;
    out->eabs = isfinite(eabs) ? eabs : INFINITY;
    out->lin = best.lin;
    out->row = best.row;
    out->col = best.col;
  }
}

template <bool SPLIT>
__device__ __forceinline__ void screen_tile_mixed(const InstDev &in, int b, int K, int64_t r0,
                                                  int nr, int64_t c0, int nc, int te, MCand *out,
                                                  ScreenSmem &sm) {
  if (te == 32) {
    if (in.gen == 0)
      screen_tile_mixed_t<SPLIT, true, 32>(in, b, K, r0, nr, c0, nc, out, sm);
    else
      screen_tile_mixed_t<SPLIT, false, 32>(in, b, K, r0, nr, c0, nc, out, sm);
  } else {
    if (in.gen == 0)
      screen_tile_mixed_t<SPLIT, true, 64>(in, b, K, r0, nr, c0, nc, out, sm);
    else
      screen_tile_mixed_t<SPLIT, false, 64>(in, b, K, r0, nr, c0, nc, out, sm);
  }
}

// state, screened, add[b] and r[b] of an instance, each word loaded by its
// own thread (one L2 round trip instead of a chain of them)
// control words of an instance read once per phase by the CTA (shared
// memory: per-thread copies would live in local memory, whose lines this
// kernel's large stack frame keeps out of L1)
struct CtrlSnap {
  int32_t state, screened;
  int32_t add[TTC_MAXB], r[TTC_MAXB];
  int32_t old_r[TTC_MAXB];  // r - add: the ranks at the start of the sweep
};

__device__ void snap_ctrl(const Ctrl &cr, int nb, CtrlSnap &out) {
  __syncthreads();
  const int k = threadIdx.x;
  if (k == 0)
    out.state = ld_cg(cr.state);
  else if (k == 1)
    out.screened = ld_cg(cr.screened);
  else if (k < 2 + nb)
    out.add[k - 2] = ld_cg(cr.add[k - 2]);
  else if (k < 2 + 2 * nb)
    out.r[k - 2 - nb] = ld_cg(cr.r[k - 2 - nb]);
  __syncthreads();
  if (k < nb) out.old_r[k] = out.r[k] - out.add[k];
  __syncthreads();
}

// ---------------------------------------------------------------------------
// phase: screen.  Tiles of every (instance, bond) pair that needs a screen
// are numbered consecutively; CTA g takes tiles g, g + G, ...
// Stored-residual instances instead hand out their tiles from a counter,
// tiles new to a superblock (A - T R, r_k FMAs per entry) first and carried
// ones (one load, one FMA, one store per entry) after, so that CTAs with a
// costly tile take fewer cheap ones.  The decide phase after the screen
// clears the counter.

// column-major linear index of superblock entry (a, c) of bond b
__device__ __forceinline__ int64_t entry_lin(const InstDev &in, int b, int64_t a, int64_t c) {
  const int64_t nb0 = in.n[b], nb1 = in.n[b + 1];
  const int64_t p = a / nb0, i = a - p * nb0;
  const int64_t q = c / nb1, j = c - q * nb1;
  return left_set(in, b).lin[p] + i * in.stride[b] + j * in.stride[b + 1] +
         right_set(in, b).lin[q];
}

// carried region of bond b: row tiles < tr0 and column tiles < tc0 lie in
// the stored extent (its rows / columns are whole prefix / suffix blocks)
__host__ __device__ __forceinline__ void carried_tiles(const InstDev &in, const TileGeo &g, int b,
                                                       int32_t sr, int32_t sc, int32_t &tr0,
                                                       int32_t &tc0) {
  tr0 = g.pr > 0 ? (sr / (int32_t)in.n[b]) * g.P.tpb : sr / g.te;
  tc0 = g.pc > 0 ? (sc / (int32_t)in.n[b + 1]) * g.Q.tpb : sc / g.te;
}

// bookkeeping of a screen (one thread, from the CTA's staged geometry):
// candidate slots per bond for the merge, and the statistics.  Stored form: sr /
// sc are the stored extents, tr0 / tc0 the carried tiles', pend whether a step is
// pending, nfs the fresh items' slots, nca the carried tiles' (the mixed forms;
// FP64 counts the candidates that it lists); the carried tiles' FMAs and bytes
// are counted as they are brought up to date, those of stored entries in tiles
// that reach beyond them here.
__device__ void screen_bookkeeping(const InstDev &in, const int32_t *r, const TileGeo *geo,
                                   const int32_t *sr, const int32_t *sc, const int32_t *tr0,
                                   const int32_t *tc0, const int32_t *pend, const int32_t *nfs,
                                   const int32_t *nca) {
  Ctrl &cw = *in.ctrl;
  int64_t entries = 0, fmas = 0, fresh = 0, bytes = 0;
  for (int b = 0; b < in.nb; ++b) {
    const int64_t e = (int64_t)geo[b].rows * geo[b].cols;
    entries += e;
    if (sr) {
      const int64_t kept = (int64_t)sr[b] * sc[b];
      fresh += e - kept;
      const int64_t cr = geo[b].pr > 0 ? sr[b] : tr0[b] * geo[b].te;  // of the carried tiles
      const int64_t cc = geo[b].pc > 0 ? sc[b] : tc0[b] * geo[b].te;
      fmas += (e - kept) * r[b] + (pend[b] ? kept - cr * cc : 0);
      bytes += 8 * (e - kept) + 16 * (kept - cr * cc);
      cw.nfresh[b] = nfs[b];
      if (in.prec != P_FP64) cw.ntiles[b] = nca[b];
    } else {
      cw.ntiles[b] = geo[b].nrt * geo[b].nct;
      fresh += e;
      fmas += e * r[b];
    }
  }
  cw.sweeps += 1;
  cw.entries += entries;
  cw.entries_fresh += fresh;
  atomicAdd((unsigned long long *)&cw.stored_bytes, (unsigned long long)bytes);
  atomicAdd((unsigned long long *)&cw.screen_fmas, (unsigned long long)fmas);
  cw.screened = 1;
}

// ---------------------------------------------------------------------------
// Lazy carried tiles (FP64).  A carried tile takes part in a screen only
// through its best |E|, and each pivot's rank-one step moves its entries by at
// most max |ew| max |erow| over the tile.  So every carried tile keeps a bound
// U on its |E| with every step so far, and its best entry with its exact value
// (one step per pivot), and its entries are left as they are, with the pivot
// index up to which their steps are applied, until U reaches L, the largest
// value among the tiles' best entries: a tile with U < L does not hold the
// argmax.  Then all pending steps are applied in order in one pass, the same
// FMAs as sweep by sweep, so every stored value that is ever read is bit for
// bit the eager one.  A screen brings up to date 58 % of the carried tiles of
// the 6D n = 256 Hilbert cross, 42 % of a 6D Maxwellian's (n = 40) and 5 % of a
// 2d2v run's, whose bonds reach their ranks early (counted on the oracle's
// residuals).  It saves passes over memory, not steps, except in tiles that
// never get that far: E's traffic goes from 241 to 44 GB and the screens from
// 137 to 97 ms in the 6D Maxwellian at ranks 256, from 36 to 8.5 GB and 41 to
// 37 ms in the 2d2v run, from 13.2 to 8.6 GB and 6.4 to 6.0 ms in the Hilbert
// cross, whose screens are bound by the FP64 pipe.  The mixed forms' top-k
// candidates need a bound on the k-th largest tile, and their steps run on a
// pipe that is not the limit: there it cost more than it saved (5.9 against
// 5.4 ms when it was tried), so they bring every tile up to date in every
// screen.
// Below LAZY_BYTES of E every carried tile is brought up to date by every screen,
// which then leaves its state as well, so that the first lazy screen finds one.
// phase_bound, before a lazy screen, moves U and the best entries through the
// newest step and leaves every CTA's largest best entry per bond; the update
// phase reads single entries through their pending steps (stored_entry).

// carried tiles of bond b that have a state: those carried by the last screen too
__device__ __forceinline__ void stateful_tiles(const InstDev &in, const Ctrl &cr, const TileGeo &g,
                                               int b, int32_t &tr, int32_t &tc) {
  carried_tiles(in, g, b, ld_cg(cr.pv_rows[b]), ld_cg(cr.pv_cols[b]), tr, tc);
}
// column tiles at the run's rank caps: the stride of the states' rows; 0 if the
// instance has none or they would not fit their slots (then every carried tile
// is brought up to date by every screen)
__device__ __forceinline__ int32_t state_stride(const InstDev &in, const TileGeo &g, int b,
                                                int32_t capL, int32_t capR) {
  if (!in.lazy) return 0;
  // (superblock extents stay below 2^31)
  const int32_t nr = g.pr > 0 ? capL * g.P.tpb : (capL * (int32_t)in.n[b] - 1) / g.te + 1;
  const int32_t nc = g.pc > 0 ? capR * g.Q.tpb : (capR * (int32_t)in.n[b + 1] - 1) / g.te + 1;
  return (int64_t)nr * nc <= in.bond[b].cand_cap ? nc : 0;
}
__device__ __forceinline__ int32_t state_stride(const InstDev &in, const Ctrl &cr, const TileGeo &g,
                                                int b) {
  return state_stride(in, g, b, b == 0 ? 1 : cr.maxr[b - 1], b == in.nb - 1 ? 1 : cr.maxr[b + 1]);
}

constexpr int LAZY_MAX = 24;  // pending steps a tile may have (a screen's pass applies them)

// E(a, c) of bond b (FP64) with every step up to pivot z1 applied, from its tile's state
__device__ __forceinline__ double stepped_entry(const BondDev &B, int64_t a, int64_t c, int z0, int z1) {
  double e = B.E[a * B.ldR + c];
  int z = z0 + 1;
  for (; z + 3 <= z1; z += 4) {
    double w[4], r[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      w[k] = B.ew[(z + k) * B.ldw + a];
      r[k] = B.erow[(z + k) * B.lde + c];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) e = __fma_rn(w[k], r[k], e);
  }
  for (; z <= z1; ++z) e = __fma_rn(B.ew[z * B.ldw + a], B.erow[z * B.lde + c], e);
  return e;
}

// what the update phase needs to find the state of an entry's tile
struct LazyGeo {
  TileGeo g;
  int32_t tr, tc, stride;
};
__device__ __forceinline__ int lazy_z(const InstDev &in, const LazyGeo &q, int b, int64_t a, int64_t c,
                                      int z1) {
  if (!in.lazy || q.stride == 0) return z1;
  const int32_t tr = row_tile_of(in, q.g, b, (int32_t)a), tc = col_tile_of(in, q.g, b, (int32_t)c);
  if (tr >= q.tr || tc >= q.tc) return z1;  // not carried by the last screen: up to date
  return ld_cg(in.bond[b].tstate[(int64_t)tr * q.stride + tc].z);
}
// as a double (update phase; the mixed forms' entries are up to date)
__device__ __forceinline__ double stored_entry(const InstDev &in, const LazyGeo &q, int b, int64_t a,
                                               int64_t c, int z1) {
  const BondDev &B = in.bond[b];
  if (in.prec == P_FP64) return stepped_entry(B, a, c, lazy_z(in, q, b, a, c, z1), z1);
  const float2 v = SV<2>::load(B.E, a * B.ldR + c);
  return __dadd_rn((double)v.x, (double)v.y);
}

// phase: bound.  The states of the carried tiles through the newest step.
__device__ void bound_bond(const InstDev &in, int b, int32_t T, int32_t tc0, int32_t stride, bool pend,
                           int z1, int64_t gt, int64_t NTOT, uint64_t &best) {
  const BondDev &B = in.bond[b];
  for (int64_t x = gt; x < T; x += NTOT) {
    const int32_t tr = (int32_t)x / tc0, tc = (int32_t)x - tr * tc0;
    TileState *ts = B.tstate + (int64_t)tr * stride + tc;
    double v = ld_cg(ts->val);
    if (pend) {
      const float U = __ldcg(&ts->U);
      const int32_t row = ld_cg(ts->row), col = ld_cg(ts->col);
      const float dw = __uint_as_float(__ldcg(&B.wmax[tr])), de = __uint_as_float(__ldcg(&B.emax[tc]));
      v = __fma_rn(B.ew[(int64_t)z1 * B.ldw + row], B.erow[(int64_t)z1 * B.lde + col], v);
      ts->val = v;
      // every rounding up, and room for the rounding of the values themselves
      ts->U = __fmul_ru(__fadd_ru(U, __fmul_ru(dw, de)), 1.000001f);
    }
    const uint64_t k = abs_key(v);
    best = best > k ? best : k;
  }
}

__device__ void phase_bound(const RunArgs &ra) {
  __shared__ CtrlSnap snap;
  __shared__ int32_t s_tr[TTC_MAXB], s_tc[TTC_MAXB], s_str[TTC_MAXB], s_pend[TTC_MAXB];
  __shared__ unsigned long long s_best[TTC_MAXB];
  const int64_t NTOT = (int64_t)gridDim.x * NT;
  const int64_t gt = (int64_t)blockIdx.x * NT + threadIdx.x;
  for (int ii = 0; ii < ra.count; ++ii) {
    const InstDev &in = inst(ra, ii);
    const Ctrl &cr = *in.ctrl;
    if (!ld_cg(cr.lazy)) continue;
    snap_ctrl(cr, in.nb, snap);
    if (snap.state != ST_SCREEN) continue;
    if (threadIdx.x < in.nb) {
      const int b = threadIdx.x;
      const TileGeo g = planned_geo(in, cr, b);
      int32_t tr, tc;
      stateful_tiles(in, cr, g, b, tr, tc);
      s_tr[b] = tr;
      s_tc[b] = tc;
      s_str[b] = state_stride(in, cr, g, b);
      s_pend[b] = ld_cg(cr.e_pend[b]);
      s_best[b] = 0ull;
    }
    __syncthreads();
    for (int b = 0; b < in.nb; ++b) {
      uint64_t best = 0;
      const int32_t T = s_tr[b] * s_tc[b];
      if (T > 0 && s_str[b] > 0) {
        bound_bond(in, b, T, s_tc[b], s_str[b], s_pend[b], snap.r[b] - 1, gt, NTOT, best);
        for (int o = 16; o > 0; o >>= 1) {
          const uint64_t k = __shfl_xor_sync(0xffffffffu, best, o);
          best = best > k ? best : k;
        }
        if ((threadIdx.x & 31) == 0 && best) atomicMax(&s_best[b], (unsigned long long)best);
      }
    }
    __syncthreads();
    if (threadIdx.x < in.nb) in.bond[threadIdx.x].low[blockIdx.x] = s_best[threadIdx.x];
    __syncthreads();
  }
}

// the largest of the CTAs' best keys of bond b (a warp)
__device__ uint64_t low_key(const InstDev &in, int b) {
  uint64_t best = 0;
  for (int c = threadIdx.x & 31; c < (int)gridDim.x; c += 32) {
    const uint64_t v = ld_cg(in.bond[b].low[c]);
    best = best > v ? best : v;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t v = __shfl_xor_sync(0xffffffffu, best, o);
    best = best > v ? best : v;
  }
  return best;
}

// A carried tile (TE = 32 or 64 wide) of bond b by one warp: lane l holds
// columns l (and l + 32); rows go in rounds of 16 (TE = 32) or 8 (TE = 64),
// every load of a round issued before its first use.  Then the pending
// rank-one steps z0 + 1..z1, E(a,c) = fma(ew_z[a], erow_z[c], E(a,c)) in
// order, and the stores; the tile's best |E| (ties: lowest linear index) goes
// to *out and, with the new state, to *ts (if any).  lin: the warp's shared
// memory (mixed forms).
template <int TE, int MIX>
__device__ __noinline__ void screen_carried_warp(const InstDev &in, int b, int64_t r0, int nr,
                                                 int64_t c0, int nc, int z0, int z1, int64_t *lin,
                                                 Cand *out, TileState *ts) {
  using V = SV<MIX>;
  using VT = typename V::T;
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int NC = TE / 32;                // columns per lane
  constexpr int RR = TE == 32 ? 16 : 8;      // rows per round
  const BondDev &B = in.bond[b];
  const int lane = threadIdx.x & 31;
  const int64_t ld = B.ldR;
  bool cok[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) cok[k] = lane + 32 * k < nc;
  // mixed forms: the parts of the linear index, the rows' in shared memory
  // (their 24-bit keys tie often; FP64 looks linear indices up after the
  // rounds); the sets' parts are loaded here and used behind the first rows
  int64_t lc[NC] = {}, lr[NC] = {};
  uint32_t ci[NC] = {}, ri[NC] = {};
  if constexpr (MIX != 0) {
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const uint32_t c = (uint32_t)(c0 + min(lane + 32 * k, nc - 1)), n1 = (uint32_t)in.n[b + 1], q = c / n1;
      const uint32_t a = (uint32_t)(r0 + min(lane + 32 * k, nr - 1)), n0 = (uint32_t)in.n[b], p = a / n0;
      ci[k] = c - q * n1;
      ri[k] = a - p * n0;
      lc[k] = right_set(in, b).lin[q];
      lr[k] = left_set(in, b).lin[p];
    }
  }
  // the mixed forms have one pending step at most: its row and column values
  // wait in registers, the row's by shuffle (FP64 loads them per round and step)
  VT wa[NC], er1[NC];
  if constexpr (MIX != 0) {
    const double *ew = B.ew + (int64_t)z1 * B.ldw + r0, *er = B.erow + (int64_t)z1 * B.lde + c0;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      wa[k] = z1 > z0 ? V::load(ew, min(lane + 32 * k, nr - 1)) : V::zero();
      er1[k] = z1 > z0 ? V::load(er, min(lane + 32 * k, nc - 1)) : V::zero();
    }
  }
  // (row brr, column lane + 32 bkk) the lane's first best; tied (FP64): another
  // of its entries has the same key (rare; the linear indices decide after the
  // rounds, where they cost the loop no registers)
  uint64_t bk = 0;
  int brr = -1, bkk = 0;
  bool tied = false;
  // the rounds stay a loop: unrolled, the body is large enough to compete for
  // the instruction cache with the fresh tiles of the SM's other CTA
  const int rl = nr - 1;
  const int cl = min(lane, nc - 1), cl1 = min(lane + 32, nc - 1);  // columns, clamped
#pragma unroll 1
  for (int r1 = 0; r1 < nr; r1 += RR) {
    VT ev[RR][NC];
    {
      // rows past the tile read its last row again
      const double *E = B.E + (r0 + r1) * ld + c0;
#pragma unroll
      for (int rr = 0; rr < RR; ++rr) {
        ev[rr][0] = V::load(E, cl);
        if (NC == 2) ev[rr][NC - 1] = V::load(E, cl1);
        if (r1 + rr < rl) E += ld;
      }
    }
    if constexpr (MIX != 0) {
      if (r1 == 0) {
#pragma unroll
        for (int k = 0; k < NC; ++k) {
          lc[k] += (int64_t)ci[k] * in.stride[b + 1];
          lin[lane + 32 * k] = lr[k] + (int64_t)ri[k] * in.stride[b];
        }
        __syncwarp();
      }
    }
    if constexpr (MIX != 0) {
      if (z1 > z0) {
#pragma unroll
        for (int rr = 0; rr < RR; ++rr) {
          const int row = r1 + rr;  // (the halves of wa: r1 is a multiple of RR <= 32)
          VT w;
          w.x = __shfl_sync(FULL, NC == 2 && r1 >= 32 ? wa[NC - 1].x : wa[0].x, row & 31);
          w.y = __shfl_sync(FULL, NC == 2 && r1 >= 32 ? wa[NC - 1].y : wa[0].y, row & 31);
#pragma unroll
          for (int k = 0; k < NC; ++k) ev[rr][k] = V::step(w, er1[k], ev[rr][k]);
        }
      }
    } else for (int z = z0 + 1; z <= z1; ++z) {
      const double *ew = B.ew + (int64_t)z * B.ldw + r0 + r1;
      const double *er = B.erow + (int64_t)z * B.lde + c0;
      VT e[NC];
      e[0] = V::load(er, cl);
      if (NC == 2) e[NC - 1] = V::load(er, cl1);
#pragma unroll
      for (int rr = 0; rr < RR; ++rr) {
        const VT w = V::load(ew, min(rr, rl - r1));
#pragma unroll
        for (int k = 0; k < NC; ++k) ev[rr][k] = V::step(w, e[k], ev[rr][k]);
      }
    }
    if (z1 > z0) {
      double *E = B.E + (r0 + r1) * ld + c0;
#pragma unroll
      for (int rr = 0; rr < RR; ++rr) {
        if (r1 + rr <= rl) {
          if (cok[0]) V::store(E, lane, ev[rr][0]);
          if (NC == 2 && cok[NC - 1]) V::store(E, lane + 32, ev[rr][NC - 1]);
        }
        E += ld;
      }
    }
#pragma unroll
    for (int rr = 0; rr < RR; ++rr)
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        if (r1 + rr > rl || !cok[k]) continue;
        const uint64_t key = V::key(ev[rr][k]);
        bool take = brr < 0 || key > bk;
        if constexpr (MIX == 0)
          tied = !take && (tied || key == bk);
        else if (!take && key == bk)
          take = lin[r1 + rr] + lc[k] < lin[brr] + lc[bkk];
        if (take) {
          bk = key;
          brr = r1 + rr;
          bkk = k;
        }
      }
  }
  int bcc = lane + 32 * bkk;
  int64_t bl = LLONG_MAX;
  if (brr >= 0) bl = MIX == 0 ? entry_lin(in, b, r0 + brr, c0 + bcc) : lin[brr] + lc[bkk];
  if (MIX == 0 && tied) {
#pragma unroll 1
    for (int row = brr; row < nr; ++row)
#pragma unroll 1
      for (int col = lane; col < nc; col += 32) {
        if (V::key(V::load(B.E, (r0 + row) * ld + c0 + col)) != bk) continue;
        const int64_t l = entry_lin(in, b, r0 + row, c0 + col);
        if (l < bl) {
          bl = l;
          brr = row;
          bcc = col;
        }
      }
  }
  const int mine = brr < 0 ? -1 : brr * 64 + bcc;
  for (int off = 16; off > 0; off >>= 1) {
    const uint64_t ok = __shfl_xor_sync(FULL, bk, off);
    const int64_t ol = __shfl_xor_sync(FULL, bl, off);
    const int orr = __shfl_xor_sync(FULL, brr, off);
    const int oc = __shfl_xor_sync(FULL, bcc, off);
    if (orr >= 0 && (brr < 0 || kb_better(KeyBest{ok, ol, orr, oc}, KeyBest{bk, bl, brr, bcc}))) {
      bk = ok;
      bl = ol;
      brr = orr;
      bcc = oc;
    }
  }
  if (lane == 0) *out = Cand{bk, bl, (int32_t)(r0 + brr), (int32_t)(c0 + bcc)};
  if constexpr (MIX == 0)
    if (ts && mine == brr * 64 + bcc) {  // the lane that holds (and stored) the best
      const double bv = B.E[(r0 + brr) * ld + c0 + bcc];
      *ts = TileState{abs_up(bv), z1, bv, bl, (int32_t)(r0 + brr), (int32_t)(c0 + bcc)};
    }
  __syncwarp();
}

__device__ __forceinline__ void carried_warp(const InstDev &in, int te, int b, int64_t r0, int nr,
                                             int64_t c0, int nc, int z0, int z1, int64_t *lin,
                                             Cand *out, TileState *ts) {
  if (in.prec == P_FP64) {
    if (te == 32)
      screen_carried_warp<32, 0>(in, b, r0, nr, c0, nc, z0, z1, lin, out, ts);
    else
      screen_carried_warp<64, 0>(in, b, r0, nr, c0, nc, z0, z1, lin, out, ts);
  } else {
    if (te == 32)
      screen_carried_warp<32, 2>(in, b, r0, nr, c0, nc, z0, z1, lin, out, ts);
    else
      screen_carried_warp<64, 2>(in, b, r0, nr, c0, nc, z0, z1, lin, out, ts);
  }
}

// carried tiles [t0, t1) of bond b by one warp (t1 - t0 <= 32; tc0 column tiles):
// a lane per tile finds the pivot its entries are at and whether a candidate
// may lie in it; those tiles are brought up to pivot cur.  low: the bond's L.
// cand: the bond's slots after the fresh items'; FP64 lists its candidates
// there (a place each from ntiles, one atomic per run), the mixed forms use a
// slot per tile.
__device__ __forceinline__ void carried_run(const InstDev &in, const TileGeo &g, int b, int32_t t0,
                                            int32_t t1, int32_t tc0, int32_t cur, int32_t pend,
                                            int32_t ptr, int32_t ptc, int32_t stride, uint64_t low,
                                            int64_t *lin, Cand *cand, unsigned long long &fma,
                                            unsigned long long &bytes) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const bool has = t0 + lane < t1;
  int32_t zt = has ? (pend ? cur - 1 : cur) : -1;  // (first time: fresh in the last screen)
  unsigned todo = __ballot_sync(FULL, has);
  if (in.prec == P_FP64) {
    bool asis = false;  // up to date as it stands, and its best entry is a candidate
    uint64_t key = 0;
    const TileState *ts = nullptr;
    if (has) {
      const int32_t tr = (t0 + lane) / tc0, tc = t0 + lane - tr * tc0;
      if (tr < ptr && tc < ptc) {
        ts = in.bond[b].tstate + (int64_t)tr * stride + tc;
        const int32_t z = ld_cg(ts->z);
        const float U = __ldcg(&ts->U);
        key = abs_key(ld_cg(ts->val));
        const bool skip = (double)U < __longlong_as_double((long long)low);
        asis = z == cur && key >= low;
        zt = (z == cur || (skip && cur - z < LAZY_MAX)) ? -1 : z;
      }
    }
    todo = __ballot_sync(FULL, zt >= 0);
    const unsigned kept = __ballot_sync(FULL, asis);
    if (!(todo | kept)) return;
    int32_t at = 0;
    if (lane == 0) at = atomicAdd(&in.ctrl->ntiles[b], __popc(todo) + __popc(kept));
    cand += __shfl_sync(FULL, at, 0);
    if (asis)
      cand[__popc(todo) + __popc(kept & ((1u << lane) - 1))] =
          Cand{key, ld_cg(ts->lin), ld_cg(ts->row), ld_cg(ts->col)};
  } else {
    cand += t0;
  }
  unsigned long long nf = 0, nb = 0;
  for (; todo; todo &= todo - 1, ++cand) {
    const int x = __ffs(todo) - 1;
    const int z0 = __shfl_sync(FULL, zt, x);
    const int32_t tr = (t0 + x) / tc0, tc = t0 + x - tr * tc0;
    int64_t r0, c0;
    int nr, nc;
    tile_rows(in, g, b, tr, r0, nr);
    tile_cols(in, g, b, tc, c0, nc);
    carried_warp(in, g.te, b, r0, nr, c0, nc, z0, cur, lin, cand,
                 stride > 0 ? in.bond[b].tstate + (int64_t)tr * stride + tc : nullptr);
    const unsigned long long e = (unsigned long long)nr * nc;
    nf += e * (unsigned long long)(cur - z0);
    nb += (cur > z0 ? 16 : 8) * e;
  }
  if (lane == 0) {
    atomicAdd(&fma, nf);
    atomicAdd(&bytes, nb);
  }
}

// A carried tile of bond b by the whole CTA, from pivot z0 to cur: an eighth of its rows
// to each warp.  Its best entry goes to the bond's next listed slot (FP64) or
// to the tile's own (mixed forms), and to its state.
__device__ __forceinline__ void carried_cta(const InstDev &in, const TileGeo &g, int b, int32_t t, int32_t tc0,
                            int32_t z0, int32_t cur, int32_t stride, int64_t *lin, Cand *cand,
                            unsigned long long &fma, unsigned long long &bytes) {
  __shared__ Cand s_cand[NT / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int32_t tr = t / tc0, tc = t - tr * tc0;
  int64_t r0, c0;
  int nr, nc;
  tile_rows(in, g, b, tr, r0, nr);
  tile_cols(in, g, b, tc, c0, nc);
  const int h = g.te / (NT / 32), nh = min(h, nr - warp * h);
  if (nh > 0)
    carried_warp(in, g.te, b, r0 + warp * h, nh, c0, nc, z0, cur, lin, &s_cand[warp], nullptr);
  else if (lane == 0)
    s_cand[warp].row = -2;
  __syncthreads();
  if (threadIdx.x == 0) {
    KeyBest best{0ull, LLONG_MAX, -1, -1};
    for (int w = 0; w < NT / 32; ++w)
      kb_take_any(best, KeyBest{s_cand[w].key, s_cand[w].lin, s_cand[w].row, s_cand[w].col});
    cand += in.prec == P_FP64 ? atomicAdd(&in.ctrl->ntiles[b], 1) : t;
    *cand = Cand{best.key, best.lin, best.row, best.col};
    if (stride > 0) {
      const double v = in.bond[b].E[best.row * in.bond[b].ldR + best.col];
      in.bond[b].tstate[(int64_t)tr * stride + tc] = TileState{abs_up(v), cur, v, best.lin, best.row, best.col};
    }
    const unsigned long long e = (unsigned long long)nr * nc;
    fma += e * (unsigned long long)(cur - z0);
    bytes += (cur > z0 ? 16 : 8) * e;
  }
}

// carried tiles a CTA below which CTAs take them one at a time
constexpr int TOGETHER = 4;

// Queue B of the stored screen (below) so taken, an item a tile: first < 0 is a CTA that
// started on the other queue.  (Out of line: inlined, its registers cost the
// large screens 1 %.)
__device__ __noinline__ void carried_together(const InstDev &in, const int32_t *r, const TileGeo *geo,
                                              const int32_t *tr0, const int32_t *tc0,
                                              const int32_t *pend, const int32_t *stride,
                                              const int32_t *nf, int32_t first, int32_t H, int32_t N,
                                              int64_t *lin, int32_t &item, unsigned long long &fma,
                                              unsigned long long &bytes) {
  int32_t nxt = 0;
  if (threadIdx.x == 0) item = first >= 0 ? first : H < N ? H + atomicAdd(&in.ctrl->steal2, 1) : N;
  for (;;) {
    __syncthreads();
    int32_t j = item;
    __syncthreads();
    if (j >= N) break;
    if (threadIdx.x == 0) nxt = H + atomicAdd(&in.ctrl->steal2, 1);
    int b = 0;
    for (; j >= tr0[b] * tc0[b]; ++b) j -= tr0[b] * tc0[b];
    const int32_t cur = r[b] - 1;
    carried_cta(in, geo[b], b, j, tc0[b], pend[b] ? cur - 1 : cur, cur, stride[b], lin,
                in.cand + in.bond[b].cand_base + nf[b], fma, bytes);
    if (threadIdx.x == 0) item = nxt;
  }
}

// The stored screen of one instance.  Work items come from two queues:
//   A: tiles new to a superblock (fresh: A - T R, r_k FMAs per entry, FP64
//      pipe or FP32 pipe in the mixed forms), one tile (or quarter) per item;
//   B: carried tiles, a run of them to a warp at a time: its lanes look up
//      which of them a candidate may lie in, and the warp brings those up to
//      date (one load, one FMA per pending step and one store per entry).
// The CTAs of the first half of the SM-spread order (one per SM) start on A,
// the others on B, so that every SM keeps its FP64 / FP32 pipe and its
// memory path busy at once; a CTA whose queue runs dry moves to the other.
// Place s takes the first item of its queue implicitly, later items come
// from the queue's counter, fetched when an item starts so that the atomic's
// round trip overlaps it.  The decide phase clears both counters.  A run is a
// sixth of a warp's even share (at most 32 tiles: its lanes; a warp's tile
// takes 40 us beside seven others and a CTA on fresh tiles, so runs of eight
// tiles per CTA left tails of half a sweep).  Where every carried tile is due and
// they are fewer than TOGETHER a CTA, CTAs take them one at a time (a warp at a tile
// each is 3D n = 70 Hilbert in 1.00 ms for 0.78, 6D n = 64 in 1.42 for 1.25, 8 of them
// in a batch 6.70 for 4.96; from two a CTA on: 1.27 and 5.19, from eight 1.25 and
// 4.96, 6D n = 64 with two pieces a mode 1.47 for 1.40).  Not the mixed forms' 32-wide
// tiles, of which a warp has but four rows: 6D n = 64 with two pieces 1.38 for 1.33 ms.
// A bond's candidate slots are its fresh items' (nfresh), then its carried
// tiles' (ntiles).

__device__ void screen_stored_instance(const InstDev &in, const int32_t *r, PhaseSmem &sm) {
  const Ctrl &cr = *in.ctrl;
  int32_t *ctr[2] = {&in.ctrl->steal, &in.ctrl->steal2};
  // per-bond geometry, stored extent and item counts, staged once
  __shared__ TileGeo s_geo[TTC_MAXB];
  __shared__ int32_t s_sr[TTC_MAXB], s_sc[TTC_MAXB], s_pend[TTC_MAXB];
  __shared__ int32_t s_tr0[TTC_MAXB], s_tc0[TTC_MAXB];
  __shared__ int32_t s_ptr[TTC_MAXB], s_ptc[TTC_MAXB], s_str[TTC_MAXB];  // tiles with a state
  __shared__ uint64_t s_low[TTC_MAXB];
  __shared__ int32_t s_item;
  __shared__ unsigned long long s_fma, s_byte;
  __syncthreads();
  if (threadIdx.x == 0) s_fma = s_byte = 0ull;
  const bool lazy = ld_cg(cr.lazy);  // carried tiles wait for their steps
  const int32_t qs = ld_cg(cr.qsplit);  // eighths of the CTAs that start on A (0: half)
  if (threadIdx.x < in.nb) {
    const int b = threadIdx.x;
    // (every word in one round of loads: each more is 0.4 us of a small sweep)
    const int32_t sr = ld_cg(cr.st_rows[b]), sc = ld_cg(cr.st_cols[b]);
    const int32_t pr = ld_cg(cr.pv_rows[b]), pc = ld_cg(cr.pv_cols[b]);
    const int32_t pend = ld_cg(cr.e_pend[b]);
    const int32_t capL = b == 0 ? 1 : ld_cg(cr.maxr[b - 1]), capR = b == in.nb - 1 ? 1 : ld_cg(cr.maxr[b + 1]);
    const TileGeo g = planned_geo(in, cr, b);
    int32_t tr0, tc0, ptr, ptc;
    carried_tiles(in, g, b, sr, sc, tr0, tc0);
    carried_tiles(in, g, b, pr, pc, ptr, ptc);
    s_geo[b] = g;
    s_sr[b] = sr;
    s_sc[b] = sc;
    s_pend[b] = pend;
    s_tr0[b] = tr0;
    s_tc0[b] = tc0;
    s_str[b] = state_stride(in, g, b, capL, capR);
    const bool has = s_str[b] > 0 && lazy;
    s_ptr[b] = has ? ptr : 0;
    s_ptc[b] = has ? ptc : 0;
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int b = warp; b < in.nb; b += NT / 32) {
    const uint64_t k = s_ptr[b] * s_ptc[b] > 0 ? low_key(in, b) : 0;
    if (lane == 0) s_low[b] = k;
  }
  // with fewer fresh tiles than CTAs, fresh tiles go out as quarters
  // (32 x 32) so that their work spreads over four times as many CTAs
  int32_t nf = 0, nc_all = 0;
  for (int b = 0; b < in.nb; ++b) {
    const int32_t nt = s_geo[b].nrt * s_geo[b].nct, nc = s_tr0[b] * s_tc0[b];
    nf += nt - nc;
    nc_all += nc;
  }
  const int32_t G = gridDim.x;
  const bool together =
      !lazy && nc_all < TOGETHER * G && (s_geo[0].te == 64 || in.prec == P_FP64);
  const int32_t run = together ? 1 : max(1, min(32, nc_all / (6 * G * (NT / 32))));  // tiles of a B item
  int32_t nB = run == 1 ? nc_all : 0;
  for (int b = 0; b < in.nb && run > 1; ++b) nB += (s_tr0[b] * s_tc0[b] + run - 1) / run;
  const bool quarters = s_geo[0].te == 64 && nf < (int32_t)gridDim.x;
  const int32_t spt = quarters ? STORED_SLOTS : 1;  // items per tile
  const int32_t nA = spt * nf;
  const int32_t HA = nA == 0 ? 0 : nB == 0 ? G : qs > 0 ? max(1, min(G - 1, G * qs / 8))
                                                         : (G + 1) / 2;
  const int32_t HB = (G - HA) * (together ? 1 : NT / 32);  // CTAs or warps that start on B
  __shared__ int32_t s_nf[TTC_MAXB], s_nc[TTC_MAXB];  // slots of the fresh items, carried tiles
  if (threadIdx.x < in.nb) {
    const int b = threadIdx.x, nc = s_tr0[b] * s_tc0[b];
    s_nc[b] = nc;
    s_nf[b] = (s_geo[b].nrt * s_geo[b].nct - nc) * spt;
  }
  __syncthreads();
  if (s_place == G - 1 && threadIdx.x == 0)  // (the place the items reach last)
    screen_bookkeeping(in, r, s_geo, s_sr, s_sc, s_tr0, s_tc0, s_pend, s_nf, s_nc);
  const bool a_first = s_place < HA;
  for (int part = 0; part < 2; ++part) {
    if ((part == 0) == a_first) {
      // queue A, the CTA together (a CTA that started on B asks only if there is
      // more than the others' first items)
      int32_t nxt = 0;
      if (threadIdx.x == 0) s_item = a_first ? s_place : HA < nA ? HA + atomicAdd(ctr[0], 1) : nA;
      for (;;) {
        __syncthreads();
        int32_t j = s_item;
        __syncthreads();
        if (j >= nA) break;
        if (threadIdx.x == 0) nxt = HA + atomicAdd(ctr[0], 1);
        // a fresh tile (or quarter q of it)
        const int32_t qt = j % spt;
        j /= spt;
        for (int b = 0; b < in.nb; ++b) {
          const TileGeo &g = s_geo[b];
          const int32_t tr0 = s_tr0[b], tc0 = s_tc0[b];
          const int32_t cnt = g.nrt * g.nct - tr0 * tc0;
          if (j >= cnt) {
            j -= cnt;
            continue;
          }
          int32_t tr, tc;
          if (j < tr0 * (g.nct - tc0)) {
            // new columns of the stored rows
            tr = j / (g.nct - tc0);
            tc = tc0 + (j - tr * (g.nct - tc0));
          } else {
            // new rows, every column
            const int32_t u = j - tr0 * (g.nct - tc0);
            tr = tr0 + u / g.nct;
            tc = u - (tr - tr0) * g.nct;
          }
          Cand *slot = in.cand + in.bond[b].cand_base + j * spt + qt;
          int64_t r0, c0;
          int nr, nc;
          tile_rows(in, g, b, tr, r0, nr);
          tile_cols(in, g, b, tc, c0, nc);
          int te = g.te;
          if (quarters) {
            // quarter qt of the tile: rows / columns [32 qr, 32 qr + 32)
            const int h = te / 2, qr = qt >> 1, qc = qt & 1;
            r0 += h * qr;
            c0 += h * qc;
            nr = min(h, nr - h * qr);
            nc = min(h, nc - h * qc);
            te = h;
          }
          if (nr > 0 && nc > 0)
            screen_tile_stored(in, b, r[b], r0, nr, c0, nc, te, s_sr[b], s_sc[b], s_pend[b], slot,
                               sm.s);
          else if (threadIdx.x == 0)
            *slot = Cand{0ull, LLONG_MAX, -2, -2};  // an empty quarter
          break;
        }
        if (threadIdx.x == 0) s_item = nxt;
      }
    } else if (together) {
      carried_together(in, r, s_geo, s_tr0, s_tc0, s_pend, s_str, s_nf, a_first ? -1 : s_place - HA, HB, nB,
                       reinterpret_cast<int64_t *>(&sm.s.op) + warp * BM, s_item, s_fma, s_byte);
    } else {
      // queue B, each warp on its own
      int64_t *lin = reinterpret_cast<int64_t *>(&sm.s.op) + warp * BM;
      int32_t item = a_first ? nB : (s_place - HA) * (NT / 32) + warp;
      if (a_first && HB < nB) {
        if (lane == 0) item = HB + atomicAdd(ctr[1], 1);
        item = __shfl_sync(0xffffffffu, item, 0);
      }
      while (item < nB) {
        int32_t nxt = lane == 0 ? HB + atomicAdd(ctr[1], 1) : 0;
        int32_t j = item;
        for (int b = 0; b < in.nb; ++b) {
          const int32_t tc0 = s_tc0[b], nc_b = s_tr0[b] * tc0;
          const int32_t cnt = (nc_b + run - 1) / run;
          if (j >= cnt) {
            j -= cnt;
            continue;
          }
          carried_run(in, s_geo[b], b, j * run, min(nc_b, (j + 1) * run), tc0, r[b] - 1, s_pend[b],
                      s_ptr[b], s_ptc[b], s_str[b], s_low[b], lin,
                      in.cand + in.bond[b].cand_base + s_nf[b], s_fma, s_byte);
          break;
        }
        item = __shfl_sync(0xffffffffu, nxt, 0);
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0 && s_byte) {
    atomicAdd((unsigned long long *)&in.ctrl->screen_fmas, s_fma);
    atomicAdd((unsigned long long *)&in.ctrl->stored_bytes, s_byte);
  }
}

// ---------------------------------------------------------------------------
// Alg. 1 with a random sample set L (recompute form, FP64).  Per screen t
// and bond b, samples j < nl are the superblock entries
//   a = floor(x rows / 2^64), c = floor(x' cols / 2^64),
//   x = SplitMix64(seed) output 2i, x' = output 2i+1, i = (t nb + b) nl + j;
// their argmax (lowest linear index on ties) is refined by whole-column and
// whole-row scans (the while loop of Alg. 1) in the refinement phases.

// E(a,c) = A(a,c) - chain(T(a,:), R(:,c)) with K terms: the contract's residual
__device__ __forceinline__ double residual_at(const InstDev &in, int b, int K, int64_t a,
                                              int64_t c) {
  const BondDev &B = in.bond[b];
  return __dsub_rn(sb_entry(in, b, a, c), chain(B.T + a, B.ldT, B.R + c, B.ldR, K));
}

__device__ __forceinline__ void take_key(KeyBest &best, double e, int64_t lin, int64_t a,
                                         int64_t c) {
  const uint64_t k = abs_key(e);
  if (best.row < 0 || k > best.key || (k == best.key && lin < best.lin)) {
    best.key = k;
    best.lin = lin;
    best.row = (int32_t)a;
    best.col = (int32_t)c;
  }
}

// CTAs that work on bond b in a sampled screen or a refinement step: every nb-th
// one (each CTA has one bond, so one block reduction instead of nb in turn), or
// all of them where a column or row is longer than 16 passes of such a share
// (wide) or the grid has fewer CTAs than there are bonds; a CTA's candidate goes to slot `rank` of the bond.
__device__ __forceinline__ int share_size(const InstDev &in, int b, bool wide) {
  return wide || (int)gridDim.x < in.nb ? (int)gridDim.x : ((int)gridDim.x - b + in.nb - 1) / in.nb;
}
__device__ __forceinline__ int share_rank(const InstDev &in, int b, bool wide) {
  if (wide || (int)gridDim.x < in.nb) return blockIdx.x;
  return (int)blockIdx.x % in.nb == b ? (int)blockIdx.x / in.nb : -1;
}
__device__ __forceinline__ bool share_wide(const InstDev &in, const int32_t *r) {
  int64_t longest = 0;
  for (int b = 0; b < in.nb; ++b) longest = max(longest, max(rows_of(in, r, b), cols_of(in, r, b)));
  return longest > (int64_t)16 * NT * max(1, (int)gridDim.x / in.nb);
}

// chain(row ra of A, row rb of Bm) over K terms for every lane of a warp, the rows
// contiguous (lda, ldb entries apart): sixteen entries at a time, the warp loads
// its 32 lanes' rows together, two rows per instruction, into shared memory
// (32 x 17 doubles), and each lane runs the contract's chain on its own two (a
// thread reading its own rows touches 32 lines per load).
__device__ __forceinline__ double warp_chain_rows(const double *A, int64_t ra, int64_t lda,
                                                  const double *Bm, int64_t rb, int64_t ldb, int K,
                                                  double *buf) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, half = lane >> 4, el = lane & 15;
  double acc = 0.0;
  for (int c = 0; c < K; c += 16) {
    const bool has = c + el < K;
    double xv[16], yv[16];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const double *tab = (side == 0 ? A : Bm) + c + el;
      const int64_t o = side == 0 ? ra * lda : rb * ldb;
      double v[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int64_t os = __shfl_sync(FULL, o, 2 * q + half);
        v[q] = has ? tab[os] : 0.0;
      }
      __syncwarp();  // the previous rows are read
#pragma unroll
      for (int q = 0; q < 16; ++q) buf[(2 * q + half) * 17 + el] = v[q];
      __syncwarp();
#pragma unroll
      for (int t = 0; t < 16; ++t) {
        if (side == 0)
          xv[t] = buf[lane * 17 + t];
        else
          yv[t] = buf[lane * 17 + t];
      }
    }
#pragma unroll
    for (int t = 0; t < 16; ++t)
      if (c + t < K) acc = __fma_rn(xv[t], yv[t], acc);
  }
  return acc;
}

// The CTA's best of its share of the samples of every bond, into the bond's
// slot (thread x of the bond's share takes samples x, x + share NT, ...).  A
// sample's row of T and column of R come from copies that keep them
// contiguous: from the t-major factors every entry is a 32-byte sector of its
// own (2 GB of L2 traffic a screen of 2^18 samples per bond at ranks 24).  An
// instance that had no memory for the copies reads the factors.
__device__ void screen_sampled_instance(const InstDev &in, const int32_t *r, int64_t t,
                                        PhaseSmem &sm) {
  double *buf = sm.sw.rows[threadIdx.x >> 5];
  for (int b = 0; b < in.nb; ++b) {
    const int rank = share_rank(in, b, false);
    if (rank < 0) continue;
    const int64_t NTOT = (int64_t)share_size(in, b, false) * NT, gt = (int64_t)rank * NT + threadIdx.x;
    __syncthreads();  // (the rows share memory with the reduction below)
    const BondDev &B = in.bond[b];
    const int64_t rows = rows_of(in, r, b), cols = cols_of(in, r, b);
    KeyBest best{0ull, LLONG_MAX, -1, -1};
    for (int64_t j = gt;; j += NTOT) {
      const bool valid = j < in.nl;
      if (!__any_sync(0xffffffffu, valid)) break;
      const uint64_t i = (uint64_t)((t * in.nb + b) * in.nl + (valid ? j : 0));
      const int64_t a = (int64_t)__umul64hi(splitmix64_at(in.lseed, 2 * i), (uint64_t)rows);
      const int64_t c = (int64_t)__umul64hi(splitmix64_at(in.lseed, 2 * i + 1), (uint64_t)cols);
      const double acc = B.Tr ? warp_chain_rows(B.Tr, a, B.ldr, B.Rr, c, B.ldr, r[b], buf)
                              : chain(B.T + a, B.ldT, B.R + c, B.ldR, r[b]);
      if (!valid) continue;
      const double e = __dsub_rn(sb_entry(in, b, a, c), acc);
      if (best.row < 0 || abs_key(e) >= best.key) take_key(best, e, entry_lin(in, b, a, c), a, c);
    }
    best = block_best(best, sm.s.sk, sm.s.sl, sm.s.sr, sm.s.sc);
    if (threadIdx.x == 0) {
      Cand *slot = in.cand + in.bond[b].cand_base + rank;
      *slot = best.row >= 0 ? Cand{best.key, best.lin, best.row, best.col}
                            : Cand{0ull, LLONG_MAX, -2, -2};
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    Ctrl &cw = *in.ctrl;
    int64_t fmas = 0;
    for (int b = 0; b < in.nb; ++b) fmas += in.nl * r[b];
    cw.sweeps += 1;
    cw.entries += in.nl * in.nb;
    cw.entries_fresh += in.nl * in.nb;
    cw.screen_fmas += fmas;
    cw.screened = 1;
  }
}

__device__ void phase_screen(const RunArgs &ra, PhaseSmem &sm) {
  __shared__ CtrlSnap snap;
  const int32_t G = gridDim.x;
  int64_t base = 0;
  int32_t boff = 0;  // base mod G
  for (int ii = 0; ii < ra.count; ++ii) {
    const InstDev &in = inst(ra, ii);
    const Ctrl &cr = *in.ctrl;
    snap_ctrl(cr, in.nb, snap);
    if (blockIdx.x == 0 && threadIdx.x == 0)
      in.ctrl->dkind = snap.state == ST_SCREEN ? DK_BONDS : snap.state == ST_VERIFY ? DK_VERIFY
                                                                                   : DK_NONE;
    if (snap.state != ST_SCREEN) continue;
    const int32_t *r = snap.r;
    if (in.stored) {
      screen_stored_instance(in, r, sm);
      continue;
    }
    if (in.nl > 0) {
      // the screen counter is advanced by the decide phase, never here
      screen_sampled_instance(in, r, ld_cg(cr.screen_t), sm);
      continue;
    }
    // every bond's tile geometry, one bond per thread
    __shared__ TileGeo s_pg[TTC_MAXB];
    __syncthreads();
    if (threadIdx.x < in.nb) s_pg[threadIdx.x] = planned_geo(in, cr, threadIdx.x);
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0)
      screen_bookkeeping(in, r, s_pg, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr);
    for (int b = 0; b < in.nb; ++b) {
      const TileGeo &g = s_pg[b];
      const int32_t nt = g.nrt * g.nct;
      for (int32_t lt = ((int32_t)blockIdx.x - boff + G) % G; lt < nt; lt += G) {
        const int32_t tr = lt / g.nct, tc = lt - tr * g.nct;
        int64_t r0, c0;
        int nr, nc;
        tile_rows(in, g, b, tr, r0, nr);
        tile_cols(in, g, b, tc, c0, nc);
        if (in.prec == P_SPLIT)
          screen_tile_mixed<true>(in, b, r[b], r0, nr, c0, nc, g.te,
                                  in.mcand + in.bond[b].cand_base + lt, sm.s);
        else if (in.prec == P_FP32)
          screen_tile_mixed<false>(in, b, r[b], r0, nr, c0, nc, g.te,
                                   in.mcand + in.bond[b].cand_base + lt, sm.s);
        else
          screen_tile_fp64(in, b, r[b], r0, nr, c0, nc, g.te, in.cand + in.bond[b].cand_base + lt,
                           sm.s);
      }
      base += nt;
      boff = (int32_t)((boff + nt) % G);
    }
  }
}

// ---------------------------------------------------------------------------
// decide: append the pivot (a*, c*) to bond b (block-wide).  I_{<=k} gets
// (alpha*, i*), J_{>k} gets (j*, beta*) (eq. nestedpivots); the history of
// step z keeps c_z = R(:, c*), T(a*, :) and delta.  P^{-1} is bordered in the
// update phase (border_inverse): no decision reads it.
__device__ bool append_pivot(const InstDev &in, Ctrl &cr, int b, int64_t as, int64_t cs, int z,
                             DecideSmem &sm) {
  const BondDev &B = in.bond[b];
  const int cap = B.cap;
  const int tid = threadIdx.x;
  const int64_t nb0 = in.n[b], nb1 = in.n[b + 1];
  const int64_t p = as / nb0, i = as - p * nb0;
  const int64_t q = cs / nb1, j = cs - q * nb1;
  const SetDev &L = left_set(in, b);
  const SetDev &Rset = right_set(in, b);
  const bool hil = in.gen == 0;
  // one round of independent loads: warp 1 appends the index sets (a lane
  // per index), threads t < z gather the history (R(t, c*), T(a*, t))
  if (tid >= 32 && tid < 64) {
    const int lane = tid - 32;
    const int wl = b, wj = in.d - 1 - b;
    if (lane < wl) B.I.idx[(int64_t)z * (wl + 1) + lane] = L.idx[p * wl + lane];
    if (lane == wl) B.I.idx[(int64_t)z * (wl + 1) + wl] = (int32_t)i;
    if (lane == 0) B.J.idx[(int64_t)z * wj] = (int32_t)j;
    if (lane >= 1 && lane < wj) B.J.idx[(int64_t)z * wj + lane] = Rset.idx[q * (wj - 1) + lane - 1];
    if (lane == 16) B.I.lin[z] = L.lin[p] + i * in.stride[b];
    if (lane == 17) B.I.sum[z] = L.sum[p] + (int32_t)i;
    if (lane == 18) B.J.lin[z] = j * in.stride[b + 1] + Rset.lin[q];
    if (lane == 19) B.J.sum[z] = (int32_t)j + Rset.sum[q];
    if (lane == 20) {
      B.prow[z] = (int32_t)as;
      B.pcol[z] = (int32_t)cs;
    }
  }
  double *hc = B.hc + (int64_t)z * cap;
  double *hp = B.hpiv + (int64_t)z * cap;
  for (int t = tid; t < z; t += NT) {
    const double c = B.R[(int64_t)t * B.ldR + cs], v = B.T[(int64_t)t * B.ldT + as];
    hc[t] = c;
    hp[t] = v;
    sm.hcs[t] = c;
    sm.hps[t] = v;
  }
  // the pivot entry A(a*, c*), by a thread of its own beside the gathers
  if (tid == NT - 1)
    sm.apiv = hil ? in.hilb[L.sum[p] + (int32_t)i + (int32_t)j + Rset.sum[q]] : sb_entry(in, b, as, cs);
  __syncthreads();
  if (tid == 0) {
    const double piv = __dsub_rn(sm.apiv, chain(sm.hps, 1, sm.hcs, 1, z));
    const double delta = 1.0 / piv;
    // 1: a usable pivot; 0: the residual formed afresh at the pivot is zero
    // (or its reciprocal overflows), so the screened value was rounding
    // noise and the bond takes no pivot; -1: not finite
    sm.flag = isfinite(delta) ? 1 : isfinite(piv) ? 0 : -1;
    // (several CTAs append pivots of one instance at once)
    if (sm.flag == 1) atomicMax((unsigned long long *)&cr.piv_max, (unsigned long long)abs_key(piv));
    B.delta[z] = delta;
  }
  __syncthreads();
  return sm.flag == 1;
}

// update: P^{-1} of bond b bordered by the pivot of step z (block-wide, one
// CTA): [[U + d U a b U, -d U a], [-d b U, d]] with a = R(:, c*) and b the
// pivot row A(a*, c_t), t < z (Sec. 3.1.1).  Nothing but the getters reads U,
// so it is not on the decide phase's critical path: there its two rounds of
// chains and the z^2 update on one SM took most of a decide at high ranks
// (100 us a sweep at ranks 256; beside the replays they cost nothing).
__device__ __noinline__ void border_inverse(const InstDev &in, int b, int z, DecideSmem &sm) {
  const BondDev &B = in.bond[b];
  const int cap = B.cap;
  const int tid = threadIdx.x;
  const int64_t as = B.prow[z];
  const bool ustage = z <= DEC_US;
  double *U = B.U;
  const double delta = B.delta[z];
  __syncthreads();
  for (int t = tid; t < z; t += NT) {
    sm.hcs[t] = B.hc[(int64_t)z * cap + t];
    sm.brow[t] = sb_entry(in, b, as, B.pcol[t]);
  }
  if (ustage)
    for (int x = tid; x < z * z; x += NT) {
      const int t = x / z, u = x - t * z;
      sm.us[x] = U[(int64_t)t * cap + u];
    }
  __syncthreads();
  const double *Ur = ustage ? sm.us : U;
  const int64_t ldu = ustage ? z : cap;
  // U a and b U side by side: lanes [0, z) take the rows, [z, 2z) the columns
  for (int x = tid; x < 2 * z; x += NT) {
    if (x < z)
      sm.ua[x] = chain(Ur + (int64_t)x * ldu, 1, sm.hcs, 1, z);
    else
      sm.bu[x - z] = chain(sm.brow, 1, Ur + (x - z), ldu, z);
  }
  __syncthreads();
  for (int x = tid; x < z * z; x += NT) {
    const int t = x / z, u = x - t * z;
    const double du = __dmul_rn(delta, sm.ua[t]);
    U[(int64_t)t * cap + u] = __fma_rn(du, sm.bu[u], Ur[(int64_t)t * ldu + u]);
  }
  for (int t = tid; t < z; t += NT) {
    U[(int64_t)t * cap + z] = -__dmul_rn(delta, sm.ua[t]);
    U[(int64_t)z * cap + t] = -__dmul_rn(delta, sm.bu[t]);
  }
  if (tid == 0) {
    U[(int64_t)z * cap + z] = delta;
    in.ctrl->u_rank[b] = z + 1;
  }
  __syncthreads();
}

// FP64 residual of superblock entry (a, c) with the contract's chain
__device__ double residual64(const InstDev &in, const Ctrl &cr, int b, int64_t a, int64_t c) {
  if (a < 0 || c < 0) return __longlong_as_double(0x7FF8000000000000ll);  // no entry: NaN
  const BondDev &B = in.bond[b];
  double acc = 0.0;
  const int K = ld_cg(cr.r[b]);
  for (int t = 0; t < K; ++t)
    acc = __fma_rn(B.T[(int64_t)t * B.ldT + a], B.R[(int64_t)t * B.ldR + c], acc);
  return __dsub_rn(sb_entry(in, b, a, c), acc);
}

__device__ void fail_instance(Ctrl &cr, int32_t status) {
  if (threadIdx.x == 0) {
    cr.status = status;
    cr.state = ST_DONE;
  }
}

// stored-residual form: the rank-one step of eq. aca_approx_E for pivot
// (a*, c*) of bond b is applied by the next screen to the stored extent:
//   ew[a] = -(E(a,c*) / E(a*,c*)) (exactly -1 at a*), erow[c] = E(a*,c);
// the decide phase only marks it pending, the update phase (every CTA, as
// thread items) fills ew and erow from E, which the screen left unchanged
__device__ void stored_step(Ctrl &cr, int b) {
  if (threadIdx.x == 0) cr.e_pend[b] = 1;
}

// stop test and pivot append for bond b on its merged best (block-wide): add
// the pivot while the best |E| exceeds tau * rms(X) and the cap allows.  The
// bond's own rank is the only rank this touches, so bonds decide in parallel.
// The values come from the caller (every thread holds the same ones).
__device__ void finalize_bond_v(const InstDev &in, Ctrl &cr, int b, DecideSmem &sm, uint64_t key,
                                int32_t row, int32_t col, int32_t rb, double tau, double xrms,
                                int32_t maxr) {
  __syncthreads();
  if (key > KEY_INF || row < 0) {
    fail_instance(cr, 4);  // TTC_ERR_NONFINITE
    if (threadIdx.x == 0) cr.add[b] = 0;
    __syncthreads();
    return;
  }
  const double v = __longlong_as_double((long long)key);
  const bool add = v > tau * xrms && v > 0.0 && rb < maxr;
  bool ok = true;
  if (add) ok = append_pivot(in, cr, b, row, col, rb, sm);
  if (add && ok && in.stored) stored_step(cr, b);
  if (add && !ok && sm.flag < 0) fail_instance(cr, 4);
  __syncthreads();
  if (threadIdx.x == 0) {
    cr.add[b] = (add && ok) ? 1 : 0;
    cr.r[b] = rb + ((add && ok) ? 1 : 0);
  }
  __syncthreads();
}

// the same with the best and the words read from the control block
__device__ void finalize_bond(const InstDev &in, Ctrl &cr, int b, DecideSmem &sm) {
  const uint64_t key = ld_cg(cr.best_key[b]);
  const int32_t row = ld_cg(cr.best_row[b]), col = ld_cg(cr.best_col[b]);
  finalize_bond_v(in, cr, b, sm, key, row, col, ld_cg(cr.r[b]), ld_cg(cr.tau), ld_cg(cr.xrms),
                  ld_cg(cr.maxr[b]));
}

// stored forms, once a bond's candidates are merged (one thread): the screen
// has stored every entry of the superblock; its list of candidates, item
// counters and pending step are cleared for the next
__device__ __forceinline__ void close_screen(Ctrl &cr, int b, const DecideSmem &sm) {
  cr.pv_rows[b] = ld_cg(cr.st_rows[b]);
  cr.pv_cols[b] = ld_cg(cr.st_cols[b]);
  cr.st_rows[b] = sm.q_prow;
  cr.st_cols[b] = sm.q_pcol;
  cr.e_pend[b] = 0;
  cr.ntiles[b] = 0;
  if (b == 0) cr.steal = cr.steal2 = 0;  // item counters of the next screen
}
// the step maxima, cleared for the update phase's next step (block-wide); the
// extents are the run's caps (ldT / ldR bound the tile counts)
__device__ __forceinline__ void clear_maxima(const InstDev &in, int b) {
  const BondDev &B = in.bond[b];
  const Ctrl &cr = *in.ctrl;
  const int32_t nr = ld_cg(cr.plan_nrt[b]), nc = ld_cg(cr.plan_nct[b]);
  for (int x = threadIdx.x; x < nr; x += NT) B.wmax[x] = 0u;
  for (int x = threadIdx.x; x < nc; x += NT) B.emax[x] = 0u;
}

// FP64 decide item of bond b: the control words it needs in one round of
// parallel loads, the merge of the tile candidates (the Allgather of Alg. 3),
// then the stop test on the merged best as it stands
template <bool STORED>
__device__ void decide_bond_fp64(const InstDev &in, Ctrl &cr, int b, DecideSmem &sm) {
  const int tid = threadIdx.x;
  if (tid == 0) sm.q_nt = ld_cg(cr.ntiles[b]);
  if (tid == 1) sm.q_r = ld_cg(cr.r[b]);
  if (tid == 2) sm.q_tau = ld_cg(cr.tau);
  if (tid == 3) sm.q_xrms = ld_cg(cr.xrms);
  if (tid == 4) sm.q_maxr = ld_cg(cr.maxr[b]);
  if (tid == 5 && STORED) sm.q_prow = ld_cg(cr.plan_rows[b]);
  if (tid == 6 && STORED) sm.q_pcol = ld_cg(cr.plan_cols[b]);
  if (tid == 7) sm.q_nf = STORED ? ld_cg(cr.nfresh[b]) : 0;
  __syncthreads();
  const int64_t nt = sm.q_nt + sm.q_nf;
  if (STORED && tid == 0) close_screen(cr, b, sm);
  if (STORED && in.lazy) clear_maxima(in, b);
  KeyBest best{0ull, LLONG_MAX, -1, -1};
  const Cand *cand = in.cand + in.bond[b].cand_base;
  int bad = 0;
  // four slots' loads in flight before their compares
  int64_t t = tid;
  for (; t + 3 * NT < nt; t += 4 * NT) {
    KeyBest o[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const Cand &c = cand[t + u * NT];
      o[u] = KeyBest{c.key, c.lin, c.row, c.col};
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      bad += o[u].row == -1;  // -2 marks a slot left empty on purpose
      STORED ? kb_take_any(best, o[u]) : kb_take(best, o[u]);
    }
  }
  for (; t < nt; t += NT) {
    KeyBest o{cand[t].key, cand[t].lin, cand[t].row, cand[t].col};
    bad += o.row == -1;
    STORED ? kb_take_any(best, o) : kb_take(best, o);
  }
  if (bad) atomicAdd((unsigned long long *)&cr.unscreened, (unsigned long long)bad);
  best = block_best<STORED>(best, sm.rk, sm.rl, sm.rr, sm.rc);
  if (tid == 0) {
    cr.best_key[b] = best.key;
    cr.best_lin[b] = best.lin;
    cr.best_row[b] = best.row;
    cr.best_col[b] = best.col;
    sm.rk[0] = best.key;
    sm.rr[0] = best.row;
    sm.rc[0] = best.col;
  }
  __syncthreads();
  finalize_bond_v(in, cr, b, sm, sm.rk[0], sm.rr[0], sm.rc[0], sm.q_r, sm.q_tau, sm.q_xrms,
                  sm.q_maxr);
}

constexpr int RS_K = 8;  // candidates re-scored per bond in the mixed stored form

// The k best (k <= RS_K) of the lanes' sorted lists loc[0..L-1]: k rounds of
// a butterfly argmax of the list heads, the winning lane popping its head;
// lane j < k returns the j-th (the others an empty candidate).
template <int L>
__device__ KeyBest warp_topk(KeyBest (&loc)[L], int k) {
  const int lane = threadIdx.x & 31;
  KeyBest mine{0ull, LLONG_MAX, -1, -1};
  for (int j = 0; j < k; ++j) {
    KeyBest w = loc[0];
    for (int off = 16; off > 0; off >>= 1) {
      KeyBest o;
      o.key = __shfl_xor_sync(0xffffffffu, w.key, off);
      o.lin = __shfl_xor_sync(0xffffffffu, w.lin, off);
      o.row = __shfl_xor_sync(0xffffffffu, w.row, off);
      o.col = __shfl_xor_sync(0xffffffffu, w.col, off);
      if (o.row >= 0 && (w.row < 0 || key_better(o.key, o.lin, w.key, w.lin))) w = o;
    }
    if (lane == j) mine = w;
    if (w.row >= 0 && loc[0].row == w.row && loc[0].col == w.col) {
#pragma unroll
      for (int q = 0; q + 1 < L; ++q) loc[q] = loc[q + 1];
      loc[L - 1] = KeyBest{0ull, LLONG_MAX, -1, -1};
    }
  }
  return mine;
}

// a candidate slot read through L2 (other SMs wrote it in this launch)
__device__ __forceinline__ Cand ld_cand(const Cand *p) {
  Cand c;
  c.key = __ldcg(&p->key);
  c.lin = __ldcg(&p->lin);
  const int2 rc = __ldcg(reinterpret_cast<const int2 *>(&p->row));
  c.row = rc.x;
  c.col = rc.y;
  return c;
}

// The k best (k <= RS_K; key, then lowest linear index) of slots [t0, t1)
// into sm.skey / slin / srow / scol [0, k), missing ones with row -1;
// block-wide.  Up to 2 NT slots: every slot's rank is the number of better
// slots (the slots are distinct entries).  More: every thread keeps its own
// k best in one pass, each warp merges its lanes' lists, one warp the warps'.
__device__ void topk_of_slots(const Cand *src, int64_t t0, int64_t t1, int k, DecideSmem &sm,
                              int &bad) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t m = t1 - t0;
  if (tid < RS_K) sm.srow[tid] = -1;
  if (m <= 2 * NT) {
    Cand c[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int64_t i = tid + u * NT;
      c[u] = i < m ? ld_cand(src + t0 + i) : Cand{0ull, LLONG_MAX, -2, -2};
      bad += c[u].row == -1;
      const bool v = c[u].row >= 0;
      sm.tk[i] = v ? c[u].key : 0ull;
      sm.tl[i] = v ? c[u].lin : LLONG_MAX;  // never better than a real slot
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (c[u].row < 0) continue;
      int rank = 0;
      for (int j = 0; j < (int)m; ++j) rank += key_better(sm.tk[j], sm.tl[j], c[u].key, c[u].lin);
      if (rank < k) {
        sm.skey[rank] = c[u].key;
        sm.slin[rank] = c[u].lin;
        sm.srow[rank] = c[u].row;
        sm.scol[rank] = c[u].col;
      }
    }
    __syncthreads();
    return;
  }
  KeyBest loc[RS_K];
#pragma unroll
  for (int j = 0; j < RS_K; ++j) loc[j] = KeyBest{0ull, LLONG_MAX, -1, -1};
  for (int64_t t = t0 + tid; t < t1; t += NT) {
    const Cand c = ld_cand(src + t);
    bad += c.row == -1;
    if (c.row < 0) continue;
    // most slots lose to the list's last entry: one comparison
    KeyBest o{c.key, c.lin, c.row, c.col};
    if (k == RS_K && loc[RS_K - 1].row >= 0 &&
        !key_better(o.key, o.lin, loc[RS_K - 1].key, loc[RS_K - 1].lin))
      continue;
    // insertion into the sorted list loc[0..k-1]
#pragma unroll
    for (int j = 0; j < RS_K; ++j) {
      if (j >= k) break;
      if (loc[j].row < 0 || key_better(o.key, o.lin, loc[j].key, loc[j].lin)) {
        const KeyBest tmp = loc[j];
        loc[j] = o;
        o = tmp;
        if (o.row < 0) break;
      }
    }
  }
  const KeyBest wb = warp_topk<RS_K>(loc, k);
  __syncthreads();  // the srow marks above are written before warp 0's results
  if (lane < RS_K) {
    sm.wk[warp * RS_K + lane] = wb.key;
    sm.wl[warp * RS_K + lane] = wb.lin;
    sm.wr[warp * RS_K + lane] = wb.row;
    sm.wc[warp * RS_K + lane] = wb.col;
  }
  __syncthreads();
  if (warp == 0) {
    KeyBest l2[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = lane + 32 * h;
      l2[h] = i < NT / 32 * RS_K ? KeyBest{sm.wk[i], sm.wl[i], sm.wr[i], sm.wc[i]}
                                 : KeyBest{0ull, LLONG_MAX, -1, -1};
    }
    if (l2[1].row >= 0 && (l2[0].row < 0 || key_better(l2[1].key, l2[1].lin, l2[0].key, l2[0].lin))) {
      const KeyBest tmp = l2[0];
      l2[0] = l2[1];
      l2[1] = tmp;
    }
    const KeyBest g = warp_topk<2>(l2, k);
    if (lane < k) {
      sm.skey[lane] = g.key;
      sm.slin[lane] = g.lin;
      sm.srow[lane] = g.row;
      sm.scol[lane] = g.col;
    }
  }
  __syncthreads();
}

// Mixed stored form, decide item (bond b, part of P): the part takes the k
// best of its share of the tile slots by stored |E| (k = topk, at most RS_K;
// entries new to the superblock formed on the FP32 pipe) into the bond's
// partial results, the Allgather of Alg. 3.  The last part to finish takes
// the k best of the partials, re-scores them in FP64 as A - chain(T(a,:),
// R(:,c)) with the current factors, and takes the best FP64 value (same tie
// rule) to the stop test and the pivot step.
__device__ __noinline__ void decide_bond_rescore(const InstDev &in, Ctrl &cr, int b, int part,
                                                 int P, DecideSmem &sm) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = max(1, min(in.topk, RS_K));
  if (tid == 0) sm.q_nt = ld_cg(cr.ntiles[b]);
  if (tid == 1) sm.q_r = ld_cg(cr.r[b]);
  if (tid == 2) sm.q_tau = ld_cg(cr.tau);
  if (tid == 3) sm.q_xrms = ld_cg(cr.xrms);
  if (tid == 4) sm.q_maxr = ld_cg(cr.maxr[b]);
  if (tid == 5) sm.q_prow = ld_cg(cr.plan_rows[b]);
  if (tid == 6) sm.q_pcol = ld_cg(cr.plan_cols[b]);
  if (tid == 7) sm.q_nf = ld_cg(cr.nfresh[b]);
  __syncthreads();
  const int64_t nt = sm.q_nt + sm.q_nf, L = (nt + P - 1) / P;
  const int64_t t0 = min(nt, (int64_t)part * L), t1 = min(nt, t0 + L);
  const Cand *cand = in.cand + in.bond[b].cand_base;
  Cand *pb = in.refine_cand + in.bond[b].cand_base;  // the parts' results, [P][k]
  int bad = 0;
  topk_of_slots(cand, t0, t1, k, sm, bad);
  if (P > 1) {
    if (tid < k)
      pb[part * k + tid] = sm.srow[tid] >= 0
                               ? Cand{sm.skey[tid], sm.slin[tid], sm.srow[tid], sm.scol[tid]}
                               : Cand{0ull, LLONG_MAX, -2, -2};
    // the last of the P parts to arrive finishes the bond
    __syncthreads();
    if (tid == 0) {
      __threadfence();  // the part's results before its arrival
      sm.last = atomicAdd(&cr.dcount[b], 1) == P - 1;
      if (sm.last) {
        cr.dcount[b] = 0;
        __threadfence();  // the other parts' results after theirs
      }
    }
    __syncthreads();
    if (!sm.last) {
      if (bad) atomicAdd((unsigned long long *)&cr.unscreened, (unsigned long long)bad);
      return;
    }
    topk_of_slots(pb, 0, (int64_t)P * k, k, sm, bad);
  }
  if (tid == 0) close_screen(cr, b, sm);
  if (bad) atomicAdd((unsigned long long *)&cr.unscreened, (unsigned long long)bad);
  // FP64 re-score of the k candidates, a lane each of warp 0 (the chains run
  // side by side instead of queueing warps on the SM's FP64 units)
  if (warp == 0 && lane < k && sm.srow[lane] >= 0)
    sm.skey[lane] = abs_key(residual_at(in, b, sm.q_r, sm.srow[lane], sm.scol[lane]));
  __syncthreads();
  if (tid == 0) {
    KeyBest best{0ull, LLONG_MAX, -1, -1};
    for (int j = 0; j < k; ++j) {
      KeyBest o{sm.skey[j], sm.slin[j], sm.srow[j], sm.scol[j]};
      kb_take(best, o);
    }
    cr.best_key[b] = best.key;
    cr.best_lin[b] = best.lin;
    cr.best_row[b] = best.row;
    cr.best_col[b] = best.col;
    atomicAdd((unsigned long long *)&cr.tiles_refined, (unsigned long long)min((int64_t)k, nt));
    sm.rk[0] = best.key;
    sm.rr[0] = best.row;
    sm.rc[0] = best.col;
  }
  __syncthreads();
  finalize_bond_v(in, cr, b, sm, sm.rk[0], sm.rr[0], sm.rc[0], sm.q_r, sm.q_tau, sm.q_xrms,
                  sm.q_maxr);
}

// mixed forms, part 1 for bond b: re-score the top-k tile bests in FP64,
// then queue for the FP64 refinement every tile whose bound reaches the best
// exact value (when that exceeds the threshold theta: the tile could hold the
// FP64 argmax, or an equal residual with a lower index) or exceeds theta
// (otherwise: the tile could hold an entry that must become a pivot).
__device__ void merge_bond_mixed(const InstDev &in, Ctrl &cr, int b, DecideSmem &sm) {
  __syncthreads();
  if (threadIdx.x == 0) sm.flag = 0;
  __syncthreads();
  const int64_t nt = ld_cg(cr.ntiles[b]);
  const MCand *mc = in.mcand + in.bond[b].cand_base;
  int32_t *list = in.refine_list + 2 * in.bond[b].cand_base;
  const int k = (int)min((int64_t)min(in.topk, TOPK_MAX), nt);
  // one pass: every thread keeps its k best tiles, the block merges them
  KeyBest loc[TOPK_MAX];
  for (int j = 0; j < k; ++j) loc[j] = KeyBest{0ull, LLONG_MAX, -1, -1};
  int bad = 0, badtile = 0;
  for (int64_t t = threadIdx.x; t < nt; t += NT) {
    const float v = mc[t].v;
    if (mc[t].row < 0) {
      // never written (NaN sentinel): count, do not use; written without an
      // entry (every residual of the tile non-finite): the instance fails
      if (!(v == v)) ++bad; else ++badtile;
      continue;
    }
    KeyBest o{(v == v) ? (uint64_t)__float_as_uint(v) : 0xFFFFFFFFull, mc[t].lin, 0, (int32_t)t};
    for (int j = 0; j < k; ++j) {
      if (loc[j].row < 0 || key_better(o.key, o.lin, loc[j].key, loc[j].lin)) {
        const KeyBest tmp = loc[j];
        loc[j] = o;
        o = tmp;
        if (o.row < 0) break;
      }
    }
  }
  if (bad) atomicAdd((unsigned long long *)&cr.unscreened, (unsigned long long)bad);
  if (badtile) atomicExch(&sm.flag, 1);
  for (int j = 0; j < k; ++j) {
    // the block's j-th best: the best head among the threads' lists
    KeyBest head = loc[0];
    KeyBest win = block_best(head, sm.rk, sm.rl, sm.rr, sm.rc);
    if (threadIdx.x == 0) sm.sel[j] = win.row >= 0 ? win.col : -1;
    __syncthreads();
    if (loc[0].row >= 0 && loc[0].col == sm.sel[j]) {
      for (int q = 0; q + 1 < k; ++q) loc[q] = loc[q + 1];
      loc[k - 1] = KeyBest{0ull, LLONG_MAX, -1, -1};
    }
    __syncthreads();
  }
  if (sm.flag) {
    // a tile without a finite residual: the FP64 screen would report it
    fail_instance(cr, 4);  // TTC_ERR_NONFINITE
    if (threadIdx.x == 0) {
      cr.best_key[b] = KEY_INF + 1;
      cr.best_row[b] = -1;
      cr.nrefine_bond[b] = 0;
      cr.pending[b] = 1;
    }
    __syncthreads();
    return;
  }
  if (threadIdx.x < k) {
    const int32_t t = sm.sel[threadIdx.x];
    if (t >= 0) {
      const MCand &c = mc[t];
      sm.skey[threadIdx.x] = abs_key(residual64(in, cr, b, c.row, c.col));
      sm.slin[threadIdx.x] = c.lin;
      sm.srow[threadIdx.x] = c.row;
      sm.scol[threadIdx.x] = c.col;
    } else {
      sm.skey[threadIdx.x] = 0ull;
      sm.slin[threadIdx.x] = LLONG_MAX;
      sm.srow[threadIdx.x] = -1;
      sm.scol[threadIdx.x] = -1;
    }
  }
  if (threadIdx.x == 0) sm.cnt = 0;
  __syncthreads();
  KeyBest vb{0ull, LLONG_MAX, -1, -1};
  for (int j = 0; j < k; ++j) {
    KeyBest o{sm.skey[j], sm.slin[j], sm.srow[j], sm.scol[j]};
    kb_take(vb, o);
  }
  const double vstar = __longlong_as_double((long long)(vb.key > KEY_INF ? KEY_INF : vb.key));
  const double theta = ld_cg(cr.tau) * ld_cg(cr.xrms);
  const bool strict = !(vstar > theta);
  const double thr = strict ? theta : vstar;
  const double g = 1.0 + 4.0 * 5.9604644775390625e-8;
  for (int64_t t = threadIdx.x; t < nt; t += NT) {
    const MCand &c = mc[t];
    bool taken = false;
    for (int q = 0; q < k; ++q) taken |= sm.sel[q] == (int32_t)t;
    if (c.row < 0 && !(c.v == c.v)) continue;  // never written (counted above)
    const double top = taken ? (double)c.rest : fmax((double)c.v, (double)c.rest);
    const double U = top * g + c.eabs;
    if (!(U == U) || (strict ? U > thr : U >= thr)) {
      const int slot = atomicAdd(&sm.cnt, 1);
      list[2 * slot] = b;
      list[2 * slot + 1] = (int32_t)t;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    cr.best_key[b] = vb.key;
    cr.best_lin[b] = vb.lin;
    cr.best_row[b] = vb.row;
    cr.best_col[b] = vb.col;
    cr.nrefine_bond[b] = sm.cnt;
    cr.pending[b] = 1;
    atomicAdd((unsigned long long *)&cr.tiles_refined, (unsigned long long)sm.cnt);
  }
  __syncthreads();
}

// sampled-error verification of an instance whose bonds all stopped (Sec. 5)
__device__ void verify_instance(const InstDev &in, Ctrl &cr, DecideSmem &sm) {
  double part = 0.0;
  for (int c = threadIdx.x; c < (int)gridDim.x; c += NT) part += in.err_part[c];
  const double num = block_sum(part, sm.red);
  if (threadIdx.x == 0) {
    cr.screened = 0;
    const double err = sqrt(num / ld_cg(cr.den));
    cr.err = err;
    int32_t rr[TTC_MAXD];
    for (int b = 0; b < in.nb; ++b) rr[b] = ld_cg(cr.r[b]);
    cr.error_fmas += error_fmas(in, rr);
    for (int b = 0; b < in.nb; ++b) cr.add[b] = 0;
    sm.flag = 0;
    if (!isfinite(err)) {
      cr.status = 4;
      cr.state = ST_DONE;
    } else if (cr.eps == 0.0 || err <= cr.eps) {
      cr.status = 0;
      cr.state = ST_DONE;
    } else {
      sm.flag = 1;
    }
  }
  __syncthreads();
  // tau /= 10 until a bond adds, the caps are hit or the refinements run out
  while (sm.flag) {
    __syncthreads();
    if (threadIdx.x == 0) {
      bool capped = true;
      for (int b = 0; b < in.nb; ++b)
        if (ld_cg(cr.r[b]) < ld_cg(cr.maxr[b])) capped = false;
      if (capped || ld_cg(cr.refinements) >= ld_cg(cr.max_refine)) {
        cr.status = 7;  // TTC_NOT_CONVERGED
        cr.state = ST_DONE;
        sm.flag = 0;
      } else {
        cr.tau = ld_cg(cr.tau) / 10.0;
        cr.refinements = ld_cg(cr.refinements) + 1;
        cr.state = ST_SCREEN;
        // the mixed recompute forms certified their bests only against the
        // old threshold: they screen again; the FP64 and stored forms keep
        // FP64 values of their bests
        // (a sampled screen draws new samples, as its reference does)
        sm.flag = ((in.prec == P_FP64 || in.stored) && in.nl == 0) ? 1 : 0;
      }
    }
    __syncthreads();
    if (!sm.flag) return;
    // FP64: the cached bests are exact, decide again at the new threshold
    int nadd = 0;
    for (int b = 0; b < in.nb; ++b) {
      finalize_bond(in, cr, b, sm);
      nadd += cr.add[b];
    }
    if (nadd > 0 || cr.state == ST_DONE) return;
  }
}

// decide work items.  Every instance contributes nb + 1 items, numbered
// alike by every CTA whatever the instance's state: item 0 the verification
// (instance, -1), items 1..nb the bonds; place g takes items g, g + G, ...
// Each item checks its own eligibility against the decide kind the screen
// phase fixed.  The numbering must not depend on words that items rewrite
// during the phase (state, screened, pending): a CTA that read them late
// would number the items differently, and one bond would be decided twice.
// item kinds of for_decide_items
enum ItemMode { IM_DECIDE = 0, IM_PENDING = 1, IM_FINALIZE = 2 };

// CTAs that share one bond's decide: the mixed stored form of a single
// instance merges its tile slots' k best in DPARTS parts (the last part to
// finish re-scores, takes the stop test and the pivot step); everything else
// in one part (the FP64 best of the slots is one short pass)
constexpr int DPARTS = 32;
__device__ __forceinline__ int decide_parts(const RunArgs &ra, const InstDev &in, int mode) {
  return (mode == IM_DECIDE && ra.count == 1 && in.stored && in.nl == 0 && in.prec != P_FP64)
             ? DPARTS
             : 1;
}

template <class F>
__device__ void for_decide_items(const RunArgs &ra, int mode, F &&f) {
  __shared__ int s_take;
  const int64_t G = gridDim.x;
  int64_t first = 0;
  for (int ii = 0; ii < ra.count; ++ii) {
    const InstDev &in = inst(ra, ii);
    const Ctrl &cr = *in.ctrl;
    const int P = decide_parts(ra, in, mode);
    const int64_t end = first + (int64_t)in.nb * P + 1;
    for (int64_t x = first + ((s_place - first) % G + G) % G; x < end; x += G) {
      const int slot = x == first ? -1 : (int)((x - first - 1) / P);
      const int part = x == first ? 0 : (int)((x - first - 1) % P);
      // one thread decides and the CTA follows: the words it reads can be
      // rewritten by other CTAs' items during the phase (a failing bond ends
      // the instance), and every thread of the CTA must take the same branch
      __syncthreads();
      if (threadIdx.x == 0) {
        const int kind = ld_cg(cr.dkind);
        bool take;
        if (slot < 0) {
          take = mode == IM_DECIDE && kind == DK_VERIFY;
        } else {
          take = kind == DK_BONDS && ld_cg(cr.state) != ST_DONE;
          if (mode == IM_PENDING) take = take && ld_cg(cr.pending[slot]);
          if (mode == IM_FINALIZE) take = take && in.nl > 0;
        }
        s_take = take ? 1 : 0;
      }
      __syncthreads();
      if (s_take) f(ii, slot, part, P);
    }
    first = end;
  }
}

__device__ void phase_decide(const RunArgs &ra, PhaseSmem &sm) {
  for_decide_items(ra, IM_DECIDE, [&](int ii, int b, int part, int P) {
    const InstDev &in = inst(ra, ii);
    Ctrl &cr = *in.ctrl;
    if (b < 0) {
      verify_instance(in, cr, sm.d);
    } else if (in.nl > 0) {
      decide_bond_sampled(in, cr, b, sm.d);
    } else if (in.prec == P_FP64) {
      if (in.stored)
        decide_bond_fp64<true>(in, cr, b, sm.d);
      else
        decide_bond_fp64<false>(in, cr, b, sm.d);
    } else if (in.stored) {
      decide_bond_rescore(in, cr, b, part, P, sm.d);
    } else {
      merge_bond_mixed(in, cr, b, sm.d);
    }
  });
}

// mixed forms, part 2: the FP64 results of the refined tiles join the
// re-scored candidates; the best is the FP64 argmax of the screen.
__device__ void phase_decide2(const RunArgs &ra, PhaseSmem &sm) {
  for_decide_items(ra, IM_PENDING, [&](int ii, int b, int, int) {
    const InstDev &in = inst(ra, ii);
    Ctrl &cr = *in.ctrl;
    DecideSmem &d = sm.d;
    const int32_t cnt = ld_cg(cr.nrefine_bond[b]);
    const Cand *rc = in.refine_cand + in.bond[b].cand_base;
    KeyBest best{ld_cg(cr.best_key[b]), ld_cg(cr.best_lin[b]), ld_cg(cr.best_row[b]),
                 ld_cg(cr.best_col[b])};
    int bad = 0;
    for (int32_t t = threadIdx.x; t < cnt; t += NT) {
      KeyBest o{rc[t].key, rc[t].lin, rc[t].row, rc[t].col};
      bad += o.row < 0;
      kb_take(best, o);
    }
    if (bad) atomicAdd((unsigned long long *)&cr.unscreened, (unsigned long long)bad);
    best = block_best(best, d.rk, d.rl, d.rr, d.rc);
    if (threadIdx.x == 0) {
      cr.best_key[b] = best.key;
      cr.best_lin[b] = best.lin;
      cr.best_row[b] = best.row;
      cr.best_col[b] = best.col;
    }
    __syncthreads();
    finalize_bond(in, cr, b, d);
  });
}

// merge of the first nt candidate slots of bond b (block-wide; the best is valid
// in every thread)
__device__ KeyBest merge_slots(const InstDev &in, Ctrl &cr, int b, int64_t nt, DecideSmem &sm) {
  const Cand *cand = in.cand + in.bond[b].cand_base;
  KeyBest best{0ull, LLONG_MAX, -1, -1};
  int bad = 0;
  for (int64_t t = threadIdx.x; t < nt; t += NT) {
    const Cand c = ld_cand(cand + t);
    const KeyBest o{c.key, c.lin, c.row, c.col};
    bad += o.row == -1;
    kb_take(best, o);
  }
  if (bad) atomicAdd((unsigned long long *)&cr.unscreened, (unsigned long long)bad);
  best = block_best(best, sm.rk, sm.rl, sm.rr, sm.rc);
  __syncthreads();
  if (threadIdx.x == 0) {
    sm.rk[0] = best.key;
    sm.rl[0] = best.lin;
    sm.rr[0] = best.row;
    sm.rc[0] = best.col;
  }
  __syncthreads();
  return KeyBest{sm.rk[0], sm.rl[0], sm.rr[0], sm.rc[0]};
}

// sampled screen, decide item of bond b: the argmax over the samples becomes
// the pivot candidate, and its refinement starts (column step first)
__device__ void decide_bond_sampled(const InstDev &in, Ctrl &cr, int b, DecideSmem &sm) {
  const KeyBest best = merge_slots(in, cr, b, share_size(in, b, false), sm);
  if (threadIdx.x == 0) {
    cr.best_key[b] = best.key;
    cr.best_lin[b] = best.lin;
    cr.best_row[b] = best.row;
    cr.best_col[b] = best.col;
    const bool go = in.max_rook > 0 && best.row >= 0 && best.key <= KEY_INF;
    cr.rook_stage[0][b] = go ? 1 : 0;  // (step 0 reads this copy)
    cr.rook_round[b] = 0;
    cr.rook_moved[b] = 0;
    if (b == 0) cr.screen_t = ld_cg(cr.screen_t) + 1;
  }
  __syncthreads();
}

// some bond of a sampled instance is in a refinement step k.  Step k reads the
// stages' copy k mod 2 (here and in the step itself) and writes the other one,
// for every bond.  That copy's readers were step k - 1's, and a CTA that writes
// it has passed the grid barrier behind them; the copy read here is written
// again by step k + 1, behind the barrier of step k, at which a CTA that is
// still here has not arrived.  So every CTA reads the same stages and all of
// them leave the loop after the same step.
__device__ bool any_rook(const RunArgs &ra, int k) {
  __shared__ int hit;
  __syncthreads();
  if (threadIdx.x == 0) {
    hit = 0;
    for (int ii = 0; ii < ra.count; ++ii) {
      const InstDev &in = inst(ra, ii);
      if (in.nl == 0) continue;
      const Ctrl &cr = *in.ctrl;
      if (ld_cg(cr.state) == ST_DONE || ld_cg(cr.dkind) != DK_BONDS) continue;
      for (int b = 0; b < in.nb; ++b)
        if (ld_cg(cr.rook_stage[k & 1][b])) hit = 1;
    }
  }
  __syncthreads();
  return hit != 0;
}

// refinement step: the pivot's column (step 1) or row (step 2) of every bond in
// a refinement step, each CTA's best of its share to its slot; the last CTA of a
// bond's share to arrive merges them (no grid barrier and second phase in
// between) and the pivot moves to a strictly larger |E|.  A round is step 1
// then step 2, and the refinement ends after a round that moved nothing or
// after max_rook rounds.  A CTA reads a bond's best only if it has a share of
// it, before it arrives; the stages have two copies (any_rook).  A step is latency (a few thousand residuals of up to
// 40 terms on the whole grid): as a scan of all bonds by every CTA, a barrier, a
// merge of all slots and a second barrier it took about 20 us, so this form and
// the row copies took the screen of Hilbert d=6, n=256, rank 40, 64 k samples, 8
// rounds from 5.1-5.4 to 3.5 ms over 24 sweeps (4.8 with the copies alone).
__device__ void phase_rook_step(const RunArgs &ra, PhaseSmem &sm, int k) {
  __shared__ CtrlSnap snap;
  __shared__ int32_t s_stage, s_row, s_col, s_last;
  for (int ii = 0; ii < ra.count; ++ii) {
    const InstDev &in = inst(ra, ii);
    if (in.nl == 0) continue;
    Ctrl &cr = *in.ctrl;
    snap_ctrl(cr, in.nb, snap);
    if (snap.state == ST_DONE || ld_cg(cr.dkind) != DK_BONDS) continue;
    const int32_t *r = snap.r;  // the sweep-start ranks (no pivot added yet)
    const bool wide = share_wide(in, r);
    for (int b = 0; b < in.nb; ++b) {
      const int rank = share_rank(in, b, wide);
      if (rank < 0) continue;
      if (threadIdx.x == 0) s_stage = ld_cg(cr.rook_stage[k & 1][b]);
      if (threadIdx.x == 1) s_row = ld_cg(cr.best_row[b]);
      if (threadIdx.x == 2) s_col = ld_cg(cr.best_col[b]);
      __syncthreads();
      const int st = s_stage;
      const int size = share_size(in, b, wide);
      const int64_t rows = rows_of(in, r, b), cols = cols_of(in, r, b);
      const int64_t a0 = s_row, c0 = s_col, len = st == 1 ? rows : cols;
      int32_t *const next = &cr.rook_stage[(k + 1) & 1][b];
      if (!st && rank == 0 && threadIdx.x == 0) *next = 0;
      if (st) {
        KeyBest best{0ull, LLONG_MAX, -1, -1};
        for (int64_t x = (int64_t)rank * NT + threadIdx.x; x < len; x += (int64_t)size * NT) {
          const int64_t a = st == 1 ? x : a0, c = st == 1 ? c0 : x;
          take_key(best, residual_at(in, b, r[b], a, c), entry_lin(in, b, a, c), a, c);
        }
        best = block_best(best, sm.s.sk, sm.s.sl, sm.s.sr, sm.s.sc);
        if (threadIdx.x == 0) {
          in.cand[in.bond[b].cand_base + rank] = best.row >= 0
                                                     ? Cand{best.key, best.lin, best.row, best.col}
                                                     : Cand{0ull, LLONG_MAX, -2, -2};
          __threadfence();  // the slot before the arrival
          s_last = atomicAdd(&cr.dcount[b], 1) == size - 1;
          if (s_last) {
            cr.dcount[b] = 0;
            __threadfence();  // the other slots after theirs
          }
        }
        __syncthreads();
        if (s_last) {
          const KeyBest line = merge_slots(in, cr, b, size, sm.d);
          if (threadIdx.x == 0) {
            const uint64_t cur = ld_cg(cr.best_key[b]);
            int moved = ld_cg(cr.rook_moved[b]);
            // several CTAs decide bonds of one instance at once: atomic counts
            atomicAdd((unsigned long long *)&cr.entries, (unsigned long long)len);
            atomicAdd((unsigned long long *)&cr.entries_fresh, (unsigned long long)len);
            atomicAdd((unsigned long long *)&cr.screen_fmas, (unsigned long long)(len * r[b]));
            if (line.row >= 0 && line.key > cur) {
              cr.best_key[b] = line.key;
              cr.best_lin[b] = line.lin;
              if (st == 1)
                cr.best_row[b] = line.row;
              else
                cr.best_col[b] = line.col;
              moved = 1;
            }
            if (line.key > KEY_INF) cr.best_key[b] = line.key;  // a non-finite residual ends the bond
            if (st == 1) {
              *next = 2;
              cr.rook_moved[b] = moved;
            } else {
              const int round = ld_cg(cr.rook_round[b]) + 1;
              cr.rook_round[b] = round;
              const bool again = moved && round < in.max_rook && ld_cg(cr.best_key[b]) <= KEY_INF;
              *next = again ? 1 : 0;
              cr.rook_moved[b] = 0;
            }
          }
        }
      }
      __syncthreads();
    }
  }
}

// sampled screen: the stop test and the pivot append of every bond, on the
// refined pivots
__device__ void phase_finalize(const RunArgs &ra, PhaseSmem &sm) {
  for_decide_items(ra, IM_FINALIZE, [&](int ii, int b, int, int) {
    const InstDev &in = inst(ra, ii);
    finalize_bond(in, *in.ctrl, b, sm.d);
  });
}

// ---------------------------------------------------------------------------
// update: items of one instance, in this order per bond b
//   C: replay rows of the new prefix (Alg. 4)                 n_b items
//   A: eq. aca_approx_T_sub on the sweep-start rows           rows_old items
//   B: new row z of R on the sweep-start columns              cols_old items
//   D: new columns of R for the new suffix                    r_new * n_{b+1}
// stores into T / R keep the FP32 (hi, lo) shadows of the mixed forms
// (and the copies by row / column of the sampled screen)
__device__ __forceinline__ void putT(const InstDev &in, const BondDev &B, int64_t t, int64_t a,
                                     double v) {
  const int64_t o = t * B.ldT + a;
  B.T[o] = v;
  if (B.Tr) B.Tr[a * B.ldr + t] = v;
  if (in.prec != P_FP64) {
    float hi, lo;
    split2(v, hi, lo);
    B.Thi[o] = hi;
    B.Tlo[o] = lo;
  }
}
__device__ __forceinline__ void putR(const InstDev &in, const BondDev &B, int64_t t, int64_t c,
                                     double v) {
  const int64_t o = t * B.ldR + c;
  B.R[o] = v;
  if (B.Rr) B.Rr[c * B.ldr + t] = v;
  if (in.prec != P_FP64) {
    float hi, lo;
    split2(v, hi, lo);
    B.Rhi[o] = hi;
    B.Rlo[o] = lo;
  }
}

// A(a, c_z) for z < nz: superblock row a of bond b against the columns of
// its first nz pivots, all issued before any is used (the replay and the row
// update need them inside serial chains).  Hilbert: the entry is the table
// value at the row's index sum plus the pivot's J_{>k} index sum.
__device__ __forceinline__ void pivot_col_entries(const InstDev &in, int b, int64_t a, int z0,
                                                  int nz, double *ent) {
  const BondDev &B = in.bond[b];
  if (in.gen == 0) {
    const int64_t nb0 = in.n[b];
    const int64_t p = a / nb0, i = a - p * nb0;
    const int32_t rs = left_set(in, b).sum[p] + (int32_t)i;
    for (int z = z0; z < nz; ++z) ent[z - z0] = in.hilb[rs + B.J.sum[z]];
  } else {
    for (int z = z0; z < nz; ++z) ent[z - z0] = sb_entry(in, b, a, B.pcol[z]);
  }
}

// Alg. 4 for up to 32 / LPR rows of bond b by one warp, LPR lanes a row: the
// steps of update_row, the same FMAs in the same order.  The contract's chain
// of step z is z dependent FMAs; its operands T(a, t) and c_z(t) come from
// shared memory as broadcasts, eight of each ahead of their FMAs, and one
// chain instruction serves all the warp's rows.  A row's lanes then share the
// step's z independent updates.  The history rows come by asynchronous copies
// RB_STAGES - 1 steps ahead.
// A warp issues one FP64 instruction per 63 cycles whatever its lanes do, so a
// row of nz pivots takes nz^2 / 2 (1 + 1 / LPR) of them and the floor is
// nz^2 / 2: eight rows a warp (LPR 4) keep the number of replay warps small
// where rows are many and short (1024 rows of 23 pivots on the 6D n = 256
// cross: 36 us a sweep with a row per lane, which runs its updates serially
// and in local memory), one row a warp (LPR 32) where they are long.  (With
// the row in registers and two shuffles per chain element a row of 256 pivots
// took 2.3 times its floor: 200 ms of update phases in the 6D Maxwellian.)
template <int LPR, int NZM>  // NZM: pivots at most
__device__ __noinline__ void replay_group(const InstDev &in, int b, int64_t a0, int nrows, int nz,
                                          double *buf) {
  constexpr int RPW = 32 / LPR;                                // rows of the warp
  constexpr int LD = LPR == 32 ? NZM : NZM + 1;                // row stride (bank spread)
  const BondDev &B = in.bond[b];
  const int lane = threadIdx.x & 31, s = lane % LPR, rI = min(lane / LPR, nrows - 1);
  const int64_t cap = B.cap, a = a0 + rI;
  double *row = buf + (lane / LPR) * LD, *ent = buf + RPW * LD + (lane / LPR) * LD;
  double *dl = buf + 2 * RPW * LD, *hcr = dl + NZM, *hpr = hcr + RB_STAGES * NZM;
  auto fetch = [&](int z) {
    if (z < nz) {
      double *c = hcr + (z % RB_STAGES) * NZM, *p = hpr + (z % RB_STAGES) * NZM;
      for (int t = lane; t < z; t += 32) {
        const uint32_t sc = (uint32_t)__cvta_generic_to_shared(c + t);
        const uint32_t sp = (uint32_t)__cvta_generic_to_shared(p + t);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sc), "l"(B.hc + z * cap + t) : "memory");
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sp), "l"(B.hpiv + z * cap + t) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int z = 0; z < RB_STAGES - 1; ++z) fetch(z);
  for (int t = lane; t < nz; t += 32) dl[t] = B.delta[t];
  // the row's entries at the pivot columns
  if (in.gen == 0) {
    const int64_t nb0 = in.n[b];
    const int64_t p = a / nb0, i = a - p * nb0;
    const int32_t rs = left_set(in, b).sum[p] + (int32_t)i;
    for (int t0 = s; t0 < nz; t0 += 8 * LPR) {
      int32_t js[8];
      double v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) js[k] = t0 + k * LPR < nz ? B.J.sum[t0 + k * LPR] : 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = t0 + k * LPR < nz ? in.hilb[rs + js[k]] : 0.0;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (t0 + k * LPR < nz) ent[t0 + k * LPR] = v[k];
    }
  } else {
    for (int t = s; t < nz; t += LPR) ent[t] = sb_entry(in, b, a, B.pcol[t]);
  }
  for (int z = 0; z < nz; ++z) {
    fetch(z + RB_STAGES - 1);
    asm volatile("cp.async.wait_group %0;" ::"n"(RB_STAGES - 1) : "memory");
    __syncwarp();  // every lane's copies of step z have landed; the rows are whole
    const double *c = hcr + (z % RB_STAGES) * NZM, *p = hpr + (z % RB_STAGES) * NZM;
    double acc = 0.0;
    int t = 0;
    for (; t + 8 <= z; t += 8) {
      double x[8], y[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        x[k] = row[t + k];
        y[k] = c[t + k];
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) acc = __fma_rn(x[k], y[k], acc);
    }
    for (; t < z; ++t) acc = __fma_rn(row[t], c[t], acc);
    const double w = __dmul_rn(dl[z], __dsub_rn(acc, ent[z]));
    __syncwarp();  // the chains have read the rows
    for (t = s; t < z; t += LPR) row[t] = __fma_rn(w, p[t], row[t]);
    if (s == z % LPR) row[z] = -w;
    __syncwarp();  // step z's buffers are free for step z + RB_STAGES
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  // neighbouring rows are neighbours in T: lanes take rows first
  for (int x = lane; x < nz * RPW; x += 32) {
    const int rr = x % RPW, t = x / RPW;
    if (rr < nrows) putT(in, B, t, a0 + rr, buf[rr * LD + t]);
  }
  __syncwarp();
}

// rows of bond b's replays that one warp takes, and the warps they need
__device__ __forceinline__ int replay_rows_per_warp(int nz) { return nz <= RB_SMALL ? 8 : 1; }
__device__ __forceinline__ int replay_warps(const InstDev &in, int b, int nz) {
  const int rpw = replay_rows_per_warp(nz);
  return (int)((in.n[b] + rpw - 1) / rpw);
}

// group g of the replays of the n_b rows that prefix p of bond b-1 adds to bond b
__device__ void replay_rows(const InstDev &in, int b, int64_t p, int nz, int g, double *buf) {
  const int64_t nit = in.n[b], i0 = (int64_t)g * replay_rows_per_warp(nz);
  if (nz <= RB_SMALL)
    replay_group<4, RB_SMALL>(in, b, p * nit + i0, (int)min((int64_t)8, nit - i0), nz, buf);
  else
    replay_group<32, RCAP>(in, b, p * nit + i0, 1, nz, buf);
}

__device__ void update_row(const InstDev &in, int b, int64_t a, int z) {
  const BondDev &B = in.bond[b];
  const int cap = B.cap;
  const double *hc = B.hc + (int64_t)z * cap;
  const double *hp = B.hpiv + (int64_t)z * cap;
  double *T = B.T + a;
  const int64_t ld = B.ldT;
  double ent;
  pivot_col_entries(in, b, a, z, z + 1, &ent);
  const double s = __dsub_rn(chain(T, ld, hc, 1, z), ent);
  const double w = __dmul_rn(B.delta[z], s);
  if (in.prec == P_FP64 && in.nl == 0) {
    for (int t = 0; t < z; ++t) T[t * ld] = __fma_rn(w, hp[t], T[t * ld]);
  } else {
    for (int t = 0; t < z; ++t) putT(in, B, t, a, __fma_rn(w, hp[t], T[t * ld]));
  }
  putT(in, B, z, a, -w);
}

// first item >= base that thread gt of NTOT takes when items are dealt
// round-robin (32-bit arithmetic while the counts allow)
__device__ __forceinline__ int64_t first_item(int64_t base, int64_t gt, int64_t NTOT) {
  if (base < ((int64_t)1 << 31) && NTOT < ((int64_t)1 << 31)) {
    const int32_t n = (int32_t)NTOT;
    return base + (((int32_t)gt - (int32_t)base % n) % n + n) % n;
  }
  return base + ((gt - base) % NTOT + NTOT) % NTOT;
}

// ---------------------------------------------------------------------------
// sampled error (Sec. 5).  X~(i) = G_1(i_1) ... G_d(i_d), cores read from T
// (core m < d: element (p, i, u) = T_m[u][p n_m + i]) and R (last core).
// The leading pL and trailing pR cores are contracted once for every index
// combination of their modes (tables tabL, tabR), so a sample pays only the
// middle cores and one dot product.  (pL, pR) minimise
//   NL * s_{pL-1} s_pL + NR * s_{d-pR} s_{d-pR+1} + ns * (middle + s_{d-pR})
// within the table capacities; every CTA evaluates the same choice.

// core size s_m (s_0 = s_d = 1, s_m = r_{m-1})
__device__ __forceinline__ int64_t core_s(const InstDev &in, const int32_t *r, int m) {
  return (m == 0 || m == in.d) ? 1 : r[m - 1];
}

// FMAs of the error evaluation with tables of pL / pR modes (the last table
// level dominates; the chunked build adds its lower levels once per chunk)
// (in FP32: a cost estimate, identical on every thread; FP64 operations are
// long-latency on this GPU and every thread evaluates the choice)
__device__ double split_cost(const InstDev &in, const int32_t *r, int pL, int pR) {
  const int d = in.d;
  float NL = 1.f, NR = 1.f;
  for (int m = 0; m < pL; ++m) NL *= (float)in.n[m];
  for (int m = d - pR; m < d; ++m) NR *= (float)in.n[m];
  const float tl = pL >= 2 ? NL * (float)core_s(in, r, pL - 1) * (float)core_s(in, r, pL) : 0.f;
  const float tr =
      pR >= 2 ? NR * (float)core_s(in, r, d - pR) * (float)core_s(in, r, d - pR + 1) : 0.f;
  float mid = (float)core_s(in, r, d - pR);
  for (int m = pL; m < d - pR; ++m) mid += (float)core_s(in, r, m) * (float)core_s(in, r, m + 1);
  return (double)(tl + tr + (float)in.nsamples * mid);
}

__device__ void choose_split(const InstDev &in, const int32_t *r, int &pL, int &pR) {
  const int d = in.d;
  double best = 1e300;
  pL = 1;
  pR = 1;
  float NL = 1.f;
  for (int a = 1; a < d; ++a) {
    NL *= (float)in.n[a - 1];
    if (a >= 2 && NL * (float)core_s(in, r, a) > (float)in.tabL_cap) break;
    float NR = 1.f;
    for (int c = 1; a + c <= d; ++c) {
      NR *= (float)in.n[d - c];
      if (c >= 2 && NR * (float)core_s(in, r, d - c) > (float)in.tabR_cap) break;
      const double cost = split_cost(in, r, a, c);
      if (cost < best) {
        best = cost;
        pL = a;
        pR = c;
      }
    }
  }
}

// v (length s_m) <- v G_m(i) for a middle core 1 <= m <= d-2
__device__ __forceinline__ int mul_core(const InstDev &in, const int32_t *r, int m, int64_t i,
                                        double *v, double *w) {
  const BondDev &B = in.bond[m];
  const int rl = (int)core_s(in, r, m), rr = (int)core_s(in, r, m + 1);
  contract4(v, rl, B.T + i, B.ldT, in.n[m], w, rr);
  for (int u = 0; u < rr; ++u) v[u] = w[u];
  return rr;
}

// w (length s_{m+1}) <- G_m(i) w for a core 1 <= m <= d-2 (right to left)
__device__ __forceinline__ int mul_core_right(const InstDev &in, const int32_t *r, int m,
                                              int64_t i, double *w, double *t) {
  const BondDev &B = in.bond[m];
  const int rl = (int)core_s(in, r, m), rr = (int)core_s(in, r, m + 1);
  contract4(w, rr, B.T + i, in.n[m], B.ldT, t, rl);
  for (int p = 0; p < rl; ++p) w[p] = t[p];
  return rl;
}

}  // namespace ttc

#include "ttc_error.cuh"

namespace ttc {

// last-mode indices per table work item: 8 share the vector of their prefix;
// fewer (down to 2) when that leaves most threads without an item (the 6D
// n = 256 tables: 8192 items of 8 rows for 77824 threads)
__device__ __forceinline__ int64_t table_chunk(int64_t prefixes, int64_t n, int64_t threads) {
  int64_t c = 8;
  while (c > 2 && prefixes * ((n + c - 1) / c) * 2 <= threads) c /= 2;
  return c;
}

// tables of the verifying instances: a work item is a prefix of pL-1 modes
// (suffix of pR-1 modes) and a chunk of values of the next mode
__device__ void phase_tables(const RunArgs &ra) {
  // items are dealt a warp's worth per CTA in turn (lane l of warp w of CTA
  // c is number (w G + c) 32 + l): when there are fewer items than threads
  // every SM still gets an equal share of this FP64-bound phase, and the
  // lanes of a warp keep neighbouring items (the same core rows)
  const int64_t NTOT = (int64_t)gridDim.x * blockDim.x;
  const int64_t gt = ((int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31);
  __shared__ CtrlSnap snap;
  int64_t base = 0;
  for (int ii = 0; ii < ra.count; ++ii) {
    const InstDev &in = inst(ra, ii);
    const Ctrl &cr = *in.ctrl;
    snap_ctrl(cr, in.nb, snap);
    if (snap.state == ST_DONE) continue;
    if (!snap.screened) continue;
    const int32_t *r = snap.r;
    int nadd = 0;
    for (int b = 0; b < in.nb; ++b) nadd += snap.add[b];
    if (nadd) continue;
    // the plan: the same on every CTA; CTA 0 leaves it for the later phases
    __shared__ TcPlan plan;
    __syncthreads();
    if (threadIdx.x == 0) {
      tc_plan(in, r, plan);
      if (blockIdx.x == 0) *in.tcp = plan;
    }
    __syncthreads();
    // the tables made here: pL / pR modes, one fewer where the last mode runs
    // on the tensor cores (phase_stages); fixed-point rows where those read them
    const int d = in.d;
    const int pL = plan.pL - plan.tl, pR = plan.pR - plan.tr;
    const bool fixL = plan.on || plan.tl, fixR = plan.tr;
    double v[RCAP], w[RCAP];
    double *const tabL = fixL ? in.ews + plan.L : in.tabL;
    double *const tabR = plan.on || fixR ? in.ews + plan.R : in.tabR;
    int32_t *const Le = reinterpret_cast<int32_t *>(in.ews + plan.Le);
    int32_t *const Re = reinterpret_cast<int32_t *>(in.ews + plan.Re);
    const int64_t sl = core_s(in, r, pL), ll = fixL ? tc_up(sl, 16) : sl;      // a prefix row
    const int64_t sr = core_s(in, r, d - pR), lr = fixR ? tc_up(sr, 16) : sr;  // a suffix row
    if (fixL && pL == 1) {
      const BondDev &B0 = in.bond[0];
      for (int64_t x = first_item(base, gt, NTOT); x < base + in.n[0]; x += NTOT) {
        double *row = tabL + (x - base) * ll;
        copy8(row, B0.T + (x - base), B0.ldT, (int)sl);
        Le[x - base] = tc_fix_row(row, (int)sl, (int)ll);
      }
      base += in.n[0];
    }
    if (fixR && pR == 1) {
      const BondDev &BL = in.bond[d - 2];
      for (int64_t x = first_item(base, gt, NTOT); x < base + in.n[d - 1]; x += NTOT) {
        double *row = tabR + (x - base) * lr;
        copy8(row, BL.R + (x - base), BL.ldR, (int)sr);
        Re[x - base] = tc_fix_row(row, (int)sr, (int)lr);
      }
      base += in.n[d - 1];
    }
    if (pL >= 2) {
      int64_t np = 1;
      for (int m = 0; m < pL - 1; ++m) np *= in.n[m];
      const int64_t nl = in.n[pL - 1], chunk = table_chunk(np, nl, NTOT / 2);
      const int64_t nch = (nl + chunk - 1) / chunk;
      const int64_t items = np * nch;
      for (int64_t x = first_item(base, gt, NTOT); x < base + items; x += NTOT) {
        const int64_t pre = (x - base) / nch, ch = (x - base) - pre * nch;
        int64_t l = pre;
        int32_t idx[TTC_MAXD];
        for (int m = 0; m < pL - 1; ++m) {
          idx[m] = (int32_t)(l % in.n[m]);
          l /= in.n[m];
        }
        const BondDev &B0 = in.bond[0];
        int len = (int)core_s(in, r, 1);
        copy8(v, B0.T + idx[0], B0.ldT, len);
        for (int m = 1; m < pL - 1; ++m) len = mul_core(in, r, m, idx[m], v, w);
        // last mode of the prefix: core pL-1 (a middle core, pL-1 <= d-2)
        const BondDev &B = in.bond[pL - 1];
        for (int64_t i = ch * chunk; i < min(nl, (ch + 1) * chunk); ++i) {
          double *row = tabL + (pre + i * np) * ll;
          contract4(v, len, B.T + i, B.ldT, nl, row, (int)sl);
          if (fixL) Le[pre + i * np] = tc_fix_row(row, (int)sl, (int)ll);
        }
      }
      base += items;
    }
    if (pR >= 2) {
      int64_t np = 1;
      for (int m = d - pR + 1; m < d; ++m) np *= in.n[m];
      const int mf = d - pR;  // first mode of the suffix
      const int64_t nf = in.n[mf], chunk = table_chunk(np, nf, NTOT / 2);
      const int64_t nch = (nf + chunk - 1) / chunk;
      const int64_t items = np * nch;
      for (int64_t x = first_item(base, gt, NTOT); x < base + items; x += NTOT) {
        const int64_t suf = (x - base) / nch, ch = (x - base) - suf * nch;
        int64_t l = suf;
        int32_t idx[TTC_MAXD];
        for (int m = mf + 1; m < d; ++m) {
          idx[m] = (int32_t)(l % in.n[m]);
          l /= in.n[m];
        }
        const BondDev &BL = in.bond[d - 2];
        int len = (int)core_s(in, r, d - 1);
        copy8(w, BL.R + idx[d - 1], BL.ldR, len);
        for (int m = d - 2; m > mf; --m) len = mul_core_right(in, r, m, idx[m], w, v);
        const BondDev &B = in.bond[mf];
        for (int64_t i = ch * chunk; i < min(nf, (ch + 1) * chunk); ++i) {
          double *row = tabR + (i + nf * suf) * lr;
          contract4(w, len, B.T + i, nf, B.ldT, row, (int)sr);
          if (fixR) Re[i + nf * suf] = tc_fix_row(row, (int)sr, (int)lr);
        }
      }
      base += items;
    }
    if (plan.on)
      for (int m = pL; m < d - pR; ++m) tc_columns(in, r, plan, m, false, base, gt, NTOT);
    if (plan.tl) tc_columns(in, r, plan, pL, false, base, gt, NTOT);
    if (plan.tr) tc_columns(in, r, plan, d - 1 - pR, true, base, gt, NTOT);
  }
}

// FP64 FMAs of an error check: the tables', then the chains per sample, or the
// samples' products with the suffix rows where the middle cores run on the
// tensor cores
__device__ int64_t error_fmas(const InstDev &in, const int32_t *r) {
  const TcPlan &p = *in.tcp;
  const int pL = ld_cg(p.pL), pR = ld_cg(p.pR);
  const int tl = ld_cg(p.tl), tr = ld_cg(p.tr);
  double per = 0.0;
  if (!ld_cg(p.on))
    per = split_cost(in, r, pL, pR) - (double)tc_table_cost(in, r, pL, pR);
  else
    per = (double)in.nsamples * (double)core_s(in, r, in.d - pR);
  return (int64_t)((double)tc_table_cost(in, r, pL - tl, pR - tr) + per);
}

// the middle cores of the checks planned on the tensor cores, a grid barrier
// after every stage of every step (all instances' stages side by side)
__device__ bool phase_stages(const RunArgs &ra, PhaseSmem &sm) {
  __shared__ CtrlSnap snap;
  __shared__ TcPlan plan;
  const int NW = (int)gridDim.x * (NT / 32);
  const int gw = (int)blockIdx.x * (NT / 32) + (threadIdx.x >> 5);
  for (int step = 0;; ++step) {
    bool any = false;
    for (int ii = 0; ii < ra.count; ++ii) {
      const InstDev &in = inst(ra, ii);
      if (!in.tc_perm) continue;
      snap_ctrl(*in.ctrl, in.nb, snap);
      if (snap.state == ST_DONE || !snap.screened) continue;
      int nadd = 0;
      for (int b = 0; b < in.nb; ++b) nadd += snap.add[b];
      if (nadd) continue;
      for (int k = threadIdx.x; k < (int)(sizeof(TcPlan) / 4); k += NT)
        reinterpret_cast<int32_t *>(&plan)[k] = __ldcg(reinterpret_cast<const int32_t *>(in.tcp) + k);
      __syncthreads();
      if (step == 0 && (plan.tl || plan.tr)) {
        any = true;
        if (plan.tl) tc_extend(in, snap.r, plan, 0, gw, NW);
        if (plan.tr) tc_extend(in, snap.r, plan, 1, gw, NW);
        continue;
      }
      if (!plan.on || step >= plan.nst * plan.nsb) continue;
      any = true;
      const int st = step % plan.nst, sb = step / plan.nst;
      const double part = tc_stage(in, snap.r, plan, st, sb, gw, NW);
      if (st == plan.nst - 1) {
        const double s = block_sum(part, sm.red);
        if (threadIdx.x == 0) in.err_part[blockIdx.x] = sb == 0 ? s : __dadd_rn(in.err_part[blockIdx.x], s);
        __syncthreads();
      }
    }
    if (!any) return true;
    if (!grid_barrier(ra, 13)) return false;
  }
}

// error of one sample: X(i) - X~(i), using the tables of (pL, pR)
__device__ double sample_residual(const InstDev &in, const int32_t *r, int pL, int pR, int64_t k) {
  const double xk = in.xs[k];
  double v[RCAP], w[RCAP];
  const int d = in.d;
  int len;
  const double *src;   // the prefix vector in memory (stride sv)
  int64_t sv;
  if (pL >= 2) {
    int64_t e = 0, st = 1;
    for (int m = 0; m < pL; ++m) {
      e += sample_coord(in, k, m) * st;
      st *= in.n[m];
    }
    len = (int)core_s(in, r, pL);
    src = in.tabL + e * len;
    sv = 1;
  } else {
    const BondDev &B0 = in.bond[0];
    len = (int)core_s(in, r, 1);
    src = B0.T + sample_coord(in, k, 0);
    sv = B0.ldT;
  }
  if (pL + pR < d) {
    // middle cores: the vector goes to local memory
    copy8(v, src, sv, len);
    for (int m = pL; m < d - pR; ++m) len = mul_core(in, r, m, sample_coord(in, k, m), v, w);
    src = v;
    sv = 1;
  }
  double xt;
  if (pR >= 2) {
    int64_t e = 0, st = 1;
    for (int m = d - pR; m < d; ++m) {
      e += sample_coord(in, k, m) * st;
      st *= in.n[m];
    }
    const double *y = in.tabR + e * len;
    if (len <= 16) {
      // both rows in flight at once (a round trip to L2 each otherwise per
      // eight entries), then the contract's chain
      double xv[16], yv[16];
#pragma unroll
      for (int t = 0; t < 16; ++t) {
        xv[t] = t < len ? src[t * sv] : 0.0;
        yv[t] = t < len ? y[t] : 0.0;
      }
      double acc = 0.0;
#pragma unroll
      for (int t = 0; t < 16; ++t)
        if (t < len) acc = __fma_rn(xv[t], yv[t], acc);
      xt = acc;
    } else {
      xt = chain(src, sv, y, 1, len);
    }
  } else {
    const BondDev &BL = in.bond[d - 2];
    xt = chain(src, sv, BL.R + sample_coord(in, k, d - 1), BL.ldR, len);
  }
  return __dsub_rn(xk, xt);
}


// The error's samples when the prefix and suffix tables meet (pL + pR = d,
// rows of len): lane l of a warp takes the l-th of 32 consecutive samples, as
// in the thread dealing of the plain loop, and the warp loads their rows
// together.  The operations and their order per thread are those of
// sample_residual.
__device__ __noinline__ double samples_joined(const InstDev &in, int pL, int pR, int len,
                                              int64_t base, int64_t ns, int64_t gs, int64_t NTOT,
                                              SampleSmem &sw) {
  constexpr unsigned FULL = 0xffffffffu;
  double *buf = sw.rows[threadIdx.x >> 5];
  const int d = in.d;
  double part = 0.0;
  for (int64_t x = first_item(base, gs, NTOT);; x += NTOT) {
    const int valid = x < base + ns;
    if (!__any_sync(FULL, valid)) break;
    const int64_t k = valid ? x - base : 0;
    const double xk = valid ? in.xs[k] : 0.0;
    int64_t eL = 0, eR = 0, st = 1;
    for (int m = 0; m < pL; ++m) {
      eL += sample_coord(in, k, m) * st;
      st *= in.n[m];
    }
    st = 1;
    for (int m = d - pR; m < d; ++m) {
      eR += sample_coord(in, k, m) * st;
      st *= in.n[m];
    }
    const double acc = warp_chain_rows(in.tabL, eL, len, in.tabR, eR, len, len, buf);
    if (valid) {
      const double e = __dsub_rn(xk, acc);
      part = __fma_rn(e, e, part);
    }
  }
  return part;
}

__device__ void phase_update(const RunArgs &ra, PhaseSmem &sm) {
  __shared__ CtrlSnap snap;
  const int64_t NTOT = (int64_t)gridDim.x * NT;
  // items that each write their own outputs are dealt over the places; the
  // error's samples by blockIdx, so that the partial sums (and their
  // rounding) do not depend on where the CTAs run
  const int64_t gt = (int64_t)s_place * NT + threadIdx.x;
  const int64_t gs = (int64_t)blockIdx.x * NT + threadIdx.x;
  int64_t base = 0;
  for (int ii = 0; ii < ra.count; ++ii) {
    const InstDev &in = inst(ra, ii);
    const Ctrl &cr = *in.ctrl;
    // the work follows from the decisions (every CTA reads the same flags;
    // the state word is rewritten by the owner CTA during this phase)
    snap_ctrl(cr, in.nb, snap);
    const int st = snap.state;
    const int32_t *ro = snap.old_r, *rn = snap.r, *ad = snap.add;
    if (st == ST_DONE) {
      // a bond whose residual is not finite ends the run; the inverses of the
      // bonds that took a pivot in that decision are bordered all the same (not
      // every bond's flag is of that decision, so the inverses' ranks tell)
      for (int b = 0; b < in.nb; ++b)
        if (s_place == b % (int)gridDim.x && ld_cg(cr.u_rank[b]) < rn[b])
          border_inverse(in, b, rn[b] - 1, sm.d);
      continue;
    }
    int nadd = 0;
    for (int b = 0; b < in.nb; ++b) nadd += ad[b];
    const bool screened = snap.screened != 0;
    if (blockIdx.x == ii % gridDim.x && threadIdx.x < 32) {
      if (nadd == 0 && screened && threadIdx.x == 0) in.ctrl->state = ST_VERIFY;
      if (nadd > 0) write_plan_warp(in, *in.ctrl, rn, gridDim.x);  // next screen's tiles
    }
    if (nadd > 0) {
      // The replays are the longest items: RB_WARPS warps of a CTA take them,
      // the groups of all bonds numbered in order.  One instance on a grid of
      // two CTAs per SM: they go to the first places (distinct SMs), at most
      // three quarters of them, whose SMs take no other item, so that their
      // dependent FP64 chains do not queue behind other warps' FP64 work on
      // the SM's shared unit (362 cycles a step instead of 63 beside seven busy
      // warps); the thread-dealt items go to the other places.  Otherwise the
      // groups are dealt over all places, and the items start on the place
      // after the last.
      const int32_t S = s_sm2, G = gridDim.x;
      int32_t ng = 0;
      for (int b = 1; b < in.nb; ++b)
        if (ad[b - 1]) ng += replay_warps(in, b, rn[b]);
      const int32_t nsr = (ng + RB_WARPS - 1) / RB_WARPS;  // CTAs they take
      const bool iso = ra.count == 1 && S > 0 && G == 2 * S && 4 * nsr <= 3 * S;
      int64_t gti = gt, NTI = NTOT;
      const int32_t cb0 = iso ? 0 : (int32_t)((base / NT) % G);  // first replay place
      bool idle = false;  // a thread of a replay SM: no thread-dealt item
      const int warp = threadIdx.x >> 5;
      if (warp < RB_WARPS) {
        for (int32_t ch = (s_place - cb0 + G) % G; ch < nsr; ch += G) {
          int32_t g = ch * RB_WARPS + warp;
          for (int b = 1; b < in.nb; ++b) {
            if (!ad[b - 1]) continue;
            const int32_t nw = replay_warps(in, b, rn[b]);
            if (g < nw) {
              replay_rows(in, b, ro[b - 1], rn[b], g, sm.rp.buf[warp]);
              break;
            }
            g -= nw;
          }
        }
      }
      if (iso) {
        const int32_t pl = s_place;
        idle = pl < nsr || (pl >= S && pl < S + nsr);
        // item threads: the places of the other SMs, renumbered from 0
        NTI = (int64_t)(G - 2 * nsr) * NT;
        gti = idle ? 0 : (int64_t)(pl < S ? pl - nsr : pl - 2 * nsr) * NT + threadIdx.x;
      } else {
        base += (int64_t)nsr * NT;
      }
      // P^{-1} of every bond that added, a CTA each, counted back from the
      // first replay: places the replays reach last
      for (int b = 0; b < in.nb; ++b)
        if (ad[b] && s_place == (cb0 + G - 1 - b % G) % G)
          border_inverse(in, b, ro[b], sm.d);
      // where the stored entries' pending steps are found (the carried tiles of
      // the last screen; only a lazy screen leaves steps pending, and only for a
      // lazy one are the new step's maxima formed)
      __shared__ LazyGeo s_lazy[TTC_MAXB];
      __shared__ bool s_bounds;
      const bool lazy = in.lazy != 0;
      if (lazy) __syncthreads();
      if (lazy && threadIdx.x == NT - 1) s_bounds = lazy_at(in, rn);
      if (lazy && threadIdx.x < in.nb) {
        const int b = threadIdx.x;
        // (the owner CTA writes the next plan's rows, columns and counts meanwhile)
        LazyGeo q;
        q.g = planned_cut(in, cr, b);
        stateful_tiles(in, cr, q.g, b, q.tr, q.tc);
        q.stride = lazy_at(in, ro) ? state_stride(in, cr, q.g, b) : 0;
        s_lazy[b] = q;
      }
      if (lazy) __syncthreads();
      auto item0 = [&](int64_t bs) -> int64_t {
        return idle ? LLONG_MAX : first_item(bs, gti, NTI);
      };
      for (int b = 0; b < in.nb; ++b) {
        const BondDev &B = in.bond[b];
        // a thread with no item of this bond skips it whole: no load of the
        // pivot's coordinates or entries reaches its path
        {
          const int64_t rc = ad[b] ? rows_of(in, ro, b) + cols_of(in, ro, b) : 0;
          const int64_t tot = (in.stored ? 2 : 1) * rc +
                              (b < in.nb - 1 && ad[b + 1] ? (int64_t)rn[b] * in.n[b + 1] : 0);
          if (item0(base) >= base + tot) {
            base += tot;
            continue;
          }
        }
        if (ad[b] && in.stored) {
          // the rank-one step of the new pivot, from the residual of the
          // sweep-start superblock (its entries through their pending steps),
          // and its largest values per tile
          const int z = ro[b];
          const int64_t rows = rows_of(in, ro, b), cols = cols_of(in, ro, b);
          const int64_t as = B.prow[z], cs = B.pcol[z];
          const LazyGeo &lg = s_lazy[b];
          const bool bounds = lazy && s_bounds;
          double *ew = B.ew + (int64_t)z * B.ldw, *erow = B.erow + (int64_t)z * B.lde;
          if (item0(base) < base + rows) {
            const double ep = stored_entry(in, lg, b, as, cs, z - 1);
            for (int64_t x = item0(base); x < base + rows; x += NTI) {
              const int64_t a = x - base;
              const double w = -(stored_entry(in, lg, b, a, cs, z - 1) / ep);
              sv_put(in, ew, a, w);
              if (bounds)
                atomicMax(&B.wmax[row_tile_of(in, lg.g, b, (int32_t)a)],
                          __float_as_uint(abs_up(w)));
            }
          }
          base += rows;
          for (int64_t x = item0(base); x < base + cols; x += NTI) {
            const int64_t c = x - base;
            if (lazy) {
              const double e = stepped_entry(B, as, c, lazy_z(in, lg, b, as, c, z - 1), z - 1);
              erow[c] = e;
              if (bounds)
                atomicMax(&B.emax[col_tile_of(in, lg.g, b, (int32_t)c)], __float_as_uint(abs_up(e)));
            } else {
              erow[c] = B.E[as * B.ldR + c];  // as it is, a float-float pair too
            }
          }
          base += cols;
        }
        if (ad[b]) {
          const int z = ro[b];
          const int64_t rows = rows_of(in, ro, b), cols = cols_of(in, ro, b);
          for (int64_t x = item0(base); x < base + rows; x += NTI)
            update_row(in, b, x - base, z);
          base += rows;
          for (int64_t x = item0(base); x < base + cols; x += NTI)
            putR(in, B, z, x - base, sb_entry(in, b, B.prow[z], x - base));
          base += cols;
        }
        if (b < in.nb - 1 && ad[b + 1]) {
          const int64_t nb1 = in.n[b + 1];
          const int64_t q = ro[b + 1];
          const int64_t nit = (int64_t)rn[b] * nb1;
          for (int64_t x = item0(base); x < base + nit; x += NTI) {
            const int64_t l = x - base, t = l / nb1, jj = l - t * nb1;
            const int64_t c = q * nb1 + jj;
            putR(in, B, t, c, sb_entry(in, b, B.prow[t], c));
          }
          base += nit;
        }
      }
    } else if (screened) {
      if (ld_cg(in.tcp->on)) continue;  // done by phase_stages
      double part = 0.0;
      const int64_t ns = in.nsamples;
      const int pL = ld_cg(in.tcp->pL), pR = ld_cg(in.tcp->pR);
      const int jl = pL >= 2 && pR >= 2 && pL + pR == in.d ? (int)core_s(in, rn, pL) : 0;
      if (jl > 0) {
        part = samples_joined(in, pL, pR, jl, base, ns, gs, NTOT, sm.sw);
      } else {
        for (int64_t x = first_item(base, gs, NTOT); x < base + ns; x += NTOT) {
          const double e = sample_residual(in, rn, pL, pR, x - base);
          part = __fma_rn(e, e, part);
        }
      }
      base += ns;
      const double s = block_sum(part, sm.red);
      if (threadIdx.x == 0) in.err_part[blockIdx.x] = s;
      __syncthreads();
    }
  }
}

// ---------------------------------------------------------------------------
// init.  The start pivot is Alg. 1 line 1 with a zero approximation: the
// argmax of |X| over the error's random samples and the origin (ties: lowest
// linear index).  Every bond takes it as its first pivot (ranks 1).
//   init1 (all CTAs): X at the samples, partial sums of X^2, per-CTA argmax
//   init2 (owner CTA): reduce; pivot sets, delta_0, U = [delta_0]
//   init3 (all CTAs): T(:,0) and R(0,:) of every bond
__device__ void phase_init1(const RunArgs &ra, PhaseSmem &sm) {
  const int64_t NTOT = (int64_t)gridDim.x * NT;
  const int64_t gt = (int64_t)blockIdx.x * NT + threadIdx.x;
  int64_t base = 0;
  for (int ii = 0; ii < ra.count; ++ii) {
    const InstDev &in = inst(ra, ii);
    double part = 0.0;
    KeyBest best{0ull, LLONG_MAX, -1, -1};
    const int64_t ns = in.nsamples;
    for (int64_t x = first_item(base, gt, NTOT); x < base + ns; x += NTOT) {
      int32_t idx[TTC_MAXD];
      sample_index(in, x - base, idx);
      // user generator: the samples' values were filled by the callback
      const double v = in.gen == 4 ? in.xs[x - base] : gen_full(in, idx);
      in.xs[x - base] = v;
      part = __fma_rn(v, v, part);
      const uint64_t k = abs_key(v);
      if (best.row < 0 || k >= best.key) {
        int64_t l = 0;
        for (int m = 0; m < in.d; ++m) l += (int64_t)idx[m] * in.stride[m];
        if (best.row < 0 || k > best.key || l < best.lin) {
          best.key = k;
          best.lin = l;
          best.row = 0;
          best.col = (int32_t)(x - base);
        }
      }
    }
    base += ns;
    const double s = block_sum(part, sm.red);
    __shared__ uint64_t sk[NT / 32];
    __shared__ int64_t sl[NT / 32];
    __shared__ int32_t sr[NT / 32], sc[NT / 32];
    best = block_best(best, sk, sl, sr, sc);
    if (threadIdx.x == 0) {
      in.err_part[blockIdx.x] = s;
      in.start_part[blockIdx.x].key = best.key;
      in.start_part[blockIdx.x].lin = best.lin;
      in.start_part[blockIdx.x].row = best.row;
      in.start_part[blockIdx.x].col = best.col;  // the sample's number
    }
    __syncthreads();
  }
}

__device__ void phase_init2(const RunArgs &ra, PhaseSmem &sm) {
  for (int ii = blockIdx.x; ii < ra.count; ii += gridDim.x) {
    const InstDev &in = inst(ra, ii);
    Ctrl &cr = *in.ctrl;
    double part = 0.0;
    KeyBest best{0ull, LLONG_MAX, -1, -1};
    for (int c = threadIdx.x; c < (int)gridDim.x; c += NT) {
      part += in.err_part[c];
      const Cand &cd = in.start_part[c];
      KeyBest o{cd.key, cd.lin, cd.row, cd.col};
      kb_take(best, o);
    }
    const double den = block_sum(part, sm.d.red);
    best = block_best(best, sm.d.rk, sm.d.rl, sm.d.rr, sm.d.rc);
    if (threadIdx.x == 0) {
      cr.den = den;
      cr.xrms = sqrt(den / (double)in.nsamples);
      int32_t zero[TTC_MAXD] = {0};
      // user generator: the origin's value follows the samples in xs
      const double x0 = in.gen == 4 ? in.xs[in.nsamples] : gen_full(in, zero);
      KeyBest o{abs_key(x0), 0, 0, (int32_t)in.nsamples};
      kb_take(best, o);
      int32_t st[TTC_MAXD];
      int64_t l = best.lin;
      for (int m = 0; m < in.d; ++m) {
        st[m] = (int32_t)(l % in.n[m]);
        l /= in.n[m];
      }
      const double xs0 = in.gen == 4 ? in.xs[best.col] : gen_full(in, st);
      if (!isfinite(den) || !isfinite(xs0)) {
        cr.status = 4;
        cr.state = ST_DONE;
      } else if (xs0 == 0.0) {
        cr.status = 3;
        cr.state = ST_DONE;
      }
      for (int b = 0; b < in.nb && cr.state != ST_DONE; ++b) {
        const BondDev &B = in.bond[b];
        int64_t ll = 0;
        int32_t ss = 0;
        for (int m = 0; m <= b; ++m) {
          B.I.idx[m] = st[m];
          ll += (int64_t)st[m] * in.stride[m];
          ss += st[m];
        }
        B.I.lin[0] = ll;
        B.I.sum[0] = ss;
        ll = 0;
        ss = 0;
        for (int m = b + 1; m < in.d; ++m) {
          B.J.idx[m - b - 1] = st[m];
          ll += (int64_t)st[m] * in.stride[m];
          ss += st[m];
        }
        B.J.lin[0] = ll;
        B.J.sum[0] = ss;
        B.prow[0] = st[b];
        B.pcol[0] = st[b + 1];
        cr.r[b] = 1;
        cr.r_old[b] = 1;
        cr.add[b] = 0;
      }
      if (cr.state != ST_DONE) {
        // the pivot entry of every superblock is X(start)
        const double delta = 1.0 / __dsub_rn(xs0, 0.0);
        cr.piv_max = abs_key(xs0);
        if (!isfinite(delta)) {
          cr.status = 4;
          cr.state = ST_DONE;
        }
        for (int b = 0; b < in.nb; ++b) {
          in.bond[b].delta[0] = delta;
          in.bond[b].U[0] = delta;
          cr.u_rank[b] = 1;
        }
      }
    }
    __syncthreads();
    if (threadIdx.x < 32 && cr.state != ST_DONE) write_plan_warp(in, cr, cr.r, gridDim.x);
    __syncthreads();
  }
}

__device__ void phase_init3(const RunArgs &ra, PhaseSmem &sm) {
  const int64_t NTOT = (int64_t)gridDim.x * NT;
  const int64_t gt = (int64_t)blockIdx.x * NT + threadIdx.x;
  int64_t base = 0;
  for (int ii = 0; ii < ra.count; ++ii) {
    const InstDev &in = inst(ra, ii);
    const Ctrl &cr = *in.ctrl;
    if (ld_cg(cr.state) == ST_DONE) continue;
    if (in.lazy)
      for (int b = 0; b < in.nb; ++b) {
        const BondDev &B = in.bond[b];
        for (int64_t x = gt; x < B.ldT; x += NTOT) B.wmax[x] = 0u;
        for (int64_t x = gt; x < B.ldR; x += NTOT) B.emax[x] = 0u;
      }
    for (int b = 0; b < in.nb; ++b) {
      const BondDev &B = in.bond[b];
      const int64_t rows = in.n[b], cols = in.n[b + 1];
      const double delta = B.delta[0];
      const int64_t a0 = B.prow[0], c0 = B.pcol[0];
      for (int64_t x = first_item(base, gt, NTOT); x < base + rows; x += NTOT) {
        const int64_t a = x - base;
        const double s = __dsub_rn(0.0, sb_entry(in, b, a, c0));
        putT(in, B, 0, a, -__dmul_rn(delta, s));
      }
      base += rows;
      for (int64_t x = first_item(base, gt, NTOT); x < base + cols; x += NTOT)
        putR(in, B, 0, x - base, sb_entry(in, b, a0, x - base));
      base += cols;
    }
  }
}

// refine (mixed forms): FP64 screen of the queued tiles
__device__ void phase_refine(const RunArgs &ra, PhaseSmem &sm) {
  const int64_t G = gridDim.x;
  int64_t base = 0;
  for (int ii = 0; ii < ra.count; ++ii) {
    const InstDev &in = inst(ra, ii);
    const Ctrl &cr = *in.ctrl;
    if (ld_cg(cr.state) == ST_DONE) continue;
    if (!ld_cg(cr.screened)) continue;
    int32_t r[TTC_MAXD];
    for (int b = 0; b < in.nb; ++b) r[b] = ld_cg(cr.r[b]);
    for (int b = 0; b < in.nb; ++b) {
      if (!ld_cg(cr.pending[b])) continue;
      const int64_t cnt = ld_cg(cr.nrefine_bond[b]);
      const int32_t *list = in.refine_list + 2 * in.bond[b].cand_base;
      Cand *out = in.refine_cand + in.bond[b].cand_base;
      const TileGeo g = planned_geo(in, cr, b);
      for (int64_t t = base + ((blockIdx.x - base) % G + G) % G; t < base + cnt; t += G) {
        const int64_t li = t - base;
        const int32_t tile = list[2 * li + 1];
        const int32_t tr = tile / g.nct, tc = tile - tr * g.nct;
        int64_t r0, c0;
        int nr, nc;
        tile_rows(in, g, b, tr, r0, nr);
        tile_cols(in, g, b, tc, c0, nc);
        screen_tile_fp64(in, b, r[b], r0, nr, c0, nc, g.te, out + li, sm.s);
      }
      base += cnt;
    }
  }
}

// what the coming sweep is: 0 none (every instance is done), 1 one without, 2 one
// with tiles that wait for their steps
__device__ int sweep_kind(const RunArgs &ra) {
  __shared__ int kind;
  __syncthreads();
  if (threadIdx.x == 0) {
    kind = 0;
    for (int ii = 0; ii < ra.count; ++ii) {
      const Ctrl &cr = *inst(ra, ii).ctrl;
      const int32_t state = ld_cg(cr.state), lazy = ld_cg(cr.lazy);
      if (state != ST_DONE) kind = max(kind, lazy ? 2 : 1);
    }
  }
  __syncthreads();
  return kind;
}

// ---------------------------------------------------------------------------
// kernels

extern __shared__ __align__(16) unsigned char dyn_smem[];



// CTA 0 accounts the time between barrier exits to the phase that ran
struct PhaseClock {
  uint64_t t;
  __device__ void start() {
    if (blockIdx.x == 0 && threadIdx.x == 0) t = globaltimer_ns();
  }
  __device__ void lap(const RunArgs &ra, int slot) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      const uint64_t now = globaltimer_ns();
      ra.bar->phase_ns[slot] += now - t;
      t = now;
    }
  }
};

// some instance evaluates its sampled error in the coming update phase
__device__ bool any_verify(const RunArgs &ra) {
  __shared__ int hit;
  __syncthreads();
  if (threadIdx.x == 0) {
    hit = 0;
    for (int ii = 0; ii < ra.count; ++ii) {
      const Ctrl &cr = *inst(ra, ii).ctrl;
      if (ld_cg(cr.state) == ST_DONE) continue;
      if (!ld_cg(cr.screened)) continue;
      int nadd = 0;
      for (int b = 0; b < inst(ra, ii).nb; ++b) nadd += ld_cg(cr.add[b]);
      if (nadd == 0) hit = 1;
    }
  }
  __syncthreads();
  return hit != 0;
}

__device__ __forceinline__ int32_t sm_id() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(r));
  return (int32_t)r;
}

// s_place from the table of SM ids (written by every CTA before a grid
// barrier): with cnt[s] CTAs on SM s and this CTA the k-th on its SM sm,
//   place = sum_s min(cnt[s], k) + #{s < sm : cnt[s] > k},
// its rank when the CTAs are sorted by (k, SM) - a bijection onto [0, G).
// Ids outside the table keep the identity order.
__device__ void spread_order(const RunArgs &ra, PhaseSmem &sm) {
  SpreadSmem &sp = sm.sp;
  const int G = gridDim.x, me = sm_id();
  for (int s = threadIdx.x; s < SPREAD_MAXSM; s += NT) sp.cnt[s] = 0;
  if (threadIdx.x == 0) {
    sp.k = 0;
    sp.place = 0;
    sp.bad = me >= SPREAD_MAXSM;
    sp.nsm = 0;
    sp.not2 = 0;
  }
  __syncthreads();
  int k = 0;
  for (int j = threadIdx.x; j < G; j += NT) {
    const int s = ld_cg(ra.smid[j]);
    if (s >= 0 && s < SPREAD_MAXSM)
      atomicAdd(&sp.cnt[s], 1);
    else
      sp.bad = 1;
    k += (j < (int)blockIdx.x && s == me);
  }
  if (k) atomicAdd(&sp.k, k);
  __syncthreads();
  const int kk = sp.k;
  int part = 0, used = 0, odd = 0;
  for (int s = threadIdx.x; s < SPREAD_MAXSM; s += NT) {
    const int c = sp.cnt[s];
    part += min(c, kk) + (s < me && c > kk);
    used += c > 0;
    odd += c != 0 && c != 2;
  }
  if (part) atomicAdd(&sp.place, part);
  if (used) atomicAdd(&sp.nsm, used);
  if (odd) atomicAdd(&sp.not2, odd);
  __syncthreads();
  if (threadIdx.x == 0) {
    s_place = sp.bad ? (int32_t)blockIdx.x : sp.place;
    s_sm2 = (sp.bad || sp.not2) ? 0 : sp.nsm;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(NT, 2) k_persistent(RunArgs ra) {
  PhaseSmem &sm = *reinterpret_cast<PhaseSmem *>(dyn_smem);
  cache_inst0(ra);
  PhaseClock clk;
  clk.start();
  if (threadIdx.x == 0) ra.smid[blockIdx.x] = sm_id();
  phase_init1(ra, sm);
  if (!grid_barrier(ra, 1)) return;
  spread_order(ra, sm);
  phase_init2(ra, sm);
  if (!grid_barrier(ra, 2)) return;
  phase_init3(ra, sm);
  if (!grid_barrier(ra, 6)) return;
  clk.lap(ra, T_INIT);
  for (int it = 0;; ++it) {
    const int kind = sweep_kind(ra);
    if (kind == 0) break;
    if (it >= ra.max_iters) {
      if (blockIdx.x == 0 && threadIdx.x == 0) atomicExch(&ra.bar->overrun, 1);
      break;
    }
    if (kind == 2) {
      phase_bound(ra);
      if (!grid_barrier(ra, 14)) return;
    }
    phase_screen(ra, sm);
    if (!grid_barrier(ra, 3)) return;
    clk.lap(ra, T_SCREEN);
    phase_decide(ra, sm);
    if (!grid_barrier(ra, 4)) return;
    clk.lap(ra, T_DECIDE);
    if (ra.sampled) {
      // the refinement of Alg. 1, step by step, then the stop tests on the
      // refined pivots
      for (int k = 0; k < 2 * ra.max_rook && any_rook(ra, k); ++k) {
        phase_rook_step(ra, sm, k);
        if (!grid_barrier(ra, 10)) return;
      }
      clk.lap(ra, T_SCREEN);
      phase_finalize(ra, sm);
      if (!grid_barrier(ra, 12)) return;
      clk.lap(ra, T_DECIDE);
    }
    if (ra.mixed) {
      phase_refine(ra, sm);
      if (!grid_barrier(ra, 7)) return;
      clk.lap(ra, T_REFINE);
      phase_decide2(ra, sm);
      if (!grid_barrier(ra, 8)) return;
      clk.lap(ra, T_DECIDE);
    }
    const bool verify = any_verify(ra);
    if (verify) {
      phase_tables(ra);
      if (!grid_barrier(ra, 9)) return;
      if (!phase_stages(ra, sm)) return;
    }
    phase_update(ra, sm);
    if (!grid_barrier(ra, 5)) return;
    clk.lap(ra, verify ? T_VERIFY : T_UPDATE);
  }
}

__global__ void __launch_bounds__(NT, 2) k_init1(RunArgs ra) {
  cache_inst0(ra);
  phase_init1(ra, *reinterpret_cast<PhaseSmem *>(dyn_smem));
}
__global__ void __launch_bounds__(NT, 2) k_init2(RunArgs ra) {
  cache_inst0(ra);
  phase_init2(ra, *reinterpret_cast<PhaseSmem *>(dyn_smem));
}
__global__ void __launch_bounds__(NT, 2) k_init3(RunArgs ra) {
  cache_inst0(ra);
  phase_init3(ra, *reinterpret_cast<PhaseSmem *>(dyn_smem));
}
__global__ void __launch_bounds__(NT, 2) k_bound(RunArgs ra) {
  cache_inst0(ra);
  phase_bound(ra);
}
__global__ void __launch_bounds__(NT, 2) k_screen(RunArgs ra) {
  cache_inst0(ra);
  phase_screen(ra, *reinterpret_cast<PhaseSmem *>(dyn_smem));
}
__global__ void __launch_bounds__(NT, 2) k_decide(RunArgs ra) {
  cache_inst0(ra);
  phase_decide(ra, *reinterpret_cast<PhaseSmem *>(dyn_smem));
}
__global__ void __launch_bounds__(NT, 2) k_refine(RunArgs ra) {
  cache_inst0(ra);
  phase_refine(ra, *reinterpret_cast<PhaseSmem *>(dyn_smem));
}
__global__ void __launch_bounds__(NT, 2) k_decide2(RunArgs ra) {
  cache_inst0(ra);
  phase_decide2(ra, *reinterpret_cast<PhaseSmem *>(dyn_smem));
}
__global__ void __launch_bounds__(NT, 2) k_rook_step(RunArgs ra) {
  cache_inst0(ra);
  phase_rook_step(ra, *reinterpret_cast<PhaseSmem *>(dyn_smem), ra.rook_step);
}
__global__ void __launch_bounds__(NT, 2) k_finalize(RunArgs ra) {
  cache_inst0(ra);
  phase_finalize(ra, *reinterpret_cast<PhaseSmem *>(dyn_smem));
}
// the error check up to its samples' FP64 chains (a cooperative launch: its
// phases meet at grid barriers); nothing when no instance verifies
__global__ void __launch_bounds__(NT, 2) k_verify(RunArgs ra) {
  cache_inst0(ra);
  if (!any_verify(ra)) return;
  phase_tables(ra);
  if (!grid_barrier(ra, 9)) return;
  phase_stages(ra, *reinterpret_cast<PhaseSmem *>(dyn_smem));
}
__global__ void __launch_bounds__(NT, 2) k_update(RunArgs ra) {
  cache_inst0(ra);
  phase_update(ra, *reinterpret_cast<PhaseSmem *>(dyn_smem));
}

// cores: G_k = reshape(T_k, [s_{k-1}, n_k, s_k]) (eq. corereshape) written
// row-major from the t-major T; the last core is R of the last bond.
__global__ void k_core(const InstDev *inp, int m, double *dst) {
  const InstDev &in = *inp;
  const Ctrl &cr = *in.ctrl;
  const int d = in.d;
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t NTOT = (int64_t)gridDim.x * blockDim.x;
  if (m < d - 1) {
    const BondDev &B = in.bond[m];
    const int rr = cr.r[m];
    const int64_t rows = (int64_t)(m == 0 ? 1 : cr.r[m - 1]) * in.n[m];
    for (int64_t x = gt; x < rows * rr; x += NTOT) {
      const int64_t a = x / rr, t = x - a * rr;
      dst[x] = B.T[t * B.ldT + a];
    }
  } else {
    const BondDev &B = in.bond[d - 2];
    const int rl = cr.r[d - 2];
    const int64_t nn = in.n[d - 1];
    for (int64_t x = gt; x < rl * nn; x += NTOT) {
      const int64_t t = x / nn, j = x - t * nn;
      dst[x] = B.R[t * B.ldR + j];
    }
  }
}

// ---------------------------------------------------------------------------
// host-side launch helpers (declared in ttc_launch.h)

size_t phase_smem_bytes() { return sizeof(PhaseSmem); }

static int64_t host_piece_tiles(int64_t n, int32_t C, int64_t T) {
  const int64_t q = n / C, rem = n - q * C;  // the balanced split of make_pieces
  return rem * ((q + 1 + T - 1) / T) + (C - rem) * ((q + T - 1) / T);
}

int64_t host_tiles(int64_t n_b, int64_t n_b1, int64_t rl, int64_t rr, int32_t pr, int32_t pc) {
  const int64_t nrt = pr > 0 ? rl * host_piece_tiles(n_b, pr, BM) : (rl * n_b + BM - 1) / BM;
  const int64_t nct = pc > 0 ? rr * host_piece_tiles(n_b1, pc, BN) : (n_b1 * rr + BN - 1) / BN;
  return nrt * nct;
}

// Host replay of the screens' tile arithmetic for bond b at ranks r: the
// kernels' own tile_geo_e / tile_rows / tile_cols / carried_tiles, run on
// the host.  Counts the violations: a tile that is empty, wider than te or
// outside the superblock; a tile that crosses a piece of the subtensor grid
// (the pieces recomputed here from the balanced split); a superblock row or
// column that the tiles cover other than exactly once; with r_stored (the
// ranks the stored residual was written at), a carried tile outside the
// stored extent.
int64_t host_check_bond_tiles(int d, const int64_t *n, const int32_t *r, const int32_t *r_stored,
                              const int32_t *grid, int b, int te, int64_t *ntiles) {
  std::unique_ptr<InstDev> in(new InstDev());
  std::unique_ptr<Ctrl> cr(new Ctrl());
  in->d = d;
  in->nb = d - 1;
  for (int m = 0; m < d; ++m) {
    in->n[m] = n[m];
    cr->grid[m] = grid ? grid[m] : 0;
  }
  const TileGeo g = tile_geo_e(*in, *cr, r, b, te);
  int64_t bad = 0;
  auto side = [&](int64_t len, int64_t nm, int32_t pieces, int32_t count, bool rows) {
    std::vector<int32_t> cov((size_t)len, 0);
    for (int32_t t = 0; t < count; ++t) {
      int64_t s0;
      int nl;
      if (rows)
        tile_rows(*in, g, b, t, s0, nl);
      else
        tile_cols(*in, g, b, t, s0, nl);
      if (nl < 1 || nl > te || s0 < 0 || s0 + nl > len) {
        ++bad;
        continue;
      }
      if (pieces > 0) {
        const int64_t i0 = s0 % nm, q = nm / pieces, rem = nm % pieces;
        int64_t k = 0;
        while (k + 1 < pieces && (k + 1) * q + std::min<int64_t>(k + 1, rem) <= i0) ++k;
        const int64_t st = k * q + std::min<int64_t>(k, rem), sz = q + (k < rem ? 1 : 0);
        if ((s0 + nl - 1) / nm != s0 / nm || i0 + nl > st + sz) ++bad;
      }
      for (int64_t x = s0; x < s0 + nl; ++x) ++cov[(size_t)x];
    }
    for (int64_t x = 0; x < len; ++x) bad += cov[(size_t)x] != 1;
  };
  side(g.rows, n[b], g.pr, g.nrt, true);
  side(g.cols, n[b + 1], g.pc, g.nct, false);
  if (r_stored) {
    // stored form: the carried rectangle (row tiles < tr0, column tiles <
    // tc0) lies inside the stored extent at the ranks the residual was last
    // written with, so the carried warp tiles read only carried entries
    const int32_t sr = (int32_t)rows_of(*in, r_stored, b), sc = (int32_t)cols_of(*in, r_stored, b);
    int32_t tr0, tc0;
    carried_tiles(*in, g, b, sr, sc, tr0, tc0);
    if (tr0 < 0 || tr0 > g.nrt || tc0 < 0 || tc0 > g.nct) ++bad;
    for (int32_t t = 0; t < std::min(tr0, g.nrt); ++t) {
      int64_t s0;
      int nl;
      tile_rows(*in, g, b, t, s0, nl);
      if (s0 + nl > sr) ++bad;
    }
    for (int32_t t = 0; t < std::min(tc0, g.nct); ++t) {
      int64_t s0;
      int nl;
      tile_cols(*in, g, b, t, s0, nl);
      if (s0 + nl > sc) ++bad;
    }
  }
  if (ntiles) *ntiles = (int64_t)g.nrt * g.nct;
  return bad;
}

cudaError_t persistent_occupancy(int *blocks_per_sm) {
  cudaError_t e = cudaFuncSetAttribute(k_persistent, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(PhaseSmem));
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_persistent, NT,
                                                       sizeof(PhaseSmem));
}

cudaError_t launch_persistent(const RunArgs &ra, int grid, cudaStream_t s) {
  void *args[] = {(void *)&ra};
  return cudaLaunchCooperativeKernel((const void *)k_persistent, dim3(grid), dim3(NT), args,
                                     sizeof(PhaseSmem), s);
}

static cudaError_t prep(const void *f) {
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)sizeof(PhaseSmem));
}

cudaError_t launch_phase(int phase, const RunArgs &ra, int grid, cudaStream_t s) {
  const void *f = nullptr;
  switch (phase) {
    case PH_INIT1: f = (const void *)k_init1; break;
    case PH_INIT2: f = (const void *)k_init2; break;
    case PH_INIT3: f = (const void *)k_init3; break;
    case PH_BOUND: f = (const void *)k_bound; break;
    case PH_SCREEN: f = (const void *)k_screen; break;
    case PH_DECIDE: f = (const void *)k_decide; break;
    case PH_UPDATE: f = (const void *)k_update; break;
    case PH_REFINE: f = (const void *)k_refine; break;
    case PH_DECIDE2: f = (const void *)k_decide2; break;
    case PH_VERIFY: f = (const void *)k_verify; break;
    case PH_ROOK_STEP: f = (const void *)k_rook_step; break;
    case PH_FINALIZE: f = (const void *)k_finalize; break;
    default: return cudaErrorInvalidValue;
  }
  cudaError_t e = prep(f);
  if (e != cudaSuccess) return e;
  void *args[] = {(void *)&ra};
  if (phase == PH_VERIFY) {
    // its grid barriers count from zero
    e = cudaMemsetAsync(&ra.bar->count, 0, sizeof ra.bar->count, s);
    if (e != cudaSuccess) return e;
    return cudaLaunchCooperativeKernel(f, dim3(grid), dim3(NT), args, sizeof(PhaseSmem), s);
  }
  return cudaLaunchKernel(f, dim3(grid), dim3(NT), args, sizeof(PhaseSmem), s);
}

// ---------------------------------------------------------------------------
// Core construction from the pivot sets alone (Alg. 5, second loop; Sec.
// 3.2.2 and eq. corereshape): the history of Alg. 4 is rebuilt for every
// bond, then every superblock row of T_k is replayed from it, sliced over the
// grid (replay_group), and the last bond's R is formed from the entries.
// By the arithmetic contract every value equals the one the sweeps kept.

// history of bond blockIdx.x (one CTA per bond).  M starts as the entries
// A(a_z, c_u) of the pivot rows and columns (k_rebuild_start); before step t
// row z >= t holds T(a_z, :t) in its first t places.  Step t takes its column
// c_t = A(a_u, c_t) (u < t), its snapshot T(a_t, :t) and delta_t, a thread per
// row z >= t runs the chain over c_t (z = t gives the pivot), and the updates
// of the later rows are dealt over the CTA.  Serial in t: a step is a chain of t
// FMAs (63 cycles each), a divide and three CTA barriers, so M lies in
// shared memory where it fits (up to RB_SMALL pivots).
__global__ void __launch_bounds__(NT) k_rebuild_history(const InstDev *inp, double *scratch) {
  const InstDev &in = *inp;
  const int b = blockIdx.x;
  if (b >= in.nb) return;
  const BondDev &B = in.bond[b];
  const int r = in.ctrl->r[b];
  const int64_t cap = B.cap;
  const bool small = r <= RB_SMALL;
  const int64_t ld = small ? RB_SMALL + 1 : RCAP;
  double *M = small ? reinterpret_cast<double *>(dyn_smem) : scratch + (int64_t)b * RCAP * RCAP;
  __shared__ double s_hc[RCAP], s_hp[RCAP], s_w[RCAP];
  __shared__ double s_delta;
  __shared__ int s_ok;
  for (int x = threadIdx.x; small && x < r * r; x += NT) {
    const int z = x / r, u = x - z * r;
    M[z * ld + u] = scratch[((int64_t)b * RCAP + z) * RCAP + u];
  }
  __syncthreads();
  for (int t = 0; t < r; ++t) {
    // c_t restricted to the earlier pivots, and row a_t's snapshot
    for (int u = threadIdx.x; u < t; u += NT) {
      s_hc[u] = M[u * ld + t];
      s_hp[u] = M[t * ld + u];
      B.hc[(int64_t)t * cap + u] = s_hc[u];
      B.hpiv[(int64_t)t * cap + u] = s_hp[u];
    }
    __syncthreads();
    for (int z = t + threadIdx.x; z < r; z += NT) {
      const double acc = chain(M + z * ld, 1, s_hc, 1, t), e = M[z * ld + t];
      if (z == t) {
        s_delta = 1.0 / __dsub_rn(e, acc);
        s_ok = isfinite(s_delta) ? 1 : 0;
        B.delta[t] = s_delta;
      } else {
        s_w[z] = __dsub_rn(acc, e);
      }
    }
    __syncthreads();
    if (!s_ok) return;  // no such pivot was taken (the sweeps check the same value)
    const double dt = s_delta;
    // step t on the later pivot rows z > t
    for (int x = threadIdx.x; x < (r - t - 1) * (t + 1); x += NT) {
      const int z = t + 1 + x / (t + 1), u = x % (t + 1);
      const double w = __dmul_rn(dt, s_w[z]);
      M[z * ld + u] = u < t ? __fma_rn(w, s_hp[u], M[z * ld + u]) : -w;
    }
    __syncthreads();
  }
}

// every superblock row of every bond replayed through its whole history
// (Alg. 4), groups of rows dealt over the grid; then R of the last bond (its
// core) from the entries.  FP64 issue bounds it where rows are many: a warp's
// instruction costs the same for one row as for eight, so up to RB_SMALL pivots
// a warp takes eight rows (6D Hilbert n = 300, ranks 15..18, history and rows
// with the clearing: 0.34 -> 0.11 ms; a random TT of ranks 48: 22.5 -> 1.5 ms).
// Rows that fill at most a quarter of the grid's warps (four warps keep an SM's
// FP64 pipe busy) take a warp each, which is shorter.
__global__ void __launch_bounds__(NT, 2) k_rebuild_rows(const InstDev *inp, int words) {
  const InstDev &in = *inp;
  double *buf = reinterpret_cast<double *>(dyn_smem) + (threadIdx.x >> 5) * words;
  const int64_t nwarps = (int64_t)gridDim.x * (NT / 32);
  // neighbouring groups on different CTAs: few groups still use every SM
  const int64_t gw = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  int64_t base = 0;
  for (int b = 0; b < in.nb; ++b) {
    const int r = in.ctrl->r[b];
    const int64_t rows = (int64_t)(b == 0 ? 1 : in.ctrl->r[b - 1]) * in.n[b];
    const bool wide = r <= RB_SMALL && rows > nwarps / 4;
    const int rpw = wide ? 8 : 1;
    const int64_t groups = (rows + rpw - 1) / rpw;
    for (int64_t g = ((gw - base) % nwarps + nwarps) % nwarps; g < groups; g += nwarps) {
      const int64_t a0 = g * rpw;
      if (wide)
        replay_group<4, RB_SMALL>(in, b, a0, (int)min((int64_t)8, rows - a0), r, buf);
      else if (r <= RB_SMALL)
        replay_group<32, RB_SMALL>(in, b, a0, 1, r, buf);
      else
        replay_group<32, RCAP>(in, b, a0, 1, r, buf);
    }
    base += groups;
  }
  const int bl = in.nb - 1;
  const BondDev &B = in.bond[bl];
  const int r = in.ctrl->r[bl];
  const int64_t nn = in.n[in.d - 1];
  const int64_t gt = (int64_t)blockIdx.x * NT + threadIdx.x, NTOT = (int64_t)gridDim.x * NT;
  for (int64_t x = gt; x < r * nn; x += NTOT) {
    const int64_t t = x / nn, c = x - t * nn;
    putR(in, B, t, c, sb_entry(in, bl, B.prow[t], c));
  }
}

// the factors and histories go, so that the cores come from the pivot sets
// alone (one launch; a memset per buffer was 4 per bond), and the entries of
// the pivot rows and columns are formed over the whole grid
__global__ void __launch_bounds__(NT) k_rebuild_start(const InstDev *inp, double *scratch) {
  const InstDev &in = *inp;
  const int64_t gt = (int64_t)blockIdx.x * NT + threadIdx.x, NTOT = (int64_t)gridDim.x * NT;
  for (int b = 0; b < in.nb; ++b) {
    const BondDev &B = in.bond[b];
    const int64_t cap = B.cap;
    for (int64_t x = gt; x < cap * B.ldT; x += NTOT) B.T[x] = 0.0;
    for (int64_t x = gt; x < cap * cap; x += NTOT) {
      B.hc[x] = 0.0;
      B.hpiv[x] = 0.0;
    }
    for (int64_t x = gt; x < cap; x += NTOT) B.delta[x] = 0.0;
    if (b == in.nb - 1)
      for (int64_t x = gt; x < cap * B.ldR; x += NTOT) B.R[x] = 0.0;
    const int r = in.ctrl->r[b];
    for (int64_t x = gt; x < r * r; x += NTOT) {
      const int z = (int)x / r, u = (int)x - z * r;
      scratch[((int64_t)b * RCAP + z) * RCAP + u] = sb_entry(in, b, B.prow[z], B.pcol[u]);
    }
  }
}

// rmax: the largest rank (sizes the replay buffers: two CTAs a SM up to RB_SMALL)
cudaError_t launch_rebuild_cores(const InstDev *d_inst, int nb, int rmax, double *scratch,
                                 int grid, cudaStream_t s) {
  const int words = rmax <= RB_SMALL ? RB_BUF_SMALL : RB_BUF;
  const int bytes = words * (NT / 32) * (int)sizeof(double);
  const int hist = RB_SMALL * (RB_SMALL + 1) * (int)sizeof(double);  // 33 KB
  cudaError_t e = cudaFuncSetAttribute((const void *)k_rebuild_rows,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       RB_BUF * (NT / 32) * (int)sizeof(double));
  if (e != cudaSuccess) return e;
  k_rebuild_start<<<grid, NT, 0, s>>>(d_inst, scratch);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_rebuild_history<<<nb, NT, hist, s>>>(d_inst, scratch);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_rebuild_rows<<<grid, NT, bytes, s>>>(d_inst, words);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// user generator: the entries that enter the superblocks after a decision.
// For bond b with old / new ranks the superblock grows from ro x co to
// rn x cn (rows, columns); its new entries are, in this order,
//   rows ro..rn-1 x columns 0..cn-1, then rows 0..ro-1 x columns co..cn-1.
// k_user_count sums them per bond (first: every entry of the rank-one
// superblocks), and says whether the run is over or an error check is due; k_user_gather writes their multi-indices, k_user_scatter
// puts the callback's values into the cache at (a, c).

__device__ void user_extent(const InstDev &in, const Ctrl &cr, int b, int first, int64_t &ro,
                            int64_t &co, int64_t &rn, int64_t &cn) {
  const int32_t *r = cr.r, *ad = cr.add;
  const int64_t pl = b == 0 ? 1 : r[b - 1], ql = b == in.nb - 1 ? 1 : r[b + 1];
  const int64_t pa = b == 0 ? 0 : ad[b - 1], qa = b == in.nb - 1 ? 0 : ad[b + 1];
  rn = pl * in.n[b];
  cn = in.n[b + 1] * ql;
  ro = first ? 0 : (pl - pa) * in.n[b];
  co = first ? 0 : in.n[b + 1] * (ql - qa);
}

__global__ void k_user_count(const InstDev *inp, int first, int64_t *counts) {
  const InstDev &in = *inp;
  const Ctrl &cr = *in.ctrl;
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  int64_t tot = 0;
  for (int b = 0; b < in.nb; ++b) {
    counts[b] = tot;
    int64_t ro, co, rn, cn;
    user_extent(in, cr, b, first, ro, co, rn, cn);
    if (cr.state != ST_DONE) tot += rn * cn - ro * co;
  }
  counts[in.nb] = tot;
  int nadd = 0;
  for (int b = 0; b < in.nb; ++b) nadd += cr.add[b];
  int nu = 0;  // inverses to be bordered yet
  for (int b = 0; b < in.nb; ++b) nu += cr.u_rank[b] < cr.r[b];
  counts[in.nb + 1] = cr.state == ST_DONE ? 1 + nu : 0;
  counts[in.nb + 2] = cr.state != ST_DONE && cr.screened && nadd == 0;
}

// entry x of the new entries of bond b -> superblock (a, c)
__device__ __forceinline__ void user_entry(int64_t x, int64_t ro, int64_t co, int64_t rn,
                                           int64_t cn, int64_t &a, int64_t &c) {
  const int64_t top = (rn - ro) * cn;
  if (x < top) {
    a = ro + x / cn;
    c = x - (a - ro) * cn;
  } else {
    const int64_t y = x - top, w = cn - co;
    a = y / w;
    c = co + (y - a * w);
  }
}

__global__ void k_user_gather(const InstDev *inp, int first, const int64_t *counts, int32_t *idx) {
  const InstDev &in = *inp;
  const Ctrl &cr = *in.ctrl;
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t NTOT = (int64_t)gridDim.x * blockDim.x;
  for (int b = 0; b < in.nb; ++b) {
    int64_t ro, co, rn, cn;
    user_extent(in, cr, b, first, ro, co, rn, cn);
    const int64_t base = counts[b], cnt = counts[b + 1] - base;
    const SetDev &L = left_set(in, b), &Rs = right_set(in, b);
    const int wl = b, wr = in.d - b - 2;
    for (int64_t x = gt; x < cnt; x += NTOT) {
      int64_t a, c;
      user_entry(x, ro, co, rn, cn, a, c);
      const int64_t p = a / in.n[b], i = a - p * in.n[b];
      const int64_t q = c / in.n[b + 1], j = c - q * in.n[b + 1];
      int32_t *o = idx + (base + x) * in.d;
      for (int m = 0; m < wl; ++m) o[m] = L.idx[p * wl + m];
      o[b] = (int32_t)i;
      o[b + 1] = (int32_t)j;
      for (int m = 0; m < wr; ++m) o[b + 2 + m] = Rs.idx[q * wr + m];
    }
  }
}

__global__ void k_user_scatter(const InstDev *inp, int first, const int64_t *counts,
                               const double *vals) {
  const InstDev &in = *inp;
  const Ctrl &cr = *in.ctrl;
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t NTOT = (int64_t)gridDim.x * blockDim.x;
  for (int b = 0; b < in.nb; ++b) {
    int64_t ro, co, rn, cn;
    user_extent(in, cr, b, first, ro, co, rn, cn);
    const int64_t base = counts[b], cnt = counts[b + 1] - base;
    const BondDev &B = in.bond[b];
    for (int64_t x = gt; x < cnt; x += NTOT) {
      int64_t a, c;
      user_entry(x, ro, co, rn, cn, a, c);
      B.A[a * B.ldR + c] = vals[base + x];
    }
  }
}

// the error samples' multi-indices, then the origin's
__global__ void k_user_samples(const InstDev *inp, int32_t *idx) {
  const InstDev &in = *inp;
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t NTOT = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = gt; k <= in.nsamples; k += NTOT) {
    int32_t *o = idx + k * in.d;
    if (k == in.nsamples) {
      for (int m = 0; m < in.d; ++m) o[m] = 0;
    } else {
      for (int m = 0; m < in.d; ++m) o[m] = sample_coord(in, k, m);
    }
  }
}

cudaError_t launch_user_count(const InstDev *d_inst, int first, int64_t *counts, cudaStream_t s) {
  k_user_count<<<1, 32, 0, s>>>(d_inst, first, counts);
  return cudaGetLastError();
}
cudaError_t launch_user_gather(const InstDev *d_inst, int first, const int64_t *counts,
                               int32_t *idx, cudaStream_t s) {
  k_user_gather<<<152 * 4, 256, 0, s>>>(d_inst, first, counts, idx);
  return cudaGetLastError();
}
cudaError_t launch_user_scatter(const InstDev *d_inst, int first, const int64_t *counts,
                                const double *vals, cudaStream_t s) {
  k_user_scatter<<<152 * 4, 256, 0, s>>>(d_inst, first, counts, vals);
  return cudaGetLastError();
}
cudaError_t launch_user_samples(const InstDev *d_inst, int32_t *idx, cudaStream_t s) {
  k_user_samples<<<152 * 4, 256, 0, s>>>(d_inst, idx);
  return cudaGetLastError();
}

// The samples of block blockIdx.x in the order of their index of mode
// m = 1 + blockIdx.y (stable), and their tiles (create time; the tile slots
// are all TC_NO_TILE before).  PW warps take equal parts of the block: each
// counts its samples per index, the counts (and the tiles they make) are
// scanned over (index, warp), each warp places its samples.  A warp's steps are
// serial, so as many warps as the counts' shared memory has room for: 32 up to
// 512 indices, 8 up to TC_NMAX; the second pass takes the indices and the places
// among the warp's equal ones from registers (1e6 samples, four middle modes of
// 64: 63 us, 71 with them formed again; two of 1024: 141 and 158; a ballot per bit in
// place of the match was slower).
template <int PW, int NM>
__global__ void __launch_bounds__(32 * PW, 1) k_tc_perm(const InstDev *inp, uint16_t *perm,
                                                     uint32_t *const *tiles) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int SEG = TC_BLOCK / PW;
  constexpr uint32_t NONE = 0xffffffffu;
  __shared__ uint16_t cnt[PW][NM];
  __shared__ int32_t wsum[PW], wtile[PW];
  const InstDev &in = *inp;
  const int m = 1 + blockIdx.y, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int n = (int)in.n[m];
  const int64_t k0 = (int64_t)blockIdx.x * TC_BLOCK;
  uint32_t held[SEG / 32];  // index, whether the last of its lanes, place among them
  for (int x = threadIdx.x; x < PW * n; x += blockDim.x) cnt[x / n][x % n] = 0;
  __syncthreads();
#pragma unroll
  for (int s = 0; s < SEG / 32; ++s) {
    const int id = w * SEG + s * 32 + lane;
    const bool ok = k0 + id < in.nsamples;
    const int key = ok ? sample_coord(in, k0 + id, m) : n;
    const unsigned peers = __match_any_sync(FULL, key);
    const int rank = __popc(peers & ((1u << lane) - 1)), many = __popc(peers);
    held[s] = ok ? (uint32_t)(key << 16 | (rank + 1 == many) << 8 | rank) : NONE;
    if (ok && rank == 0) cnt[w][key] += (uint16_t)many;
    __syncwarp();
  }
  __syncthreads();
  // exclusive scan in (index, warp) order: thread x takes indices [x c, (x + 1) c)
  const int c = (n + (int)blockDim.x - 1) / (int)blockDim.x;
  const int i0 = min(n, (int)threadIdx.x * c), i1 = min(n, i0 + c);
  int sum = 0, nti = 0;
  for (int i = i0; i < i1; ++i) {
    int v = 0;
    for (int q = 0; q < PW; ++q) v += cnt[q][i];
    sum += v;
    nti += (v + 15) / 16;
  }
  int inc = sum, tinc = nti;
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(FULL, inc, o), u = __shfl_up_sync(FULL, tinc, o);
    if (lane >= o) {
      inc += v;
      tinc += u;
    }
  }
  if (lane == 31) {
    wsum[w] = inc;
    wtile[w] = tinc;
  }
  __syncthreads();
  int at = inc - sum, ta = tinc - nti;
  for (int q = 0; q < w; ++q) {
    at += wsum[q];
    ta += wtile[q];
  }
  uint32_t *tl = tiles[m] + (int64_t)blockIdx.x * (TC_BLOCK / 16 + n);
  for (int i = i0; i < i1; ++i) {
    const int first = at;
    for (int q = 0; q < PW; ++q) {
      const int v = cnt[q][i];
      cnt[q][i] = (uint16_t)at;
      at += v;
    }
    for (int o = first; o < at; o += 16)
      tl[ta++] = ((uint32_t)i << 19) | ((uint32_t)o << 4) | (uint32_t)(min(16, at - o) - 1);
  }
  __syncthreads();
  uint16_t *pm = perm + (int64_t)(m - 1) * in.tc_stride + k0;
#pragma unroll
  for (int s = 0; s < SEG / 32; ++s) {
    const uint32_t h = held[s];
    const int key = h >> 16, rank = h & 0xff;
    const int to = h == NONE ? 0 : cnt[w][key] + rank;
    if (h != NONE) pm[to] = (uint16_t)(w * SEG + s * 32 + lane);
    __syncwarp();
    if (h != NONE && (h >> 8 & 1)) cnt[w][key] = (uint16_t)(to + 1);
    __syncwarp();
  }
}

cudaError_t launch_tc_perm(const InstDev *d_inst, int d, int64_t nmax, int64_t blocks, uint16_t *perm,
                           uint32_t *const *tiles) {
  const dim3 g((unsigned)blocks, (unsigned)(d - 2));
  if (nmax <= 512)
    k_tc_perm<32, 512><<<g, 32 * 32>>>(d_inst, perm, tiles);
  else
    k_tc_perm<8, TC_NMAX><<<g, 32 * 8>>>(d_inst, perm, tiles);
  return cudaGetLastError();
}

size_t tc_plan_bytes() { return sizeof(TcPlan); }

// Maxwellian tables of an instance (create time)
__global__ void k_maxwellian_tables(const InstDev *inp, double *coef, double *nh, double *uv) {
  const InstDev &in = *inp;
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t NTOT = (int64_t)gridDim.x * blockDim.x;
  if (in.gen == 3) {
    for (int m = 0; m < in.d; ++m)
      for (int64_t i = gt; i < in.n[m]; i += NTOT)
        maxwellian_xv_table_entry(in, m, i, coef + in.mx_off[m] + i, nh + in.mx_off[m] + i);
    return;
  }
  int64_t ncombo = 1;
  for (int m = 0; m < in.dx; ++m) ncombo *= in.n[m];
  for (int64_t c = gt; c < ncombo; c += NTOT) maxwellian_table_entry(in, c, coef + c, nh + c);
  const double two_pi = 6.283185307179586476925286766559;
  for (int m = 0; m < in.dx; ++m)
    for (int64_t i = gt; i < in.n[m]; i += NTOT)
      uv[in.mx_off[m] + i] = __dmul_rn(in.a_u, cos(__dmul_rn(two_pi, (double)i) / (double)in.n[m]));
  for (int m = in.dx; m < in.d; ++m)
    for (int64_t i = gt; i < in.n[m]; i += NTOT)
      uv[in.mx_off[m] + i] =
          __dadd_rn(in.vmin, __dmul_rn(__dsub_rn(in.vmax, in.vmin), (double)i) / (double)(in.n[m] - 1));
}

cudaError_t launch_maxwellian_tables(const InstDev *d_inst, double *coef, double *nh, double *uv) {
  k_maxwellian_tables<<<152 * 4, 256>>>(d_inst, coef, nh, uv);
  return cudaGetLastError();
}

cudaError_t launch_core(const InstDev *d_inst, int m, double *dst, cudaStream_t s) {
  k_core<<<152, 256, 0, s>>>(d_inst, m, dst);
  return cudaGetLastError();
}


}  // namespace ttc

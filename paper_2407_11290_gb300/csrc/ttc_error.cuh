// ttc_error.cuh -- the sampled error's middle cores on the tensor cores.
//
// X~(i) = G_1(i_1) ... G_d(i_d) at up to millions of samples is a chain of
// vector x matrix products, one middle core G_m(i_m) after the other, and in
// FP64 it is bound by the FP64 pipe (two FMAs per clock and SM on this GPU:
// 1.1e9 FMAs took 2.26 ms of the 6D n = 256 Hilbert cross, 8.8e10 took 160 ms
// of the 6D Maxwellian at ranks 256).  Samples that share i_m share the matrix,
// so the samples are kept sorted by every middle index (within blocks of
// TC_BLOCK samples, ttcross_create) and each middle core becomes a small GEMM
// per value of i_m.
//
// The products are exact integer arithmetic: a vector (a table row, or the
// result of the previous core) and each column of G_m(i) are scaled to 63-bit
// integers by a power of two (the exponent of their largest entry), split
// into eight signed base-256 digits, and the digit products of weight
// 256^-(i+j), i + j <= 7, run as f16 mma.sync with FP32 accumulation: digits
// are at most 128 in magnitude, so eight levels' sums over K <= 128 terms stay
// within 2^24 and every FP32 sum is exact.  (This is the splitting of Ozaki,
// Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication
// by using fast routines of matrix multiplication", 2012, with digits in fixed
// point.)  What is dropped lies 2^-61 below the largest product of a sum and below:
// X~ is as exact as the FP64 chains' (each of which rounds K times) as long as
// its terms are not far smaller than the largest ones of T and R.  An entry 2^-40
// of its row's largest keeps 22 bits where FP64 kept 53.  In a cross T's entries
// are about one and R's as large as the pivots, so what counts is the largest
// pivot against rms(X) (TC_PEAK): beyond it the chains do the check.
//
// The same products extend the prefix / suffix tables by their last mode where
// its rows are fewer than the samples (n^3 rows for 1e6 samples at n = 64).
//
// f16 and not s8: s8 mma.sync runs at a quarter of the f16 rate here (237
// against 951 MACs per clock and SM, measured).  mma.sync and not tcgen05: an
// output needs eight f32 accumulators, a warp's tile is 16 rows gathered from
// anywhere, and the digits are made in registers right before their use.  At
// kp = 32 a warp spends its time on L2 latency and integer work about as much
// as on the tensor pipe (18 % busy, ncu), at four warps an SM quarter (the
// register budget of the cross kernel).
//
// Measured (error check, 1e6 samples; FP64 chains -> this): 2.26 -> 0.91 ms
// (6D n = 256, ranks 21..23), 160 -> 8.0 ms (6D Maxwellian n = 64, ranks up to
// 256), 0.41 -> 0.32 ms (6D n = 64), 174 -> 52 ms (37 checks of a batch of 12
// Maxwellians).  The error against extended precision is below the FP64
// chains' in each of six Hilbert cases (7.8e-8 against 4.0e-7 relative at
// n = 256, where err itself is 7e-12 of the norm).
//
// Layout: fixed-point rows are K rounded up to 16 (kp) integers, biased by
// 0x8080808080808080 so that every byte is an unsigned digit + 128 (zero is
// the bias itself), and stored as pairs of neighbours with their bytes
// interleaved, most significant first: the 16 bytes of a pair (x, y) are
// x7 y7 x6 y6 ... x0 y0, so that one byte permutation with 0x64 makes the f16
// pair (1024 + x_k, 1024 + y_k).  Columns of G_m(i) lie as [i][u][p].
#pragma once

#include "ttc_split.cuh"

namespace ttc {

// the error check's plan for the current ranks, one per instance (InstDev::tcp)
struct TcPlan {
  int32_t on;              // 1: the middle cores run here; 0: the FP64 chains
  int32_t pL, pR;          // modes in the prefix / suffix tables
  int32_t nst;             // middle cores (stages)
  int32_t blocks;          // sample blocks per step
  int32_t nsb;             // steps' sample ranges: ceil(sample blocks / blocks)
  int32_t tl, tr;          // on = 0: the prefix / suffix table's last mode runs here
  // workspace offsets (8-byte words): prefix rows and their exponents (on, tl),
  // suffix rows (on: doubles; tr: fixed point) and their exponents (tr)
  int64_t L, Le, R, Re;
  int64_t G[TTC_MAXD], Ge[TTC_MAXD];  // per mode: columns, their exponents
  int64_t C[2], Ce[2];     // results of the stages (ping-pong) and exponents
};

// a row of len doubles (16-byte aligned, room for kp) to fixed point in place;
// returns the exponent of its units
__device__ int32_t tc_fix_row(double *row, int len, int kp) {
  int emax = 0;
  for (int t = 0; t < len; ++t) emax = max(emax, tc_expo(row[t]));
  for (int t = 0; t < kp; t += 2) {
    const uint64_t x = t < len ? tc_fix(row[t], emax) : TC_BIAS;
    const uint64_t y = t + 1 < len ? tc_fix(row[t + 1], emax) : TC_BIAS;
    *reinterpret_cast<uint4 *>(row + t) = tc_pack(x, y);
  }
  return tc_unit(emax);
}

// ---------------------------------------------------------------------------
// the plan

// FP64 FMAs of the tables of pL / pR modes (their last level)
__device__ __forceinline__ float tc_table_cost(const InstDev &in, const int32_t *r, int pL, int pR) {
  const int d = in.d;
  float NL = 1.f, NR = 1.f;
  for (int m = 0; m < pL; ++m) NL *= (float)in.n[m];
  for (int m = d - pR; m < d; ++m) NR *= (float)in.n[m];
  const float tl = pL >= 2 ? NL * (float)core_s(in, r, pL - 1) * (float)core_s(in, r, pL) : 0.f;
  const float tr =
      pR >= 2 ? NR * (float)core_s(in, r, d - pR) * (float)core_s(in, r, d - pR + 1) : 0.f;
  return tl + tr;
}

// Offsets of the plan (pL, pR) in the workspace; false if it does not fit.
__device__ bool tc_layout(const InstDev &in, const int32_t *r, int pL, int pR, TcPlan &p) {
  const int d = in.d;
  int64_t NL = 1, NR = 1, o = 0;
  for (int m = 0; m < pL; ++m) NL *= in.n[m];
  for (int m = d - pR; m < d; ++m) NR *= in.n[m];
  if (NL > TC_TABLE_MAX || NR > TC_TABLE_MAX) return false;
  p.pL = pL;
  p.pR = pR;
  p.tl = p.tr = 0;
  p.nst = d - pL - pR;
  p.L = o;
  o += NL * tc_up(core_s(in, r, pL), 16);
  p.Le = o;
  o += tc_up(NL, 4) / 2;
  p.R = o;
  o += tc_up(NR * core_s(in, r, d - pR), 4);
  int64_t kmax = 0;
  for (int m = pL; m < d - pR; ++m) {
    const int64_t kp = tc_up(core_s(in, r, m), 16), np = tc_up(core_s(in, r, m + 1), 8);
    p.G[m] = o;
    o += in.n[m] * np * kp;
    p.Ge[m] = o;
    o += tc_up(in.n[m] * np, 4) / 2;
    if (m > pL) kmax = max(kmax, kp);
  }
  // the stages' results: one buffer between two stages, two beyond
  const int nbuf = p.nst >= 3 ? 2 : p.nst == 2 ? 1 : 0;
  const int64_t nblk = (in.nsamples + TC_BLOCK - 1) / TC_BLOCK;
  int64_t per = 0;  // words of one sample block in all buffers
  if (nbuf) per = nbuf * (TC_BLOCK * kmax + TC_BLOCK / 2);
  if (o > in.ews_cap || (nbuf && o + per > in.ews_cap)) return false;
  // as many samples at a time as the workspace holds results of, in even steps
  int64_t nb = nblk;
  if (nbuf) {
    nb = min(nblk, (in.ews_cap - o) / per);
    nb = (nblk + (nblk + nb - 1) / nb - 1) / ((nblk + nb - 1) / nb);
  }
  p.blocks = (int32_t)nb;
  p.nsb = (int32_t)((nblk + nb - 1) / nb);
  for (int k = 0; k < 2; ++k) {
    p.C[k] = o;
    o += k < nbuf ? nb * TC_BLOCK * kmax : 0;
    p.Ce[k] = o;
    o += k < nbuf ? nb * TC_BLOCK / 2 : 0;
  }
  return true;
}

// Costs in FP64 FMAs at the pipe's rate (half a clock of an SM each).  A K x N
// product of one row here: 36 K N / 951 clocks of tensor time; with the loads,
// the digits and the rescaling 0.16 K N + 75 (measured: 0.70 ms for the two
// 21..23-wide cores of the 6D n = 256 check, 23 ms for the 256 x 256 and
// 86 x 256 cores of the 6D Maxwellian).  FP64 chains and tables run at about
// two thirds of the pipe; a sample's gather and dot cost its length and 30.
__device__ __forceinline__ float tc_cost(int64_t K, int64_t N) {
  return 0.16f * (float)tc_up(K, 16) * (float)tc_up(N, 8) + 75.f;
}
constexpr float TC_FP64 = 1.5f;

// The plan with every sample's chain in FP64 and tables of pL / pR modes,
// their last mode on the tensor cores where that is cheaper; its cost.
__device__ float tc_tables(const InstDev &in, const int32_t *r, int pL, int pR, TcPlan &p) {
  const int d = in.d;
  p.on = p.nst = p.tl = p.tr = 0;
  p.pL = pL;
  p.pR = pR;
  int64_t o = tc_up(in.tabL_cap, 32) + tc_up(in.tabR_cap, 32);
  float cost = 0.f;
  for (int side = 0; side < 2; ++side) {
    const int w = side ? pR : pL;
    if (w < 2) continue;
    // rows before the last mode m, its contraction K x N, the rows before
    const int m = side ? d - pR : pL - 1;
    int64_t base = 1;
    for (int q = 1; q < w; ++q) base *= in.n[side ? d - q : q - 1];
    const int64_t K = core_s(in, r, side ? m + 1 : m), N = core_s(in, r, side ? m : m + 1);
    const float rows = (float)base * (float)in.n[m];
    float f64 = TC_FP64 * rows * (float)K * (float)N;
    float tc = rows * tc_cost(K, N) + 1.2e7f;
    if (w >= 3) tc += TC_FP64 * (float)base * (float)K * (float)core_s(in, r, side ? m + 2 : m - 1);
    const int64_t kp = tc_up(K, 16), np = tc_up(N, 8);
    const int64_t need = base * kp + tc_up(base, 4) / 2 + in.n[m] * np * kp + tc_up(in.n[m] * np, 4) / 2;
    if (tc < f64 && o + need <= in.ews_cap && base * in.n[m] < ((int64_t)1 << 30)) {
      f64 = tc;
      (side ? p.tr : p.tl) = 1;
      (side ? p.R : p.L) = o;
      o += base * kp;
      (side ? p.Re : p.Le) = o;
      o += tc_up(base, 4) / 2;
      p.G[m] = o;
      o += in.n[m] * np * kp;
      p.Ge[m] = o;
      o += tc_up(in.n[m] * np, 4) / 2;
    }
    cost += f64;
  }
  float per = (float)core_s(in, r, d - pR) + 30.f;
  for (int m = pL; m < d - pR; ++m)
    per += TC_FP64 * (float)core_s(in, r, m) * (float)core_s(in, r, m + 1);
  return cost + (float)in.nsamples * per;
}

// The cheapest plan for ranks r: tables and FP64 chains, or the middle cores
// of every sample here (the extra phases cost about 20 us, 1.2e7).
__device__ void tc_plan(const InstDev &in, const int32_t *r, TcPlan &p) {
  const int d = in.d;
  const double peak = __longlong_as_double((long long)ld_cg(in.ctrl->piv_max));
  if (!in.tc_perm || !(peak <= TC_PEAK * ld_cg(in.ctrl->xrms))) {
    p.on = p.nst = p.tl = p.tr = 0;
    choose_split(in, r, p.pL, p.pR);
    return;
  }
  float best = 3e38f;
  int on = 0, bl = 1, br = 1;
  float NL = 1.f;
  for (int a = 1; a < d; ++a) {
    NL *= (float)in.n[a - 1];
    if (a >= 2 && NL * (float)core_s(in, r, a) > (float)in.tabL_cap) break;
    float NR = 1.f;
    for (int c = 1; a + c <= d; ++c) {
      NR *= (float)in.n[d - c];
      if (c >= 2 && NR * (float)core_s(in, r, d - c) > (float)in.tabR_cap) break;
      const float cost = tc_tables(in, r, a, c, p);
      if (cost < best) {
        best = cost;
        bl = a;
        br = c;
      }
    }
  }
  for (int a = 1; a <= 2; ++a)
    for (int c = 1; c <= 2; ++c) {
      if (a + c >= d || !tc_layout(in, r, a, c, p)) continue;
      float per = (float)core_s(in, r, d - c) + 30.f;
      for (int m = a; m < d - c; ++m) per += tc_cost(core_s(in, r, m), core_s(in, r, m + 1));
      const float cost = TC_FP64 * tc_table_cost(in, r, a, c) + (float)in.nsamples * per + 1.2e7f;
      if (cost < best) {
        best = cost;
        on = 1;
        bl = a;
        br = c;
      }
    }
  if (on)
    tc_layout(in, r, bl, br, p);
  else
    tc_tables(in, r, bl, br, p);
  p.on = on;
}

// ---------------------------------------------------------------------------
// The columns of G_m(i) in fixed point.  right: its rows (the core applied to
// suffix vectors, K = s_{m+1} wide); else its columns (K = s_m).  A thread per
// (i, u) reads its K entries (coalesced over i) and writes their kp words.
__device__ void tc_columns(const InstDev &in, const int32_t *r, const TcPlan &p, int m, bool right,
                           int64_t &base, int64_t gt, int64_t NTOT) {
  uint64_t *ws = reinterpret_cast<uint64_t *>(in.ews);
  const BondDev &B = in.bond[m];
  const int K = (int)core_s(in, r, right ? m + 1 : m), N = (int)core_s(in, r, right ? m : m + 1);
  const int kp = (int)tc_up(K, 16), np = (int)tc_up(N, 8);
  const int64_t n = in.n[m], items = n * np;
  const int64_t sk = right ? B.ldT : n, su = right ? n : B.ldT;
  int32_t *ge = reinterpret_cast<int32_t *>(ws + p.Ge[m]);
  for (int64_t x = first_item(base, gt, NTOT); x < base + items; x += NTOT) {
    const int64_t u = (x - base) / n, i = (x - base) - u * n;
    uint4 *o = reinterpret_cast<uint4 *>(ws + p.G[m] + (i * np + u) * kp);
    const double *src = B.T + u * su + i;
    int emax = 0;
    if (u < N)
      for (int q = 0; q < K; q += 8) {
        double v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = q + k < K ? src[(q + k) * sk] : 0.0;
#pragma unroll
        for (int k = 0; k < 8; ++k) emax = max(emax, tc_expo(v[k]));
      }
    for (int q = 0; q < kp; q += 8) {
      uint64_t w[8];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        w[k] = u < N && q + k < K ? tc_fix(src[(q + k) * sk], emax) : TC_BIAS;
#pragma unroll
      for (int k = 0; k < 8; k += 2) o[(q + k) / 2] = tc_pack(w[k], w[k + 1]);
    }
    ge[i * np + u] = tc_unit(emax);
  }
  base += items;
}

// ---------------------------------------------------------------------------
// one tile: 16 samples' rows times G_m(i)

// The four outputs of a lane (rows g, g + 8; columns 2t, 2t + 1 of one 8-wide
// column tile) of rows x G_m(i): out * 2^(units of the row and of the column
// + 88 - sh).  a0 / a1: the rows' pairs at the lane's place (pair t of every
// eight); b: the column's.
__device__ __forceinline__ void tc_product(const uint64_t *a0, const uint64_t *a1,
                                           const uint64_t *b, int kp, int sh, int64_t (&out)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) out[q] = 0;
  const bool magic = kp <= 32;
  for (int k0 = 0; k0 < kp; k0 += 128) {
    float acc[8][4];
#pragma unroll
    for (int l = 0; l < 8; ++l)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[l][q] = magic ? TC_MAGIC : 0.f;
    const int k1 = min(kp, k0 + 128);
    for (int ks = k0; ks < k1; ks += 16) {
      const uint4 x0 = *reinterpret_cast<const uint4 *>(a0 + ks);
      const uint4 x1 = *reinterpret_cast<const uint4 *>(a0 + ks + 8);
      const uint4 y0 = *reinterpret_cast<const uint4 *>(a1 + ks);
      const uint4 y1 = *reinterpret_cast<const uint4 *>(a1 + ks + 8);
      const uint4 z0 = *reinterpret_cast<const uint4 *>(b + ks);
      const uint4 z1 = *reinterpret_cast<const uint4 *>(b + ks + 8);
      // the column's digits first, then the rows' a level at a time (fewer live
      // registers than the other way round)
      uint32_t db[8][2];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        db[j][0] = tc_digits(z0, j);
        db[j][1] = tc_digits(z1, j);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const uint32_t da[4] = {tc_digits(x0, k), tc_digits(y0, k), tc_digits(x1, k),
                                tc_digits(y1, k)};
#pragma unroll
        for (int j = 0; k + j < 8; ++j) tc_mma(acc[k + j], da, db[j][0], db[j][1]);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t hi = tc_join(tc_int(acc[0][q], magic), tc_int(acc[1][q], magic),
                                 tc_int(acc[2][q], magic), tc_int(acc[3][q], magic));
      const int64_t lo = tc_join(tc_int(acc[4][q], magic), tc_int(acc[5][q], magic),
                                 tc_int(acc[6][q], magic), tc_int(acc[7][q], magic));
      out[q] += (hi << sh) + ((lo + (1ll << (31 - sh))) >> (32 - sh));  // to nearest: no bias
    }
  }
}

// A tile of the sorted samples, packed: its index i of the mode (bits 19..29),
// its first place in the block's order (bits 4..18), its rows - 1 (bits 0..3)
__device__ __forceinline__ int tc_tile_i(uint32_t t) { return (int)(t >> 19); }
__device__ __forceinline__ int tc_tile_at(uint32_t t) { return (int)(t >> 4) & 0x7fff; }
__device__ __forceinline__ int tc_tile_rows(uint32_t t) { return (int)(t & 15) + 1; }

// lane l's row of a tile (l mod 16; the last row again beyond the tile's rows)
struct TcRow {
  int32_t k;   // the sample
  int32_t ri;  // its row of the first stage's table
};

// Stage st of step sb: every warp takes tiles of up to 16 samples with one
// index i of mode m = pL + st, one after the other; neighbouring warps take
// neighbouring tiles, so that a CTA's warps mostly share G_m(i) in L1.  The
// first stage reads the prefix table's rows, later ones the previous stage's
// results; the last stage's results meet the suffix rows in FP64 and the
// squared residuals are added to the sum returned.  The next tile's samples
// are looked up before this tile's products, off their critical path.
__device__ __noinline__ double tc_stage(const InstDev &in, const int32_t *r, const TcPlan &p,
                                        int st, int sb, int gw, int NW) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int d = in.d, m = p.pL + st;
  const bool last = st == p.nst - 1;
  uint64_t *ws = reinterpret_cast<uint64_t *>(in.ews);
  const int K = (int)core_s(in, r, m), N = (int)core_s(in, r, m + 1);
  const int kp = (int)tc_up(K, 16), np = (int)tc_up(N, 8), kq = (int)tc_up(N, 16);
  // the words are below 2^62, so the sums stay below kp 2^36 2^88: sh keeps
  // them below 2^61 2^(88 - sh)
  int lg = 4;
  while ((1 << lg) < kp) ++lg;
  const int sh = 25 - lg;
  const int blk0 = sb * p.blocks;
  const int nblk = min(p.blocks, (int)((in.nsamples + TC_BLOCK - 1) / TC_BLOCK) - blk0);
  const int kbase = blk0 * TC_BLOCK;
  const int n = (int)in.n[m];
  const int32_t *ge = reinterpret_cast<const int32_t *>(ws + p.Ge[m]);
  const uint64_t *src = ws + (st == 0 ? p.L : p.C[(st - 1) & 1]);
  const int32_t *srce = reinterpret_cast<const int32_t *>(ws + (st == 0 ? p.Le : p.Ce[(st - 1) & 1]));
  uint64_t *dst = ws + p.C[st & 1];
  int32_t *dste = reinterpret_cast<int32_t *>(ws + p.Ce[st & 1]);
  const int ntb = TC_BLOCK / 16 + n;  // tile slots of a block
  const uint32_t *tiles = in.tc_tile[m] + (int64_t)blk0 * ntb;
  const uint16_t *perm = in.tc_perm + (int64_t)(m - 1) * in.tc_stride + kbase;
  const int items = nblk * ntb;
  auto row_of = [&](uint32_t tl, int x) {
    TcRow o{0, 0};
    if (tl != TC_NO_TILE) {
      const int b = x / ntb;
      o.k = kbase + b * TC_BLOCK +
            perm[b * TC_BLOCK + tc_tile_at(tl) + min(lane & 15, tc_tile_rows(tl) - 1)];
      if (st == 0) {
        int s = 1;
        for (int mm = 0; mm < p.pL; ++mm) {
          o.ri += sample_coord(in, o.k, mm) * s;
          s *= (int)in.n[mm];
        }
      } else {
        o.ri = o.k - kbase;
      }
    }
    return o;
  };
  double part = 0.0;
  uint32_t nt = gw < items ? tiles[gw] : TC_NO_TILE;
  TcRow nr = row_of(nt, gw);
  for (int x = gw; x < items; x += NW) {
    const uint32_t tl = nt;
    const TcRow row = nr;
    nt = x + NW < items ? tiles[x + NW] : TC_NO_TILE;
    nr = row_of(nt, x + NW);
    if (tl == TC_NO_TILE) continue;
    const int i = tc_tile_i(tl), rows = tc_tile_rows(tl);
    const uint64_t *Gi = ws + p.G[m] + (int64_t)i * np * kp + g * kp + 2 * t;
    const int32_t *gei = ge + i * np + 2 * t;
    const int rg = __shfl_sync(FULL, row.ri, g), rh = __shfl_sync(FULL, row.ri, g + 8);
    const uint64_t *a0 = src + (int64_t)rg * kp + 2 * t, *a1 = src + (int64_t)rh * kp + 2 * t;
    const int32_t e0 = srce[rg], e1 = srce[rh];
    if (!last) {
      const int kg = __shfl_sync(FULL, row.k, g) - kbase, kh = __shfl_sync(FULL, row.k, g + 8) - kbase;
      uint64_t *o0 = dst + (int64_t)kg * kq + 2 * t, *o1 = dst + (int64_t)kh * kq + 2 * t;
      // the raw results, and the highest bit of each row in units of 2^-exponent
      int top0 = INT_MIN, top1 = INT_MIN;
      bool bad = false;
      for (int c = 0; c < np; c += 8) {
        int64_t out[4];
        tc_product(a0, a1, Gi + c * kp, kp, sh, out);
        const int32_t ea = gei[c], eb = gei[c + 1];
        bad |= ea == TC_BAD || eb == TC_BAD;
        if (out[0]) top0 = max(top0, ea + 64 - __clzll(llabs(out[0])));
        if (out[1]) top0 = max(top0, eb + 64 - __clzll(llabs(out[1])));
        if (out[2]) top1 = max(top1, ea + 64 - __clzll(llabs(out[2])));
        if (out[3]) top1 = max(top1, eb + 64 - __clzll(llabs(out[3])));
        if (g < rows) *reinterpret_cast<longlong2 *>(o0 + c) = make_longlong2(out[0], out[1]);
        if (g + 8 < rows) *reinterpret_cast<longlong2 *>(o1 + c) = make_longlong2(out[2], out[3]);
      }
      for (int o = 1; o < 4; o <<= 1) {
        top0 = max(top0, __shfl_xor_sync(FULL, top0, o));
        top1 = max(top1, __shfl_xor_sync(FULL, top1, o));
      }
      bad = __any_sync(FULL, bad);
      // rescale to 62 bits below the row's largest (each lane its own words)
      for (int c = 0; c < kq; c += 8) {
        const bool in_np = c < np;
        const int32_t ea = in_np ? gei[c] : 0, eb = in_np ? gei[c + 1] : 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (g + 8 * h >= rows) continue;
          longlong2 *o = reinterpret_cast<longlong2 *>((h ? o1 : o0) + c);
          const int top = h ? top1 : top0;
          // (a row of zeros: top is INT_MIN and nothing is shifted)
          const bool nz = in_np && top != INT_MIN;
          const longlong2 v = nz ? *o : make_longlong2(0, 0);
          const int s0 = nz ? 62 - (top - ea) : 0, s1 = nz ? 62 - (top - eb) : 0;
          *reinterpret_cast<uint4 *>(o) = tc_pack((uint64_t)tc_shift(v.x, s0) + TC_BIAS,
                                                  (uint64_t)tc_shift(v.y, s1) + TC_BIAS);
        }
      }
      if (t == 0) {
        if (g < rows)
          dste[kg] = bad || e0 == TC_BAD ? TC_BAD : top0 == INT_MIN ? 0 : e0 + 88 - sh + top0 - 62;
        if (g + 8 < rows)
          dste[kh] = bad || e1 == TC_BAD ? TC_BAD : top1 == INT_MIN ? 0 : e1 + 88 - sh + top1 - 62;
      }
    } else {
      // the suffix rows: lane l < 16 finds row l's (as an offset)
      const double *Y = p.pR >= 2 ? in.ews + p.R : in.bond[d - 2].R;
      const int64_t sy = p.pR >= 2 ? 1 : in.bond[d - 2].ldR;
      int e = 0, s = 1;
      for (int mm = d - p.pR; mm < d; ++mm) {
        e += sample_coord(in, row.k, mm) * s;
        s *= (int)in.n[mm];
      }
      const double *yg = Y + (int64_t)__shfl_sync(FULL, e, g) * (p.pR >= 2 ? N : 1);
      const double *yh = Y + (int64_t)__shfl_sync(FULL, e, g + 8) * (p.pR >= 2 ? N : 1);
      double v0 = 0.0, v1 = 0.0;
      bool bad = e0 == TC_BAD || e1 == TC_BAD;
      for (int c = 0; c < np; c += 8) {
        int64_t out[4];
        tc_product(a0, a1, Gi + c * kp, kp, sh, out);
        const int u = c + 2 * t;
        const int32_t ea = gei[c], eb = gei[c + 1];
        bad |= ea == TC_BAD || eb == TC_BAD;
        const double q0a = u < N ? yg[u * sy] : 0.0, q0b = u + 1 < N ? yg[(u + 1) * sy] : 0.0;
        const double q1a = u < N ? yh[u * sy] : 0.0, q1b = u + 1 < N ? yh[(u + 1) * sy] : 0.0;
        v0 = __fma_rn(tc_real(out[0], e0 + ea + 88 - sh), q0a, v0);
        v0 = __fma_rn(tc_real(out[1], e0 + eb + 88 - sh), q0b, v0);
        v1 = __fma_rn(tc_real(out[2], e1 + ea + 88 - sh), q1a, v1);
        v1 = __fma_rn(tc_real(out[3], e1 + eb + 88 - sh), q1b, v1);
      }
      bad = __any_sync(FULL, bad);
      for (int o = 1; o < 4; o <<= 1) {
        v0 = __dadd_rn(v0, __shfl_xor_sync(FULL, v0, o));
        v1 = __dadd_rn(v1, __shfl_xor_sync(FULL, v1, o));
      }
      // lane t = 0 closes row g, lane t = 1 row g + 8
      const int kk = __shfl_sync(FULL, row.k, g + 8 * (t & 1));
      if (t < 2 && g + 8 * t < rows) {
        const double e2 = bad ? __longlong_as_double(0x7FF8000000000000ll)
                              : __dsub_rn(in.xs[kk], t ? v1 : v0);
        part = __fma_rn(e2, e2, part);
      }
    }
  }
  return part;
}

// The last mode of a table (side 0: prefix, 1: suffix) from the rows before it:
// row e times G_m(i) for every row and index, a warp per 16 rows of one index,
// the results as doubles in the table's layout.
__device__ __noinline__ void tc_extend(const InstDev &in, const int32_t *r, const TcPlan &p,
                                       int side, int gw, int NW) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int d = in.d, m = side ? d - p.pR : p.pL - 1;
  uint64_t *ws = reinterpret_cast<uint64_t *>(in.ews);
  const int K = (int)core_s(in, r, side ? m + 1 : m), N = (int)core_s(in, r, side ? m : m + 1);
  const int kp = (int)tc_up(K, 16), np = (int)tc_up(N, 8);
  int lg = 4;
  while ((1 << lg) < kp) ++lg;
  const int sh = 25 - lg;
  const int n = (int)in.n[m];
  int64_t rows = 1;
  for (int q = 1; q < (side ? p.pR : p.pL); ++q) rows *= in.n[side ? d - q : q - 1];
  const uint64_t *src = ws + (side ? p.R : p.L);
  const int32_t *srce = reinterpret_cast<const int32_t *>(ws + (side ? p.Re : p.Le));
  const int32_t *ge = reinterpret_cast<const int32_t *>(ws + p.Ge[m]);
  double *dst = side ? in.tabR : in.tabL;
  const int64_t nt = (rows + 15) / 16;
  for (int64_t x = gw; x < nt * n; x += NW) {
    const int i = (int)(x / nt);
    const int64_t q = (x - i * nt) * 16;
    const int64_t rg = min(q + g, rows - 1), rh = min(q + g + 8, rows - 1);
    const uint64_t *a0 = src + rg * kp + 2 * t, *a1 = src + rh * kp + 2 * t;
    const uint64_t *Gi = ws + p.G[m] + (int64_t)i * np * kp + g * kp + 2 * t;
    const int32_t *gei = ge + i * np + 2 * t;
    const int32_t e0 = srce[rg], e1 = srce[rh];
    double *o0 = dst + (side ? i + n * rg : rg + rows * i) * N + 2 * t;
    double *o1 = dst + (side ? i + n * rh : rh + rows * i) * N + 2 * t;
    for (int c = 0; c < np; c += 8) {
      int64_t out[4];
      tc_product(a0, a1, Gi + c * kp, kp, sh, out);
      const int32_t ea = gei[c], eb = gei[c + 1];
      const double nan = __longlong_as_double(0x7FF8000000000000ll);
      const bool ba = ea == TC_BAD, bb = eb == TC_BAD, b0 = e0 == TC_BAD, b1 = e1 == TC_BAD;
      const bool ua = c + 2 * t < N, ub = c + 2 * t + 1 < N;
      if (ua && q + g < rows) o0[c] = ba || b0 ? nan : tc_real(out[0], e0 + ea + 88 - sh);
      if (ub && q + g < rows) o0[c + 1] = bb || b0 ? nan : tc_real(out[1], e0 + eb + 88 - sh);
      if (ua && q + g + 8 < rows) o1[c] = ba || b1 ? nan : tc_real(out[2], e1 + ea + 88 - sh);
      if (ub && q + g + 8 < rows) o1[c + 1] = bb || b1 ? nan : tc_real(out[3], e1 + eb + 88 - sh);
    }
  }
}

}  // namespace ttc

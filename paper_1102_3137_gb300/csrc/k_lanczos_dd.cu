// Lanczos step of the mixed form (Sec. 2.1 recurrence in the bilinear form,
// CGS2 re-orthogonalisation, Eq. 9 assembly) with its dot products and
// basis updates in double-float arithmetic on the FP32 pipe.
//
// The basis Q is stored as double-floats (cdfl: hi + lo binary32 per real
// part, 47 significant bits, 16 bytes per complex entry like binary64), so the
// passes over it read the split form directly; the X-matvec output u, the
// running diagonal and every scalar of T stay in binary64.  What moves off the
// binary64 pipe (GB300 issues binary32 FMAs at ~64x its binary64 rate) is the
// arithmetic of the passes over Q: products accumulated with
// TwoProduct/TwoSum (~2^-47 relative per operation); u is split by integer
// operations where it is read.
//
// Classical Gram-Schmidt twice, with the three-term part folded in and the
// second pass's coefficients taken from the Gram matrix of the stored basis:
//   pass A:  g  = Q_j^T u                     (alpha_j = g_j)
//            M's column j: Q_j^T q_j
//            h  = g - M g,  M = Q_j^T Q_j     (M kept per frequency, binary64)
//   pass B:  r  = u - Q_j (g + h)             (formed in binary64, stored split)
// In exact arithmetic h = Q_j^T (u - Q_j g) is the second pass's coefficient
// vector, so r is the classical Gram-Schmidt residual orthogonalised twice;
// reading Q_j^T Q_j from M instead of re-projecting u - Q_j g saves a sweep
// over the basis: two reads of Q per step, the new column of M coming from the
// entries that pass A has in registers anyway.  With the unit diagonal of M
// exact, M - I holds the basis's measured loss of orthogonality, which h
// removes to second order (one-reduce CGS2 in the Gram-matrix form); the
// remaining error is the rounding of g, ~2^-47 ||u|| / |beta_{j+1}|.
//
// What bounds it: the double-float multiply-accumulates (48 instructions per
// complex one, three per basis entry) and the reads of Q (32 bytes per entry)
// cost about the same, so neither may be spent on anything else.  Thread
// layout: a thread has its own sites in both passes.  Pass A takes BV = 4
// vectors at a time over T sites of every lane, the sums g and M in registers,
// then folds the eight sums of the 32 lanes by a halving butterfly (nine
// complex adds a lane instead of forty) into the warp's own row of shared
// memory; no barrier until all vectors are done.  u and q_j of the T sites are
// read again for each four vectors, from L1 (the basis itself bypasses it).
// Pass B sums a site's basis entries in its thread.  Per-CTA sums are added
// over the cluster in a fixed order in binary64, so every CTA of a frequency
// holds bit-identical coefficients.  Rank caps up to 64; larger caps take the
// binary64 kernel.  The running sums are double-floats updated by TwoProduct
// and TwoSum without renormalising the low word.
// Measured (average of the 16 steps at k = 16, cold L2): 256^2 x 16 frequencies
// 0.77 -> 0.22 ms, 512^2 x 16 2.85 -> 0.79 ms, 101^2 x 21 0.16 -> 0.11 ms, against a
// kernel that gave each warp whole vectors (its index work and barriers were most of
// its instructions; 1.6x the instructions and half the SMs idle at 256^2).
#include "solve_device.cuh"

namespace {

constexpr int LDD_MAX = 64;              // largest j + 1 this kernel takes
constexpr int BV = 4;                    // basis vectors at a time in pass A (g and M sums: eight values)
constexpr int T = 8;                     // sites of a thread between two folds
// A strip is shared by 2 or 4 CTAs where each keeps this many sites: below, the folds
// and the wider cluster's barriers cost what the split saves (64^2 x 16 solve, strips of
// 1024: 5.7 ms unsplit, 5.9 in two, 6.1 in four; 101^2 x 63, 2525: 18.4 / 19.5 / 22.7);
// above, one CTA a strip leaves SMs idle (256^2 x 16, 8192: 0.31 ms a step, 0.22 in two).
constexpr int SPLIT_MIN = 2048;
constexpr int MAX_RANKS = 16;            // CTAs of a cluster
// The Lanczos thresholds scaled to double-float arithmetic: the same multiples of the
// unit roundoff as TERM_TOL and BRK_TOL are of binary64's (2^-47 / 2^-53 = 64).
constexpr double TERM_TOL_DD = 64.0 * TERM_TOL;
constexpr double BRK_TOL_DD = 64.0 * BRK_TOL;
// A step re-projects r when ||r|| < REORTH_ETA ||u||: the Gram form's orthogonality is
// ~2^-47 ||u|| / ||r||, held below ~1.5e-13 this way.
constexpr double REORTH_ETA = 0.05;

__device__ __forceinline__ cdfl czero() { return {dfl(0.f, 0.f), dfl(0.f, 0.f)}; }

__device__ __forceinline__ void cmac(cdfl& acc, const cdfl& a, const cdfl& b) {
  dfl_mac(acc.x, a.x, b.x);
  dfl_mac(acc.x, dfl(-a.y.hi, -a.y.lo), b.y);
  dfl_mac(acc.y, a.x, b.y);
  dfl_mac(acc.y, a.y, b.x);
}
// renormalised sum / difference of two double-floats
__device__ __forceinline__ cdfl cadd(const cdfl& a, const cdfl& b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ cdfl csub(const cdfl& a, const cdfl& b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ cdfl cnorm(const cdfl& a) { return {dfl_fast(a.x.hi, a.x.lo), dfl_fast(a.y.hi, a.y.lo)}; }

struct LanDDSmem {
  cdfl wred[DY_WARPS][2 * LDD_MAX];      // per warp: Q^T u, then Q^T v, of its sites
  cxd vpart[2 * LDD_MAX];                // this CTA's sums (read by its peers)
  cxd vres[2 * LDD_MAX];                 // the cluster totals
  cdfl coef[LDD_MAX];                    // g + h, double-float
};

// v[0..7] summed over the warp; lane 4 i holds the sum of v[i] on return.  The first
// three steps halve the values as they add (a lane keeps the half its bit selects).
__device__ __forceinline__ cdfl warp_fold8(cdfl (&v)[8]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = cnorm(v[i]);
#pragma unroll
  for (int h = 4, off = 16; h > 0; h >>= 1, off >>= 1) {
    const bool up = lane & off;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (i >= h) break;
      const cdfl give = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
      v[i] = {keep.x + shfl_xor_any(give.x, off), keep.y + shfl_xor_any(give.y, off)};
    }
  }
#pragma unroll
  for (int off = 2; off > 0; off >>= 1)
    v[0] = {v[0].x + shfl_xor_any(v[0].x, off), v[0].y + shfl_xor_any(v[0].y, off)};
  return v[0];
}

// The basis is read once per pass: past L1, which keeps u and q_j.
__device__ __forceinline__ cdfl ld_basis(const cdfl* p) {
  const float4 v = __ldcg(reinterpret_cast<const float4*>(p));
  return {dfl(v.x, v.y), dfl(v.z, v.w)};
}

// Totals over the cluster's CTAs of this CTA's sites e in [e0, e1) of Q_l^T u and
// Q_l^T v, l <= j (v a double-float vector): sm.vres[l] and sm.vres[LDD_MAX + l].
__device__ __noinline__ void basis_dots(cg::cluster_group& cl, LanDDSmem& sm, const Geo& g, int i, int P, int e0,
                                        int e1, const cdfl* Q, const cxd* u, const cdfl* v, int j) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nsub = g.Lx * g.W;
  const size_t Ndd = g.Ndd;
  cdfl* row = sm.wred[w];
  for (int l = lane; l < 2 * LDD_MAX; l += 32) row[l] = czero();
  __syncwarp();
  // a warp's sites: 32 consecutive ones every DY_THREADS
  for (int eb = e0 + 32 * w; eb < e1; eb += DY_THREADS * T) {
    for (int lb = 0; lb <= j; lb += BV) {
      cdfl a[2 * BV];
#pragma unroll
      for (int m = 0; m < 2 * BV; ++m) a[m] = czero();
      const cdfl* Qb = Q + (size_t)lb * Ndd;
      for (int t = 0; t < T; ++t) {
        const int e = eb + t * DY_THREADS + lane;
        if (e >= e1) break;
        const size_t k = own_idx(g, i, e, nsub);
        cdfl qv[BV];
#pragma unroll
        for (int m = 0; m < BV; ++m) qv[m] = lb + m <= j ? ld_basis(Qb + (size_t)m * Ndd + k) : czero();
        const cdfl ud = csplit(u[k]), vd = v[k];
#pragma unroll
        for (int m = 0; m < BV; ++m)
          if (lb + m <= j) {
            cmac(a[m], qv[m], ud);
            cmac(a[BV + m], qv[m], vd);
          }
      }
      __syncwarp();
      const cdfl s = warp_fold8(a);
      if ((lane & 3) == 0) {
        const int m = lane >> 2, l = lb + (m & (BV - 1)) + (m / BV) * LDD_MAX;
        row[l] = cadd(row[l], s);
      }
    }
  }
  __syncthreads();
  // two threads a value, each half the warps, then half the cluster's CTAs
  const int x = tid >> 1, hf = tid & 1;
  const bool act = (x & (LDD_MAX - 1)) <= j;
  {
    cxd s = {0, 0};
#pragma unroll
    for (int k = 0; k < DY_WARPS / 2; ++k) s = s + cwiden(sm.wred[2 * k + hf][x]);
    s = {s.x + __shfl_xor_sync(0xffffffffu, s.x, 1), s.y + __shfl_xor_sync(0xffffffffu, s.y, 1)};
    if (hf == 0) sm.vpart[x] = s;
  }
  cl.sync();
  cxd rv[MAX_RANKS / 2];
#pragma unroll
  for (int k = 0; k < MAX_RANKS / 2; ++k) {
    const int r = 2 * k + hf;
    rv[k] = cxd{0, 0};
    if (act && r < P) rv[k] = cl.map_shared_rank(sm.vpart, r)[x];
  }
  cxd s = {0, 0};
#pragma unroll
  for (int k = 0; k < MAX_RANKS / 2; ++k) s = s + rv[k];
  s = {s.x + __shfl_xor_sync(0xffffffffu, s.x, 1), s.y + __shfl_xor_sync(0xffffffffu, s.y, 1)};
  if (hf == 0) sm.vres[x] = s;
  __syncthreads();
}
static_assert(DY_THREADS == 4 * LDD_MAX && DY_WARPS % 2 == 0 && BV == 4, "basis_dots' sums");

// sum over l < n of Q_l[k] c_l (double-float): the entries of eight vectors are
// loaded before any is used (eight loads in flight per thread), then summed in two
// interleaved chains
__device__ __forceinline__ cdfl basis_sum(const cdfl* Q, size_t Ndd, size_t k, int n, const cdfl* coef) {
  cdfl s0 = czero(), s1 = czero();
  for (int lb = 0; lb < n; lb += 8) {
    cdfl qv[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) qv[m] = lb + m < n ? ld_basis(Q + (size_t)(lb + m) * Ndd + k) : czero();
#pragma unroll
    for (int m = 0; m < 8; m += 2) {
      if (lb + m < n) cmac(s0, qv[m], coef[lb + m]);
      if (lb + m + 1 < n) cmac(s1, qv[m + 1], coef[lb + m + 1]);
    }
  }
  return cadd(cnorm(s0), cnorm(s1));
}

// Three CTAs an SM: with two, 14 clusters of 16 fit the chip and the 16 of a 512^2 group
// ran in two waves (1.02 ms a step, 0.79 with three; 256^2 0.29 and 0.22).
__global__ void __launch_bounds__(DY_THREADS, 3) k_lanczos_dd(Geo g, Bufs b, int j) {
  cg::cluster_group cl = cg::this_cluster();
  __shared__ RedSmem rs;
  __shared__ LanDDSmem sm;
  // a strip's entries in `split` runs of whole 32s, one a CTA
  const int P = gridDim.x, split = P / g.p;
  const int i = blockIdx.x / split, part = blockIdx.x - i * split, kf = blockIdx.y;
  const int tid = threadIdx.x;
  int* stt = b.st + (size_t)kf * ST_N;
  if (stt[ST_DONE]) return;
  int phase = 0;
  const size_t Ndd = g.Ndd;
  const int nsub = g.Lx * g.W, n = own_count(g, i);
  const int n32 = (n + 31) / 32;
  const int e0 = n32 * part / split * 32, e1 = min(n, n32 * (part + 1) / split * 32);
  // the basis is stored as double-floats (Geo::qsplit)
  cdfl* Q = reinterpret_cast<cdfl*>(b.Q + (size_t)kf * (g.k_max + g.nb) * Ndd);
  const cdfl* qj = Q + (size_t)j * Ndd;
  const cdfl* qm = (j > 0) ? Q + (size_t)(j - 1) * Ndd : nullptr;
  cdfl* r = Q + (size_t)(j + 1) * Ndd;
  const cxd* u = b.u + (size_t)kf * Ndd;
  cxd* acc = b.acc + (size_t)kf * Ndd;
  cxd* lan = b.lan + (size_t)kf * (g.k_max + g.nb) * 2;
  const int K1 = g.k_max + 1;
  cxd* gram = b.gram + (size_t)kf * K1 * K1;
  const cxd beta_j = (j > 0) ? lan[2 * j + 1] : cxd{0, 0};
  // read before the first cluster barrier: CTA 0 updates it once all CTAs passed the last one
  const double maxT_prev = b.maxT[kf];

  // ---- pass A: g = Q^T u, M's column j = Q^T q_j
  basis_dots(cl, sm, g, i, P, e0, e1, Q, u, qj, j);
  const cxd* gv = sm.vres;
  const cxd* mj = sm.vres + LDD_MAX;
  const cxd alpha = gv[j];
  // ---- second Gram-Schmidt coefficients from the Gram matrix M = Q_j^T Q_j of the
  // stored basis: h = Q_j^T (u - Q_j g) = g - M g, so g + h = g - (M - I) g (the unit
  // diagonal of M taken as exact; binary64); four threads a row
  {
    const int l = tid >> 2;
    cxd s = {0, 0};
    if (l <= j)
      for (int m = tid & 3; m <= j; m += 4) {
        if (m == l) continue;
        const int lo = min(l, m), hi = max(l, m);
        s = cfma(hi == j ? mj[lo] : gram[(size_t)hi * K1 + lo], gv[m], s);
      }
#pragma unroll
    for (int off = 1; off < 4; off <<= 1)
      s = {s.x + __shfl_xor_sync(0xffffffffu, s.x, off), s.y + __shfl_xor_sync(0xffffffffu, s.y, off)};
    if (l <= j && (tid & 3) == 0) sm.coef[l] = csplit(gv[l] - s);
  }
  if (blockIdx.x == 0 && tid < j) gram[(size_t)j * K1 + tid] = mj[tid];
  __syncthreads();

  // ---- pass B: r = u - Q (g + h) per site, finished in binary64 and stored split,
  // with r^T r, ||r||^2 and the Eq. 9 three-vector update
  cxd v2[3] = {{0, 0}, {0, 0}, {0, 0}};   // r^T r, ||r||^2, ||u||^2
  {
    const cdfl ad = csplit(alpha), bd = csplit(2.0 * beta_j);
    for (int e = e0 + tid; e < e1; e += DY_THREADS) {
      const size_t k = own_idx(g, i, e, nsub);
      const cxd uv = u[k], av = acc[k];
      const cdfl qjd = qj[k], qmd = qm ? ld_basis(qm + k) : czero();
      cdfl tot = basis_sum(Q, Ndd, k, j - 1, sm.coef), last = czero();
      cmac(last, qjd, sm.coef[j]);
      if (qm) cmac(last, qmd, sm.coef[j - 1]);
      tot = cadd(tot, cnorm(last));
      const cxd rv = {(uv.x - f2d_bits(tot.x.hi)) - f2d_bits(tot.x.lo),
                      (uv.y - f2d_bits(tot.y.hi)) - f2d_bits(tot.y.lo)};
      r[k] = csplit(rv);
      v2[0] = cfma(rv, rv, v2[0]);
      v2[1].x += cabs2(rv);
      v2[2].x += cabs2(uv);
      cdfl sq = czero(), d = czero();
      cmac(sq, qjd, qjd);
      cmac(d, ad, cnorm(sq));
      if (qm) {
        cdfl pr = czero();
        cmac(pr, qmd, qjd);
        cmac(d, bd, cnorm(pr));
      }
      d = cnorm(d);
      acc[k] = cxd{(av.x + f2d_bits(d.x.hi)) + f2d_bits(d.x.lo), (av.y + f2d_bits(d.y.hi)) + f2d_bits(d.y.lo)};
    }
  }
  cluster_sum<3>(cl, rs, phase, P, v2);
  cxd rr = v2[0];
  double rn2 = v2[1].x;
  // ---- pass C, only when r lost most of u (||r|| < REORTH_ETA ||u||, near an
  // invariant subspace): the Gram form leaves r's rounding error ~2^-47 ||u|| in
  // place, so project r once more onto the complement, r -= Q (Q^T r), as the
  // classical second pass would (the selective test of Daniel, Gragg, Kaufman and
  // Stewart, 1976)
  if (rn2 < REORTH_ETA * REORTH_ETA * v2[2].x) {
    basis_dots(cl, sm, g, i, P, e0, e1, Q, u, r, j);
    if (tid <= j) sm.coef[tid] = csplit(mj[tid]);
    __syncthreads();
    cxd w2[2] = {{0, 0}, {0, 0}};
    for (int e = e0 + tid; e < e1; e += DY_THREADS) {
      const size_t k = own_idx(g, i, e, nsub);
      const cdfl rn = csub(r[k], basis_sum(Q, Ndd, k, j + 1, sm.coef));
      r[k] = rn;
      const cxd rv = cwiden(rn);
      w2[0] = cfma(rv, rv, w2[0]);
      w2[1].x += cabs2(rv);
    }
    cluster_sum<2>(cl, rs, phase, P, w2);
    rr = w2[0];
    rn2 = w2[1].x;
  }
  const cxd beta = csqrt_principal(rr);
  const double maxT = fmax(maxT_prev, sqrt(cabs2(alpha)));
  const double babs = sqrt(cabs2(beta));
  int done = 0, flag = 0;
  if (j == g.k_max - 1) {
    done = 1;
  } else if (sqrt(rn2) <= TERM_TOL_DD * maxT) {         // r vanished: invariant subspace
    done = 1;
    flag = 1;
  } else if (sqrt(cabs2(rr)) <= BRK_TOL_DD * rn2) {     // r != 0, (r, r)_C ~ 0: breakdown
    done = 1;
    flag = 2;
  }
  if (!done) {
    // q_{j+1} = r / beta in double-float
    const cdfl ib = csplit(cinv(beta));
    for (int e = e0 + tid; e < e1; e += DY_THREADS) {
      const size_t k = own_idx(g, i, e, nsub);
      cdfl q = czero();
      cmac(q, r[k], ib);
      r[k] = cnorm(q);
    }
  }
  if (blockIdx.x == 0 && tid == 0) {
    lan[2 * j] = alpha;
    stt[ST_STEPS] = j + 1;
    if (done) {
      stt[ST_DONE] = 1;
      stt[ST_STATUS] |= flag;
    } else {
      lan[2 * (j + 1) + 1] = beta;
      b.maxT[kf] = fmax(maxT, babs);
    }
  }
  cl.sync();          // no CTA exits while a peer may still read its shared memory
}

}  // namespace

// The mixed form's Lanczos step (rank caps up to 64; the binary64 kernel otherwise).
cudaError_t launch_lanczos_dd(const Geo& g, const Bufs& b, int K, int j, cudaStream_t st) {
  if (g.k_max > LDD_MAX || g.nb != 1 || g.p > MAX_RANKS) return cudaErrorInvalidValue;
  int split = 1;
  while (2 * split * g.p <= MAX_RANKS && g.Lx * g.W / (2 * split) >= SPLIT_MIN) split *= 2;
  return launch_cluster(k_lanczos_dd, dim3(split * g.p, K), split * g.p, 0, st, g, b, j);
}

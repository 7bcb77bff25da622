// Lanczos-based low-rank correction: device code shared by the per-step
// kernels (included by k_solve.cu and the two k_xmatvec_*.cu units).
//
// Every kernel here runs one thread-block cluster per frequency with one CTA
// per subdomain (cluster = p CTAs, grid = p x K).  CTA i owns subdomain i's
// slice block of every DD-layout vector and interface layer i (i < p-1).
// Reductions over a frequency's lattice are two-level: a fixed-order
// block reduction, then every CTA reads the p partials from distributed
// shared memory in rank order, so all CTAs of a cluster hold bit-identical
// scalars and take identical branch decisions (no CTA can leave a cluster
// barrier behind).  Every kernel that reads peers' shared memory ends with a
// cluster barrier, so no CTA exits while a peer may still be reading it.
//
// X-"matvec" (Sec. 2.3, Eqs. 6-8).  The paper defines u = v - w with
// H v = q and w = blkdiag(B^-1, 0) q.  Eliminating the subdomain unknowns
// of H v = q gives, without ever forming S = C - E^T B^-1 E (Eq. 4),
//     y   = S^-1 (E^T B^-1 q_B - q_C),
//     u_B = B^-1 E y,   u_C = -y,
// which is exactly v - w with no cancellation.  S y = r is solved by COCG
// (conjugate orthogonal CG: CG in the bilinear form, valid for complex
// symmetric S) whose S-products are subdomain solves with boundary-only
// right-hand sides.
#pragma once
#include <cooperative_groups.h>

#include "dyson.h"
#include "dyson_common.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr double TERM_TOL = 1e-12;    // ||r||_2 <= TERM_TOL * max|T|: invariant subspace
constexpr double BRK_TOL = 1e-14;     // |r^T r| <= BRK_TOL * ||r||^2: breakdown
constexpr int KMAX_SMEM = 256;        // largest Lanczos rank cap
// refinement stops early once a pass no longer shrinks the squared FP64
// residual 16-fold (the residual has reached its rounding floor)
constexpr double REFINE_STALL = 1.0 / 16.0;

__device__ __forceinline__ size_t own_idx(const Geo& g, int i, int e, int nsub) {
  return e < nsub ? (size_t)i * nsub + e : (size_t)g.ifc_off + (size_t)i * g.A + (e - nsub);
}
__device__ __forceinline__ int own_count(const Geo& g, int i) {
  return g.Lx * g.W + (i < g.p - 1 ? g.A : 0);
}

// ---------------------------------------------------------------- reductions
constexpr int RED_WARPS = 18;            // most warps of a CTA that reduces
struct RedSmem {
  cxd wred[RED_WARPS * 8];
  cxd slot[2 * 8];
  cxd res[8];
};

__device__ __forceinline__ cxd warp_sum(cxd v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, off);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, off);
  }
  return v;
}

// Sum NV complex partials over the whole cluster; every thread gets the totals.
template <int NV>
__device__ void cluster_sum(cg::cluster_group& cl, RedSmem& rs, int& phase, int p, cxd (&v)[NV]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = warp_sum(v[k]);
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) rs.wred[wid * 8 + k] = v[k];
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    cxd s = {0, 0};
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s = s + rs.wred[w * 8 + threadIdx.x];
    rs.slot[phase * 8 + threadIdx.x] = s;
  }
  cl.sync();
  if (threadIdx.x < NV) {
    cxd s = {0, 0};
    for (int r = 0; r < p; ++r) {
      const cxd* rem = cl.map_shared_rank(rs.slot, r);
      s = s + rem[phase * 8 + threadIdx.x];
    }
    rs.res[threadIdx.x] = s;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = rs.res[k];
  phase ^= 1;
}

// CTA-local sum (no cluster exchange)
template <int NV>
__device__ void block_sum(RedSmem& rs, cxd (&v)[NV]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = warp_sum(v[k]);
  __syncthreads();
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) rs.wred[wid * 8 + k] = v[k];
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    cxd s = {0, 0};
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s = s + rs.wred[w * 8 + threadIdx.x];
    rs.res[threadIdx.x] = s;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = rs.res[k];
  __syncthreads();
}

// ---------------------------------------------------------------- async copies
// g_s blocks stream from HBM into a ring of shared-memory slots with 1D bulk
// copies (cp.async.bulk, completion counted on an mbarrier per slot).  Every
// wait is bounded by the global timer: on time-out the kernel records
// DYSON_ST_WAIT_TIMEOUT and goes on (no CTA may leave its cluster's barriers);
// the thread then waits on the ring no more in that sweep, and no thread of the
// CTA waits in its later sweeps.
constexpr unsigned long long WAIT_LIMIT_NS = 2000000000ull;   // 2 s
constexpr int ST_WAIT_TIMEOUT = DYSON_ST_WAIT_TIMEOUT;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes) : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}" : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ bool mbar_wait_for(uint64_t* bar, uint32_t parity, unsigned long long limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  while (!mbar_try_wait(bar, parity))
    if (global_ns() - t0 > limit_ns) return false;
  return true;
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  return mbar_wait_for(bar, parity, WAIT_LIMIT_NS);
}
// A copy-ring wait that gives up for good: once one of this thread's waits has
// run out (dead, a register flag, seeded from the CTA's shared flag at the start
// of each sweep), its later waits return at once, so a lost copy costs the
// kernel one wait limit per thread and sweep instead of one per slice step.
__device__ __forceinline__ void ring_wait(uint64_t* bar, uint32_t parity, bool& dead, int* err) {
  if (dead) return;
  if (!mbar_wait(bar, parity)) {
    dead = true;
    *err = 1;
  }
}

// Per-CTA copy pipeline: S slots of one W x W block each, one mbarrier per slot.
struct Pipe {
  uint64_t* bar;   // [S] in static shared memory: a slot's copy has landed
  uint64_t* empty; // [S] a slot's block has been read (the wide form, one arrival per compute warp)
  void* ring;      // S slots in dynamic shared memory
  void* ybuf;      // forward intermediates in shared memory, or null (global scratch)
  int S;
  int CR;          // rows of a slice block per streamed chunk (= W unless W > 64)
  unsigned seq;    // blocks issued (= consumed) so far by this CTA
  int* err;        // shared flag: a bounded wait ran out
};

constexpr int MAX_STAGES = 8;
constexpr int WIDE_WARPS = 16;                    // compute warps of the wide sweep, one more issues the copies
constexpr int WIDE_THREADS = 32 * (WIDE_WARPS + 1);
template <int WF>
constexpr int solve_threads() { return WF == 0 ? WIDE_THREADS : DY_THREADS; }
// groups of compute threads of the wide sweep: W / V threads cover a block row
// 16 bytes each (V entries)
template <typename R>
__host__ __device__ inline int wide_groups(int W) { return 32 * WIDE_WARPS / (W * (int)sizeof(cx<R>) / 16); }
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ void pipe_init(Pipe& pp) {
  if (threadIdx.x == 0) {
    for (int k = 0; k < pp.S; ++k) {
      mbar_init(pp.bar + k, 1);
      mbar_init(pp.empty + k, WIDE_WARPS);
    }
    *pp.err = 0;
    fence_mbar_init();
  }
  __syncthreads();
}

// ---------------------------------------------------------------- block sweep
// Solve B_i x = rhs by block forward/back substitution with the stored
// left-connected inverses g_s (Eq. 7 and the S-products):
//   forward  y_s = g_s (rhs_s - t y_{s-1})
//   backward x_s = y_s - t g_s x_{s+1}
// The right-hand side is either a full DD block (src) or boundary-only,
// t times an interface-layer vector on the first/last slow rows (E y).
// The 2 Lx - 1 blocks the two passes read stream through the copy ring.
template <typename R>
struct SweepArgs {
  const cx<R>* g;      // [Lx][W][W] this subdomain's factors
  cx<R>* y;            // [Lx][W] scratch for the forward intermediates
  const cxd* src;      // full right-hand side (subdomain block) or null
  const cx<R>* lay_lo; // interface layer below (i-1), boundary mode
  const cx<R>* lay_hi; // interface layer above (i), boundary mode
  cxd* dst;            // full solution out (subdomain block) or null
  int dst_op;          // 0 store, 1 add, 2 subtract, 3 store negated
  double in_scale;     // src is multiplied by this when rounded to R
  double out_scale;    // x is multiplied by this when written to dst
  cx<R>* bnd_lo;       // solution on the lowest slow row, layer layout (or null)
  cx<R>* bnd_hi;       // solution on the highest slow row
};

// Thread layout of the block products y = g_s z (g_s complex symmetric, so its
// row r is also its column r and rows are read contiguously): warp w owns rows
// [w*RPW, (w+1)*RPW); inside the warp lane = rr*G + cg, row group rr, column
// class cg (columns cg, cg+G, ...: CPG of them); the G partial sums of a row
// are added with log2(G) butterfly shuffles and lane rr*G finishes the row.
struct SweepLayout {
  int RPW, G, CPG;
};
__host__ __device__ inline SweepLayout sweep_layout(int rows, int W) {
  int rpw = (rows + DY_WARPS - 1) / DY_WARPS, p2 = 1;
  while (p2 < rpw) p2 <<= 1;
  SweepLayout L;
  L.RPW = p2;
  L.G = 32 / p2;
  L.CPG = (W + L.G - 1) / L.G;
  return L;
}

// The sequential slice loop touches only shared memory (or the per-unit
// scratch) and R-precision registers: a parallel pre-pass converts the
// right-hand side into the row buffer yb (rhs_s in row s), the forward pass
// overwrites row s with y_s, the backward pass with x_s, and a parallel
// post-pass converts the rows to FP64 and writes the requested outputs.  On
// GB300 FP64 issue is ~1/64 of FP32, so keeping conversions out of the
// dependent chain matters as much as keeping global loads out of it.
template <typename R>
__device__ void sweep_chunked(const Geo& g, int i, const SweepArgs<R>& a, cx<R>* sm, Pipe& pp,
                              unsigned long long* cnt);

// Pre-pass of a sweep (all threads): the right-hand side rows in precision R
// into the row buffer yb [Lx][W] (zero on padding columns).
template <typename R>
__device__ __forceinline__ void sweep_prepass(const Geo& g, int i, const SweepArgs<R>& a, cx<R>* yb) {
  const int W = g.W, Lx = g.Lx, T = g.T, w = T * g.h[i], nrow = Lx * W;
  const R t = (R)g.t;
  for (int e = threadIdx.x; e < nrow; e += (int)blockDim.x) {
    const int s = e / W, j = e - s * W;
    cxd v = {0, 0};
    if (j < w) {
      if (a.src) {
        v = a.in_scale * a.src[e];
      } else {
        cx<R> u = {0, 0};
        if (a.lay_lo && j < T) u = u + t * a.lay_lo[s + Lx * j];
        if (a.lay_hi && j >= w - T) u = u + t * a.lay_hi[s + Lx * (j - (w - T))];
        yb[e] = u;
        continue;
      }
    }
    yb[e] = cconv<R>(v);
  }
}

// Post-pass of a sweep (all threads): the solution rows x_s in yb to the FP64
// outputs and the boundary-row copies.
template <typename R>
__device__ __forceinline__ void sweep_postpass(const Geo& g, int i, const SweepArgs<R>& a,
                                               const cx<R>* yb) {
  const int W = g.W, Lx = g.Lx, T = g.T, w = T * g.h[i], nrow = Lx * W;
  for (int e = threadIdx.x; e < nrow; e += (int)blockDim.x) {
    const int s = e / W, j = e - s * W;
    if (j >= w) continue;
    const cx<R> xr = yb[e];
    if (a.dst) {
      const cxd xd = a.out_scale * cconv<double>(xr);
      cxd* d = a.dst + e;
      if (a.dst_op == 0) *d = xd;
      else if (a.dst_op == 1) *d = *d + xd;
      else if (a.dst_op == 2) *d = *d - xd;
      else *d = -xd;
    }
    if (a.bnd_lo && j < T) a.bnd_lo[s + Lx * j] = xr;
    if (a.bnd_hi && j >= w - T) a.bnd_hi[s + Lx * (j - (w - T))] = xr;
  }
}

// WF selects the sweep form at compile time, so each kernel carries only its
// own: 0 = row-chunked (W > 64, either precision); otherwise the 8-warp form of
// the FP64 strips (W <= 64).  The mixed form's strips: xmatvec_mixed.cuh.
template <typename R, int WF>
__device__ void sweep(const Geo& g, int i, const SweepArgs<R>& a, cx<R>* sm, Pipe& pp,
                      unsigned long long* cnt) {
  if constexpr (WF == 0) {
    sweep_chunked<R>(g, i, a, sm, pp, cnt);
    return;
  }
  bool dead = *pp.err != 0;              // an earlier wait of this CTA ran out
  const int W = g.W, Lx = g.Lx;
  const SweepLayout L = sweep_layout(W, W);
  cx<R>* zbuf = sm;                      // [2][W]: z of the current and of the next slice
  cx<R>* ring = reinterpret_cast<cx<R>*>(pp.ring);
  cx<R>* yb = pp.ybuf ? reinterpret_cast<cx<R>*>(pp.ybuf) : a.y;   // [Lx][W] row buffer
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int rr = lane / L.G, cg = lane - rr * L.G;
  const int row = wid * L.RPW + rr;      // the row this lane works on
  const bool rvalid = row < W;
  const bool owner = rvalid && cg == 0;  // finishes the row
  // rows of one warp are W entries apart, i.e. in the same banks; starting each
  // row group at a different multiple of G spreads a warp's accesses over all banks
  const int rot = (W % L.G == 0) ? (rr * L.G) % W : 0;
  const R t = (R)g.t;
  const int WW = W * W;
  const uint32_t bytes = (uint32_t)(WW * sizeof(cx<R>));
  const int NL = 2 * Lx - 1;
  const int S = pp.S;
  auto slice_of = [&](int n) { return n < Lx ? n : 2 * Lx - 2 - n; };
  auto issue = [&](int n) {
    const unsigned q = pp.seq + n;
    const int slot = (int)(q % S);
    bulk_load(ring + (size_t)slot * WW, a.g + (size_t)slice_of(n) * WW, bytes, pp.bar + slot);
  };

  __syncthreads();                       // previous users of ring, zbuf and yb are done
  if (tid == 0) {
    fence_proxy_async();
    for (int n = 0; n < S && n < NL; ++n) issue(n);
  }
  sweep_prepass<R>(g, i, a, yb);
  __syncthreads();
  if (owner) zbuf[row] = yb[row];
  // Rows are read two slices ahead into ping-pong registers: with yb in shared
  // memory this costs nothing, with the global scratch it hides the latency.
  cx<R> fA = {0, 0}, fB = {0, 0};
  if (owner) {
    if (Lx > 1) fA = yb[W + row];
    if (Lx > 2) fB = yb[2 * W + row];
  }
  __syncthreads();

  // one slice of either pass: wait for g_s, row products, butterfly
  auto product = [&](int n) -> cx<R> {
    const unsigned q = pp.seq + n;
    const int slot = (int)(q % S);
    ring_wait(pp.bar + slot, (q / S) & 1u, dead, pp.err);
    const cx<R>* grow = ring + (size_t)slot * WW + (size_t)row * W;
    const cx<R>* zc = zbuf + (n & 1) * W;
    cx<R> acc = {0, 0};
    if (rvalid) {
#pragma unroll 4
      for (int k = 0; k < L.CPG; ++k) {
        const int base = cg + L.G * k;   // columns interleaved over the group's lanes
        if (base < W) {
          int col = base + rot;          // rotated per row group: no bank conflicts
          if (col >= W) col -= W;
          acc = cfma(grow[col], zc[col], acc);
        }
      }
    }
    for (int off = L.G >> 1; off > 0; off >>= 1) {
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, off);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, off);
    }
    return acc;
  };
  auto finish = [&](int n) {
    __syncthreads();                     // slot n and z of slice n fully read; z of n+1 written
    if (tid == 0 && n + S < NL) {
      fence_proxy_async();
      issue(n + S);
    }
  };
  // forward: y_s = g_s (rhs_s - t y_{s-1}); row s of yb becomes y_s
  auto fwd = [&](int s, cx<R>& f) {
    const cx<R> m = product(s);
    if (owner) {
      cx<R>* zn = zbuf + ((s + 1) & 1) * W;
      yb[(size_t)s * W + row] = m;
      zn[row] = (s + 1 < Lx) ? f - t * m : m;   // x_{Lx-1} = y_{Lx-1}
      if (s + 3 < Lx) f = yb[(size_t)(s + 3) * W + row];
    }
    finish(s);
  };
  for (int s = 0; s < Lx; s += 2) {
    fwd(s, fA);
    if (s + 1 < Lx) fwd(s + 1, fB);
  }
  // backward: x_s = y_s - t g_s x_{s+1}; row s of yb becomes x_s
  cx<R> yA = {0, 0}, yB = {0, 0};
  if (owner && Lx > 1) {
    yA = yb[(size_t)(Lx - 2) * W + row];
    if (Lx > 2) yB = yb[(size_t)(Lx - 3) * W + row];
  }
  auto bwd = [&](int s, cx<R>& yv) {
    const int n = 2 * Lx - 2 - s;
    const cx<R> m = product(n);
    if (owner) {
      cx<R>* zn = zbuf + ((n + 1) & 1) * W;
      const cx<R> xv = yv - t * m;
      yb[(size_t)s * W + row] = xv;
      zn[row] = xv;
      if (s >= 2) yv = yb[(size_t)(s - 2) * W + row];
    }
    finish(n);
  };
  for (int s = Lx - 2; s >= 0; s -= 2) {
    bwd(s, yA);
    if (s - 1 >= 0) bwd(s - 1, yB);
  }
  sweep_postpass<R>(g, i, a, yb);
  pp.seq += NL;
  if (tid == 0 && cnt) *cnt += 1;
}

// Wide slices (W > 64, 3D slabs): a slice block streams as NC = W / CR chunks
// of CR rows.  The blocks are symmetric, so a chunk's rows are read as columns:
// thread (grp, rv) owns the outputs rv V .. rv V + V - 1 (16 bytes of a row, V = 2
// in complex64) and adds up the chunk rows grp, grp + ng, ... of every chunk of the
// slice in registers; the ng partial sums of an output meet once a slice.  Nothing
// synchronises the CTA between chunks: a warp waits for a chunk's copy, and its
// arrival on the slot's second barrier lets the producer warp refill it.  (Finishing
// a chunk's rows with shuffles and a CTA barrier each, in 256 threads, took 12.8 k
// cycles a slice at W = 128, 16.6 k at 144, several times the copies' time.)
// The row buffer yb is always on chip on this path.
template <typename R>
__device__ void sweep_chunked(const Geo& g, int i, const SweepArgs<R>& a, cx<R>* sm, Pipe& pp,
                              unsigned long long* cnt) {
  using C = cx<R>;
  constexpr int V = 16 / (int)sizeof(C), NTC = 32 * WIDE_WARPS;
  bool dead = *pp.err != 0;              // an earlier wait of this CTA ran out
  const int W = g.W, Lx = g.Lx;
  const int CR = pp.CR, NC = W / CR, WV = W / V, ng = wide_groups<R>(W);
  C* zbuf = sm;                          // [2][W]
  C* part = sm + 2 * W;                  // [ng][W]
  C* ring = reinterpret_cast<C*>(pp.ring);
  C* yb = reinterpret_cast<C*>(pp.ybuf);
  const int tid = threadIdx.x, lane = tid & 31;
  const int grp = tid / WV, rv = (tid - grp * WV) * V;
  const bool active = tid < NTC && grp < ng;
  const R t = (R)g.t;
  const int CW = CR * W;
  const uint32_t bytes = (uint32_t)(CW * sizeof(C));
  const int NL = 2 * Lx - 1, NQ = NL * NC;
  const int S = pp.S;
  auto slice_of = [&](int n) { return n < Lx ? n : 2 * Lx - 2 - n; };
  auto csync = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(NTC) : "memory"); };

  // the producer's next chunk: q-th of the sweep, chunk pc of step pn
  int q = 0, pn = 0, pc = 0;
  auto issue = [&]() {
    const unsigned qq = pp.seq + q, u = qq / S;
    const int slot = (int)(qq - u * S);
    if (u > 0) ring_wait(pp.empty + slot, (u - 1) & 1u, dead, pp.err);
    bulk_load(ring + (size_t)slot * CW, a.g + ((size_t)slice_of(pn) * NC + pc) * CW, bytes, pp.bar + slot);
    ++q;
    if (++pc == NC) {
      pc = 0;
      ++pn;
    }
  };
  __syncthreads();                       // previous users of zbuf and yb are done
  if (tid == NTC) {                      // the first S chunks: their slots were read in the last sweep
    fence_proxy_async();
    while (q < S && q < NQ) issue();
  }
  sweep_prepass<R>(g, i, a, yb);
  __syncthreads();
  if (tid == NTC)
    while (q < NQ) issue();
  if (tid < NTC) {
    if (tid < W) zbuf[tid] = yb[tid];
    csync();
    unsigned qq = pp.seq, u = qq / S;
    int slot = (int)(qq - u * S);
    uint32_t ph = u & 1u;
    for (int n = 0; n < NL; ++n) {
      const int s = slice_of(n);
      const C* zc = zbuf + (n & 1) * W;
      C* zn = zbuf + ((n + 1) & 1) * W;
      C acc[2][V] = {};
      for (int c = 0; c < NC; ++c) {
        ring_wait(pp.bar + slot, ph, dead, pp.err);
        if (active) {
          const C* blk = ring + (size_t)slot * CW + rv;
          const C* zk = zc + c * CR;
          auto term = [&](int r, int k) {
            const C z = zk[r];
            if constexpr (V == 2) {
              const float4 m = *reinterpret_cast<const float4*>(blk + r * W);
              acc[k][0] = cfma(C{m.x, m.y}, z, acc[k][0]);
              acc[k][1] = cfma(C{m.z, m.w}, z, acc[k][1]);
            } else {
              acc[k][0] = cfma(blk[r * W], z, acc[k][0]);
            }
          };
          int r = grp;
          for (; r + 3 * ng < CR; r += 4 * ng) {
            term(r, 0);
            term(r + ng, 1);
            term(r + 2 * ng, 0);
            term(r + 3 * ng, 1);
          }
          for (; r < CR; r += ng) term(r, 0);
        }
        __syncwarp();                    // the warp's reads of the slot are done
        if (lane == 0) mbar_arrive(pp.empty + slot);
        if (++slot == S) {
          slot = 0;
          ph ^= 1u;
        }
      }
      if (active) {
#pragma unroll
        for (int v = 0; v < V; ++v) part[grp * W + rv + v] = acc[0][v] + acc[1][v];
      }
      csync();
      if (tid < W) {
        C y = part[tid];
        for (int k = 1; k < ng; ++k) y = y + part[k * W + tid];
        if (n < Lx) {                    // forward: row s of yb becomes y_s
          yb[(size_t)s * W + tid] = y;
          zn[tid] = (s + 1 < Lx) ? yb[(size_t)(s + 1) * W + tid] - t * y : y;
        } else {                         // backward: row s of yb becomes x_s
          const C xv = yb[(size_t)s * W + tid] - t * y;
          yb[(size_t)s * W + tid] = xv;
          zn[tid] = xv;
        }
      }
      csync();
    }
  }
  __syncthreads();
  sweep_postpass<R>(g, i, a, yb);
  pp.seq += NQ;
  if (tid == 0 && cnt) *cnt += 1;
}

template <typename R>
__device__ __forceinline__ SweepArgs<R> sweep_base(const Geo& g, const Bufs& b, int vs, int i) {
  SweepArgs<R> a;
  const size_t nsub = (size_t)g.Lx * g.W;
  a.g = reinterpret_cast<const cx<R>*>(b.g) + ((size_t)slot_freq(g, vs) * g.p + i) * nsub * g.W;
  a.y = reinterpret_cast<cx<R>*>(b.yscr) + ((size_t)vs * g.p + i) * nsub;
  a.src = nullptr;
  a.lay_lo = a.lay_hi = nullptr;
  a.dst = nullptr;
  a.dst_op = 0;
  a.in_scale = a.out_scale = 1.0;
  a.bnd_lo = a.bnd_hi = nullptr;
  return a;
}

__device__ __forceinline__ unsigned long long* sweep_cnt(const Geo& g, const Bufs& b, int vs, int i) {
  return b.sweeps ? b.sweeps + (size_t)vs * g.p + i : nullptr;
}
// boundary-row values and interface vectors are kept in the sweep precision R
// (their buffers are sized for complex128, so either precision fits)
template <typename R>
__device__ __forceinline__ cx<R>* bnd_ptr(const Geo& g, const Bufs& b, int vs, int i, int hi) {
  return reinterpret_cast<cx<R>*>(b.bnd) + (((size_t)vs * g.p + i) * 2 + hi) * g.A;
}
template <typename R>
__device__ __forceinline__ cx<R>* ifv_ptr(const Geo& g, const Bufs& b, int vs, int slot) {
  return reinterpret_cast<cx<R>*>(b.ifv) + ((size_t)vs * IF_N + slot) * nifc(g);
}

// ---------------------------------------------------------------- interface pieces
template <typename R>
__device__ __forceinline__ cx<R> shfl_up_c(cx<R> v, int d) {
  return {__shfl_up_sync(0xffffffffu, v.x, d), __shfl_up_sync(0xffffffffu, v.y, d)};
}
template <typename R>
__device__ __forceinline__ cx<R> shfl_down_c(cx<R> v, int d) {
  return {__shfl_down_sync(0xffffffffu, v.x, d), __shfl_down_sync(0xffffffffu, v.y, d)};
}

// Affine map on a pair of complex values: (s0, s1) -> (a s0 + b s1 + u, c s0 + d s1 + v).
template <typename R>
struct Aff2 {
  cx<R> a, b, c, d, u, v;
};
template <typename R>
__device__ __forceinline__ Aff2<R> aff_id() {
  return {{1, 0}, {0, 0}, {0, 0}, {1, 0}, {0, 0}, {0, 0}};
}
// o after in
template <typename R>
__device__ __forceinline__ Aff2<R> aff_after(const Aff2<R>& o, const Aff2<R>& in) {
  return {o.a * in.a + o.b * in.c, o.a * in.b + o.b * in.d, o.c * in.a + o.d * in.c,
          o.c * in.b + o.d * in.d, o.a * in.u + o.b * in.v + o.u, o.c * in.u + o.d * in.v + o.v};
}
template <typename R>
__device__ __forceinline__ Aff2<R> aff_shfl_up(const Aff2<R>& f, int d) {
  return {shfl_up_c(f.a, d), shfl_up_c(f.b, d), shfl_up_c(f.c, d),
          shfl_up_c(f.d, d), shfl_up_c(f.u, d), shfl_up_c(f.v, d)};
}
template <typename R>
__device__ __forceinline__ Aff2<R> aff_shfl_down(const Aff2<R>& f, int d) {
  return {shfl_down_c(f.a, d), shfl_down_c(f.b, d), shfl_down_c(f.c, d),
          shfl_down_c(f.d, d), shfl_down_c(f.u, d), shfl_down_c(f.v, d)};
}

// Apply the banded interface preconditioner along the x lines of layer i:
// z = M^-1 r with M = L D L^T (complex symmetric, no conjugation; L unit lower
// with sub-diagonals l1, l2, l2 = 0 where only the tridiagonal part is kept):
//   forward   y_x = r_x - l1_x y_{x-1} - l2_x y_{x-2},   w_x = y_x / d_x
//   backward  z_x = w_x - l1_{x+1} z_{x+1} - l2_{x+2} z_{x+2}
// Each recurrence is a chain of affine maps on the pair state (y_x, y_{x-1})
// (resp. (z_x, z_{x+1})): one warp per line, 128 sites (4 per lane) per pass
// with the state carried from pass to pass; each lane composes its 4 sites'
// maps, a 5-step warp scan composes across lanes, then the lanes finish
// their sites.  Factors per site: 1/d_x, l1_x, l2_x.
//
// r is the COCG residual, rewritten in this kernel between calls: it must be
// read through the coherent path, never as const __restrict__ (which lets the
// compiler use non-coherent loads whose cached lines can be stale by the next
// iteration).  The preconditioner factors are read-only for the kernel's life.
//
// Not inlined: the scan's state would otherwise compete for registers with the
// whole X-matvec kernel (capped at 128 per thread for two CTAs per SM) and
// spill inside the sweeps.
template <typename R>
__device__ __noinline__ void precond_apply(const Geo& g, const Bufs& b, int vs, int i, const cx<R>* r,
                                           cx<R>* z) {
  using C = cx<R>;
  constexpr int E = 4, CH = 32 * E;
  const int Lx = g.Lx, A = g.A;
  const C* __restrict__ pre =
      reinterpret_cast<const C*>(b.pre) + ((size_t)slot_freq(g, vs) * nifc(g) + (size_t)i * A) * 3;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const C zero = {0, 0};
  for (int tr = wid; tr < g.T; tr += (int)(blockDim.x >> 5)) {
    const int o = Lx * tr;
    const C* invd = pre + o;
    const C* l1 = pre + A + o;
    const C* l2 = pre + 2 * A + o;
    C c0v = zero, c1v = zero;              // (y, y_prev) entering the pass
    for (int c0 = 0; c0 < Lx; c0 += CH) {
      const int x0 = c0 + lane * E;
      // site x: (s0, s1) -> (-l1_x s0 - l2_x s1 + r_x, s0); the coefficients are
      // re-read in the apply pass rather than held in registers
      Aff2<R> P = aff_id<R>();
#pragma unroll
      for (int k = 0; k < E; ++k) {
        const int x = x0 + k;
        if (x < Lx) P = aff_after(Aff2<R>{-l1[x], -l2[x], {1, 0}, zero, r[o + x], zero}, P);
      }
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {   // inclusive scan: lanes l-d.. then l
        const Aff2<R> q = aff_shfl_up(P, d);
        if (lane >= d) P = aff_after(P, q);
      }
      // state entering this lane: the previous lane's prefix applied to the carry
      C s0 = P.a * c0v + P.b * c1v + P.u, s1 = P.c * c0v + P.d * c1v + P.v;
      s0 = shfl_up_c(s0, 1);
      s1 = shfl_up_c(s1, 1);
      if (lane == 0) {
        s0 = c0v;
        s1 = c1v;
      }
#pragma unroll
      for (int k = 0; k < E; ++k) {
        const int x = x0 + k;
        if (x < Lx) {
          const C y = r[o + x] - l1[x] * s0 - l2[x] * s1;
          s1 = s0;
          s0 = y;
          z[o + x] = y * invd[x];
        }
      }
      c0v = cx<R>{__shfl_sync(0xffffffffu, s0.x, 31), __shfl_sync(0xffffffffu, s0.y, 31)};
      c1v = cx<R>{__shfl_sync(0xffffffffu, s1.x, 31), __shfl_sync(0xffffffffu, s1.y, 31)};
    }
    __syncwarp();
    C e0v = zero, e1v = zero;              // (z, z_next) entering the pass from the right
    const int nch = (Lx + CH - 1) / CH;
    for (int c = nch - 1; c >= 0; --c) {
      const int x0 = c * CH + lane * E;
      // site x: (s0, s1) -> (-l1_{x+1} s0 - l2_{x+2} s1 + w_x, s0)
      auto m1 = [&](int x) { return (x + 1 < Lx) ? l1[x + 1] : zero; };
      auto m2 = [&](int x) { return (x + 2 < Lx) ? l2[x + 2] : zero; };
      Aff2<R> Q = aff_id<R>();
#pragma unroll
      for (int k = E - 1; k >= 0; --k) {
        const int x = x0 + k;
        if (x < Lx) Q = aff_after(Aff2<R>{-m1(x), -m2(x), {1, 0}, zero, z[o + x], zero}, Q);
      }
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {   // inclusive suffix scan: lanes l+d.. then l
        const Aff2<R> q = aff_shfl_down(Q, d);
        if (lane + d < 32) Q = aff_after(Q, q);
      }
      C s0 = Q.a * e0v + Q.b * e1v + Q.u, s1 = Q.c * e0v + Q.d * e1v + Q.v;
      s0 = shfl_down_c(s0, 1);
      s1 = shfl_down_c(s1, 1);
      if (lane == 31) {
        s0 = e0v;
        s1 = e1v;
      }
#pragma unroll
      for (int k = E - 1; k >= 0; --k) {
        const int x = x0 + k;
        if (x < Lx) {
          const C v = z[o + x] - m1(x) * s0 - m2(x) * s1;
          s1 = s0;
          s0 = v;
          z[o + x] = v;
        }
      }
      e0v = cx<R>{__shfl_sync(0xffffffffu, s0.x, 0), __shfl_sync(0xffffffffu, s0.y, 0)};
      e1v = cx<R>{__shfl_sync(0xffffffffu, s1.x, 0), __shfl_sync(0xffffffffu, s1.y, 0)};
    }
  }
}

// (C p)[a] on layer l: the Dyson matrix restricted to the interface layer,
// with its diagonal d_C precomputed in R precision.
template <typename R>
__device__ __forceinline__ cx<R> layer_C_apply(const Geo& g, const cx<R>* dC, const cx<R>* pv, int a) {
  const int Lx = g.Lx, x = a % Lx, tr = a / Lx;
  cx<R> nb = {0, 0};
  if (x > 0) nb = nb + pv[a - 1];
  if (x < Lx - 1) nb = nb + pv[a + 1];
  if (tr > 0) nb = nb + pv[a - Lx];
  if (tr < g.T - 1) nb = nb + pv[a + Lx];
  return dC[a] * pv[a] + (R)g.t * nb;
}

// ---------------------------------------------------------------- reductions in R
template <typename R>
__device__ __forceinline__ cx<R> warp_sum_r(cx<R> v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, off);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, off);
  }
  return v;
}
// Cluster-wide sums in R precision (partials exchanged through the same
// shared slots as cluster_sum, widened to double there).
template <typename R, int NV>
__device__ void cluster_sum_r(cg::cluster_group& cl, RedSmem& rs, int& phase, int p, cx<R> (&v)[NV]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = warp_sum_r(v[k]);
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) rs.wred[wid * 8 + k] = cconv<double>(v[k]);
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    cxd s = {0, 0};
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s = s + rs.wred[w * 8 + threadIdx.x];
    rs.slot[phase * 8 + threadIdx.x] = s;
  }
  cl.sync();
  if (threadIdx.x < NV) {
    cxd s = {0, 0};
    for (int r = 0; r < p; ++r) {
      const cxd* rem = cl.map_shared_rank(rs.slot, r);
      s = s + rem[phase * 8 + threadIdx.x];
    }
    rs.res[threadIdx.x] = s;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = cconv<R>(rs.res[k]);
  phase ^= 1;
}

// z = M_l^-1 r on interface line i with the exact layer block of S: a dense symmetric
// product (the stored inverse is symmetric, so column a is read contiguously across
// threads), its columns split over the warps: warp task (32 V outputs, one of CS
// column ranges), the CS partials added in a fixed order.  The block (2 MB at A = 512) comes from HBM on
// every application, so what counts is the bytes in flight: V = 2 outputs a lane
// by 16-byte loads where a row's length keeps them aligned, eight columns at a time.
// part: the free row buffer [Lx][W], CS x A entries of it.  r must be complete (a
// barrier after its writers) before the call.
template <typename R, int V>
__device__ __forceinline__ void lpre_apply_v(const Geo& g, const Bufs& b, int vs, int i, const cx<R>* r, cx<R>* z,
                                             cx<R>* part) {
  const int A = g.A, nw = (int)blockDim.x >> 5, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nblk = (A + 32 * V - 1) / (32 * V);
  int CS = (3 * nw + nblk - 1) / nblk;
  if (CS > g.W / g.T) CS = g.W / g.T;    // the scratch holds W / T entries per layer site
  const int per = (A + CS - 1) / CS;
  const cx<R>* M = reinterpret_cast<const cx<R>*>(b.lpm) + ((size_t)slot_freq(g, vs) * (g.p - 1) + i) * (size_t)A * A;
  constexpr int U = 8;
  for (int task = wid; task < nblk * CS; task += nw) {
    const int blk = task % nblk, ch = task / nblk, a = (blk * 32 + lane) * V;
    const int c0 = ch * per, c1 = min(A, c0 + per);
    if (a >= A) continue;
    cx<R> acc[2][V] = {};
    const cx<R>* col = M + a;
    auto mul = [&](int c, int k) {
      if constexpr (V == 2) {
        const float4 m = *reinterpret_cast<const float4*>(col + (size_t)c * A);
        const cxf rv = r[c];
        acc[k][0] = cfma(cxf{m.x, m.y}, rv, acc[k][0]);
        acc[k][1] = cfma(cxf{m.z, m.w}, rv, acc[k][1]);
      } else {
        acc[k][0] = cfma(col[(size_t)c * A], r[c], acc[k][0]);
      }
    };
    int c = c0;
    for (; c + U <= c1; c += U) {
      if constexpr (V == 2) {
        float4 m[U];
        cxf rv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) m[u] = *reinterpret_cast<const float4*>(col + (size_t)(c + u) * A);
#pragma unroll
        for (int u = 0; u < U; ++u) rv[u] = r[c + u];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          acc[u & 1][0] = cfma(cxf{m[u].x, m[u].y}, rv[u], acc[u & 1][0]);
          acc[u & 1][1] = cfma(cxf{m[u].z, m[u].w}, rv[u], acc[u & 1][1]);
        }
      } else {
        cx<R> m[U], rv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) m[u] = col[(size_t)(c + u) * A];
#pragma unroll
        for (int u = 0; u < U; ++u) rv[u] = r[c + u];
#pragma unroll
        for (int u = 0; u < U; ++u) acc[u & 1][0] = cfma(m[u], rv[u], acc[u & 1][0]);
      }
    }
    for (; c < c1; ++c) mul(c, 0);
#pragma unroll
    for (int v = 0; v < V; ++v) part[ch * A + a + v] = acc[0][v] + acc[1][v];
  }
  __syncthreads();
  for (int a = threadIdx.x; a < A; a += (int)blockDim.x) {
    cx<R> s = part[a];
    for (int ch = 1; ch < CS; ++ch) s = s + part[ch * A + a];
    z[a] = s;
  }
}
template <typename R>
__device__ __noinline__ void lpre_apply(const Geo& g, const Bufs& b, int vs, int i, const cx<R>* r, cx<R>* z,
                                        cx<R>* part) {
  if constexpr (sizeof(R) == 4) {
    if (g.A % 2 == 0) {                  // rows start on 16-byte boundaries
      lpre_apply_v<R, 2>(g, b, vs, i, r, z, part);
      return;
    }
  }
  lpre_apply_v<R, 1>(g, b, vs, i, r, z, part);
}

template <typename R>
__device__ __forceinline__ void interface_precond(const Geo& g, const Bufs& b, int vs, int i, const cx<R>* r,
                                                  cx<R>* z, cx<R>* part) {
  if (g.lpre) lpre_apply<R>(g, b, vs, i, r, z, part);
  else precond_apply<R>(g, b, vs, i, r, z);
}

// COCG for S y = b on the interface (S = C - E^T B^-1 E never formed), all in
// precision R: the FP64 form solves to krylov_tol in FP64; the mixed form's
// inner solves (refined against FP64 residuals one level up) run in complex64.
// Right-hand side in IF_B, solution y in IF_X.  Returns the iteration count;
// *conv is set to 0 if the cap was hit.  xB += xs B^-1 E y (the subdomain block; "="
// when fresh) comes along without a sweep of its own: the iteration's product
// B^-1 E p is still in the row buffer when its step length alpha is known.
template <typename R, int WF>
__device__ int schur_cocg(cg::cluster_group& cl, RedSmem& rs, int& phase, const Geo& g,
                          const Bufs& b, int vs, int i, double tol, cx<R>* sm, Pipe& pp,
                          cxd* xB, double xs, bool fresh, int* conv) {
  using C = cx<R>;
  const int p = g.p, A = g.A;
  const bool has = i < p - 1;
  C* X = ifv_ptr<R>(g, b, vs, IF_X);
  C* Rv = ifv_ptr<R>(g, b, vs, IF_R);
  C* Z = ifv_ptr<R>(g, b, vs, IF_Z);
  C* P = ifv_ptr<R>(g, b, vs, IF_P);
  C* SP = ifv_ptr<R>(g, b, vs, IF_SP);
  const C* Bv = ifv_ptr<R>(g, b, vs, IF_B);
  const C* dC = ifv_ptr<R>(g, b, vs, IF_D) + (size_t)i * A;
  const size_t o = (size_t)i * A;
  const C* bl_i = bnd_ptr<R>(g, b, vs, i, 1);
  const C* bl_n = has ? bnd_ptr<R>(g, b, vs, i + 1, 0) : nullptr;
  const R tr = (R)g.t;

  if (has) {
    for (int a = threadIdx.x; a < A; a += (int)blockDim.x) {
      X[o + a] = C{0, 0};
      Rv[o + a] = Bv[o + a];
    }
  }
  __syncthreads();
  C* yb = pp.ybuf ? reinterpret_cast<C*>(pp.ybuf) : sweep_base<R>(g, b, vs, i).y;   // the sweeps' row buffer
  const int W = g.W, wd = g.T * g.h[i], nsub = g.Lx * W;
  if (has) interface_precond<R>(g, b, vs, i, Rv + o, Z + o, yb);
  __syncthreads();
  C v2[2] = {{0, 0}, {0, 0}};
  if (has) {
    for (int a = threadIdx.x; a < A; a += (int)blockDim.x) {
      C zz = Z[o + a], r = Rv[o + a];
      P[o + a] = zz;
      v2[0] = cfma(r, zz, v2[0]);
      v2[1].x += cabs2(r);
    }
  }
  cluster_sum_r<R, 2>(cl, rs, phase, p, v2);
  C rho = v2[0];
  const R bn = v2[1].x;
  *conv = 1;
  if (bn == (R)0) {
    if (fresh)
      for (int e = threadIdx.x; e < nsub; e += (int)blockDim.x)
        if (e % W < wd) xB[e] = cxd{0, 0};
    return 0;
  }
  SweepArgs<R> sa = sweep_base<R>(g, b, vs, i);
  sa.lay_lo = (i > 0) ? P + (size_t)(i - 1) * A : nullptr;
  sa.lay_hi = has ? P + o : nullptr;
  sa.bnd_lo = bnd_ptr<R>(g, b, vs, i, 0);
  sa.bnd_hi = bnd_ptr<R>(g, b, vs, i, 1);
  const R tol2 = (R)(tol * tol);
  int it = 0;
  for (;;) {
    if (it >= g.krylov_maxit) {
      *conv = 0;
      break;
    }
    ++it;
    cl.sync();                                  // P of both neighbour layers is final
    sweep<R, WF>(g, i, sa, sm, pp, sweep_cnt(g, b, vs, i));   // B^-1 E p on this subdomain
    cl.sync();                                  // boundary values of every subdomain written
    C v1[1] = {{0, 0}};
    if (has) {
      for (int a = threadIdx.x; a < A; a += (int)blockDim.x) {
        C sp = layer_C_apply<R>(g, dC, P + o, a) - tr * (bl_i[a] + bl_n[a]);
        SP[o + a] = sp;
        v1[0] = cfma(P[o + a], sp, v1[0]);
      }
    }
    cluster_sum_r<R, 1>(cl, rs, phase, p, v1);
    const C alpha = cdiv(rho, v1[0]);
    v1[0] = C{0, 0};
    if (has) {
      for (int a = threadIdx.x; a < A; a += (int)blockDim.x) {
        X[o + a] = X[o + a] + alpha * P[o + a];
        const C r = Rv[o + a] - alpha * SP[o + a];
        Rv[o + a] = r;
        v1[0].x += cabs2(r);
      }
    }
    for (int e = threadIdx.x; e < nsub; e += (int)blockDim.x) {
      if (e % W >= wd) continue;
      const cxd d = cconv<double>(alpha * yb[e]);
      cxd x = fresh ? cxd{0, 0} : xB[e];
      x.x = fma(xs, d.x, x.x);
      x.y = fma(xs, d.y, x.y);
      xB[e] = x;
    }
    fresh = false;
    cluster_sum_r<R, 1>(cl, rs, phase, p, v1);  // also: the row buffer is free (the preconditioner's scratch)
    if (v1[0].x <= tol2 * bn) break;
    if (has) interface_precond<R>(g, b, vs, i, Rv + o, Z + o, yb);
    __syncthreads();
    v1[0] = C{0, 0};
    if (has)
      for (int a = threadIdx.x; a < A; a += (int)blockDim.x) v1[0] = cfma(Rv[o + a], Z[o + a], v1[0]);
    cluster_sum_r<R, 1>(cl, rs, phase, p, v1);
    const C beta = cdiv(v1[0], rho);
    rho = v1[0];
    if (has) {
      for (int a = threadIdx.x; a < A; a += (int)blockDim.x) P[o + a] = Z[o + a] + beta * P[o + a];
    }
  }
  return it;
}

// Layer diagonal d_C = i w + mu - V - Sigma on this CTA's interface layer, in
// precision R, computed once per launch for the interface products.
template <typename R>
__device__ void layer_diag(const Geo& g, const Bufs& b, int vs, int i) {
  if (i >= g.p - 1) return;
  cx<R>* dC = ifv_ptr<R>(g, b, vs, IF_D) + (size_t)i * g.A;
  const int f = slot_freq(g, vs);
  const cxd* hd = b.hdiag ? b.hdiag + (size_t)f * g.Ndd + g.ifc_off + (size_t)i * g.A : nullptr;
  for (int a = threadIdx.x; a < g.A; a += (int)blockDim.x)
    dC[a] = cconv<R>(hd ? hd[a] : dyson_diag(g, b, f, a + g.A * g.ylayer[i]));
}

// res = rhs - H x (mode 0: full H; mode 1: B only, no interface coupling),
// FP64, on this CTA's entries.  Returns partials (||res||^2, ||rhs||^2).
// H_ii comes from the per-solve DD-layout copy (coalesced); each thread takes
// RU sites per pass and issues all their loads before any store, so the loads
// of a pass are in flight together; every term enters by one fused
// multiply-add (the FP64 pipe is what bounds this pass when all frequencies
// run it together).
__device__ __noinline__ void residual_H(const Geo& g, const Bufs& b, int vs, int i, const cxd* rhs,
                                        const cxd* x, cxd* res, int mode, double* rn, double* qn) {
  constexpr int RU = 4;
  const int W = g.W, Lx = g.Lx, T = g.T, h = g.h[i], w = T * h, A = g.A;
  const int nsub = Lx * W, nt = (int)blockDim.x;
  const cxd* xs = x + (size_t)i * nsub;
  const cxd* rs_ = rhs + (size_t)i * nsub;
  cxd* ro = res + (size_t)i * nsub;
  const double t = g.t;
  const int f = slot_freq(g, vs);
  const cxd* hd = b.hdiag + (size_t)f * g.Ndd;
  const cxd* hs = hd + (size_t)i * nsub;
  const cxd* xlo = (mode == 0 && i > 0) ? x + g.ifc_off + (size_t)(i - 1) * A : nullptr;
  const cxd* xhi = (mode == 0 && i < g.p - 1) ? x + g.ifc_off + (size_t)i * A : nullptr;
  double sr = 0, sq = 0;
  const double mt = -t;
  for (int e0 = threadIdx.x; e0 < nsub; e0 += RU * nt) {
    cxd q[RU], rr[RU];
    bool on[RU];
#pragma unroll
    for (int u = 0; u < RU; ++u) {
      const int e = e0 + u * nt;
      const int s = e / W, j = e - s * W;
      on[u] = e < nsub && j < w;
      q[u] = rr[u] = cxd{0, 0};
      if (on[u]) {
        const int tr = j % T, sl = j / T;
        const cxd dv = hs[e], xc = xs[e];
        cxd r = rs_[e];
        q[u] = r;
        // r = q - t (sum of neighbours) - H_ii x, one fused multiply-add per term
        auto sub = [&](cxd v) {
          r.x = fma(mt, v.x, r.x);
          r.y = fma(mt, v.y, r.y);
        };
        if (s > 0) sub(xs[e - W]);
        if (s < Lx - 1) sub(xs[e + W]);
        if (tr > 0) sub(xs[e - 1]);
        if (tr < T - 1) sub(xs[e + 1]);
        if (sl > 0) sub(xs[e - T]);
        if (sl < h - 1) sub(xs[e + T]);
        if (sl == 0 && xlo) sub(xlo[s + Lx * tr]);
        if (sl == h - 1 && xhi) sub(xhi[s + Lx * tr]);
        r.x = fma(-dv.x, xc.x, fma(dv.y, xc.y, r.x));
        r.y = fma(-dv.x, xc.y, fma(-dv.y, xc.x, r.y));
        rr[u] = r;
      }
    }
#pragma unroll
    for (int u = 0; u < RU; ++u) {
      if (!on[u]) continue;
      ro[e0 + u * nt] = rr[u];
      sr += cabs2(rr[u]);
      sq += cabs2(q[u]);
    }
  }
  if (mode == 0 && i < g.p - 1) {
    const size_t o = g.ifc_off + (size_t)i * A;
    const cxd* xl = x + o;
    const cxd* xb = x + (size_t)i * nsub;         // subdomain i: its top row touches layer i
    const cxd* xa = x + (size_t)(i + 1) * nsub;   // subdomain i+1: its bottom row touches layer i
    const int hi = T * (g.h[i] - 1);
    for (int a = threadIdx.x; a < A; a += nt) {
      const int xx = a % Lx, tr = a / Lx;
      cxd nb = {0, 0};
      if (xx > 0) nb = nb + xl[a - 1];
      if (xx < Lx - 1) nb = nb + xl[a + 1];
      if (tr > 0) nb = nb + xl[a - Lx];
      if (tr < T - 1) nb = nb + xl[a + Lx];
      cxd hv = hd[o + a] * xl[a] + t * nb;
      hv = hv + t * (xb[(size_t)xx * W + hi + tr] + xa[(size_t)xx * W + tr]);
      cxd q = rhs[o + a];
      cxd rr = q - hv;
      res[o + a] = rr;
      sr += cabs2(rr);
      sq += cabs2(q);
    }
  }
  *rn = sr;
  *qn = sq;
}

// x = H^-1 rhs by elimination of the subdomain unknowns, sweeps and the
// interface solve in precision R:
//   z = B^-1 rhs_B;  y = S^-1 (rhs_C - E^T z);  x_B = z - B^-1 E y;  x_C = y.
// zero_B: rhs_B = 0 is known, so z = 0 and its sweep is skipped.
// sc: the solve runs on rhs / sc and its result is scaled back by sc, so the
// R-precision recurrences work on O(1) numbers (the squared norms of the
// shrinking refinement residuals would leave float range otherwise).
template <typename R, int WF>
__device__ int solve_H(cg::cluster_group& cl, RedSmem& rs, int& phase, const Geo& g,
                       const Bufs& b, int vs, int i, const cxd* rhs, cxd* xout, bool zero_B,
                       double sc, double tol, cx<R>* sm, Pipe& pp, int* conv) {
  const int A = g.A;
  const bool has = i < g.p - 1;
  const size_t nsub = (size_t)g.Lx * g.W;
  cx<R>* Bv = ifv_ptr<R>(g, b, vs, IF_B);
  const cxd* rc = rhs + g.ifc_off + (size_t)i * A;
  const R tr = (R)g.t;
  const double isc = 1.0 / sc;
  if (!zero_B) {
    SweepArgs<R> sa = sweep_base<R>(g, b, vs, i);
    sa.src = rhs + i * nsub;
    sa.in_scale = isc;
    sa.dst = xout + i * nsub;
    sa.out_scale = sc;
    sa.dst_op = 0;
    sa.bnd_lo = bnd_ptr<R>(g, b, vs, i, 0);
    sa.bnd_hi = bnd_ptr<R>(g, b, vs, i, 1);
    sweep<R, WF>(g, i, sa, sm, pp, sweep_cnt(g, b, vs, i));
    cl.sync();
    if (has) {
      const cx<R>* bl_i = bnd_ptr<R>(g, b, vs, i, 1);
      const cx<R>* bl_n = bnd_ptr<R>(g, b, vs, i + 1, 0);
      for (int a = threadIdx.x; a < A; a += (int)blockDim.x)
        Bv[(size_t)i * A + a] = cconv<R>(isc * rc[a]) - tr * (bl_i[a] + bl_n[a]);
    }
  } else if (has) {
    for (int a = threadIdx.x; a < A; a += (int)blockDim.x) Bv[(size_t)i * A + a] = cconv<R>(isc * rc[a]);
  }
  __syncthreads();
  int it = schur_cocg<R, WF>(cl, rs, phase, g, b, vs, i, tol, sm, pp, xout + i * nsub, -sc, zero_B, conv);
  const cx<R>* X = ifv_ptr<R>(g, b, vs, IF_X);
  if (has) {
    cxd* xc = xout + g.ifc_off + (size_t)i * A;
    for (int a = threadIdx.x; a < A; a += (int)blockDim.x) xc[a] = sc * cconv<double>(X[(size_t)i * A + a]);
  }
  return it;
}

constexpr size_t YBUF_MAX = 64 * 1024;   // forward intermediates kept on chip up to this size
constexpr size_t SMEM_LIMIT = 223 * 1024;   // dynamic shared memory per CTA, below the 227 KB cap (static: ~3 KB)

// Shared-memory plan of a sweep: ring of S slots of CR x W entries (CR = W when
// a whole slice block fits a slot, the W <= 64 strips of the FP64 form; row
// chunks otherwise), zw entries of z vectors, and the on-chip row buffer when
// it fits.  W <= 64: 256 threads at two CTAs per SM, ~100 KB each.
struct RingPlan {
  int CR, S, zw;
  size_t ybuf, smem;
};
template <typename R>
__host__ __device__ inline RingPlan ring_plan(int W, int Lx) {
  RingPlan rp;
  const size_t cs = sizeof(cx<R>);
  const size_t yb = (size_t)Lx * W * cs;
  rp.zw = 2 * W + (W > DY_MAXW_SMEM ? wide_groups<R>(W) * W : 0);
  if (W <= DY_MAXW_SMEM) {
    rp.ybuf = yb <= YBUF_MAX ? yb : 0;
    rp.CR = W;
    long S = ((long)100 * 1024 - (long)rp.ybuf - (long)(rp.zw * cs)) / (long)(W * W * cs);
    if (S > MAX_STAGES) S = MAX_STAGES;
    if (S < 2) S = 2;
    rp.S = (int)S;
  } else {
    rp.ybuf = yb;                                                       // one CTA per SM
    const long budget = (long)SMEM_LIMIT - (long)yb - (long)(rp.zw * cs);
    // largest divisor of W whose chunks are at most 32 KB and leave >= 4 ring slots
    // (>= 2, and any size, as a last resort); a chunk row is W entries, a multiple of
    // 32 bytes, so any row count keeps the bulk copies 16-byte aligned
    rp.CR = 0;
    rp.S = 0;
    for (int want = 4; want >= 2 && !rp.CR; want -= 2)
      for (int cr = W; cr >= 1; --cr) {
        if (W % cr || (want > 2 && (size_t)cr * W * cs > 32 * 1024)) continue;
        const long S = budget / (long)((size_t)cr * W * cs);
        if (S >= want) {
          rp.CR = cr;
          rp.S = (int)(S > MAX_STAGES ? MAX_STAGES : S);
          break;
        }
      }
  }
  rp.smem = rp.CR ? (size_t)rp.S * rp.CR * W * cs + (size_t)rp.zw * cs + rp.ybuf : 0;
  return rp;
}
// The plan of a geometry: the heuristic above, or the autotuner's choice of
// slots (and chunk rows for W > 64) with the same row buffer and z area.
template <typename R>
__host__ __device__ inline RingPlan ring_plan(const Geo& g) {
  RingPlan rp = ring_plan<R>(g.W, g.Lx);
  if (g.ring_S > 0 && rp.CR > 0) {
    rp.S = g.ring_S;
    if (g.W > DY_MAXW_SMEM && g.ring_CR > 0) rp.CR = g.ring_CR;
    rp.smem = (size_t)rp.S * rp.CR * g.W * sizeof(cx<R>) + (size_t)rp.zw * sizeof(cx<R>) + rp.ybuf;
  }
  return rp;
}
// Configurations the autotuner times: the heuristic's first, then every slot
// count 2..MAX_STAGES that fits, and for W > 64 the chunk heights (divisors of
// W) with the most slots that fit.
template <typename R>
inline int ring_candidates(const Geo& g, int* S, int* CR, int max) {
  const RingPlan h = ring_plan<R>(g.W, g.Lx);
  if (h.CR == 0 || max < 1) return 0;
  int n = 0;
  S[n] = h.S;
  CR[n] = h.CR;
  ++n;
  const size_t cs = sizeof(cx<R>), fixed = (size_t)h.zw * cs + h.ybuf;
  auto fits = [&](int s, int cr) { return (size_t)s * cr * g.W * cs + fixed <= SMEM_LIMIT; };
  auto add = [&](int s, int cr) {
    for (int k = 0; k < n; ++k)
      if (S[k] == s && CR[k] == cr) return;
    if (n < max && fits(s, cr)) {
      S[n] = s;
      CR[n] = cr;
      ++n;
    }
  };
  if (g.W <= DY_MAXW_SMEM) {
    for (int s = 2; s <= MAX_STAGES; ++s) add(s, g.W);
  } else {
    for (int cr = g.W; cr >= 1; --cr) {            // chunks of 8 to 64 KB
      const size_t bytes = (size_t)cr * g.W * cs;
      if (g.W % cr || bytes > 64 * 1024 || bytes < 8 * 1024) continue;
      int best = 0;
      for (int s = MAX_STAGES; s >= 2; --s)
        if (fits(s, cr)) {
          best = s;
          break;
        }
      if (best >= 3) add(best, cr);
      if (n >= max) break;
    }
  }
  return n;
}

// ---------------------------------------------------------------- kernels
// u = X q_j  (Sec. 2.3 Eqs. 6-8), with u = v - w computed as the solution of
// H u = q - H w = [0; q_C - E^T w_B]  (w = blkdiag(B^-1, 0) q, so B w_B = q_B),
// i.e. y = S^-1 (E^T w_B - q_C), u_B = B^-1 E y, u_C = -y: no cancellation.
//   mixed = 0: every sweep in R (= double), the interface solve to krylov_tol.
//   mixed = 1: sweeps in complex64 (R = float).  w_B is refined against FP64
//              residuals of B, u against FP64 residuals of H, each until the
//              relative residual is below refine_tol.
template <typename R, int WF>
__global__ void __launch_bounds__(solve_threads<WF>(), WF == 0 ? 1 : 2) k_xmatvec(Geo g, Bufs b, int j, int mixed, int ncols) {
  cg::cluster_group cl = cg::this_cluster();
  __shared__ RedSmem rs;
  __shared__ __align__(8) uint64_t bars[2 * MAX_STAGES];
  __shared__ int err;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  // one cluster per (frequency, block column): slot vs = f * nb + c
  const int i = blockIdx.x, vs = blockIdx.y, p = g.p, A = g.A;
  const int f = slot_freq(g, vs), c = vs - f * g.nb;
  if (c >= ncols) return;                  // same values in every CTA of the cluster
  int* st = b.st + (size_t)f * ST_N;
  if (st[ST_DONE]) return;
  Pipe pp;
  pp.bar = bars;
  pp.empty = bars + MAX_STAGES;
  const RingPlan rp = ring_plan<R>(g);
  pp.S = rp.S;
  pp.CR = rp.CR;
  pp.ring = smem_raw;
  pp.seq = 0;
  pp.err = &err;
  pipe_init(pp);
  cx<R>* sm = reinterpret_cast<cx<R>*>(smem_raw + (size_t)rp.S * rp.CR * g.W * sizeof(cx<R>));
  pp.ybuf = rp.ybuf ? (void*)(sm + rp.zw) : nullptr;
  layer_diag<R>(g, b, vs, i);
  int phase = 0;
  const bool has = i < p - 1;
  const size_t Ndd = g.Ndd, nsub = (size_t)g.Lx * g.W;
  const cxd* q = b.Q + ((size_t)f * (g.k_max + g.nb) + (size_t)j * g.nb + c) * Ndd;
  cxd* u = b.u + (size_t)vs * Ndd;
  if (g.qsplit) {
    // the basis is stored as double-floats: widen this CTA's entries of q_j into u,
    // which is free until the first H solve writes it, and read q_j from there
    const cdfl* qs = reinterpret_cast<const cdfl*>(q);
    const int n = own_count(g, i);
    for (int e = threadIdx.x; e < n; e += (int)blockDim.x) {
      const size_t k = own_idx(g, i, e, (int)nsub);
      u[k] = cwiden(qs[k]);
    }
    __syncthreads();
    q = u;
  }
  int iters = 0, solves = 0, refines = 0, conv_all = 1, conv = 1;

  if (!mixed) {
    // w = B^-1 q_B, only its boundary rows are needed: E^T w
    SweepArgs<R> sa = sweep_base<R>(g, b, vs, i);
    sa.src = q + i * nsub;
    sa.bnd_lo = bnd_ptr<R>(g, b, vs, i, 0);
    sa.bnd_hi = bnd_ptr<R>(g, b, vs, i, 1);
    sweep<R, WF>(g, i, sa, sm, pp, sweep_cnt(g, b, vs, i));
    cl.sync();
    cx<R>* Bv = ifv_ptr<R>(g, b, vs, IF_B);
    if (has) {
      const cx<R>* bl_i = bnd_ptr<R>(g, b, vs, i, 1);
      const cx<R>* bl_n = bnd_ptr<R>(g, b, vs, i + 1, 0);
      const cxd* qc = q + g.ifc_off + (size_t)i * A;
      for (int a = threadIdx.x; a < A; a += (int)blockDim.x)
        Bv[(size_t)i * A + a] = (R)g.t * (bl_i[a] + bl_n[a]) - cconv<R>(qc[a]);
    }
    __syncthreads();
    iters += schur_cocg<R, WF>(cl, rs, phase, g, b, vs, i, g.krylov_tol, sm, pp, u + i * nsub, 1.0, true, &conv);
    conv_all &= conv;
    solves = 1;
    const cx<R>* X = ifv_ptr<R>(g, b, vs, IF_X);
    if (has) {
      cxd* uc = u + g.ifc_off + (size_t)i * A;
      for (int a = threadIdx.x; a < A; a += (int)blockDim.x) uc[a] = -cconv<double>(X[(size_t)i * A + a]);
    }
  } else {
    cxd* wv = b.v1 + (size_t)vs * Ndd;   // w_B, later the refinement corrections
    cxd* rv = b.v2 + (size_t)vs * Ndd;   // FP64 residuals
    cxd* hr = b.v3 + (size_t)vs * Ndd;   // right-hand side [0; q_C - E^T w_B]
    // ---- w_B = B^-1 q_B, refined against FP64 residuals of B (subdomain-local)
    {
      SweepArgs<R> sa = sweep_base<R>(g, b, vs, i);
      sa.src = q + i * nsub;
      sa.dst = wv + i * nsub;
      sa.dst_op = 0;
      sweep<R, WF>(g, i, sa, sm, pp, sweep_cnt(g, b, vs, i));
      double prev = INFINITY;
      for (int r = 0; r < g.refine_max; ++r) {
        __syncthreads();
        double rn, qn;
        residual_H(g, b, vs, i, q, wv, rv, 1, &rn, &qn);
        cxd v2[2] = {{rn, 0}, {qn, 0}};
        block_sum<2>(rs, v2);
        if (v2[0].x <= g.refine_tol * g.refine_tol * v2[1].x) break;
        if (v2[0].x > REFINE_STALL * prev) break;        // at the FP64 rounding floor
        prev = v2[0].x;
        SweepArgs<R> sc = sweep_base<R>(g, b, vs, i);
        sc.src = rv + i * nsub;
        sc.dst = wv + i * nsub;
        sc.dst_op = 1;
        sweep<R, WF>(g, i, sc, sm, pp, sweep_cnt(g, b, vs, i));
      }
    }
    cl.sync();                             // w_B of the neighbour subdomains is final
    {
      const int n = own_count(g, i);
      const int hi = g.T * (g.h[i] - 1);
      for (int e = threadIdx.x; e < n; e += (int)blockDim.x) {
        size_t k = own_idx(g, i, e, (int)nsub);
        cxd v = {0, 0};
        if (e >= (int)nsub) {
          const int a = e - (int)nsub, xx = a % g.Lx, tr = a / g.Lx;
          const cxd ew = wv[i * nsub + (size_t)xx * g.W + hi + tr] +
                         wv[(i + 1) * nsub + (size_t)xx * g.W + tr];
          v = q[k] - g.t * ew;
        }
        hr[k] = v;
      }
    }
    __syncthreads();                       // interface entries of hr are written by other threads
    double hn;
    {
      cxd v1[1] = {{0, 0}};
      if (has)
        for (int a = threadIdx.x; a < A; a += (int)blockDim.x)
          v1[0].x += cabs2(hr[g.ifc_off + (size_t)i * A + a]);
      cluster_sum<1>(cl, rs, phase, p, v1);   // also: every CTA has read w_B before it is reused
      hn = sqrt(v1[0].x);
    }
    if (hn > 0.0) {
      iters += solve_H<R, WF>(cl, rs, phase, g, b, vs, i, hr, u, true, hn, g.krylov_tol, sm, pp, &conv);
      conv_all &= conv;
      ++solves;
    } else {
      const int n = own_count(g, i);
      for (int e = threadIdx.x; e < n; e += (int)blockDim.x) u[own_idx(g, i, e, (int)nsub)] = cxd{0, 0};
    }
    double prev = INFINITY;
    for (int r = 0; r < g.refine_max && hn > 0.0; ++r) {
      cl.sync();
      double rn, qn;
      residual_H(g, b, vs, i, hr, u, rv, 0, &rn, &qn);
      cxd v2[2] = {{rn, 0}, {qn, 0}};
      cluster_sum<2>(cl, rs, phase, p, v2);
      if (v2[0].x <= g.refine_tol * g.refine_tol * v2[1].x) break;
      if (v2[0].x > REFINE_STALL * prev) break;          // at the FP64 rounding floor
      prev = v2[0].x;
      ++refines;
      iters += solve_H<R, WF>(cl, rs, phase, g, b, vs, i, rv, wv, false, sqrt(v2[0].x), g.krylov_tol, sm,
                          pp, &conv);
      conv_all &= conv;
      ++solves;
      __syncthreads();
      const int n = own_count(g, i), nt = (int)blockDim.x;
      for (int e0 = threadIdx.x; e0 < n; e0 += 4 * nt) {   // four entries' loads in flight
        cxd a4[4], b4[4];
        size_t k4[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int e = e0 + m * nt;
          k4[m] = e < n ? own_idx(g, i, e, (int)nsub) : 0;
          a4[m] = e < n ? u[k4[m]] : cxd{0, 0};
          b4[m] = e < n ? wv[k4[m]] : cxd{0, 0};
        }
#pragma unroll
        for (int m = 0; m < 4; ++m)
          if (e0 + m * nt < n) u[k4[m]] = a4[m] + b4[m];
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && err) atomicOr(st + ST_STATUS, ST_WAIT_TIMEOUT);
  if (i == 0 && threadIdx.x == 0) {       // the nb clusters of a frequency share its counters
    atomicAdd(st + ST_ITERS, iters);
    atomicAdd(st + ST_SOLVES, solves);
    atomicAdd(st + ST_REFINE, refines);
    if (!conv_all) atomicOr(st + ST_STATUS, 4);
  }
  cl.sync();          // no CTA exits while a peer may still read its shared memory
}

// w = blkdiag(B^-1, 0) q for DD-layout vectors (Eq. 7), one CTA per subdomain.
template <typename R, int WF>
__global__ void __launch_bounds__(solve_threads<WF>(), WF == 0 ? 1 : 2) k_bsolve(Geo g, Bufs b, const cxd* q, cxd* w) {
  __shared__ __align__(8) uint64_t bars[2 * MAX_STAGES];
  __shared__ int err;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int i = blockIdx.x, kf = blockIdx.y, vs = kf * g.nb;   // scratch of the frequency's first slot
  const size_t nsub = (size_t)g.Lx * g.W;
  Pipe pp;
  pp.bar = bars;
  pp.empty = bars + MAX_STAGES;
  const RingPlan rp = ring_plan<R>(g);
  pp.S = rp.S;
  pp.CR = rp.CR;
  pp.ring = smem_raw;
  pp.seq = 0;
  pp.err = &err;
  pipe_init(pp);
  cx<R>* sm = reinterpret_cast<cx<R>*>(smem_raw + (size_t)rp.S * rp.CR * g.W * sizeof(cx<R>));
  pp.ybuf = rp.ybuf ? (void*)(sm + rp.zw) : nullptr;
  SweepArgs<R> sa = sweep_base<R>(g, b, vs, i);
  sa.src = q + (size_t)kf * g.Ndd + i * nsub;
  sa.dst = w + (size_t)kf * g.Ndd + i * nsub;
  sa.dst_op = 0;
  sweep<R, WF>(g, i, sa, sm, pp, sweep_cnt(g, b, vs, i));
  if (i < g.p - 1)
    for (int a = threadIdx.x; a < g.A; a += (int)blockDim.x)
      w[(size_t)kf * g.Ndd + g.ifc_off + (size_t)i * g.A + a] = cxd{0, 0};
  __syncthreads();
  if (threadIdx.x == 0 && err) atomicOr(b.st + (size_t)kf * ST_N + ST_STATUS, ST_WAIT_TIMEOUT);
}

template <typename Kern, typename... Args>
cudaError_t launch_cluster_nt(Kern kern, dim3 grid, int cx_, int threads, size_t smem, cudaStream_t st,
                              Args... args) {
  cudaError_t e = raise_smem_limit((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  if (cx_ > 8) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cx_;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <typename Kern, typename... Args>
cudaError_t launch_cluster(Kern kern, dim3 grid, int cx_, size_t smem, cudaStream_t st, Args... args) {
  return launch_cluster_nt(kern, grid, cx_, DY_THREADS, smem, st, args...);
}

template <typename R>
size_t sweep_smem(const Geo& g) { return ring_plan<R>(g).smem; }

}  // namespace

// One X-matvec / subdomain-solve variant (precision R, sweep form WF) per
// entry point; each is defined by DY_SOLVE_VARIANT in the translation unit
// that compiles it, so the variants build in parallel.
template <typename R, int WF>
cudaError_t run_xmatvec(const Geo& g, const Bufs& b, int K, int j, int mixed, int ncols, cudaStream_t st);
template <typename R, int WF>
cudaError_t run_bsolve(const Geo& g, const Bufs& b, int K, const cxd* q_dd, cxd* w_dd, cudaStream_t st);

#define DY_SOLVE_VARIANT(R, WF)                                                                   \
  template <>                                                                                     \
  cudaError_t run_xmatvec<R, WF>(const Geo& g, const Bufs& b, int K, int j, int mixed, int ncols, \
                                 cudaStream_t st) {                                               \
    return launch_cluster_nt(k_xmatvec<R, WF>, dim3(g.p, K * g.nb), g.p, solve_threads<WF>(),     \
                             sweep_smem<R>(g), st, g, b, j, mixed, ncols);                        \
  }                                                                                               \
  template <>                                                                                     \
  cudaError_t run_bsolve<R, WF>(const Geo& g, const Bufs& b, int K, const cxd* q_dd, cxd* w_dd,   \
                                cudaStream_t st) {                                                \
    const size_t smem = sweep_smem<R>(g);                                                         \
    cudaError_t e = raise_smem_limit((const void*)k_bsolve<R, WF>, smem);                         \
    if (e != cudaSuccess) return e;                                                               \
    k_bsolve<R, WF><<<dim3(g.p, K), solve_threads<WF>(), smem, st>>>(g, b, q_dd, w_dd);           \
    return cudaGetLastError();                                                                    \
  }

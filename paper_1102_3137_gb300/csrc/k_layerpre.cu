// Exact interface-layer preconditioner for 2D strips: M = blkdiag_l(S_ll),
// the diagonal blocks of the Schur complement S = C - E^T B^-1 E (Eq. 4) on
// each interface line, inverted once per solve.  The paper leaves the
// interface solver open and credits ARMS-type approximate Schur complements;
// here S_ll is formed without approximation,
//
//   S_ll = C_ll - t^2 (P_top(l) + P_bot(l+1)),
//
// P_top(i) / P_bot(i) the restriction of B_i^-1 to the top / bottom row of
// strip i, its "surface" Green's function along the row.  Only the coupling
// between different lines (through a whole strip) is left out, which is
// small, so COCG on S needs one or two iterations.  S itself is never formed.
//
// The preconditioner may be inexact, so everything here runs in complex64:
//   k_surface_two  per (strip, side, frequency): P[s][s'] from the factorization's
//                two-sided factors and boundary columns of G_ss, by chains of
//                products towards the two ends of the strip.
//   k_layer_inv  per (interface line, frequency): S_ll and its inverse by the
//                sweep operator, symmetrised so that COCG sees a complex
//                symmetric M^-1.
// Layers of more than DY_LPRE_MAXLX (160) sites do not fit shared memory; there
//   k_layer_inv_g forms S_ll in place of P_top(l) and inverts it there by the
//                block sweep operator (32 x 32 pivots, rank-32 updates of the
//                upper 64 x 64 tiles), then writes the mirrored inverse.
// 3D slabs (slice width W = T h, T = Ly > 1) have interface layers of
// A = Lx T sites, S_ll is A x A (in-plane hopping along x and y), and
//   k_surface_3d forms P_bot(i), P_top(i) from the factorization's
//                left-connected g_s (read in binary64), by the backward
//                recursion G_ss = g_s + t^2 g_s G_{s+1,s+1} g_s and the chains
//                G_{s,c} = -t g_s G_{s+1,c} carried on the T boundary columns
//                of each slice c, with 32 x 32 tiles through shared memory
//                multiplied on the tensor cores (3xTF32; persistent grid, one
//                (slab, frequency) at a time per cluster);
//   k_layer_inv_g  inverts the A x A blocks (A <= 1024).
#include <type_traits>

#include "solve_device.cuh"
#include "tc_tf32.cuh"

namespace {

using cxf_ = cx<float>;

// In-place inverse of an n x n complex64 matrix (row stride n) in shared
// memory by the sweep operator on the full matrix (pivots on the diagonal;
// Im of the Dyson diagonal keeps them away from zero).  Thread t owns column
// t % n and every (256 / n)-th row from t / n.
__device__ __forceinline__ void sweep_invert_f(cxf_* A, int n, cxf_* prow, cxf_* fcol) {
  const int nrp = DY_THREADS / n;
  const int c = threadIdx.x % n, r0 = threadIdx.x / n;
  const bool act = r0 < nrp;
  for (int k = 0; k < n; ++k) {
    __syncthreads();
    for (int e = threadIdx.x; e < n; e += DY_THREADS) {
      const cxf_ piv = cinv(A[k * n + k]);
      prow[e] = A[k * n + e];
      fcol[e] = (e == k) ? cxf_{-piv.x, -piv.y} : A[e * n + k] * piv;
    }
    __syncthreads();
    if (act) {
      const cxf_ pc = prow[c];
      for (int r = r0; r < n; r += nrp) {
        cxf_& a = A[r * n + c];
        if (c == k) a = fcol[r];                                    // a_rk / a_kk; -1 / a_kk at r = k
        else if (r == k) a = pc * cxf_{-fcol[k].x, -fcol[k].y};     // a_kc / a_kk
        else a = cfma(cxf_{-fcol[r].x, -fcol[r].y}, pc, a);         // a_rc - a_rk a_kc / a_kk
      }
    }
  }
  __syncthreads();
  // the sweep ends at -A^-1
  for (int e = threadIdx.x; e < n * n; e += DY_THREADS) A[e] = cxf_{-A[e].x, -A[e].y};
  __syncthreads();
}

constexpr int SURF_MAXW = 32;
// The surface Green's functions of the 2D strips, from the two-sided factors g_s (S:
// complex64 or binary64) and the boundary columns of G_ss that the factorization leaves
// in b.lpg, in complex64: no recursion of its own.  With m the middle slice
// and rb the boundary row, per side:
//   pairs of one half:  G_{s,c} e_rb = -t g_s G_{s+-1,c} e_rb   (towards the ends, all c at once)
//   pairs across:       G_{s,c} = G_{s,m} N_c^T,  G_{s,m} = -t g_s G_{s+1,m} (s < m),
//                       N_c = -t g_c N_{c-1}, N_m = 1 (c > m)
// so a half is one chain of products of the 32 x 32 block -t g_s with its boundary
// columns plus W columns of G_{.,m} or N, and the across pairs are dot products of the
// rows rb of the two.  A cluster of two CTAs (left, right) per (side, strip, frequency),
// lane = row with its row of g_s in registers, a warp's columns two at a time by 16-byte
// broadcasts from shared memory.  The one-CTA form ran its own complex64 recursion and a
// chain of Lx slices: 4.0 ms at 128^2 x 32 with 128 CTAs.
template <typename S, int WT>
__global__ void __launch_bounds__(DY_THREADS, 2) k_surface_two(Geo g, Bufs b) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cg::cluster_group cl = cg::this_cluster();
  const int half = (int)cl.block_rank(), u = blockIdx.x / 2, i = u / 2, sd = u - 2 * i, f = blockIdx.y;
  const int W = WT ? WT : g.W, Lx = g.Lx, w = g.h[i], n = W * W, m = Lx / 2;
  if (sd == 0 ? i == g.p - 1 : i == 0) return;                  // no layer on that side (the whole cluster)
  const int steps = half == 0 ? m : Lx - 1 - m, rb = sd == 0 ? w - 1 : 0;
  cxf_* gb[2] = {reinterpret_cast<cxf_*>(smem_raw), reinterpret_cast<cxf_*>(smem_raw) + n};
  cxf_* M = gb[1] + n;                            // [W columns][W]: G_{s,m} or N_s
  cxf_* V = M + n;                                // [steps][W]: the boundary columns, by distance from the middle
  const size_t unit = (size_t)f * g.p + i;
  const cx<S>* gsrc = reinterpret_cast<const cx<S>*>(b.g) + unit * (size_t)Lx * n;   // complex64: column pairs interleaved
  const cxf_* bc = b.lpg + unit * lpg_entries(g);
  cxf_* Rr = b.lpg + unit * lpg_entries(g) + (size_t)(2 + sd) * Lx * W;   // [Lx][W] rows rb of G_{s,m} / N_s
  cxf_* P = b.lpt + (unit * 2 + sd) * (size_t)Lx * Lx;
  const float t = d2f_bits(g.t);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int n4 = n / 2;                           // words of two entries of a block
  auto slice = [&](int k) { return half == 0 ? m - 1 - k : m + 1 + k; };     // k-th step's slice
  constexpr int NF = (SURF_MAXW * SURF_MAXW / 2 + DY_THREADS - 1) / DY_THREADS;
  float4 nx[NF];
  auto fetch = [&](int s) {
#pragma unroll
    for (int q = 0; q < NF; ++q)
      if (tid + DY_THREADS * q < n4) {
        if constexpr (sizeof(S) == 4) {
          nx[q] = reinterpret_cast<const float4*>(gsrc + (size_t)s * n)[tid + DY_THREADS * q];
        } else {                                  // columns 2 k2, 2 k2 + 1 of row r (symmetric) into the same order
          const int e = tid + DY_THREADS * q, k2 = e / W, r = e - k2 * W;
          const cxd v0 = gsrc[(size_t)s * n + (size_t)(2 * k2) * W + r], v1 = gsrc[(size_t)s * n + (size_t)(2 * k2 + 1) * W + r];
          nx[q] = make_float4(d2f_bits(v0.x), d2f_bits(v0.y), d2f_bits(v1.x), d2f_bits(v1.y));
        }
      }
  };
  auto put = [&](cxf_* d) {
#pragma unroll
    for (int q = 0; q < NF; ++q)
      if (tid + DY_THREADS * q < n4) reinterpret_cast<float4*>(d)[tid + DY_THREADS * q] = nx[q];
  };
  // M: G_mm (slot m; symmetric, so its rows are its columns) or 1
  for (int e = tid; e < n; e += DY_THREADS) {
    const int c = e / W, r = e - c * W;
    if (half == 1) {
      M[e] = cxf_{r == c ? 1.f : 0.f, 0.f};
    } else if constexpr (sizeof(S) == 4) {
      M[e] = gsrc[(size_t)m * n + ((size_t)(c >> 1) * W + r) * 2 + (c & 1)];
    } else {
      const cxd v = gsrc[(size_t)m * n + e];
      M[e] = cxf_{d2f_bits(v.x), d2f_bits(v.y)};
    }
  }
  if (steps > 0) {
    fetch(slice(0));
    put(gb[0]);
  }
  __syncthreads();
  if (half == 0) {                                // s = m: row rb of G_mm, and P[m][m]
    for (int c = tid; c < W; c += DY_THREADS) Rr[(size_t)m * W + c] = M[c * W + rb];
    if (tid == 0) P[(size_t)m * Lx + m] = M[rb * W + rb];
  }
  for (int k = 0; k < steps; ++k) {
    const int s = slice(k);
    const cxf_* G = gb[k & 1];
    if (k + 1 < steps) fetch(slice(k + 1));
    cxf_ gr[SURF_MAXW];                           // row `lane` of -t g_s
#pragma unroll
    for (int q = 0; q < SURF_MAXW / 2; ++q) {
      const float4 v = lane < W && 2 * q < W ? reinterpret_cast<const float4*>(G)[q * W + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
      gr[2 * q] = cxf_{-t * v.x, -t * v.y};
      gr[2 * q + 1] = cxf_{-t * v.z, -t * v.w};
    }
    // this step's columns: W of M, then the boundary columns of the k slices nearer the middle
    const int nc = W + k;
    for (int c0 = 2 * wid; c0 < nc; c0 += 2 * DY_WARPS) {
      const bool b2 = c0 + 1 < nc;
      cxf_* x0 = M + (size_t)c0 * W;              // M and V are contiguous: column c at M + c W
      cxf_* x1 = b2 ? x0 + W : x0;
      cxf_ a0 = {0.f, 0.f}, a1 = {0.f, 0.f}, d0 = {0.f, 0.f}, d1 = {0.f, 0.f};
#pragma unroll
      for (int q = 0; q < SURF_MAXW / 2; ++q) {
        if (2 * q < W) {
          const float4 v = reinterpret_cast<const float4*>(x0)[q], y = reinterpret_cast<const float4*>(x1)[q];
          a0 = cfma(gr[2 * q], cxf_{v.x, v.y}, a0);
          d0 = cfma(gr[2 * q], cxf_{y.x, y.y}, d0);
          a1 = cfma(gr[2 * q + 1], cxf_{v.z, v.w}, a1);
          d1 = cfma(gr[2 * q + 1], cxf_{y.z, y.w}, d1);
        }
      }
      a0 = a0 + a1;
      d0 = d0 + d1;
      __syncwarp();                               // both columns are read before they are rewritten
      auto out = [&](int c, cxf_* x, cxf_ v) {
        if (lane >= W) return;
        x[lane] = v;
        if (lane != rb) return;
        if (c < W) {
          Rr[(size_t)s * W + c] = v;
          if (half == 0 && c == rb) P[(size_t)s * Lx + m] = P[(size_t)m * Lx + s] = v;
        } else {
          const int sc = slice(c - W);
          P[(size_t)s * Lx + sc] = P[(size_t)sc * Lx + s] = v;
        }
      };
      out(c0, x0, a0);
      if (b2) out(c0 + 1, x1, d0);
    }
    // the chain of column s starts with the boundary column of G_ss
    for (int r = tid; r < W; r += DY_THREADS) {
      const cxf_ v = bc[((size_t)s * 2 + sd) * W + r];
      V[(size_t)k * W + r] = v;
      if (r == rb) P[(size_t)s * Lx + s] = v;
    }
    if (k + 1 < steps) put(gb[(k + 1) & 1]);
    __syncthreads();
  }
  cl.sync();                                      // the rows of both halves are written
  // pairs across the middle: P[s][c] = row_s . row_c, s <= m < c
  const int na = m + 1, ncr = Lx - 1 - m;
  cxf_* tb = reinterpret_cast<cxf_*>(smem_raw);   // [W][33] rows of 32 slices c, transposed (the chain's space)
  for (int c0 = 0; c0 < ncr; c0 += 32) {
    __syncthreads();
    for (int e = tid; e < 32 * W; e += DY_THREADS) {
      const int q = e / W, x = e - q * W;
      tb[x * 33 + q] = c0 + q < ncr ? Rr[(size_t)(m + 1 + c0 + q) * W + x] : cxf_{0.f, 0.f};
    }
    __syncthreads();
    for (int s = half * DY_WARPS + wid; s < na; s += 2 * DY_WARPS) {
      cxf_ a = {0.f, 0.f}, d = {0.f, 0.f};
      const cxf_* row = Rr + (size_t)s * W;
      for (int x = 0; x < W; x += 2) {
        a = cfma(row[x], tb[x * 33 + lane], a);
        d = cfma(row[x + 1], tb[(x + 1) * 33 + lane], d);
      }
      a = a + d;
      const int c = m + 1 + c0 + lane;
      if (c < Lx) P[(size_t)s * Lx + c] = P[(size_t)c * Lx + s] = a;
    }
  }
}

// C (M x N, row stride ldc) = alpha X Y (+ D), X: M x K, Y: K x N, D: M x N, all in
// global memory in any of binary64 / complex64 (converted to complex64 on load),
// 32 x 32 tiles staged through shared memory and multiplied on the tensor cores
// (3xTF32, binary32 accuracy): warp w forms the 16 x 8 sub-tile at rows 16 (w / 4),
// columns 8 (w % 4) of each output tile.  Callers keep C apart from X, Y.  The
// output tiles are shared out over CN CTAs (this one is ci); the next k block's
// loads are in flight during a block's products.
template <typename TX, typename TY, typename TD>
__device__ void gmm_c64(cxf_* C, int ldc, const TX* X, int ldx, const TY* Y, int ldy, const TD* D, int ldd,
                        int M, int N, int K, float alpha, cxf_ (&tx)[32][32], cxf_ (&ty)[32][32], int ci, int CN) {
  auto f32 = [](auto v) -> cxf_ {
    using V = decltype(v);
    if constexpr (std::is_same_v<V, cxd>) return cxf_{d2f_bits(v.x), d2f_bits(v.y)};
    else if constexpr (std::is_same_v<V, cx<dfl>>) return cxf_{v.x.hi + v.x.lo, v.y.hi + v.y.lo};
    else return v;
  };
  static_assert(DY_THREADS == 256, "eight 16 x 8 tensor-core tiles per 32 x 32 output tile");
  const int lr = threadIdx.x >> 5, lc = threadIdx.x & 31;
  const int tm = 16 * (lr >> 2), tn = 8 * (lr & 3);
  const int nr = (M + 31) / 32, ncol = (N + 31) / 32;
  for (int tile = ci; tile < nr * ncol; tile += CN) {
    const int r0 = (tile / ncol) * 32, c0 = (tile % ncol) * 32;
    tc::CTile acc = {};
    cxf_ px[4], py[4];
    auto fetch = [&](int k0) {
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int r = lr + 8 * m;
        px[m] = (r0 + r < M && k0 + lc < K) ? f32(X[(size_t)(r0 + r) * ldx + k0 + lc]) : cxf_{0.f, 0.f};
        py[m] = (k0 + r < K && c0 + lc < N) ? f32(Y[(size_t)(k0 + r) * ldy + c0 + lc]) : cxf_{0.f, 0.f};
      }
    };
    fetch(0);
    for (int k0 = 0; k0 < K; k0 += 32) {
      __syncthreads();                     // previous tiles fully read
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        tx[lr + 8 * m][lc] = px[m];
        ty[lr + 8 * m][lc] = py[m];
      }
      __syncthreads();
      if (k0 + 32 < K) fetch(k0 + 32);
      tc::cgemm_tile_3xtf32(acc, &tx[0][0], &ty[0][0], 32, tm, tn);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      int r, c;
      tc::tile_pos(e, tm, tn, r, c);
      if (r0 + r < M && c0 + c < N) {
        cxf_ v = {alpha * acc.re[e], alpha * acc.im[e]};
        if (D) v = v + f32(D[(size_t)(r0 + r) * ldd + c0 + c]);
        C[(size_t)(r0 + r) * ldc + c0 + c] = v;
      }
    }
  }
}

// Surface Green's functions of 3D slabs (see the top of the file).  Chains are kept
// as one W x NV matrix per CTA, NV = 2 Lx T columns: [side][slice c][boundary column b]
// (side 0 top, 1 bottom), updated by one product per step into the other half of
// the ping-pong pair.  G_{s+1,s+1} and the product g_s G_{s+1,s+1} (complex64) use
// the factor's workspace, free once the factorization has run.  A unit's products
// are shared by a cluster of CTAs (as in k_factor_wide): with one CTA a unit the 64
// units of 24^3 x 16 kept 64 SMs waiting on their tiles' loads.
template <typename FT>   // the factors' element: binary64 (FP64 form) or double-float (mixed)
__global__ void __launch_bounds__(DY_THREADS, 2) k_surface_3d(Geo g, Bufs b, int K) {
  cg::cluster_group cl = cg::this_cluster();
  const int CN = (int)cl.num_blocks(), ci = (int)cl.block_rank();
  const int clu = blockIdx.x / CN, nclu = gridDim.x / CN;
  const int gt = ci * DY_THREADS + threadIdx.x, gn = CN * DY_THREADS;
  auto sync = [&]() {
    if (CN > 1) cl.sync();
    else __syncthreads();
  };
  __shared__ __align__(16) cxf_ tx[32][32];
  __shared__ __align__(16) cxf_ ty[32][32];
  const int W = g.W, Lx = g.Lx, T = g.T, A = g.A;
  const size_t n = (size_t)W * W, NV = (size_t)2 * Lx * T;
  cxf_* Gd = reinterpret_cast<cxf_*>(b.fwork + (size_t)clu * 2 * n);   // G_{s+1,s+1}
  cxf_* Tm = Gd + n;
  cxf_* Va = b.lpw + (size_t)clu * 2 * W * NV;
  cxf_* Vb = Va + (size_t)W * NV;
  const float t = d2f_bits(g.t), t2 = t * t;
  for (int unit = clu; unit < g.p * K; unit += nclu) {
    const int i = unit % g.p, f = unit / g.p, w = T * g.h[i];
    const FT* gs = reinterpret_cast<const FT*>(b.g64 ? (const void*)b.g64 : b.g) + ((size_t)f * g.p + i) * (size_t)Lx * n;
    cxf_* P[2] = {b.lpt + (((size_t)f * g.p + i) * 2 + 0) * (size_t)A * A,
                  b.lpt + (((size_t)f * g.p + i) * 2 + 1) * (size_t)A * A};
    const bool need[2] = {i < g.p - 1, i > 0};
    // boundary row / column j of slice for side sd and in-plane index b: top rows
    // (slow row h-1) and bottom rows (slow row 0); its layer index is x + Lx b
    auto bj = [&](int sd, int bb) { return sd == 0 ? w - T + bb : bb; };
    cxf_* V = Va;
    cxf_* Vn = Vb;
    for (int s = Lx - 1; s >= 0; --s) {
      const FT* g_s = gs + (size_t)s * n;
      if (s < Lx - 1) {
        // G_{s,c}[:, bnd(c)] = -t g_s G_{s+1,c}[:, bnd(c)] for every c > s, both sides
        const int c0 = (s + 1) * T, nc = (Lx - 1 - s) * T;
        for (int sd = 0; sd < 2; ++sd) {
          if (!need[sd]) continue;
          const size_t off = (size_t)sd * Lx * T + c0;
          gmm_c64(Vn + off, (int)NV, g_s, W, V + off, (int)NV, (const cxf_*)nullptr, 0, W, nc, W, -t, tx, ty, ci, CN);
        }
        sync();
        cxf_* tmp = V;
        V = Vn;
        Vn = tmp;
        // P[s][c] = rows bnd(s) of the chains, and its mirror (G is complex symmetric)
        for (int sd = 0; sd < 2; ++sd) {
          if (!need[sd]) continue;
          for (int e = gt; e < T * nc; e += gn) {
            const int ra = e / nc, q = e - ra * nc;            // row b_s, chain column (c, b_c)
            const int c = s + 1 + q / T, bc = q % T;
            const cxf_ v = V[(size_t)bj(sd, ra) * NV + (size_t)sd * Lx * T + c0 + q];
            const size_t a = (size_t)s + (size_t)Lx * ra, a2 = (size_t)c + (size_t)Lx * bc;
            P[sd][a * A + a2] = v;
            P[sd][a2 * A + a] = v;
          }
        }
      }
      // G_ss = g_s + t^2 g_s G_{s+1,s+1} g_s  (g_{Lx-1} itself at the end of the slab)
      if (s == Lx - 1) {
        for (size_t e = gt; e < n; e += gn) {
          if constexpr (std::is_same_v<FT, cxd>) Gd[e] = cxf_{d2f_bits(g_s[e].x), d2f_bits(g_s[e].y)};
          else Gd[e] = cxf_{g_s[e].x.hi + g_s[e].x.lo, g_s[e].y.hi + g_s[e].y.lo};
        }
      } else {
        gmm_c64(Tm, W, g_s, W, Gd, W, (const cxf_*)nullptr, 0, W, W, W, 1.f, tx, ty, ci, CN);
        sync();
        gmm_c64(Gd, W, Tm, W, g_s, W, g_s, W, W, W, W, t2, tx, ty, ci, CN);
      }
      sync();
      // start the chains of column c = s, and the diagonal block P[s][s]
      for (int sd = 0; sd < 2; ++sd) {
        if (!need[sd]) continue;
        for (int e = gt; e < W * T; e += gn) {
          const int r = e / T, bc = e - r * T;
          V[(size_t)r * NV + (size_t)sd * Lx * T + (size_t)s * T + bc] = Gd[(size_t)r * W + bj(sd, bc)];
        }
        for (int e = gt; e < T * T; e += gn) {
          const int ra = e / T, bc = e - ra * T;
          P[sd][((size_t)s + (size_t)Lx * ra) * A + (size_t)s + (size_t)Lx * bc] = Gd[(size_t)bj(sd, ra) * W + bj(sd, bc)];
        }
      }
      sync();
    }
  }
}

// S_ll and its inverse for layers larger than the shared-memory form takes, in
// place of P_top(l) (only line l reads it): A = S_ll, then the block form of the
// symmetric sweep operator with NB x NB pivots on the upper 64 x 64 tiles,
//   P = A_kk^-1;  F_i = A_ik P;  A_ij -= F_i A_kj;  A_ik <- F_i;  A_kk <- -P   (i, j != k),
// which leaves -A^-1 (pivots by the sweep operator on the diagonal block; Im S_ll > 0
// keeps them away from zero), and is written mirrored in the form's precision.
// F_i and the old A_ik go through P_bot(l+1)'s space (read once, while A is formed),
// k-major, so that a tile's update reads 64 consecutive entries of each.
// A rank-32 update of a 64 x 64 tile is 2 x 2 KB in and 32 KB out and back for 524 k
// FMAs: 16 bytes a clock and SM, below the HBM share, so the matrix may stream.  Each
// thread holds 4 x 4 complex accumulators in binary32 (64 FMAs for four 16-byte
// shared loads).  The CTAs of a cluster share the tiles of one matrix (as many as keep
// the grid within DY_FACTOR_CTAS): 7 x 16 matrices of 1024 x 1024 had one SM each.
constexpr int LINV_NB = 32;
template <typename R>
__global__ void __launch_bounds__(DY_THREADS, 2) k_layer_inv_g(Geo g, Bufs b) {
  constexpr int NB = LINV_NB, TU = 64;
  __shared__ __align__(16) cxf_ Pk[NB * NB];
  __shared__ __align__(16) cxf_ FO[2][NB][TU];               // F and O of a tile, k-major
  __shared__ cxf_ prow[NB], fcol[NB];
  cxf_ (*tx)[NB + 1] = reinterpret_cast<cxf_ (*)[NB + 1]>(&FO[0][0][0]);   // panel tile (before the update)
  static_assert(sizeof(cxf_) * NB * (NB + 1) <= sizeof(FO), "the panel tile shares the update tiles' space");
  cg::cluster_group cl = cg::this_cluster();
  const int CN = (int)cl.num_blocks(), ci = (int)cl.block_rank();
  auto sync = [&]() {
    if (CN > 1) cl.sync();
    else __syncthreads();
  };
  const int l = blockIdx.x / CN, f = blockIdx.y, n = g.A, lx = g.Lx;   // layer index a = x + Lx y
  const size_t n2 = (size_t)n * n;
  cxf_* A = b.lpt + (((size_t)f * g.p + l) * 2 + 0) * n2;          // P_top(l), overwritten
  cxf_* Pb = b.lpt + (((size_t)f * g.p + l + 1) * 2 + 1) * n2;     // P_bot(l+1), then F and O
  cxf_ *Ft = Pb, *Ot = Pb + (size_t)NB * n;                        // [NB][n] each
  const float t = d2f_bits(g.t), t2 = t * t;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (size_t e = (size_t)ci * DY_THREADS + tid; e < n2; e += (size_t)CN * DY_THREADS) {
    const int r = (int)(e / n), c = (int)(e - (size_t)r * n);
    cxf_ v = {0.f, 0.f};
    if (r == c) {
      const cxd d = dyson_diag(g, b, f, r + g.A * g.ylayer[l]);
      v = cxf_{d2f_bits(d.x), d2f_bits(d.y)};
    } else if (((r == c + 1 || c == r + 1) && r / lx == c / lx) || r == c + lx || c == r + lx) {
      v = cxf_{t, 0.f};                                             // in-plane neighbours along x and y
    }
    A[e] = cfma(cxf_{-t2, 0.f}, A[e] + Pb[e], v);
  }
  sync();
  const int nbk = (n + NB - 1) / NB, ntu = (n + TU - 1) / TU;
  const int ty = tid >> 4, txi = tid & 15;                          // 16 x 16 threads of a tile, 4 x 4 entries each
  for (int kb = 0; kb < nbk; ++kb) {
    const int k0 = kb * NB;
    for (int e = tid; e < NB * NB; e += DY_THREADS) {
      const int r = e / NB, c = e - r * NB;
      Pk[e] = k0 + r < n && k0 + c < n ? A[(size_t)(k0 + r) * n + k0 + c] : (r == c ? cxf_{1.f, 0.f} : cxf_{0.f, 0.f});
    }
    sweep_invert_f(Pk, NB, prow, fcol);                   // every CTA for itself
    // panel: O = A_ik (from the upper triangle), F_i = O P
    for (int q = ci; q < nbk - 1; q += CN) {
      const int ib = q < kb ? q : q + 1, i0 = ib * NB;
      __syncthreads();
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int rr = wid + 8 * m;
        if (ib < kb) tx[rr][lane] = i0 + rr < n && k0 + lane < n ? A[(size_t)(i0 + rr) * n + k0 + lane] : cxf_{0.f, 0.f};
        else tx[lane][rr] = k0 + rr < n && i0 + lane < n ? A[(size_t)(k0 + rr) * n + i0 + lane] : cxf_{0.f, 0.f};
      }
      __syncthreads();
      cxf_ acc[4] = {};
#pragma unroll 8
      for (int k = 0; k < NB; ++k) {
        const cxf_ x = tx[lane][k];
#pragma unroll
        for (int m = 0; m < 4; ++m) acc[m] = cfma(x, Pk[k * NB + wid * 4 + m], acc[m]);
      }
      if (i0 + lane < n) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          Ft[(size_t)(wid * 4 + m) * n + i0 + lane] = acc[m];
          Ot[(size_t)(wid * 4 + m) * n + i0 + lane] = tx[lane][wid * 4 + m];
        }
      }
    }
    sync();                                               // F and O complete, the old panel is not read any more
    int tile = 0;
    for (int ti = 0; ti < ntu; ++ti)
      for (int tj = ti; tj < ntu; ++tj, ++tile) {
        if (tile % CN != ci) continue;
        const int r0 = ti * TU, c0 = tj * TU, rt = r0 + ty * 4, ct = c0 + txi * 4;
        cxf_ acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int c = 0; c < 4; ++c)
            acc[a][c] = rt + a < n && ct + c < n ? A[(size_t)(rt + a) * n + ct + c] : cxf_{0.f, 0.f};
        __syncthreads();
#pragma unroll
        for (int m = 0; m < 8; ++m) {
          const int e = tid + DY_THREADS * m, k = e / TU, x = e % TU;
          FO[0][k][x] = r0 + x < n ? -Ft[(size_t)k * n + r0 + x] : cxf_{0.f, 0.f};
          FO[1][k][x] = c0 + x < n ? Ot[(size_t)k * n + c0 + x] : cxf_{0.f, 0.f};
        }
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < NB; ++k) {
          const float4* fp = reinterpret_cast<const float4*>(&FO[0][k][ty * 4]);
          const float4* op = reinterpret_cast<const float4*>(&FO[1][k][txi * 4]);
          const float4 f0 = fp[0], f1 = fp[1], o0 = op[0], o1 = op[1];
          const cxf_ fv[4] = {{f0.x, f0.y}, {f0.z, f0.w}, {f1.x, f1.y}, {f1.z, f1.w}};
          const cxf_ ov[4] = {{o0.x, o0.y}, {o0.z, o0.w}, {o1.x, o1.y}, {o1.z, o1.w}};
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[a][c] = cfma(fv[a], ov[c], acc[a][c]);
        }
        // a thread's four rows (columns) lie in one pivot block
        const bool rk = rt / NB == kb, ck = ct / NB == kb;
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int r = rt + a, cc = ct + c;
            if (r >= n || cc >= n) continue;
            cxf_ v = acc[a][c];
            if (rk && ck) v = -Pk[(r - k0) * NB + cc - k0];
            else if (ck) v = Ft[(size_t)(cc - k0) * n + r];
            else if (rk) v = Ft[(size_t)(r - k0) * n + cc];
            A[(size_t)r * n + cc] = v;
          }
      }
    sync();
  }
  cx<R>* M = reinterpret_cast<cx<R>*>(b.lpm) + ((size_t)f * (g.p - 1) + l) * n2;
  for (size_t e = (size_t)ci * DY_THREADS + tid; e < n2; e += (size_t)CN * DY_THREADS) {
    const int r = (int)(e / n), c = (int)(e - (size_t)r * n);
    const cxf_ a = r <= c ? A[e] : A[(size_t)c * n + r];
    M[e] = cx<R>{(R)-a.x, (R)-a.y};
  }
}

// S_ll = C_ll - t^2 (P_top(l) + P_bot(l+1)) and M_l^-1, symmetrised, in the form's precision.
template <typename R>
__global__ void __launch_bounds__(DY_THREADS) k_layer_inv(Geo g, Bufs b) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int l = blockIdx.x, f = blockIdx.y, Lx = g.A, lx = g.Lx, n = Lx * Lx;   // layer index a = x + lx y
  cxf_* S = reinterpret_cast<cxf_*>(smem_raw);
  cxf_* prow = S + n;
  cxf_* fcol = prow + Lx;
  const cxf_* Pt = b.lpt + (((size_t)f * g.p + l) * 2 + 0) * (size_t)n;
  const cxf_* Pb = b.lpt + (((size_t)f * g.p + l + 1) * 2 + 1) * (size_t)n;
  const float t = d2f_bits(g.t), t2 = t * t;
  for (int e = threadIdx.x; e < n; e += DY_THREADS) {
    const int r = e / Lx, c = e - r * Lx;
    cxf_ v = {0.f, 0.f};
    if (r == c) {
      const cxd d = dyson_diag(g, b, f, r + g.A * g.ylayer[l]);
      v = cxf_{d2f_bits(d.x), d2f_bits(d.y)};
    } else if (((r == c + 1 || c == r + 1) && r / lx == c / lx) || r == c + lx || c == r + lx) {
      v = cxf_{t, 0.f};                                             // in-plane neighbours along x and y
    }
    S[e] = cfma(cxf_{-t2, 0.f}, Pt[e] + Pb[e], v);
  }
  sweep_invert_f(S, Lx, prow, fcol);
  cx<R>* M = reinterpret_cast<cx<R>*>(b.lpm) + ((size_t)f * (g.p - 1) + l) * (size_t)n;
  for (int e = threadIdx.x; e < n; e += DY_THREADS) {
    const int r = e / Lx, c = e - r * Lx;
    const cxf_ a = S[e], at = S[c * Lx + r];
    const cxf_ v = {0.5f * (a.x + at.x), 0.5f * (a.y + at.y)};
    M[e] = cx<R>{(R)v.x, (R)v.y};
  }
}

}  // namespace

size_t dyson_internal_layer_inv_smem(const Geo& g) {
  if (g.A > DY_LPRE_MAXLX) return 0;                       // global-memory form
  return ((size_t)g.A * g.A + 2 * (size_t)g.A) * sizeof(cxf_);
}

cudaError_t launch_surface(const Geo& g, const Bufs& b, int K, cudaStream_t st) {
  if (!g.lpre) return cudaSuccess;
  if (g.T > 1) {                           // 3D slabs: persistent grid over (slab, frequency)
    if (!b.lpw || !b.fwork || g.W <= DY_MAXW_SMEM || g.A > DY_LPRE_MAXLX_G) return cudaErrorInvalidValue;
    const int units = g.p * K;
    const int C = unit_cluster(units);
    const int grid = C * (units < DY_FACTOR_CTAS / C ? units : DY_FACTOR_CTAS / C);
    if (b.g64) return launch_clustered(k_surface_3d<cx<dfl>>, dim3(grid), C, 0, st, g, b, K);   // mixed: double-float factors
    return launch_clustered(k_surface_3d<cxd>, dim3(grid), C, 0, st, g, b, K);
  }
  if (g.W > SURF_MAXW || g.Lx > DY_LPRE_MAXLX_G) return cudaErrorInvalidValue;
  size_t smem = (3 * (size_t)g.W * g.W + (size_t)(g.Lx / 2) * g.W) * sizeof(cxf_);
  const size_t tb = (size_t)33 * g.W * sizeof(cxf_);
  if (smem < tb) smem = tb;
  const dim3 grid(4 * g.p, K);
  if (b.g64) return launch_clustered(g.W == 32 ? k_surface_two<float, 32> : k_surface_two<float, 0>, grid, 2, smem, st, g, b);
  return launch_clustered(g.W == 32 ? k_surface_two<double, 32> : k_surface_two<double, 0>, grid, 2, smem, st, g, b);
}

template <typename R>
cudaError_t launch_layer_inv(const Geo& g, const Bufs& b, int K, cudaStream_t st) {
  if (!g.lpre) return cudaSuccess;
  if (g.A > DY_LPRE_MAXLX) {               // also: k_layer_inv_g keeps its panels in 64 A <= A^2 entries
    const int C = unit_cluster((g.p - 1) * K);
    return launch_clustered(k_layer_inv_g<R>, dim3((g.p - 1) * C, K), C, 0, st, g, b);
  }
  const size_t smem = dyson_internal_layer_inv_smem(g);
  cudaError_t e = raise_smem_limit((const void*)k_layer_inv<R>, smem);
  if (e != cudaSuccess) return e;
  k_layer_inv<R><<<dim3(g.p - 1, K), DY_THREADS, smem, st>>>(g, b);
  return cudaGetLastError();
}
template cudaError_t launch_layer_inv<float>(const Geo&, const Bufs&, int, cudaStream_t);
template cudaError_t launch_layer_inv<double>(const Geo&, const Bufs&, int, cudaStream_t);

// Subdomain factorization: diag(B^-1) and the slice factors used by every
// subdomain solve (Sec. 2.3: "the diagonal of B^-1 ... needs to be
// calculated only once at the very beginning of the Lanczos steps"; Eq. 7).
//
// One CTA per (subdomain, frequency).  B_i is block tridiagonal along x with
// slice blocks D_s (diag(H_jj) + t * in-slice hopping) and couplings t*I:
//   forward   g_s  = (D_s - t^2 g_{s-1})^-1          (left-connected inverse)
//   backward  G_ss = g_s + t^2 g_s G_{s+1,s+1} g_s
// The g_s are stored for the block forward/back substitutions; diag(G_ss) is
// diag(B^-1) on that slice.  Matrices live in shared memory (W <= 64);
// inversion is in-place Gauss-Jordan without pivoting, which is safe here
// because every pivot block has a positive-definite imaginary part
// (Im H_jj >= w_0 > 0 and -t^2 Im g_{s-1} is positive semi-definite), so
// all Schur complements stay non-singular.
#include <cooperative_groups.h>

#include <type_traits>

#include "dyson_common.cuh"

namespace cg = cooperative_groups;

namespace {

template <typename R>
__device__ __forceinline__ bool slice_adjacent(int r, int c, int T) {
  int tr_r = r % T, sl_r = r / T, tr_c = c % T, sl_c = c / T;
  if (sl_r == sl_c) return abs(tr_r - tr_c) == 1;
  return tr_r == tr_c && abs(sl_r - sl_c) == 1;
}

// In-place inverse of the complex symmetric W x W matrix A (row-major, shared)
// by the symmetric sweep operator (symmetric Gauss-Jordan): sweeping pivot k
// maps a_kk -> -1/a_kk, a_rk, a_kr -> a_rk / a_kk and the rest to
// a_rc - a_rk a_kc / a_kk, which keeps the matrix symmetric, so only the upper
// triangle is updated (W^2/2 complex FMAs per step, half of plain
// Gauss-Jordan); after all W pivots it holds -A^-1.  Step k: W threads cache
// column k unscaled in prow and scaled by the pivot inverse in fcol (with
// -1/a_kk at fcol[k]); every other entry has one owner thread.  Every block
// inverted here is complex symmetric (D_s and the g_s are), without pivoting
// because Im A is positive definite (leading minors never vanish).
template <typename R>
__device__ void gj_invert(cx<R>* A, int W, cx<R>* prow, cx<R>* fcol) {
  const int n = W * W;
  for (int k = 0; k < W; ++k) {
    __syncthreads();                         // step k-1 finished by every thread
    for (int e = threadIdx.x; e < W; e += DY_THREADS) {
      const cx<R> piv = cinv(A[k * W + k]);
      const cx<R> a = (e < k) ? A[e * W + k] : A[k * W + e];   // a_ek from the upper triangle
      prow[e] = a;
      fcol[e] = (e == k) ? -piv : a * piv;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < n; e += DY_THREADS) {
      const int r = e / W, c = e - r * W;
      if (c < r) continue;
      if (r == k || c == k) A[e] = fcol[r == k ? c : r];
      else A[e] = cfma(-fcol[r], prow[c], A[e]);
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n; e += DY_THREADS) {   // -(-A^-1), upper triangle
    const int r = e / W, c = e - r * W;
    if (c >= r) A[e] = -A[e];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n; e += DY_THREADS) {   // mirror to the lower triangle
    const int r = e / W, c = e - r * W;
    if (c < r) A[e] = A[c * W + r];
  }
  __syncthreads();
}

// C = X * Y for W x W shared matrices
template <typename R>
__device__ __forceinline__ void smem_matmul(cx<R>* C, const cx<R>* X, const cx<R>* Y, int W) {
  const int n = W * W;
  for (int e = threadIdx.x; e < n; e += DY_THREADS) {
    int r = e / W, c = e - r * W;
    cx<R> acc = {0, 0};
    const cx<R>* xr = X + r * W;
    for (int k = 0; k < W; ++k) acc = cfma(xr[k], Y[k * W + c], acc);
    C[e] = acc;
  }
}

// One CTA per (subdomain, frequency), binary64, DY_TWO_MAXW64 < W <= 64 (the other
// strips run k_factor_two): g_s left-connected for every s, stored row-major for the
// 8-warp sweeps.
template <typename R>
__global__ void __launch_bounds__(DY_THREADS) k_factor(Geo g, Bufs b) {
  using C = cx<R>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int i = blockIdx.x, kf = blockIdx.y;
  const int W = g.W, Lx = g.Lx, T = g.T, w = T * g.h[i];
  const int n = W * W;
  C* A = reinterpret_cast<C*>(smem_raw);
  C* Bm = A + n;
  C* Cm = Bm + n;
  C* prow = Cm + n;                          // Gauss-Jordan pivot row / column caches
  C* fcol = prow + W;
  C* Gprev = fcol + W;                       // [2][W] columns of the last off-diagonal block at the boundary rows
  const size_t uoff = ((size_t)kf * g.p + i) * (size_t)Lx * n;
  C* gout = reinterpret_cast<C*>(b.g) + uoff;
  cxd* dB = b.diagB + (size_t)kf * g.Ndd + (size_t)i * Lx * W;
  const R t = (R)g.t, t2 = (R)(g.t * g.t);

  // A = D_s - t^2 pa; pa may be A itself (each entry is read and written by the
  // same thread) or null
  auto form = [&](int s, const C* pa) {
    for (int e = threadIdx.x; e < n; e += DY_THREADS) {
      int r = e / W, c = e - r * W;
      C v = {0, 0};
      if (pa) v = v - t2 * pa[e];
      if (r < w && c < w) {
        if (r == c) {
          cxd d = dyson_diag(g, b, kf, sub_nat(g, i, s, r));
          v = v + cconv<R>(d);
        } else if (slice_adjacent<R>(r, c, T)) {
          v.x += t;
        }
      } else {
        v = (r == c) ? C{1, 0} : C{0, 0};
      }
      A[e] = v;
    }
  };
  // invert A in place, zero its padding and store it in slot s
  auto invert_store = [&](int s) {
    gj_invert<R>(A, W, prow, fcol);
    for (int e = threadIdx.x; e < n; e += DY_THREADS) {
      int r = e / W, c = e - r * W;
      C v = A[e];
      if (r >= w || c >= w) v = C{0, 0};
      A[e] = v;
      gout[(size_t)s * n + e] = v;
    }
    __syncthreads();
  };
  auto diag_out = [&](int s) {
    for (int r = threadIdx.x; r < W; r += DY_THREADS)
      dB[(size_t)s * W + r] = (r < w) ? cconv<double>(A[r * W + r]) : cxd{0, 0};
  };
  cxd* oB = b.offB ? b.offB + ((size_t)kf * g.p + i) * (size_t)Lx * W : nullptr;
  // distance-2 couplings on the two boundary rows (2D strips: row 0 below,
  // row w-1 above): G_{s,s2} = -t g_s G_{sn,s2} with s2 = 2 sn - s, from the
  // columns of the previous step's off-diagonal block G_{sn,s2}
  cxd* o2 = (b.off2 && T == 1) ? b.off2 + ((size_t)kf * g.p + i) * (size_t)Lx * W : nullptr;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // A <- g_s + t^2 g_s A g_s with g_s from slot s (A = G of the neighbour toward
  // the start, slice sn); -t g_s A is the off-diagonal block G_{s,sn}, whose
  // diagonal the interface preconditioner uses (stored at min(s, sn)).
  // prevc: boundary columns of G_{sn,s2} (null if s2 is outside the strip)
  auto grow_G = [&](int s, int sn, const C* prevc) {
    for (int e = threadIdx.x; e < n; e += DY_THREADS) Bm[e] = gout[(size_t)s * n + e];
    __syncthreads();
    smem_matmul<R>(Cm, Bm, A, W);
    __syncthreads();
    if (oB)
      for (int r = threadIdx.x; r < W; r += DY_THREADS)
        oB[(size_t)(s < sn ? s : sn) * W + r] = (r < w) ? cconv<double>((-t) * Cm[r * W + r]) : cxd{0, 0};
    if (o2) {
      const int s2 = 2 * sn - s;
      if (prevc && wid < 2) {                // warp jj: boundary row jj ? w-1 : 0
        const int j = wid ? w - 1 : 0;
        C acc = {0, 0};
        for (int c = lane; c < W; c += 32) acc = cfma(Bm[j * W + c], prevc[wid * W + c], acc);
        for (int off = 16; off > 0; off >>= 1) {
          acc.x += shfl_xor_any(acc.x, off);
          acc.y += shfl_xor_any(acc.y, off);
        }
        if (lane == 0) o2[(size_t)(s < s2 ? s : s2) * W + j] = cconv<double>((-t) * acc);
      }
      __syncthreads();                       // prevc read before Gprev is rewritten
      for (int e = threadIdx.x; e < 2 * W; e += DY_THREADS) {
        const int jj = e / W, c = e - jj * W, j = jj ? w - 1 : 0;
        Gprev[e] = (-t) * Cm[c * W + j];
      }
    }
    // g_s + t^2 (g_s A) g_s is complex symmetric: the upper triangle, then the mirror
    for (int e = threadIdx.x; e < n; e += DY_THREADS) {
      int r = e / W, c = e - r * W;
      if (c < r) continue;
      C acc = {0, 0};
      const C* xr = Cm + r * W;
      for (int k = 0; k < W; ++k) acc = cfma(xr[k], Bm[k * W + c], acc);
      A[e] = Bm[e] + t2 * acc;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < n; e += DY_THREADS) {
      int r = e / W, c = e - r * W;
      if (c < r) A[e] = A[c * W + r];
    }
    __syncthreads();
    diag_out(s);
  };

  for (int s = 0; s < Lx; ++s) {            // forward: A holds g_{s-1} on entry
    form(s, s > 0 ? A : nullptr);
    invert_store(s);
  }
  diag_out(Lx - 1);                          // backward: A holds G_{s+1,s+1}
  for (int s = Lx - 2; s >= 0; --s) grow_G(s, s + 1, s < Lx - 2 ? Gprev : nullptr);
  // interface part of diag(B^-1) is zero (blkdiag(B^-1, 0), Eq. 9)
  if (i == g.p - 1) {
    cxd* dI = b.diagB + (size_t)kf * g.Ndd + g.ifc_off;
    size_t m = (size_t)(g.p - 1) * g.A;
    for (size_t e = threadIdx.x; e < m; e += DY_THREADS) dI[e] = cxd{0, 0};
  }
}

// ---------------------------------------------------------------- triangle inversion
// Inverse of a complex symmetric W x W block (W <= WF) by the sweep operator (see
// gj_invert) on the upper triangle, whose entries stay in the registers of warps
// 1..7 (thread t of them owns triangle entries t, t + 224, ...).  Warp 0 runs one pivot
// ahead: while the others apply pivot k it brings column k + 1 up to date itself,
// inverts pivot k + 1 and scales the column, so a pivot costs one barrier and the
// longer of the two (~650 cycles at W = 32 in double-float) instead of their sum
// (2250).  Every product is renormalised as it is added: sums without it, 48
// operations a term instead of 60, made the diagonal's error 1.2 to 1.4 times as large.
template <typename R>
struct TriSmem {
  cx<R>*prow, *fcol, *craw;                  // [2][W] each: the pivot's column, scaled by the inverse
                                             // pivot, and the column after it (one pivot behind)
};
template <int WF>
struct Tri {
  static constexpr int OWN = DY_THREADS - 32;
  static constexpr int NE = (WF * (WF + 1) / 2 + OWN - 1) / OWN;                 // triangle entries an owner holds
  static constexpr int NP = (WF * (WF + 1) / 2 + DY_THREADS - 1) / DY_THREADS;   // and a thread of all of them
};
// triangle entry number e (rows of length W, W - 1, ...) as (r, c), r <= c; false, (0, 0) past the end
__device__ __forceinline__ bool tri_entry(int e, int W, int& r, int& c) {
  r = 0;
  const bool on = e < W * (W + 1) / 2;
  while (on && e >= W - r) {
    e -= W - r;
    ++r;
  }
  c = on ? r + e : 0;
  return on;
}

// 1 / z: in double-float one Newton step from the binary32 reciprocal of |z|^2, with
// its square term (the start is off by at most 2^-24, so the result by ~2^-70 before
// rounding)
template <typename R>
__device__ __forceinline__ cx<R> inv_fast(const cx<R>& z) {
  if constexpr (std::is_same<R, dfl>::value) {
    dfl d = dfl(0.f, 0.f);
    dfl_mac(d, z.x, z.x);
    dfl_mac(d, z.y, z.y);
    d = dfl_fast(d.hi, d.lo);
    const float r0 = __frcp_rn(d.hi);
    const float e = __fmaf_rn(-d.lo, r0, __fmaf_rn(-d.hi, r0, 1.f));
    const dfl r = dfl_fast(r0, r0 * __fmaf_rn(e, e, e));
    const dfl im = z.y * r;
    return {z.x * r, dfl(-im.hi, -im.lo)};
  } else {
    return cinv(z);
  }
}

// from(r, c) (r <= c) gives the block's entries, to(r, c, v) takes the inverse's; from
// is not called after the first barrier, to not before the last one (the caller syncs
// before the results are read).  er, ec, eon: this thread's entries (tri_entry of
// tid - 32 + OWN q for warps 1..7).
template <typename R, int WF, typename From, typename To>
__device__ __forceinline__ void tri_invert(int W, const TriSmem<R>& ts, const int (&er)[Tri<WF>::NE],
                                           const int (&ec)[Tri<WF>::NE], unsigned eon, From from, To to) {
  using C = cx<R>;
  constexpr int NE = Tri<WF>::NE;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  C v[NE];
#pragma unroll
  for (int q = 0; q < NE; ++q) v[q] = wid > 0 ? from(er[q], ec[q]) : C{0, 0};
  if (wid == 0) {
    for (int e = lane; e < W; e += 32) {
      ts.prow[e] = from(0, e);
      if (W > 1) ts.craw[W + e] = from(e < 1 ? e : 1, e < 1 ? 1 : e);       // column 1
    }
    __syncwarp();
    const C piv = inv_fast<R>(ts.prow[0]);
    for (int e = lane; e < W; e += 32) ts.fcol[e] = e == 0 ? -piv : ts.prow[e] * piv;
  }
  for (int k = 0; k < W; ++k) {
    const C *pk = ts.prow + (k & 1) * W, *fk = ts.fcol + (k & 1) * W, *cr = ts.craw + ((k + 1) & 1) * W;
    C *pn = ts.prow + ((k + 1) & 1) * W, *fn = ts.fcol + ((k + 1) & 1) * W, *cn = ts.craw + (k & 1) * W;
    __syncthreads();                         // pk, fk and column k + 1 as of pivot k - 1 are complete
    if (wid == 0) {
      if (k + 1 < W) {
        const C p1 = pk[k + 1], f1 = fk[k + 1];
        for (int e = lane; e < W; e += 32) {
          // the same product the entry's owner forms (f of the row, p of the column)
          const bool up = e <= k + 1;
          C x = cfma(up ? -fk[e] : -f1, up ? p1 : pk[e], cr[e]);
          if (e == k) x = f1;
          pn[e] = x;
        }
        __syncwarp();
        const C piv = inv_fast<R>(pn[k + 1]);
        for (int e = lane; e < W; e += 32) {
          const C x = pn[e] * piv;
          fn[e] = e == k + 1 ? -piv : x;
        }
      }
    } else {
#pragma unroll
      for (int q = 0; q < NE; ++q) {
        const int r = er[q], c = ec[q];
        const C f = fk[r], x = fk[r == k ? c : r];
        const C u = cfma(-f, pk[c], v[q]);
        v[q] = r == k || c == k ? x : u;
      }
#pragma unroll
      for (int q = 0; q < NE; ++q) {         // column k + 2 for the pivot warp
        if (!(eon >> q & 1)) continue;
        if (er[q] == k + 2) cn[ec[q]] = v[q];
        else if (ec[q] == k + 2) cn[er[q]] = v[q];
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NE; ++q)               // -(-A^-1)
    if (eon >> q & 1) to(er[q], ec[q], -v[q]);
}

// ---------------------------------------------------------------- two-sided
// The recursion from both ends, so that the sweeps can run two chains at once: the
// mixed form for W <= 64 (R = dfl), the FP64 form for W <= DY_TWO_MAXW64 (binary64).  With m = Lx / 2:
//   left   g_s = (D_s - t^2 g_{s-1})^-1            s < m
//   right  g_s = (D_s - t^2 g_{s+1})^-1            s > m
//   middle G_mm = (D_m - t^2 g_{m-1} - t^2 g_{m+1})^-1
//   G_ss = g_s + t^2 g_s G_{s+1,s+1} g_s  (s < m),  g_s + t^2 g_s G_{s-1,s-1} g_s  (s > m)
// Slot s holds g_s, or G_mm for s = m.  FP64 form: in b.g.  Mixed form: in double-float
// in b.g64, and in complex64 in b.g with column pairs interleaved (entry (r, c) at
// ((c / 2) W + r) 2 + c % 2, so that a lane reads columns 2k, 2k+1 of its row as one
// 16-byte word).
// One cluster of two CTAs per (subdomain, frequency): CTA 0 the left chain, CTA 1 the
// right one, which meet at the middle block (each inverts it for itself) and go back
// separately.  One CTA running both chains in turn took 65 us a slice at W = 28 with
// 21 x 4 units on 152 SMs.

template <typename R, int WF>
__global__ void __launch_bounds__(DY_THREADS, WF <= 32 ? 2 : 1) k_factor_two(Geo g, Bufs b) {
  using cxl = cx<R>;                         // 16 bytes in either arithmetic
  constexpr bool mixed = std::is_same<R, dfl>::value;
  constexpr int NE = Tri<WF>::NE, NP = Tri<WF>::NP, OWN = Tri<WF>::OWN;
  constexpr int NB = (WF * WF + DY_THREADS - 1) / DY_THREADS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cg::cluster_group cl = cg::this_cluster();
  const int side = (int)cl.block_rank(), i = blockIdx.x / 2, kf = blockIdx.y;
  const int W = g.W, Lx = g.Lx, T = g.T, w = T * g.h[i], n = W * W, m = Lx / 2, ntri = W * (W + 1) / 2;
  cxl* A = reinterpret_cast<cxl*>(smem_raw);
  cxl* Bm = A + n;
  cxl* Cm = Bm + n;
  const TriSmem<R> ts = {Cm + n, Cm + n + 2 * W, Cm + n + 4 * W};
  cxl* dg = Cm + n + 6 * W;                    // [W] H_ii of the slice being formed
  cxl* Gprev = dg + W;                       // [2][W] columns of the last off-diagonal block at the boundary rows
  cxl* Gmid = Gprev + 2 * W;                 // [2][W] rows of G_{m+1,m} at the boundary rows (left CTA's copy is used)
  const size_t uoff = ((size_t)kf * g.p + i) * (size_t)Lx * n;
  cxl* gout = reinterpret_cast<cxl*>(mixed ? (void*)b.g64 : b.g) + uoff;
  cxf* gsw = reinterpret_cast<cxf*>(b.g) + uoff;
  cxd* dB = b.diagB + (size_t)kf * g.Ndd + (size_t)i * Lx * W;
  const cxd* hd = b.hdiag + (size_t)kf * g.Ndd + (size_t)i * Lx * W;
  // off-diagonal blocks: for the banded preconditioner only
  cxd* oB = b.offB ? b.offB + ((size_t)kf * g.p + i) * (size_t)Lx * W : nullptr;
  cxd* o2 = b.off2 && T == 1 ? b.off2 + ((size_t)kf * g.p + i) * (size_t)Lx * W : nullptr;
  const R t = (R)g.t, t2 = (R)(g.t * g.t);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;

  int er[NE], ec[NE], pr[NP], pc[NP];
  unsigned eon = 0, pon = 0;                 // bit q: entry q exists
#pragma unroll
  for (int q = 0; q < NE; ++q)
    if (tri_entry(wid > 0 ? tid - 32 + OWN * q : ntri, W, er[q], ec[q])) eon |= 1u << q;
#pragma unroll
  for (int q = 0; q < NP; ++q)
    if (tri_entry(tid + DY_THREADS * q, W, pr[q], pc[q])) pon |= 1u << q;

  // H_ii of row tid of slice s (tid < W): from the DD-layout copy in the mixed form
  auto diag_of = [&](int s) -> cxl {
    if constexpr (mixed) {
      return cconv<R>(hd[(size_t)s * W + tid]);
    } else {
      return tid < w ? dyson_diag(g, b, kf, sub_nat(g, i, s, tid)) : cxl{0, 0};
    }
  };
  // A <- (D_s - t^2 (pa + pb))^-1, zero on the padding; pa, pb (full W x W, either may be
  // null) may be A itself; stored in slot s when keep.  dg holds slice s's diagonal;
  // slice sn's (if >= 0) is fetched for the next call.
  auto invert = [&](int s, const cxl* pa, const cxl* pb, bool keep, int sn) {
    cxl hn = {0, 0};
    if (sn >= 0 && tid < W) hn = diag_of(sn);
    tri_invert<R, WF>(
        W, ts, er, ec, eon,
        [&](int r, int c) -> cxl {
          const int e = r * W + c;
          cxl x = {0, 0};
          if (pa) x = x - t2 * pa[e];
          if (pb) x = x - t2 * pb[e];
          if (r < w && c < w) {
            if (r == c) x = x + dg[r];
            else if (slice_adjacent<R>(r, c, T)) x.x += t;
          } else {
            x = r == c ? cxl{1, 0} : cxl{0, 0};
          }
          return x;
        },
        [&](int r, int c, const cxl& v) {
          const cxl x = c < w ? v : cxl{0, 0};
          A[r * W + c] = x;
          A[c * W + r] = x;
        });
    if (sn >= 0 && tid < W) dg[tid] = hn;
    __syncthreads();
    if (keep)
      for (int e = tid; e < n; e += DY_THREADS) {
        const int r = e / W, c = e - r * W;
        const cxl x = A[e];
        gout[(size_t)s * n + e] = x;
        if constexpr (mixed) gsw[(size_t)s * n + ((size_t)(c >> 1) * W + r) * 2 + (c & 1)] = cconv<float>(x);
      }
  };
  // the layer preconditioner's input: columns w - 1 and 0 of G_ss (k_surface_two)
  cxf* bc = b.lpg ? b.lpg + ((size_t)kf * g.p + i) * lpg_entries(g) : nullptr;
  auto diag_out = [&](int s) {
    for (int r = tid; r < W; r += DY_THREADS) dB[(size_t)s * W + r] = (r < w) ? cconv<double>(A[r * W + r]) : cxd{0, 0};
    if (bc)
      for (int e = tid; e < 2 * W; e += DY_THREADS) {
        const int sd = e / W, r = e - sd * W;
        bc[((size_t)s * 2 + sd) * W + r] = cconv<float>(A[r * W + (sd == 0 ? w - 1 : 0)]);
      }
  };
  cxl nb[NB];                                // the next slice's factor on its way to Bm
  auto fetch = [&](int s) {
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int e = tid + DY_THREADS * q;
      nb[q] = e < n ? gout[(size_t)s * n + e] : cxl{0, 0};
    }
  };
  // A <- g_s + t^2 g_s A g_s with g_s from nb, A = G of the neighbour towards the
  // middle, slice sn; -t g_s A is the off-diagonal block G_{s,sn}, whose diagonal (and,
  // through the boundary columns prevc of G_{sn,s2}, s2 = 2 sn - s, the distance-2
  // couplings on the two boundary rows) the banded preconditioner uses.  mid: also put
  // the boundary rows of G_{s,sn} into the left CTA's Gmid.  nx: the next slice (or -1).
  auto grow = [&](int s, int sn, const cxl* prevc, bool mid, int nx) {
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int e = tid + DY_THREADS * q;
      if (e < n) Bm[e] = nb[q];
    }
    __syncthreads();
    if (nx >= 0) fetch(nx);
    // Cm = g_s A, 2 x 2 entries a thread: rows r, r + W/2, columns c, c + W/2
    const int h = W / 2;
    for (int e = tid; e < h * h; e += DY_THREADS) {
      const int r = e / h, c = e - r * h;
      const cxl *x0 = Bm + r * W, *x1 = x0 + h * W, *y = A + c;
      cxl a00 = {0, 0}, a01 = {0, 0}, a10 = {0, 0}, a11 = {0, 0};
      for (int k0 = 0; k0 < W; k0 += 2) {
#pragma unroll
        for (int k = k0; k < k0 + 2; ++k) {
          const cxl xa = x0[k], xb = x1[k], ya = y[k * W], yb = y[k * W + h];
          a00 = cfma(xa, ya, a00);
          a01 = cfma(xa, yb, a01);
          a10 = cfma(xb, ya, a10);
          a11 = cfma(xb, yb, a11);
        }
      }
      Cm[r * W + c] = a00;
      Cm[r * W + c + h] = a01;
      Cm[(r + h) * W + c] = a10;
      Cm[(r + h) * W + c + h] = a11;
    }
    __syncthreads();
    if (oB)
      for (int r = tid; r < W; r += DY_THREADS)
        oB[(size_t)(s < sn ? s : sn) * W + r] = (r < w) ? cconv<double>((-t) * Cm[r * W + r]) : cxd{0, 0};
    if (o2) {
      const int s2 = 2 * sn - s;
      if (prevc && wid < 2) {                // warp jj: boundary row jj ? w-1 : 0
        const int j = wid ? w - 1 : 0;
        cxl acc = {0, 0};
        for (int c = lane; c < W; c += 32) acc = cfma(Bm[j * W + c], prevc[wid * W + c], acc);
        for (int off = 16; off > 0; off >>= 1) {
          acc.x += shfl_xor_any(acc.x, off);
          acc.y += shfl_xor_any(acc.y, off);
        }
        if (lane == 0) o2[(size_t)(s < s2 ? s : s2) * W + j] = cconv<double>((-t) * acc);
      }
      __syncthreads();                       // prevc read before Gprev is rewritten
      cxl* other = cl.map_shared_rank(Gmid, 0);
      for (int e = tid; e < 2 * W; e += DY_THREADS) {
        const int jj = e / W, c = e - jj * W, j = jj ? w - 1 : 0;
        Gprev[e] = (-t) * Cm[c * W + j];
        if (mid) other[e] = (-t) * Cm[j * W + c];
      }
    }
    // g_s + t^2 (g_s A) g_s on the upper triangle, mirrored; a warp without a last entry
    // leaves it out
    auto last = [&](auto nq) {
      constexpr int NQ = decltype(nq)::value;
      cxl v[NQ > 0 ? NQ : 1];
#pragma unroll
      for (int q = 0; q < NQ; ++q) v[q] = cxl{0, 0};
      for (int k0 = 0; k0 < W; k0 += 2) {
#pragma unroll
        for (int k = k0; k < k0 + 2; ++k)
#pragma unroll
          for (int q = 0; q < NQ; ++q) v[q] = cfma(Cm[pr[q] * W + k], Bm[k * W + pc[q]], v[q]);
      }
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        if (!(pon >> q & 1)) continue;
        const int r = pr[q], c = pc[q];
        const cxl x = Bm[r * W + c] + t2 * v[q];
        A[r * W + c] = x;
        A[c * W + r] = x;
      }
    };
    if (NP > 1 && wid * 32 + DY_THREADS * (NP - 1) >= ntri) last(std::integral_constant<int, NP - 1>{});
    else last(std::integral_constant<int, NP>{});
    __syncthreads();
    diag_out(s);
  };

  if (tid < W) dg[tid] = diag_of(side == 0 ? 0 : Lx - 1);
  __syncthreads();
  if (side == 0) {
    for (int s = 0; s < m; ++s) invert(s, s > 0 ? A : nullptr, nullptr, true, s + 1);
  } else {
    for (int s = Lx - 1; s > m; --s) invert(s, s < Lx - 1 ? A : nullptr, nullptr, true, s - 1);
  }
  cl.sync();                                 // both neighbours of the middle slice are stored
  invert(m, m > 0 ? gout + (size_t)(m - 1) * n : nullptr, m < Lx - 1 ? gout + (size_t)(m + 1) * n : nullptr,
         side == 0, -1);
  if (side == 0) diag_out(m);
  if (side == 1 && m + 1 < Lx) {
    fetch(m + 1);
    __syncthreads();
    grow(m + 1, m, nullptr, true, m + 2 < Lx ? m + 2 : -1);
  }
  cl.sync();                                 // Gmid is in the left CTA's shared memory
  if (side == 1) {
    for (int s = m + 2; s < Lx; ++s) grow(s, s - 1, Gprev, false, s + 1 < Lx ? s + 1 : -1);
  } else if (m > 0) {
    fetch(m - 1);
    for (int s = m - 1; s >= 0; --s) grow(s, s + 1, s < m - 1 ? Gprev : (m + 1 < Lx ? Gmid : nullptr), false, s - 1);
  }
  // interface part of diag(B^-1) is zero (blkdiag(B^-1, 0), Eq. 9)
  if (i == g.p - 1 && side == 0) {
    cxd* dI = b.diagB + (size_t)kf * g.Ndd + g.ifc_off;
    const size_t mi = (size_t)(g.p - 1) * g.A;
    for (size_t e = tid; e < mi; e += DY_THREADS) dI[e] = cxd{0, 0};
  }
}

// ---------------------------------------------------------------- wide slices
// W > 64 (3D slabs, wide strips, one subdomain): a W x W block no longer fits
// shared memory.  The same recursion runs on global memory, which at these sizes
// stays in L2, as products of 32 x 32 tiles: the inverse g_s by the block form of
// the symmetric sweep operator (gj_invert with 32 x 32 pivots: the pivot block
// inverted in shared memory, the row panel, a rank-32 update of the upper tiles),
// the backward pass as two W x W products.
//
// A (subdomain, frequency) unit is worked on by a cluster of C CTAs that share the
// tiles of every phase (wide_cluster): 32 units of 128 x 128 blocks (128 x 128 sites,
// p = 1) left 120 of the 152 SMs idle with one CTA each, and 128 unblocked pivots
// with two barriers each took most of 3.9 ms a slice; now 0.44 ms.
constexpr int TB = 32, TP = 33;          // tile edge and padded row length in shared memory

template <typename R>
__device__ __forceinline__ cx<R> mac(cx<R> a, cx<R> b, cx<R> acc) {
  if constexpr (sizeof(R) == sizeof(double) && !std::is_same<R, dfl>::value) {
    return cfma(a, b, acc);
  } else {
    // products by TwoProduct, sums by TwoSum, the low words not renormalised (see tile_done)
    dfl_mac(acc.x, a.x, b.x);
    dfl_mac(acc.x, dfl(-a.y.hi, -a.y.lo), b.y);
    dfl_mac(acc.y, a.x, b.y);
    dfl_mac(acc.y, a.y, b.x);
    return acc;
  }
}
template <typename R>
__device__ __forceinline__ cx<R> tile_done(cx<R> v) {
  if constexpr (std::is_same<R, dfl>::value) return {dfl_fast(v.x.hi, v.x.lo), dfl_fast(v.y.hi, v.y.lo)};
  else return v;
}

template <typename R>
struct TileSmem {
  cx<R> tx[TB][TP], ty[TB][TP], tp[TB][TP];
  cx<R> tri[6 * TB];
};

// tile (r0, c0) of the row-major ld-wide matrix M (n x n; identity outside) to t, or
// its transpose
template <typename R, bool TR>
__device__ __forceinline__ void tile_in(cx<R> (*t)[TP], const cx<R>* M, int n, int ld, int r0, int c0) {
  const int lc = threadIdx.x & 31, lr = threadIdx.x >> 5;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int r = lr + 8 * m, gr = r0 + r, gc = c0 + lc;
    const cx<R> v = gr < n && gc < n ? M[(size_t)gr * ld + gc] : (gr == gc ? cx<R>{1, 0} : cx<R>{0, 0});
    if (TR) t[lc][r] = v;
    else t[r][lc] = v;
  }
}
// acc[m] += sum_k tx[lr + 8 m][k] ty[k][lc], renormalised every KR terms (the low
// words stay small: without it the diagonal of 128 x 128 blocks lost a bit)
template <typename R>
__device__ __forceinline__ void tile_mac(const cx<R> (*tx)[TP], const cx<R> (*ty)[TP], cx<R> (&acc)[4]) {
  const int lc = threadIdx.x & 31, lr = threadIdx.x >> 5;
  constexpr int KR = 4;
#pragma unroll 1
  for (int k0 = 0; k0 < TB; k0 += KR) {
#pragma unroll
    for (int k = k0; k < k0 + KR; ++k) {
      const cx<R> y = ty[k][lc];
#pragma unroll
      for (int m = 0; m < 4; ++m) acc[m] = mac<R>(tx[lr + 8 * m][k], y, acc[m]);
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) acc[m] = tile_done<R>(acc[m]);
  }
}

// R: the recursion's arithmetic, binary64 (FP64 form) or double-float (mixed
// form, on the FP32 pipe), stored in b.g (FP64 form) or b.g64 (mixed: the
// double-float factors, beside their complex64 copy in b.g for the sweeps).
template <typename R, typename S>
__global__ void __launch_bounds__(DY_THREADS, 2) k_factor_wide(Geo g, Bufs b, int K) {
  using C = cx<R>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TileSmem<R>& sm = *reinterpret_cast<TileSmem<R>*>(smem_raw);
  cg::cluster_group cl = cg::this_cluster();
  constexpr bool two = sizeof(S) != sizeof(double);
  static_assert(sizeof(C) == sizeof(cxd), "factor storage holds 16 bytes per entry");
  const int CN = (int)cl.num_blocks(), ci = (int)cl.block_rank();
  const int clu = blockIdx.x / CN, nclu = gridDim.x / CN;
  const int W = g.W, Lx = g.Lx, T = g.T, nt = (W + TB - 1) / TB;
  const size_t n = (size_t)W * W;
  const R t = (R)g.t, t2 = (R)(g.t * g.t);
  C* Gw = reinterpret_cast<C*>(b.fwork) + (size_t)clu * CN * 2 * n;     // G_{s+1,s+1}
  C* Pw = Gw + n;                        // g_s G_{s+1,s+1}
  // During the forward pass the space of Gw and Pw holds the panels (2 nt 32^2 <= 2 W^2
  // entries from W = 65 on; more than the W^2 of Pw alone up to W = 76).
  C* Fb = Gw;                            // [nt][32][32] F_i = A_ik A_kk^-1
  C* Ob = Gw + (size_t)nt * TB * TB;     // [nt][32][32] A_ik before
  const int lc = threadIdx.x & 31, lr = threadIdx.x >> 5;
  const int gt = ci * DY_THREADS + threadIdx.x, gn = CN * DY_THREADS;
  const TriSmem<R> ts = {sm.tri, sm.tri + 2 * TB, sm.tri + 4 * TB};
  int er[Tri<TB>::NE], ec[Tri<TB>::NE];
  unsigned eon = 0;
#pragma unroll
  for (int q = 0; q < Tri<TB>::NE; ++q)
    if (tri_entry(threadIdx.x >= 32 ? (int)threadIdx.x - 32 + Tri<TB>::OWN * q : TB * TB, TB, er[q], ec[q])) eon |= 1u << q;
  auto sync = [&]() {
    if (CN > 1) cl.sync();
    else __syncthreads();
  };
  for (int unit = clu; unit < g.p * K; unit += nclu) {
    const int i = unit % g.p, kf = unit / g.p, w = T * g.h[i];
    const size_t uoff = ((size_t)kf * g.p + i) * (size_t)Lx * n;
    C* gout = reinterpret_cast<C*>(two ? b.g64 : b.g) + uoff;
    cx<S>* gsw = reinterpret_cast<cx<S>*>(b.g) + uoff;
    cxd* dB = b.diagB + (size_t)kf * g.Ndd + (size_t)i * Lx * W;
    // ---- forward: g_s = (D_s - t^2 g_{s-1})^-1, formed and inverted in place
    for (int s = 0; s < Lx; ++s) {
      C* A = gout + (size_t)s * n;
      const C* Ap = A - n;
      for (int e = gt; e < (int)n; e += gn) {
        const int r = e / W, c = e - r * W;
        C v = {0, 0};
        if (r < w && c < w) {
          if (s > 0) v = (-t2) * Ap[e];
          if (r == c) {
            v = v + cconv<R>(dyson_diag(g, b, kf, sub_nat(g, i, s, r)));
          } else if (slice_adjacent<R>(r, c, T)) {
            v.x += t;
          }
        } else if (r == c) {
          v = C{1, 0};                   // padding: identity, inverted to itself
        }
        A[e] = v;
      }
      sync();
      for (int k = 0; k < nt; ++k) {
        // pivot block, by every CTA for itself
        tile_in<R, false>(sm.tp, A, W, W, k * TB, k * TB);
        __syncthreads();
        tri_invert<R, TB>(
            TB, ts, er, ec, eon, [&](int r, int c) -> C { return sm.tp[r][c]; },
            [&](int r, int c, const C& v) {
              sm.tp[r][c] = v;
              sm.tp[c][r] = v;
            });
        __syncthreads();
        // panel F_i = A_ik A_kk^-1 (kept beside the old A_ik for the update)
        for (int q = ci; q < nt - 1; q += CN) {
          const int ii = q < k ? q : q + 1;
          if (ii < k) tile_in<R, false>(sm.tx, A, W, W, ii * TB, k * TB);
          else tile_in<R, true>(sm.tx, A, W, W, k * TB, ii * TB);
          __syncthreads();
          C acc[4] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
          tile_mac<R>(sm.tx, sm.tp, acc);
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const int r = lr + 8 * m;
            const C v = tile_done<R>(acc[m]);
            Fb[((size_t)ii * TB + r) * TB + lc] = v;
            Ob[((size_t)ii * TB + r) * TB + lc] = sm.tx[r][lc];
          }
          __syncthreads();
        }
        sync();                          // panels complete, nobody reads A_.k any more
        // A_ij -= F_i A_kj on the upper tiles, and the new row and column k
        int tile = 0;
        for (int ii = 0; ii < nt; ++ii) {
          for (int jj = ii; jj < nt; ++jj, ++tile) {
            if (tile % CN != ci) continue;
            const int r0 = ii * TB, c0 = jj * TB;
            if (ii == k || jj == k) {
              const int o = ii == k ? jj : ii;
#pragma unroll
              for (int m = 0; m < 4; ++m) {
                const int r = lr + 8 * m;
                if (r0 + r < W && c0 + lc < W) {
                  C v;
                  if (ii == jj) v = -sm.tp[r][lc];
                  else if (jj == k) v = Fb[((size_t)o * TB + r) * TB + lc];
                  else v = Fb[((size_t)o * TB + lc) * TB + r];      // row k: F_j transposed
                  A[(size_t)(r0 + r) * W + c0 + lc] = v;
                }
              }
              continue;
            }
            tile_in<R, false>(sm.tx, Fb + (size_t)ii * TB * TB, TB, TB, 0, 0);
            tile_in<R, true>(sm.ty, Ob + (size_t)jj * TB * TB, TB, TB, 0, 0);
            __syncthreads();
            C acc[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
              const int r = r0 + lr + 8 * m, c = c0 + lc;
              // double-float: the products summed first (the smaller error), binary64: from A_ij
              const bool from = !std::is_same<R, dfl>::value && r < W && c < W;
              acc[m] = from ? -A[(size_t)r * W + c] : C{0, 0};
            }
            tile_mac<R>(sm.tx, sm.ty, acc);
#pragma unroll
            for (int m = 0; m < 4; ++m) {
              const int r = r0 + lr + 8 * m, c = c0 + lc;
              if (r < W && c < W) {
                C* d = A + (size_t)r * W + c;
                *d = std::is_same<R, dfl>::value ? *d - acc[m] : -acc[m];
              }
            }
            __syncthreads();
          }
        }
        sync();
      }
      // -(-A^-1), mirrored from the upper triangle, zero on the padding
      for (int e = gt; e < (int)n; e += gn) {
        const int r = e / W, c = e - r * W;
        if (c < r) continue;
        C v = -A[e];
        if (r >= w || c >= w) v = C{0, 0};
        const size_t e2 = (size_t)c * W + r;
        A[e] = v;
        A[e2] = v;
        if (two) {
          const cx<S> vs = cconv<S>(v);
          gsw[(size_t)s * n + e] = vs;
          gsw[(size_t)s * n + e2] = vs;
        }
      }
      sync();
    }
    // ---- backward: Gw holds G_{s+1,s+1}
    const C* glast = gout + (size_t)(Lx - 1) * n;
    for (int e = gt; e < (int)n; e += gn) Gw[e] = glast[e];
    for (int r = gt; r < W; r += gn)
      dB[(size_t)(Lx - 1) * W + r] = (r < w) ? cconv<double>(glast[(size_t)r * W + r]) : cxd{0, 0};
    sync();
    // out = X Y on this CTA's tiles, the tiles' k range staged one 32-block at a time with
    // the next block's loads in flight
    auto product = [&](const C* X, const C* Y, int r0, int c0, C (&acc)[4]) {
      C px[4], py[4];
      auto fetch = [&](int k0) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int r = lr + 8 * m;
          px[m] = (r0 + r < W && k0 + lc < W) ? X[(size_t)(r0 + r) * W + k0 + lc] : C{0, 0};
          py[m] = (k0 + r < W && c0 + lc < W) ? Y[(size_t)(k0 + r) * W + c0 + lc] : C{0, 0};
        }
      };
      fetch(0);
      for (int k0 = 0; k0 < W; k0 += TB) {
        __syncthreads();
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          sm.tx[lr + 8 * m][lc] = px[m];
          sm.ty[lr + 8 * m][lc] = py[m];
        }
        __syncthreads();
        if (k0 + TB < W) fetch(k0 + TB);
        tile_mac<R>(sm.tx, sm.ty, acc);
      }
    };
    for (int s = Lx - 2; s >= 0; --s) {
      const C* gs = gout + (size_t)s * n;
      for (int tile = ci; tile < nt * nt; tile += CN) {       // P = g_s G_{s+1}
        const int r0 = (tile / nt) * TB, c0 = (tile % nt) * TB;
        C acc[4] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
        product(gs, Gw, r0, c0, acc);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int r = r0 + lr + 8 * m, c = c0 + lc;
          if (r >= W || c >= W) continue;
          const C v = tile_done<R>(acc[m]);
          Pw[(size_t)r * W + c] = v;
          if (r == c && b.offB)                               // diag of G_{s,s+1} = -t g_s G_{s+1}
            b.offB[((size_t)kf * g.p + i) * (size_t)Lx * W + (size_t)s * W + r] =
                (r < w) ? cconv<double>((-t) * v) : cxd{0, 0};
        }
      }
      sync();
      int tile = 0;
      for (int ii = 0; ii < nt; ++ii) {                       // G_ss = g_s + t^2 P g_s, upper tiles
        for (int jj = ii; jj < nt; ++jj, ++tile) {
          if (tile % CN != ci) continue;
          const int r0 = ii * TB, c0 = jj * TB;
          C acc[4] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
          product(Pw, gs, r0, c0, acc);
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const int r = r0 + lr + 8 * m, c = c0 + lc;
            if (r >= W || c >= W) continue;
            const C v = gs[(size_t)r * W + c] + t2 * tile_done<R>(acc[m]);
            Gw[(size_t)r * W + c] = v;
            if (ii != jj) Gw[(size_t)c * W + r] = v;
            if (r == c) dB[(size_t)s * W + r] = (r < w) ? cconv<double>(v) : cxd{0, 0};
          }
        }
      }
      sync();
    }
    if (i == g.p - 1) {
      cxd* dI = b.diagB + (size_t)kf * g.Ndd + g.ifc_off;
      const size_t m = (size_t)(g.p - 1) * g.A;
      for (size_t e = gt; e < m; e += gn) dI[e] = cxd{0, 0};
    }
    sync();                              // workspace reads done before the next unit
  }
}

// Banded preconditioner of the interface Schur system.  The Schur complement
// S = C - E^T B^-1 E (Eq. 4) is never formed; its cheap approximation keeps,
// on each x line of interface layer l, the entries of S_ll within two sites
// along x (one in 3D slabs), which need only the diagonal, first and second
// off-diagonal blocks of B^-1 on the rows next to the layer, all from the
// factorization:
//   M[x][x]   = d_C(x) - t^2 (G_{x,x}^{l,top}   + G_{x,x}^{l+1,bot})
//   M[x][x+1] = t      - t^2 (G_{x,x+1}^{l,top} + G_{x,x+1}^{l+1,bot})
//   M[x][x+2] =        - t^2 (G_{x,x+2}^{l,top} + G_{x,x+2}^{l+1,bot})
// (in 3D the in-plane y hopping is dropped).  At the lowest Matsubara frequency
// of the 128^2 workload COCG needs 16 iterations to 1e-5 with the diagonal
// correction alone, 9 with the first off-diagonal and 6 with both.  Factors
// per x line, M = L D L^T without conjugation, computed in FP64 and stored in
// precision R: 1/d_x, l1_x, l2_x.
template <typename R>
__global__ void __launch_bounds__(DY_THREADS) k_precond(Geo g, Bufs b) {
  const int l = blockIdx.x, kf = blockIdx.y;
  const int Lx = g.Lx, T = g.T, A = g.A, W = g.W;
  const cxd* dB = b.diagB + (size_t)kf * g.Ndd;
  const size_t nsub = (size_t)Lx * W;
  const cxd* oB = b.offB + (size_t)kf * g.p * nsub;
  const cxd* o2 = (g.penta && b.off2) ? b.off2 + (size_t)kf * g.p * nsub : nullptr;
  cx<R>* pre = reinterpret_cast<cx<R>*>(b.pre) + ((size_t)kf * nifc(g) + (size_t)l * A) * 3;
  const double t = g.t, t2 = g.t * g.t;
  const cxd zero = {0, 0};
  for (int tr = threadIdx.x; tr < T; tr += DY_THREADS) {
    // row just below the layer: top row of subdomain l; just above: bottom row of l+1
    const size_t jb = (size_t)l * nsub + tr + T * (g.h[l] - 1);
    const size_t ja = (size_t)(l + 1) * nsub + tr;
    auto e1 = [&](int x) {                   // M[x][x+1]
      return (x >= 0 && x + 1 < Lx) ? cxd{t, 0} - t2 * (oB[jb + (size_t)x * W] + oB[ja + (size_t)x * W]) : zero;
    };
    auto e2 = [&](int x) {                   // M[x][x+2]
      return (o2 && x >= 0 && x + 2 < Lx) ? -(t2 * (o2[jb + (size_t)x * W] + o2[ja + (size_t)x * W])) : zero;
    };
    cxd d1 = zero, d2 = zero, l1p = zero;    // d_{x-1}, d_{x-2}, l1_{x-1}
    for (int x = 0; x < Lx; ++x) {
      const int a = x + Lx * tr;
      const cxd mxx = dyson_diag(g, b, kf, a + A * g.ylayer[l]) -
                      t2 * (dB[jb + (size_t)x * W] + dB[ja + (size_t)x * W]);
      const cxd l2 = (x >= 2) ? e2(x - 2) * cinv(d2) : zero;
      const cxd l1 = (x >= 1) ? (e1(x - 1) - l2 * l1p * d2) * cinv(d1) : zero;
      const cxd dx = mxx - l1 * l1 * d1 - l2 * l2 * d2;
      pre[a] = cconv<R>(cinv(dx));
      pre[A + a] = cconv<R>(l1);
      pre[2 * A + a] = cconv<R>(l2);
      d2 = d1;
      d1 = dx;
      l1p = l1;
    }
  }
}

}  // namespace

// H_ii (Eq. 1) of every DD slot, zero on padding: the mixed form's residuals
// read it coalesced instead of gathering V and Sigma in natural order.
__global__ void __launch_bounds__(DY_THREADS) k_hdiag(Geo g, Bufs b) {
  const int kf = blockIdx.y;
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < (size_t)g.Ndd;
       k += (size_t)gridDim.x * blockDim.x) {
    const int nat = b.dd2nat[k];
    b.hdiag[(size_t)kf * g.Ndd + k] = nat >= 0 ? dyson_diag(g, b, kf, nat) : cxd{0, 0};
  }
}

// CTAs per unit of k_factor_wide with nt x nt tiles: the one with the shortest
// longest share of a slice's 32^3 tile products, two CTAs on an SM counting 1.9
// (they share its FP32 pipe but hide each other's barriers).  Measured: 32 units, nt = 4
// 56 ms with 4 CTAs, 68 with 8; 128 units, nt = 4 41 ms with 2, 43 with 1; 64 units,
// nt = 5 31.9 with 2, 32.3 with 4.
static int wide_cluster(int units, int nt) {
  int best = 1;
  double t_best = 0.0;
  for (int C = 1; C <= 8 && (C == 1 || (long long)units * C <= DY_FACTOR_CTAS); C *= 2) {
    auto share = [&](int tiles) { return (tiles + C - 1) / C; };
    const int products = nt * (share(nt * nt) + share(nt * (nt + 1) / 2)) +
                         nt * (share(nt - 1) + share(nt * (nt - 1) / 2));
    const long long ctas = (long long)units * C;
    const double per_sm = ctas <= DY_FACTOR_CTAS / 2 ? 1.0 : 1.9;
    const double t = products * per_sm;
    if (C == 1 || t < t_best) {
      best = C;
      t_best = t;
    }
  }
  return best;
}

template <typename R, typename S>
cudaError_t launch_factor(const Geo& g, const Bufs& b, int K, cudaStream_t st) {
  if (b.hdiag) {
    const size_t blocks = ((size_t)g.Ndd + DY_THREADS - 1) / DY_THREADS;
    k_hdiag<<<dim3((unsigned)(blocks < 1024 ? blocks : 1024), K), DY_THREADS, 0, st>>>(g, b);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (g.W > DY_MAXW_SMEM) {
    // wide slices: the recursion in global memory (binary64, or double-float in the
    // mixed form), a cluster of CTAs per unit where there are few units
    if constexpr (sizeof(cx<R>) == sizeof(cxd)) {
      if (g.W > DY_MAXW || !b.fwork) return cudaErrorInvalidValue;
      const int units = g.p * K;
      const int C = wide_cluster(units, (g.W + TB - 1) / TB);
      const int clusters = units < DY_FACTOR_CTAS / C ? units : DY_FACTOR_CTAS / C;
      return launch_clustered(k_factor_wide<R, S>, dim3(clusters * C), C, sizeof(TileSmem<R>), st, g, b, K);
    } else {
      return cudaErrorInvalidValue;
    }
  }
  const size_t smem2 = (3 * (size_t)g.W * g.W + 11 * (size_t)g.W) * sizeof(cx<R>);
  if constexpr (std::is_same<R, dfl>::value) {
    auto kern = g.W <= 16 ? k_factor_two<R, 16> : (g.W <= 32 ? k_factor_two<R, 32> : k_factor_two<R, 64>);
    return launch_clustered(kern, dim3(2 * g.p, K), 2, smem2, st, g, b);
  } else {
    if (g.W <= DY_TWO_MAXW64)
      return launch_clustered(g.W <= 16 ? k_factor_two<R, 16> : k_factor_two<R, 32>, dim3(2 * g.p, K), 2, smem2, st, g, b);
    const size_t smem = (3 * (size_t)g.W * g.W + 4 * (size_t)g.W) * sizeof(cx<R>);
    cudaError_t e = raise_smem_limit((const void*)k_factor<R>, smem);
    if (e != cudaSuccess) return e;
    k_factor<R><<<dim3(g.p, K), DY_THREADS, smem, st>>>(g, b);
    return cudaGetLastError();
  }
}
template cudaError_t launch_factor<double, double>(const Geo&, const Bufs&, int, cudaStream_t);
template cudaError_t launch_factor<dfl, float>(const Geo&, const Bufs&, int, cudaStream_t);

template <typename R>
cudaError_t launch_precond(const Geo& g, const Bufs& b, int K, cudaStream_t st) {
  if (g.p < 2) return cudaSuccess;
  if (g.lpre) {
    cudaError_t e = launch_surface(g, b, K, st);
    if (e != cudaSuccess) return e;
    return launch_layer_inv<R>(g, b, K, st);
  }
  k_precond<R><<<dim3(g.p - 1, K), DY_THREADS, 0, st>>>(g, b);
  return cudaGetLastError();
}
template cudaError_t launch_precond<double>(const Geo&, const Bufs&, int, cudaStream_t);
template cudaError_t launch_precond<float>(const Geo&, const Bufs&, int, cudaStream_t);

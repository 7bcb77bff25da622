// X-matvec on the two-sided factors, two chains a subdomain: the mixed form's strips
// (W <= 64, complex64 block sweeps refined against binary64 residuals) and the FP64
// form's (W <= DY_TWO_MAXW64, the same sweeps and interface solve in binary64).
//
// One cluster per (frequency, block column), one CTA per subdomain, as in
// solve_device.cuh.  What is special here:
//
// 1. The sweep.  Each of the two chains of a subdomain (left to the middle
//    slice, right to the middle slice, and back) is run by WF / 8 warps.  Four
//    lanes share a row: lane (cg = lane / 8, rr = lane % 8) of warp w holds the
//    column pairs cg, cg + 4, ... of row 8 w + rr, so a 32 x 32 block product is
//    4 16-byte loads and 32 FMAs a lane plus two shuffles, and one barrier of
//    the chain's warps a slice.  The block of the next step is read into
//    registers before that barrier, which also frees its ring slot.  A producer
//    warp per chain takes part in the same barrier: it waits for the copies (the
//    chain's warps never touch an mbarrier) and refills the freed slots, and the
//    copies run on from one sweep into the next, as every sweep reads the same
//    sequence of blocks.
// 2. Two right-hand sides in one sweep (NR = 2): the refinement's subdomain
//    residual of w and that of u go through the factors together.
// 3. No closing sweep: the interface solve's last product B^-1 E p is still in
//    the row buffer when its step length alpha is known, and u_B is the sum of
//    alpha B^-1 E p over the iterations, so B^-1 E y needs no sweep of its own.
// w, u, H_ii and the residuals are binary64, as are the sums over warps and
// CTAs: what the refinement ends at is the rounding floor of the binary64
// residual, whatever H is.  The part issues two binary64 operations per clock and
// SM, so a pass takes ~17 clocks a site (34 operations for both residuals, their
// norms and the updates); in double-float on the FP32 pipe a solve was 5 % (512^2 x 32
// 242 ms -> 229) to 9 % (64^2 x 16 6.25 ms -> 5.7) faster, but ended at 24 x 2^-53 of
// sum |H||u| instead of below 10.
#pragma once
#include "solve_device.cuh"

namespace {

constexpr int MIX_MAXS = 8;              // most ring slots of one chain
constexpr size_t MIX_SMEM_2 = 112 * 1024;   // dynamic shared memory per CTA at two CTAs per SM
constexpr size_t MIX_SMEM_1 = 226 * 1024;   // and at one

template <typename R, int WF>
struct Mix {
  static constexpr int WARPS = WF / 8;   // compute warps of one chain
  static constexpr int CT = 32 * WARPS;
  static constexpr int CU = 16 / (int)sizeof(cx<R>);   // columns in a 16-byte word of a block
  static constexpr int KP = WF / (4 * CU);   // words a lane holds (it has a quarter of a row)
  static constexpr int PROD = 2 * WARPS; // first of the two producer warps
  static constexpr int NT = WF == 16 ? 256 : 32 * (2 * WARPS + 2);   // 256, 320, 576
  static constexpr int PER_SM = WF <= (sizeof(R) == 4 ? 32 : 16) ? 2 : 1;
};
__host__ __device__ inline int mix_threads(int W) {
  return W <= 16 ? Mix<float, 16>::NT : (W <= 32 ? Mix<float, 32>::NT : Mix<float, 64>::NT);
}

// Everything but the ring and the rows, at the start of the dynamic shared memory.
template <typename R, int WF>
struct MixSmem {
  alignas(16) cx<R> z[2][2][2][WF];      // [chain][right-hand side][parity]: z of the current and next slice
  alignas(16) cx<R> zm[2][2][WF];        // [chain][right-hand side]: the chain's part of the middle z
  double wred[24 * 8];                   // per-warp partial sums
  double slot[2][DY_MAXP * 8];           // [phase][rank]: the CTAs' partial sums
  double res[8];                         // the cluster's sums
  alignas(8) uint64_t bars[2 * MIX_MAXS];
  int err;
};
template <typename R>
__host__ __device__ constexpr size_t mix_head(int W) {
  return ((W <= 16 ? sizeof(MixSmem<R, 16>) : (W <= 32 ? sizeof(MixSmem<R, 32>) : sizeof(MixSmem<R, 64>))) + 127) &
         ~(size_t)127;
}

// Shared-memory plan: S ring slots of one block for each chain, and both row
// buffers on chip or in the plan's scratch.  g.ring_S (slots of both chains)
// and g.xm_rows come from the autotuner; 0: the heuristic, which keeps the
// rows on chip when four slots a chain (two in binary64) fit beside them.
struct MixPlan {
  int S, rows;
  size_t smem;
};
template <typename R>
__host__ __device__ inline size_t mix_smem(int W, int Lx, int S, int rows) {
  return mix_head<R>(W) + ((size_t)2 * S * W * W + (rows ? 2 * (size_t)Lx * W : 0)) * sizeof(cx<R>);
}
template <typename R>
__host__ __device__ inline MixPlan mix_plan(const Geo& g) {
  MixPlan m;
  if (g.ring_S > 0) {
    m.S = g.ring_S / 2;
    m.rows = g.xm_rows > 0 ? 1 : 0;
  } else {
    const size_t lim = g.W <= 32 && sizeof(R) == 4 ? MIX_SMEM_2 : MIX_SMEM_1;
    m.rows = mix_smem<R>(g.W, g.Lx, sizeof(R) == 4 ? 4 : 2, 1) <= lim ? 1 : 0;
    m.S = 4;
    while (m.S > 2 && mix_smem<R>(g.W, g.Lx, m.S, m.rows) > lim) --m.S;
  }
  m.smem = mix_smem<R>(g.W, g.Lx, m.S, m.rows);
  return m;
}
// Configurations the autotuner times: slots a chain, rows on chip or not.
template <typename R>
inline int mix_candidates(const Geo& g, int* S, int* CR, int* ROWS, int max) {
  Geo h = g;
  h.ring_S = 0;
  const MixPlan d = mix_plan<R>(h);
  int n = 0;
  auto add = [&](int s, int rows) {
    for (int k = 0; k < n; ++k)
      if (S[k] == 2 * s && ROWS[k] == rows) return;
    if (n < max && mix_smem<R>(g.W, g.Lx, s, rows) <= MIX_SMEM_1) {
      S[n] = 2 * s;
      CR[n] = g.W;
      ROWS[n] = rows;
      ++n;
    }
  };
  add(d.S, d.rows);
  for (int rows = 1; rows >= 0; --rows)
    for (int s : {2, 3, 4, 6}) add(s, rows);
  return n;
}

// The dynamic shared memory, named here so that every function (inlined or
// not) addresses it as shared memory and not through generic pointers.
extern __shared__ __align__(128) unsigned char mix_raw[];
template <typename R, int WF>
__device__ __forceinline__ MixSmem<R, WF>& mix_sm() {
  return *reinterpret_cast<MixSmem<R, WF>*>(mix_raw);
}
template <typename R, int WF>
__device__ __forceinline__ cx<R>* mix_ring() {
  constexpr size_t head = (sizeof(MixSmem<R, WF>) + 127) & ~(size_t)127;
  return reinterpret_cast<cx<R>*>(mix_raw + head);
}

__device__ __forceinline__ void named_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// What a thread keeps from sweep to sweep (compute warps: slot; producers: the
// rest).  The addresses of the next copy and of the next wait are computed when
// the previous one is done, off the chain's critical path: after a barrier the
// producer only issues.
template <typename R>
struct MixState {
  int slot;                              // compute: slot of the next block to read; producer: next slot to fill
  int pos;                               // position of the next block to copy in the sweep's sequence
  const cx<R>* src;                      // its address
  int wslot;                             // slot of the next block to wait for
  uint32_t wph;
  bool dead;
};

// One CTA's constants and buffers.
template <typename R, int WF, bool ROWS>
struct MixCtx {
  int W, Lx, S, m;
  const cx<R>* src;                        // the subdomain's factors
  cx<R> *g0, *g1;                          // row buffers in the scratch (ROWS = false)
  unsigned long long* cnt;
  R t;

  __device__ __forceinline__ cx<R>* row(int k) const {
    if constexpr (ROWS) return mix_ring<R, WF>() + 2 * S * W * W + (k ? Lx * W : 0);
    else return k ? g1 : g0;
  }
  __device__ __forceinline__ int blocks(int chain) const { return chain == 0 ? 2 * m + 1 : 2 * (Lx - 1 - m); }
  // The sequence of a chain's slices over one sweep: left 0 .. m, m-1 .. 0, right
  // Lx-1 .. m+1, m+1 .. Lx-1; the next sweep starts with the last one's last slice.
  __device__ __forceinline__ const cx<R>* first(int chain) const { return src + (chain == 0 ? 0 : (size_t)(Lx - 1) * W * W); }
  __device__ __forceinline__ void issue(int chain, MixState<R>& st) const {
    MixSmem<R, WF>& sm = mix_sm<R, WF>();
    const int n = W * W;
    bulk_load(mix_ring<R, WF>() + (chain * S + st.slot) * n, st.src, (uint32_t)(n * sizeof(cx<R>)),
              sm.bars + chain * MIX_MAXS + st.slot);
    if (++st.slot == S) st.slot = 0;
    const int up = chain == 0 ? m : Lx - 2 - m, last = blocks(chain) - 1;   // the turn: left at m, right repeats m+1
    const int dn = chain == 0 ? n : -n;
    const int turn = chain == 0 ? 0 : 1;
    st.src += st.pos < up ? dn : (st.pos < up + turn || st.pos == last ? 0 : -dn);
    st.pos = st.pos == last ? 0 : st.pos + 1;
  }
  __device__ __forceinline__ void wait(int chain, MixState<R>& st) const {
    MixSmem<R, WF>& sm = mix_sm<R, WF>();
    ring_wait(sm.bars + chain * MIX_MAXS + st.wslot, st.wph, st.dead, &sm.err);
    if (++st.wslot == S) {
      st.wslot = 0;
      st.wph ^= 1u;
    }
  }
};

template <typename R, int WF, bool ROWS>
__device__ void mix_init(const MixCtx<R, WF, ROWS>& ctx, MixState<R>& st) {
  MixSmem<R, WF>& sm = mix_sm<R, WF>();
  const int tid = threadIdx.x, wid = tid >> 5;
  st.slot = st.pos = st.wslot = 0;
  st.src = ctx.first(wid == Mix<R, WF>::PROD + 1 ? 1 : 0);
  st.wph = 0;
  st.dead = false;
  for (int e = tid; e < 8 * WF; e += Mix<R, WF>::NT) (&sm.z[0][0][0][0])[e] = cx<R>{0, 0};
  for (int e = tid; e < 4 * WF; e += Mix<R, WF>::NT) (&sm.zm[0][0][0])[e] = cx<R>{0, 0};
  if (tid == 0) {
    for (int k = 0; k < 2 * MIX_MAXS; ++k) mbar_init(sm.bars + k, 1);
    sm.err = 0;
    fence_mbar_init();
  }
  __syncthreads();
  const int c = wid - Mix<R, WF>::PROD;
  if ((c == 0 || c == 1) && (tid & 31) == 0 && ctx.blocks(c) > 0)
    for (int k = 0; k < ctx.S; ++k) ctx.issue(c, st);
}
// Before the kernel ends: the S copies of each chain issued beyond its last
// step have landed (bounded waits, also after an earlier wait ran out; the
// first that runs out ends it).
template <typename R, int WF, bool ROWS>
__device__ void mix_drain(const MixCtx<R, WF, ROWS>& ctx, MixState<R>& st) {
  const int c = ((int)threadIdx.x >> 5) - Mix<R, WF>::PROD;
  if ((c == 0 || c == 1) && (threadIdx.x & 31) == 0 && ctx.blocks(c) > 0)
    for (int k = 0; k < ctx.S; ++k) {
      if (!mbar_wait(mix_sm<R, WF>().bars + c * MIX_MAXS + st.wslot, st.wph)) {
        mix_sm<R, WF>().err = 1;
        break;
      }
      if (++st.wslot == ctx.S) {
        st.wslot = 0;
        st.wph ^= 1u;
      }
    }
}

// B_i x = rhs for NR right-hand sides in place in the row buffers [Lx][W]
// (complex64; padding columns zero; NR = 1: buffer k0; NR = 2: both), with
// m = Lx / 2, qR = Lx - 1 - m:
//   left   y_s = g_s (rhs_s - t y_{s-1})        s = 0 .. m-1
//   right  y_s = g_s (rhs_s - t y_{s+1})        s = Lx-1 .. m+1
//   middle x_m = G_mm (rhs_m - t y_{m-1} - t y_{m+1})        (left chain's warps)
//   back   x_s = y_s - t g_s x_{s+1} (left, s = m-1 .. 0),  x_s = y_s - t g_s x_{s-1} (right)
// Block n of a chain's sequence is in registers when its step begins; step n
// reads block n + 1 after its products.  The producer has waited for block
// n + 2 when it joins the barrier of step n, and refills block n + 1's slot
// after it (block 0's after the first barrier, which starts the chain), so the
// block it waits for is always in flight with two slots or more.  Rows are read PF slices ahead into registers (the latency of a row
// buffer in the scratch), and a step's row is stored during the next step,
// behind that step's loads of z.  Every warp of the CTA calls it; the rows are
// complete and visible to the CTA on return.
template <typename R, int WF, int NR, bool ROWS>
__device__ __noinline__ void mix_sweep(const MixCtx<R, WF, ROWS>& ctx, MixState<R>& state, int k0) {
  constexpr int CT = Mix<R, WF>::CT, PF = NR == 1 && !ROWS ? 4 : 2, KP = Mix<R, WF>::KP, WARPS = Mix<R, WF>::WARPS;
  constexpr int KH = KP < 4 ? KP : 4;    // column pairs handled at a time
  using C = cx<R>;
  using U = std::conditional_t<sizeof(R) == 4, float4, double2>;   // a 16-byte word: CU columns
  constexpr int CU = Mix<R, WF>::CU;
  MixSmem<R, WF>& sm = mix_sm<R, WF>();
  const MixCtx<R, WF, ROWS> cx_ = ctx;
  MixState<R> st = state;
  const int W = cx_.W, Lx = cx_.Lx, m = cx_.m, qR = Lx - 1 - m;
  const int wid = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
  const int role = wid < 2 * WARPS ? 0 : (wid < 2 * WARPS + 2 ? 1 : 2);
  const int c = role == 0 ? wid / WARPS : (role == 1 ? wid - Mix<R, WF>::PROD : 0);
  const int NL = cx_.blocks(c), steps = c == 0 ? m : qR;
  const R t = cx_.t;
  const int cg = lane >> 3, row = (wid % WARPS) * 8 + (lane & 7);
  const bool own = role == 0 && cg == 0 && row < W;
  const int off0 = cg * W + (row < W ? row : 0), W4 = 4 * W, WW2 = W * W / CU;
  const int wu = W / CU, km = wu > cg ? (wu - cg + 3) / 4 : 0;
  const U* ring4 = reinterpret_cast<const U*>(mix_ring<R, WF>()) + (size_t)c * cx_.S * WW2 + off0;
  C* yb[2] = {cx_.row(NR == 1 ? k0 : 0), cx_.row(1)};
  U gb[KP];
  auto load = [&]() {
    const U* p = ring4 + st.slot * WW2;
#pragma unroll
    for (int q = 0; q < KP; ++q) gb[q] = q < km ? p[q * W4] : U{};
    if (++st.slot == cx_.S) st.slot = 0;
  };
  auto load_z = [&](const C* z, int h, U (&zv)[KH]) {
    const U* z4 = reinterpret_cast<const U*>(z) + cg + 16 * h;
#pragma unroll
    for (int q = 0; q < KH; ++q) zv[q] = z4[4 * q];
  };
  // this lane's part of (block row) . z, the first KH pairs of z already in zv
  auto part = [&](const C* z, U (&zv)[KH]) -> C {
    constexpr int NA = KP >= 4 ? 4 : 2;
    C a[NA];
#pragma unroll
    for (int q = 0; q < NA; ++q) a[q] = C{0, 0};
#pragma unroll
    for (int h = 0; h < KP / KH; ++h) {
      if (h > 0) load_z(z, h, zv);
#pragma unroll
      for (int q = 0; q < KH; ++q) {
        const U gv = gb[h * KH + q];
        a[(CU * q) % NA] = cfma(C{gv.x, gv.y}, C{zv[q].x, zv[q].y}, a[(CU * q) % NA]);
        if constexpr (CU == 2) a[(2 * q + 1) % NA] = cfma(C{gv.z, gv.w}, C{zv[q].z, zv[q].w}, a[(2 * q + 1) % NA]);
      }
    }
    C s = a[0] + a[1];
    if constexpr (NA == 4) s = s + (a[2] + a[3]);
    return s;
  };
  auto total = [&](C v) -> C {                           // over the row's four lanes
    if constexpr (sizeof(R) == 8) {      // one part a lane of a pair: two binary64 sums instead of four
      const bool odd = cg & 1;
      R a = odd ? v.y : v.x;
      a += __shfl_xor_sync(0xffffffffu, odd ? v.x : v.y, 8);
      a += __shfl_xor_sync(0xffffffffu, a, 16);
      const R o = __shfl_xor_sync(0xffffffffu, a, 8);
      return odd ? C{o, a} : C{a, o};
    }
    v.x += __shfl_xor_sync(0xffffffffu, v.x, 8);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, 8);
    v.x += __shfl_xor_sync(0xffffffffu, v.x, 16);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, 16);
    return v;
  };
  if (role == 1 && lane == 0) {
    if (NL > 0) cx_.wait(c, st);          // blocks 0 and 1
    if (NL > 1) cx_.wait(c, st);
  }
  __syncthreads();                       // the rows are written; earlier readers of z are done
  if (role == 0) {
    if (own) {
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        if (steps > 0) sm.z[c][r][0][row] = yb[r][(c == 0 ? 0 : Lx - 1) * W + row];
        else sm.zm[c][r][row] = c == 0 ? yb[r][row] : cx<R>{0, 0};
      }
    }
    if (NL > 0) load();
    named_sync(3 + c, CT + 32);
    // ---- towards the middle: step n is slice s0 + d n, its z needs row s0 + d (n + 1) next
    const int d = c == 0 ? W : -W;       // row step
    int o = (c == 0 ? 0 : (Lx - 1) * W) + row;           // this step's row entry
    const int nf = c == 0 ? steps : steps - 1;           // steps whose next z has a right-hand side
    C f[NR][PF], yp[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      yp[r] = cx<R>{0, 0};
#pragma unroll
      for (int u = 0; u < PF; ++u) f[r][u] = own && u < nf ? yb[r][o + d * (u + 1)] : cx<R>{0, 0};
    }
    for (int n0 = 0; n0 < steps; n0 += PF) {
#pragma unroll
      for (int u = 0; u < PF; ++u) {
        const int n = n0 + u;
        if (n < steps) {
          C y[NR];
          U zv[KH];
          load_z(sm.z[c][0][u & 1], 0, zv);
          if (own && n > 0) {            // row n - 1 out, its slot of f refilled
#pragma unroll
            for (int r = 0; r < NR; ++r) {
              yb[r][o - d] = yp[r];
              f[r][(u + PF - 1) % PF] = n - 1 + PF < nf ? yb[r][o + d * PF] : cx<R>{0, 0};
            }
          }
          y[0] = part(sm.z[c][0][u & 1], zv);
          if constexpr (NR == 2) {
            load_z(sm.z[c][1][u & 1], 0, zv);
            y[1] = part(sm.z[c][1][u & 1], zv);
          }
          if (n + 1 < NL) load();
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            y[r] = total(y[r]);
            if (own) {
              C* zn = n + 1 < steps ? sm.z[c][r][(u + 1) & 1] : sm.zm[c][r];
              zn[row] = f[r][u] - t * y[r];
            }
            yp[r] = y[r];
          }
          o += d;
          named_sync(1 + c, CT + 32);
        }
      }
    }
    if (own && steps > 0) {
#pragma unroll
      for (int r = 0; r < NR; ++r) yb[r][o - d] = yp[r];
    }
  } else if (role == 1) {
    named_sync(3 + c, CT + 32);          // block 0 has been read
    if (lane == 0 && NL > 0) cx_.issue(c, st);
    for (int n = 0; n < steps; ++n) {
      if (lane == 0 && n + 2 < NL) cx_.wait(c, st);
      __syncwarp();
      named_sync(1 + c, CT + 32);        // block n + 1 has been read
      if (lane == 0 && n + 1 < NL) cx_.issue(c, st);
    }
  }
  __syncthreads();                       // both parts of the middle z are written
  if (c == 0 && role == 0) {
    if (own) {
#pragma unroll
      for (int r = 0; r < NR; ++r) sm.z[0][r][1][row] = sm.zm[0][r][row] + sm.zm[1][r][row];
    }
    named_sync(3, CT);
    C x[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      U zv[KH];
      load_z(sm.z[0][r][1], 0, zv);
      x[r] = part(sm.z[0][r][1], zv);
    }
    if (m + 1 < NL) load();
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      x[r] = total(x[r]);
      if (own) {
        yb[r][m * W + row] = x[r];
        sm.z[0][r][0][row] = x[r];       // the first z of both ways back is z buffer 0
        sm.z[1][r][0][row] = x[r];
      }
    }
  } else if (c == 0 && role == 1 && lane == 0 && m + 2 < NL) {
    cx_.wait(c, st);
  }
  __syncthreads();                       // x_m is visible to both chains
  if (c == 0 && role == 1 && lane == 0 && m + 1 < NL) cx_.issue(c, st);
  const int n1 = c == 0 ? m + 1 : qR;
  if (role == 0) {
    // ---- back from the middle: step k is slice m -+ (k + 1)
    const int d = c == 0 ? -W : W;
    int o = (c == 0 ? m - 1 : m + 1) * W + row;
    C f[NR][PF], xp[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      xp[r] = cx<R>{0, 0};
#pragma unroll
      for (int u = 0; u < PF; ++u) f[r][u] = own && u < steps ? yb[r][o + d * u] : cx<R>{0, 0};
    }
    for (int kb = 0; kb < steps; kb += PF) {
#pragma unroll
      for (int u = 0; u < PF; ++u) {
        const int k = kb + u;
        if (k < steps) {
          C y[NR];
          U zv[KH];
          load_z(sm.z[c][0][u & 1], 0, zv);
          if (own && k > 0) {
#pragma unroll
            for (int r = 0; r < NR; ++r) {
              yb[r][o - d] = xp[r];
              f[r][(u + PF - 1) % PF] = k - 1 + PF < steps ? yb[r][o + d * (PF - 1)] : cx<R>{0, 0};
            }
          }
          y[0] = part(sm.z[c][0][u & 1], zv);
          if constexpr (NR == 2) {
            load_z(sm.z[c][1][u & 1], 0, zv);
            y[1] = part(sm.z[c][1][u & 1], zv);
          }
          if (n1 + k + 1 < NL) load();
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            y[r] = total(y[r]);
            xp[r] = f[r][u] - t * y[r];
            if (own) sm.z[c][r][(u + 1) & 1][row] = xp[r];
          }
          o += d;
          named_sync(1 + c, CT + 32);
        }
      }
    }
    if (own && steps > 0) {
#pragma unroll
      for (int r = 0; r < NR; ++r) yb[r][o - d] = xp[r];
    }
  } else if (role == 1) {
    for (int k = 0; k < steps; ++k) {
      const int n = n1 + k;
      if (lane == 0 && n + 2 < NL) cx_.wait(c, st);
      __syncwarp();
      named_sync(1 + c, CT + 32);
      if (lane == 0 && n + 1 < NL) cx_.issue(c, st);
    }
  }
  __syncthreads();
  state = st;
  if (threadIdx.x == 0 && cx_.cnt) *cx_.cnt += 1;
}

// ---------------------------------------------------------------- reductions
// Cluster-wide sums of NV values of V (every thread gets them), and this CTA's
// own totals in loc if not null.  A warp's total is formed in V, the sums over
// warps and CTAs in binary64: warp 0 adds the warps and puts the total into every
// CTA's slot for this rank; after the cluster barrier it adds the ranks' slots by
// the same tree in every CTA, so all threads of the cluster hold the same bits.
// active (the same in a warp): this warp has something to add.  `phase` alternates
// two slot sets.
template <typename R, int WF, int NV, typename V>
__device__ __forceinline__ void mix_sum(cg::cluster_group& cl, int& phase, int p, V (&v)[NV], double (&out)[NV],
                                        bool active = true, double* loc = nullptr) {
  MixSmem<R, WF>& sm = mix_sm<R, WF>();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  constexpr int NW = Mix<R, WF>::NT / 32;
  const int me = (int)cl.block_rank();
  if (active) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < NV; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  }
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) sm.wred[wid * 8 + k] = active ? (double)v[k] : 0.0;
  }
  __syncthreads();
  if (wid == 0) {
    double s[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) s[k] = lane < NW ? sm.wred[lane * 8 + k] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < NV; ++k) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
    if (lane < p) {
      double* rem = cl.map_shared_rank(&sm.slot[phase][me * 8], lane);
#pragma unroll
      for (int k = 0; k < NV; ++k) rem[k] = s[k];
    }
  }
  cl.sync();
  if (wid == 0) {
    double s[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) s[k] = lane < p ? sm.slot[phase][lane * 8 + k] : 0.0;
#pragma unroll
    for (int o = DY_MAXP / 2; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < NV; ++k) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < NV; ++k) sm.res[k] = s[k];
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) out[k] = sm.res[k];
  if (loc) {
#pragma unroll
    for (int k = 0; k < NV; ++k) loc[k] = sm.slot[phase][me * 8 + k];
  }
  phase ^= 1;
}
static_assert(DY_MAXP == 16, "mix_sum adds the ranks over 16 lanes");

// Sum of v over the CTA in binary64 (every thread gets it).
template <typename R, int WF>
__device__ __forceinline__ double cta_sum(double v) {
  MixSmem<R, WF>& sm = mix_sm<R, WF>();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  constexpr int NW = Mix<R, WF>::NT / 32;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) sm.wred[wid] = v;
  __syncthreads();
  if (wid == 0) {
    double s = lane < NW ? sm.wred[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) sm.res[0] = s;
  }
  __syncthreads();
  return sm.res[0];
}

// ---------------------------------------------------------------- interface solve
template <typename R>
struct MixSolve {
  bool useB0;                            // the subdomain part is B0 - alpha B1 (else - alpha B1)
  cx<R> alpha;
  int iters, conv;
};

// COCG on S y = IF_B (relative residual krylov_tol), S applied by one sweep in
// row buffer 1 per iteration.  The solution's subdomain part -B^-1 E y is left
// as B0 - alpha B1: each iteration but the last is folded into B0, the last one
// is the caller's.  keep0: B0 holds a vector to add to (else it counts as zero).
// IF_B is complete (a barrier after its writers) on entry.
// In binary32 IF_B may have any size: its first dot products are binary64, and from
// there the iteration runs on IF_B 2^kc with a norm of about 1 (the squares of its
// dot products would leave the range at 1e-23 and 1e19); alpha carries the factor
// 2^-kc back, so y and B^-1 E y have IF_B's own scale.
template <typename R, int WF, bool ROWS>
__device__ __noinline__ MixSolve<R> mix_cocg(const Geo& g, const Bufs& b, const MixCtx<R, WF, ROWS>& ctx, MixState<R>& st,
                                          int& phase_, int vs, bool keep0) {
  using C = cx<R>;
  cg::cluster_group cl = cg::this_cluster();
  int phase = phase_;
  constexpr int nt = Mix<R, WF>::NT;
  const int i = blockIdx.x, A = g.A, p = g.p, W = ctx.W, Lx = ctx.Lx, T = g.T, w = T * g.h[i], nsub = Lx * W;
  const int ds = nt / W, dj = nt % W;
  const bool has = i < p - 1;
  C* B0 = ctx.row(0);
  C* B1 = ctx.row(1);
  const size_t o = (size_t)i * A;
  C* X = ifv_ptr<R>(g, b, vs, IF_X) + o;
  C* Rv = ifv_ptr<R>(g, b, vs, IF_R) + o;
  C* Z = ifv_ptr<R>(g, b, vs, IF_Z) + o;
  C* P = ifv_ptr<R>(g, b, vs, IF_P);
  C* SP = ifv_ptr<R>(g, b, vs, IF_SP) + o;
  const C* Bv = ifv_ptr<R>(g, b, vs, IF_B) + o;
  const C* dC = ifv_ptr<R>(g, b, vs, IF_D) + o;
  C* blo = bnd_ptr<R>(g, b, vs, i, 0);
  C* bhi = bnd_ptr<R>(g, b, vs, i, 1);
  const C* bnx = has ? bnd_ptr<R>(g, b, vs, i + 1, 0) : nullptr;
  const C* plo = i > 0 ? P + o - A : nullptr;
  C* phi = P + o;
  const R t = ctx.t;
  const bool act = has && ((int)threadIdx.x & ~31) < A;   // this warp has interface sites
  auto precond = [&](const C* r, C* z) {
    if (g.lpre) lpre_apply<R>(g, b, vs, i, r, z, B1);
    else precond_apply<R>(g, b, vs, i, r, z);
  };
  MixSolve<R> out = {keep0, {0, 0}, 0, 1};
  if (has) precond(Bv, Z);
  __syncthreads();
  constexpr bool f32 = sizeof(R) == 4;
  auto wide = [](C v) -> cxd {
    if constexpr (f32) return c2d_bits(v);
    else return v;
  };
  double v3[3] = {0, 0, 0};
  if (has) {
    cxd rz = {0, 0};
    for (int a = threadIdx.x; a < A; a += nt) {
      const C zz = Z[a], r = Bv[a];
      X[a] = C{0, 0};
      if (!f32) Rv[a] = r;
      phi[a] = zz;
      rz = cfma(wide(r), wide(zz), rz);
      v3[2] += cabs2(wide(r));
    }
    v3[0] = rz.x;
    v3[1] = rz.y;
  }
  double s3[3];
  mix_sum<R, WF>(cl, phase, p, v3, s3, act);   // also: P of the neighbour layers is final
  C rho;
  R bn, fs = 1, back = 1;                // 2^kc, 2^-kc
  if constexpr (f32) {
    const int kc = min(126, max(-126, -norm_exp(s3[2])));
    fs = pow2f(kc);
    back = pow2f(-kc);
    rho = C{d2f_scaled(s3[0], 2 * kc), d2f_scaled(s3[1], 2 * kc)};
    bn = d2f_scaled(s3[2], 2 * kc);
    if (has)
      for (int a = threadIdx.x; a < A; a += nt) Rv[a] = fs * Bv[a];
  } else {
    rho = C{s3[0], s3[1]};
    bn = s3[2];
  }
  R pf = fs;                             // P's factor: the first direction is stored unscaled
  auto scaled = [](R c, C v) -> C {
    if constexpr (f32) return c * v;
    else return v;
  };
  const R tol2 = (R)(g.krylov_tol * g.krylov_tol);
  if (bn > 0 || bn != bn) {
    for (;;) {
      if (out.iters >= g.krylov_maxit) {
        out.conv = 0;
        break;
      }
      if (out.iters > 0) {
        // fold the last product into B0, then the next direction
        const bool z0 = !out.useB0;
        for (int e = threadIdx.x; e < nsub; e += nt) {
          const C q = out.alpha * B1[e];
          B0[e] = z0 ? -q : B0[e] - q;
        }
        out.useB0 = true;
        __syncthreads();                 // B1 is free (the preconditioner's scratch)
        if (has) precond(Rv, Z);
        __syncthreads();
        R v2[2] = {0, 0};
        if (has) {
          C rz = {0, 0};
          for (int a = threadIdx.x; a < A; a += nt) rz = cfma(Rv[a], Z[a], rz);
          v2[0] = rz.x;
          v2[1] = rz.y;
        }
        double s2[2];
        mix_sum<R, WF>(cl, phase, p, v2, s2, act);
        const C rn = {(R)s2[0], (R)s2[1]}, beta = cdiv(rn, rho);
        rho = rn;
        if (has)
          for (int a = threadIdx.x; a < A; a += nt) phi[a] = Z[a] + beta * scaled(pf, phi[a]);
        pf = 1;
        cl.sync();                       // P of the neighbour layers is final
      }
      ++out.iters;
      // B1 = E p
      const R tp = t * pf;
      for (int e = threadIdx.x, s = e / W, j = e - s * W; e < nsub; e += nt) {
        C u = {0, 0};
        if (plo && j < T) u = u + tp * plo[s + Lx * j];
        if (has && j >= w - T && j < w) u = u + tp * phi[s + Lx * (j - (w - T))];
        B1[e] = u;
        s += ds;
        j += dj;
        if (j >= W) {
          j -= W;
          ++s;
        }
      }
      mix_sweep<R, WF, 1, ROWS>(ctx, st, 1);
      for (int e = threadIdx.x; e < A; e += nt) {
        const int j = T == 1 ? 0 : e / Lx, s = e - j * Lx;
        blo[e] = B1[s * W + j];
        bhi[e] = B1[s * W + (w - T) + j];
      }
      cl.sync();                         // boundary rows of every subdomain written
      R v2[2] = {0, 0};
      if (has) {
        C ps = {0, 0};
        for (int a = threadIdx.x; a < A; a += nt) {
          const C sp = scaled(pf, layer_C_apply<R>(g, dC, phi, a)) - t * (bhi[a] + bnx[a]);
          SP[a] = sp;
          ps = cfma(scaled(pf, phi[a]), sp, ps);
        }
        v2[0] = ps.x;
        v2[1] = ps.y;
      }
      double s2[2], s1[1];
      mix_sum<R, WF>(cl, phase, p, v2, s2, act);
      const C alpha = cdiv(rho, C{(R)s2[0], (R)s2[1]});
      out.alpha = scaled(back, alpha);
      R v1[1] = {0};
      if (has) {
        for (int a = threadIdx.x; a < A; a += nt) {
          X[a] = X[a] + out.alpha * scaled(pf, phi[a]);
          const C r = Rv[a] - alpha * SP[a];
          Rv[a] = r;
          v1[0] += cabs2(r);
        }
      }
      mix_sum<R, WF>(cl, phase, p, v1, s1, act);
      if ((R)s1[0] <= tol2 * bn) break;
    }
  }
  phase_ = phase;
  return out;
}

// ---------------------------------------------------------------- the X-matvec
// r + mt x, mt = -t
__device__ __forceinline__ void sub_scaled(cxd& r, double mt, cxd x) {
  r.x = fma(mt, x.x, r.x);
  r.y = fma(mt, x.y, r.y);
}
__device__ __forceinline__ void add_norm(double& n, cxd r) { n = fma(r.x, r.x, fma(r.y, r.y, n)); }

// w = blkdiag(B^-1, 0) q and u = X q = H^-1 [0; q_C - E^T w_B] (Eqs. 6-8, no
// cancellation) are found together:
//   w  from one sweep on q_B, u from one interface solve on q_C - E^T w_B;
//   then, until both relative residuals are below refine_tol, the residuals
//     r_w = q_B - B w,   r_u = [0; q_C - E^T w] - H u       (binary64)
//   and one correction: a sweep on both subdomain residuals gives d_w and
//   z = B^-1 r_u, an interface solve on r_u,C - E^T (d_w + z) gives d_y, and
//   w += d_w,  u_B += z - B^-1 E d_y,  u_C += d_y.
// The residual pass writes its rows straight into the row buffers in complex64,
// scaled by an estimate of their size (2^20 over the last residual's norm: about
// what a complex64 correction leaves).  The scale only keeps the values inside the
// binary32 range, and must do so for any q: a vector local to one strip reaches the
// others and the interface 30 and more decades down, and a scale held as a binary32
// number overflows there (at a norm of 3e-26 in the second pass).  So every scale is an
// exponent, applied in the conversions between binary64 and binary32: kq for q_B and kw
// for r_w, this subdomain's own, ku for r_u.  Where the subdomain and the interface
// differ in size, kw is kept within 2^60 below ku, so that the two corrections add up on
// the boundary rows in binary32; ku stays within 2^120 of q's own scale, which makes
// that possible.  An interface right-hand side below 2^-120 ||q|| counts as zero: a
// Lanczos vector's entries, and 1 / beta, end at the binary32 range.
template <int WF, bool ROWS>
__global__ void __launch_bounds__(Mix<float, WF>::NT, Mix<float, WF>::PER_SM)
    k_xmatvec_m(const __grid_constant__ Geo g, const __grid_constant__ Bufs b, int j, int ncols) {
  cg::cluster_group cl = cg::this_cluster();
  constexpr int nt = Mix<float, WF>::NT;
  const int i = blockIdx.x, vs = blockIdx.y, p = g.p, A = g.A, W = g.W, Lx = g.Lx, T = g.T;
  const int f = slot_freq(g, vs), c = vs - f * g.nb;
  if (c >= ncols) return;                  // same values in every CTA of the cluster
  int* st = b.st + (size_t)f * ST_N;
  if (st[ST_DONE]) return;
  const size_t Ndd = g.Ndd;
  const int nsub = Lx * W, w = T * g.h[i], hh = g.h[i], tid = threadIdx.x;
  const int ds = nt / W, dj = nt % W, s_0 = tid / W, j_0 = tid - s_0 * W;
  MixCtx<float, WF, ROWS> cx;
  cx.W = W;
  cx.Lx = Lx;
  cx.S = mix_plan<float>(g).S;
  cx.m = Lx / 2;
  cx.src = reinterpret_cast<const cxf*>(b.g) + ((size_t)f * p + i) * (size_t)nsub * W;
  cx.g0 = reinterpret_cast<cxf*>(b.yscr) + ((size_t)vs * p + i) * nsub;
  cx.g1 = reinterpret_cast<cxf*>(b.v2 + (size_t)vs * Ndd + (size_t)i * nsub);
  cx.cnt = sweep_cnt(g, b, vs, i);
  cx.t = (float)g.t;
  MixState<float> ms;
  mix_init<float, WF, ROWS>(cx, ms);
  int phase = 0;
  cxf* B0 = cx.row(0);
  cxf* B1 = cx.row(1);
  const bool has = i < p - 1;
  const cxd* qd = b.Q + ((size_t)f * (g.k_max + g.nb) + (size_t)j * g.nb + c) * Ndd;
  const cdfl* qs = reinterpret_cast<const cdfl*>(qd);
  const bool split = g.qsplit != 0;
  const size_t qo = (size_t)i * nsub, lo = (size_t)g.ifc_off + (size_t)i * A, o = (size_t)i * A;
  cxd* u = b.u + (size_t)vs * Ndd;
  cxd* wv = b.v1 + (size_t)vs * Ndd;                               // w_B
  cxd* rc = b.v2 + (size_t)vs * Ndd + lo;                          // interface residual
  cxd *us = u + qo, *ws = wv + qo;
  const cxd* hd = b.hdiag + (size_t)f * Ndd;
  const cxd* hs = hd + qo;
  const double mt = -g.t;
  const float tf = cx.t;
  cxf* Bv = ifv_ptr<float>(g, b, vs, IF_B) + o;
  cxf* X = ifv_ptr<float>(g, b, vs, IF_X) + o;
  cxf* dC = ifv_ptr<float>(g, b, vs, IF_D) + o;
  cxf* blo = bnd_ptr<float>(g, b, vs, i, 0);
  cxf* bhi = bnd_ptr<float>(g, b, vs, i, 1);
  const cxf* bnx = has ? bnd_ptr<float>(g, b, vs, i + 1, 0) : nullptr;
  auto ldq = [&](size_t k) -> cxd { return split ? cwiden(qs[k]) : qd[k]; };

  // the neighbour subdomain's w at layer i, and the two rows next to it
  const cxd* wa = wv + (size_t)(i + 1) * nsub;
  const int top = T * (hh - 1);
  auto layer_rows = [&](int a, int& kb, int& ka) {
    const int tr = T == 1 ? 0 : a / Lx, xx = a - tr * Lx;
    kb = xx * W + top + tr;
    ka = xx * W + tr;
  };

  // ---- w_0 = B^-1 q_B
  double qn2 = 0.0;                        // ||q_B||^2 of this subdomain
  for (int e = tid, jj = j_0; e < nsub; e += nt) {
    cxf v = {0.f, 0.f};
    if (jj < w) {
      const cxd q = ldq(qo + e);
      v = c2f_bits(q);
      add_norm(qn2, q);
    }
    B0[e] = v;
    jj += dj;
    if (jj >= W) jj -= W;
  }
  if (has)
    for (int a = tid; a < A; a += nt) dC[a] = c2f_bits(hd[lo + a]);
  qn2 = cta_sum<float, WF>(qn2);
  int kq = -norm_exp(qn2);
  if (kq >= -8 && kq <= 8) {               // the usual size of a Lanczos vector: as it is
    kq = 0;
  } else {
    for (int e = tid, jj = j_0; e < nsub; e += nt) {
      if (jj < w) B0[e] = c2f_scaled(ldq(qo + e), kq);
      jj += dj;
      if (jj >= W) jj -= W;
    }
  }
  mix_sweep<float, WF, 1, ROWS>(cx, ms, 0);
  for (int e = tid; e < nsub; e += nt) ws[e] = c2d_scaled(B0[e], -kq);   // zero on the padding
  cl.sync();                               // w of the neighbour subdomains is final
  double hn2, qa2;                         // ||hr||^2, ||q||^2 (the whole vector)
  {
    double v[2] = {0.0, tid == 0 ? qn2 : 0.0}, tot[2];
    if (has)
      for (int a = tid; a < A; a += nt) {
        int kb, ka;
        layer_rows(a, kb, ka);
        cxd h = ldq(lo + a);
        add_norm(v[1], h);
        sub_scaled(h, mt, ws[kb]);
        sub_scaled(h, mt, wa[ka]);
        rc[a] = h;
        add_norm(v[0], h);
      }
    mix_sum<float, WF>(cl, phase, p, v, tot);
    hn2 = tot[0];
    qa2 = tot[1];
  }
  int iters = 0, solves = 0, refines = 0, conv_all = 1;
  constexpr int K0 = 20, KB = 120;
  constexpr double TINY2 = 0x1p-240;       // (2^-KB)^2
  const int ktop = K0 - norm_exp(qa2) + KB;
  // not live: nothing reaches the interface, or a NaN in H or q, with which X q counts as zero
  const bool live = hn2 > TINY2 * qa2 || hn2 == INFINITY;
  // ---- u_0 = H^-1 [0; hr]
  if (live) {
    const int kh = -norm_exp(hn2);
    if (has)
      for (int a = tid; a < A; a += nt) Bv[a] = c2f_scaled(rc[a], kh);
    __syncthreads();
    const MixSolve<float> sv = mix_cocg<float, WF, ROWS>(g, b, cx, ms, phase, vs, false);
    iters += sv.iters;
    conv_all &= sv.conv;
    ++solves;
    for (int e = tid; e < nsub; e += nt) {   // zero on the padding, which the Lanczos step reads too
      cxf v = sv.iters > 0 ? sv.alpha * B1[e] : cxf{0.f, 0.f};
      if (sv.useB0) v = v - B0[e];
      us[e] = c2d_scaled(-v, -kh);
    }
    if (has)
      for (int a = tid; a < A; a += nt) u[lo + a] = c2d_scaled(X[a], -kh);
  } else {
    for (int e = tid; e < nsub; e += nt) us[e] = cxd{0, 0};
    if (has)
      for (int a = tid; a < A; a += nt) u[lo + a] = cxd{0, 0};
  }
  // ---- refinement of w and u together
  const cxd* xlo = i > 0 ? u + g.ifc_off + (size_t)(i - 1) * A : nullptr;
  const cxd* xhi = u + lo;
  const double tol2 = g.refine_tol * g.refine_tol;
  int ku = min(K0 - norm_exp(hn2), ktop), kw = max(K0 - norm_exp(qn2), ku - KB / 2);   // row scales
  double prev_u = INFINITY, prev_w = INFINITY;
  bool wdone = qn2 == 0.0;
  for (int pass = 0; live && pass < g.refine_max; ++pass) {
    cl.sync();                             // u and w of the neighbours are final
    double v[3] = {0.0, 0.0, 0.0}, tot[3], own[3];   // ||r_u||^2, ||hr||^2, ||r_w||^2
    for (int e = tid, s = s_0, jj = j_0; e < nsub; e += nt) {
      cxf ru = {0.f, 0.f}, rw = {0.f, 0.f};
      if (jj < w) {
        const int tr = T == 1 ? 0 : jj % T, sl = T == 1 ? jj : jj / T;
        const cxd dv = hs[e];
        const bool pl = s > 0, pr = s < Lx - 1, dl = sl > 0, dr = sl < hh - 1;
        const cxd zero = {0, 0};
        // r - t (sum of x over the neighbours) - H_ii x, one fused multiply-add a term;
        // every load is issued before the first of them
        auto residual = [&](cxd r, const cxd* x, const cxd& lo_, const cxd& hi_) -> cxd {
          const cxd xc = x[e], n0 = pl ? x[e - W] : zero, n1 = pr ? x[e + W] : zero;
          const cxd n2 = dl ? x[e - T] : lo_, n3 = dr ? x[e + T] : hi_;
          cxd n4 = zero, n5 = zero;
          if (T > 1) {
            n4 = tr > 0 ? x[e - 1] : zero;
            n5 = tr < T - 1 ? x[e + 1] : zero;
          }
          sub_scaled(r, mt, n0);
          sub_scaled(r, mt, n1);
          sub_scaled(r, mt, n2);
          sub_scaled(r, mt, n3);
          if (T > 1) {
            sub_scaled(r, mt, n4);
            sub_scaled(r, mt, n5);
          }
          return cfma(-dv, xc, r);
        };
        // the interface layers' u stands in for the neighbour outside the subdomain
        const cxd ul = !dl && xlo ? xlo[s + Lx * tr] : zero, uh = !dr && has ? xhi[s + Lx * tr] : zero;
        cxd r = residual(zero, us, ul, uh);
        ru = c2f_scaled(r, ku);
        add_norm(v[0], r);
        if (!wdone) {
          r = residual(ldq(qo + e), ws, zero, zero);
          rw = c2f_scaled(r, kw);
          add_norm(v[2], r);
        }
      }
      B0[e] = ru;
      if (!wdone) B1[e] = rw;
      s += ds;
      jj += dj;
      if (jj >= W) {
        jj -= W;
        ++s;
      }
    }
    if (has) {
      const cxd* xa = u + (size_t)(i + 1) * nsub;    // subdomain i + 1: its bottom row touches layer i
      for (int a = tid; a < A; a += nt) {
        const int tr = T == 1 ? 0 : a / Lx, xx = a - tr * Lx;
        int kb, ka;
        layer_rows(a, kb, ka);
        cxd r = ldq(lo + a);
        sub_scaled(r, mt, ws[kb]);
        sub_scaled(r, mt, wa[ka]);             // hr = q_C - E^T w
        add_norm(v[1], r);
        sub_scaled(r, mt, us[kb]);
        sub_scaled(r, mt, xa[ka]);
        if (xx > 0) sub_scaled(r, mt, xhi[a - 1]);
        if (xx < Lx - 1) sub_scaled(r, mt, xhi[a + 1]);
        if (tr > 0) sub_scaled(r, mt, xhi[a - Lx]);
        if (tr < T - 1) sub_scaled(r, mt, xhi[a + Lx]);
        r = cfma(-hd[lo + a], xhi[a], r);
        rc[a] = r;
        add_norm(v[0], r);
      }
    }
    mix_sum<float, WF>(cl, phase, p, v, tot, true, own);
    const double rn = tot[0], wn = own[2];   // w: this subdomain's, which decides for its w alone
    if (!wdone && (wn <= tol2 * qn2 || !(wn <= REFINE_STALL * prev_w))) wdone = true;
    if (!wdone) prev_w = wn;
    if (rn != rn) {                          // the interface solve broke down: nothing left to refine
      conv_all = 0;
      break;
    }
    const bool udone = rn <= tol2 * tot[1] || rn > REFINE_STALL * prev_u;
    if (udone) {
      // u is done: go on only if some w of the cluster is not
      float go[1] = {!wdone && tid == 0 ? 1.f : 0.f};
      double any[1];
      mix_sum<float, WF>(cl, phase, p, go, any, tid < 32);
      if (any[0] == 0.0) break;
    }
    prev_u = rn;
    ++refines;
    // ---- z = B^-1 r_u in B0, d_w = B^-1 r_w in B1
    const bool wgo = !wdone;
    if (wgo) mix_sweep<float, WF, 2, ROWS>(cx, ms, 0);
    else mix_sweep<float, WF, 1, ROWS>(cx, ms, 0);
    const float ratio = pow2f(max(ku - kw, -126));   // at most 2^60; below 2^-126 it adds nothing
    if (wgo)
      for (int e = tid; e < nsub; e += nt) ws[e] = ws[e] + c2d_scaled(B1[e], -kw);
    for (int e = tid; e < A; e += nt) {
      const int jj = T == 1 ? 0 : e / Lx, s = e - jj * Lx;
      const int k0 = s * W + jj, k1 = s * W + (w - T) + jj;
      blo[e] = wgo ? B0[k0] + ratio * B1[k0] : B0[k0];
      bhi[e] = wgo ? B0[k1] + ratio * B1[k1] : B0[k1];
    }
    cl.sync();                             // boundary rows of the neighbours
    if (has)
      for (int a = tid; a < A; a += nt) Bv[a] = c2f_scaled(rc[a], ku) - tf * (bhi[a] + bnx[a]);
    __syncthreads();
    const MixSolve<float> sv = mix_cocg<float, WF, ROWS>(g, b, cx, ms, phase, vs, true);
    iters += sv.iters;
    conv_all &= sv.conv;
    ++solves;
    for (int e = tid; e < nsub; e += nt) {
      cxf v2 = B0[e];
      if (sv.iters > 0) v2 = v2 - sv.alpha * B1[e];
      us[e] = us[e] + c2d_scaled(v2, -ku);
    }
    if (has)
      for (int a = tid; a < A; a += nt) u[lo + a] = u[lo + a] + c2d_scaled(X[a], -ku);
    ku = min(K0 - norm_exp(rn), ktop);
    kw = max(K0 - norm_exp(wgo ? prev_w : qn2), ku - KB / 2);
  }
  mix_drain<float, WF, ROWS>(cx, ms);
  __syncthreads();
  if (tid == 0 && mix_sm<float, WF>().err) atomicOr(st + ST_STATUS, ST_WAIT_TIMEOUT);
  if (i == 0 && tid == 0) {               // the nb clusters of a frequency share its counters
    atomicAdd(st + ST_ITERS, iters);
    atomicAdd(st + ST_SOLVES, solves);
    atomicAdd(st + ST_REFINE, refines);
    if (!conv_all) atomicOr(st + ST_STATUS, 4);
  }
  cl.sync();          // no CTA exits while a peer may still read its shared memory
}

// The FP64 form of the strips (W <= 32): the same sweeps and interface solve in binary64,
//   w = B^-1 q_B (boundary rows only), y = S^-1 (E^T w - q_C) to krylov_tol,
//   u_B = B^-1 E y (from the interface solve's own products), u_C = -y.
// The one-chain sweep of eight warps took 255 steps of 2.5 us a sweep at 128^2; the two
// chains share the SM's binary64 pipe (2 multiply-adds a clock: 1 us a 32 x 32 product)
// and hide each other's latency.
template <int WF, bool ROWS>
__global__ void __launch_bounds__(Mix<double, WF>::NT, Mix<double, WF>::PER_SM)
    k_xmatvec_d(const __grid_constant__ Geo g, const __grid_constant__ Bufs b, int j, int ncols) {
  cg::cluster_group cl = cg::this_cluster();
  constexpr int nt = Mix<double, WF>::NT;
  const int i = blockIdx.x, vs = blockIdx.y, A = g.A, W = g.W, Lx = g.Lx, T = g.T;
  const int f = slot_freq(g, vs), c = vs - f * g.nb;
  if (c >= ncols) return;                  // same values in every CTA of the cluster
  int* st = b.st + (size_t)f * ST_N;
  if (st[ST_DONE]) return;
  const size_t Ndd = g.Ndd;
  const int nsub = Lx * W, w = T * g.h[i], tid = threadIdx.x;
  const bool has = i < g.p - 1;
  cxd* u = b.u + (size_t)vs * Ndd;
  cxd* us = u + (size_t)i * nsub;
  const cxd* q = b.Q + ((size_t)f * (g.k_max + g.nb) + (size_t)j * g.nb + c) * Ndd;
  MixCtx<double, WF, ROWS> ctx;
  ctx.W = W;
  ctx.Lx = Lx;
  ctx.S = mix_plan<double>(g).S;
  ctx.m = Lx / 2;
  ctx.src = reinterpret_cast<const cxd*>(b.g) + ((size_t)f * g.p + i) * (size_t)nsub * W;
  ctx.g0 = reinterpret_cast<cxd*>(b.yscr) + ((size_t)vs * g.p + i) * nsub;
  ctx.g1 = us;                             // the result's own place: an entry is read before it is written
  ctx.cnt = sweep_cnt(g, b, vs, i);
  ctx.t = g.t;
  MixState<double> ms;
  mix_init<double, WF, ROWS>(ctx, ms);
  int phase = 0;
  layer_diag<double>(g, b, vs, i);
  cxd* B0 = ctx.row(0);
  cxd* B1 = ctx.row(1);
  for (int e = tid; e < nsub; e += nt) B0[e] = e % W < w ? q[(size_t)i * nsub + e] : cxd{0, 0};
  mix_sweep<double, WF, 1, ROWS>(ctx, ms, 0);
  cxd* blo = bnd_ptr<double>(g, b, vs, i, 0);
  cxd* bhi = bnd_ptr<double>(g, b, vs, i, 1);
  for (int e = tid; e < A; e += nt) {
    const int jj = T == 1 ? 0 : e / Lx, s = e - jj * Lx;
    blo[e] = B0[s * W + jj];
    bhi[e] = B0[s * W + (w - T) + jj];
  }
  cl.sync();                               // boundary rows of the neighbours
  const size_t lo = (size_t)g.ifc_off + (size_t)i * A;
  if (has) {
    cxd* Bv = ifv_ptr<double>(g, b, vs, IF_B) + (size_t)i * A;
    const cxd* bnx = bnd_ptr<double>(g, b, vs, i + 1, 0);
    for (int a = tid; a < A; a += nt) Bv[a] = g.t * (bhi[a] + bnx[a]) - q[lo + a];
  }
  __syncthreads();
  const MixSolve<double> sv = mix_cocg<double, WF, ROWS>(g, b, ctx, ms, phase, vs, false);
  for (int e = tid; e < nsub; e += nt) {   // zero on the padding, which the Lanczos step reads too
    cxd v = sv.iters > 0 ? sv.alpha * B1[e] : cxd{0, 0};
    if (sv.useB0) v = v - B0[e];
    us[e] = v;
  }
  if (has) {
    const cxd* X = ifv_ptr<double>(g, b, vs, IF_X) + (size_t)i * A;
    for (int a = tid; a < A; a += nt) u[lo + a] = sv.iters > 0 ? -X[a] : cxd{0, 0};
  }
  mix_drain<double, WF, ROWS>(ctx, ms);
  __syncthreads();
  if (tid == 0 && mix_sm<double, WF>().err) atomicOr(st + ST_STATUS, ST_WAIT_TIMEOUT);
  if (i == 0 && tid == 0) {               // the nb clusters of a frequency share its counters
    atomicAdd(st + ST_ITERS, sv.iters);
    atomicAdd(st + ST_SOLVES, 1);
    if (!sv.conv) atomicOr(st + ST_STATUS, 4);
  }
  cl.sync();          // no CTA exits while a peer may still read its shared memory
}

// w = blkdiag(B^-1, 0) q for DD-layout vectors (Eq. 7), one CTA per subdomain.
template <typename R, int WF, bool ROWS>
__global__ void __launch_bounds__(Mix<R, WF>::NT, Mix<R, WF>::PER_SM)
    k_bsolve_m(const __grid_constant__ Geo g, const __grid_constant__ Bufs b, const cxd* q, cxd* w) {
  constexpr int nt = Mix<R, WF>::NT;
  const int i = blockIdx.x, kf = blockIdx.y, vs = kf * g.nb, W = g.W, nsub = g.Lx * W, wd = g.T * g.h[i];
  MixCtx<R, WF, ROWS> ctx;
  ctx.W = W;
  ctx.Lx = g.Lx;
  ctx.S = mix_plan<R>(g).S;
  ctx.m = g.Lx / 2;
  ctx.src = reinterpret_cast<const cx<R>*>(b.g) + ((size_t)kf * g.p + i) * (size_t)nsub * W;
  ctx.g0 = ctx.g1 = reinterpret_cast<cx<R>*>(b.yscr) + ((size_t)vs * g.p + i) * nsub;
  ctx.cnt = sweep_cnt(g, b, vs, i);
  ctx.t = (R)g.t;
  MixState<R> ms;
  mix_init<R, WF, ROWS>(ctx, ms);
  cx<R>* B0 = ctx.row(0);
  const cxd* qs = q + (size_t)kf * g.Ndd + (size_t)i * nsub;
  cxd* ws = w + (size_t)kf * g.Ndd + (size_t)i * nsub;
  for (int e = threadIdx.x; e < nsub; e += nt) {
    cx<R> v = {0, 0};
    if (e % W < wd) {
      if constexpr (sizeof(R) == 4) v = c2f_bits(qs[e]);
      else v = qs[e];
    }
    B0[e] = v;
  }
  mix_sweep<R, WF, 1, ROWS>(ctx, ms, 0);
  for (int e = threadIdx.x; e < nsub; e += nt)
    if (e % W < wd) {
      if constexpr (sizeof(R) == 4) ws[e] = c2d_bits(B0[e]);
      else ws[e] = B0[e];
    }
  if (i < g.p - 1)
    for (int a = threadIdx.x; a < g.A; a += nt)
      w[(size_t)kf * g.Ndd + g.ifc_off + (size_t)i * g.A + a] = cxd{0, 0};
  mix_drain<R, WF, ROWS>(ctx, ms);
  __syncthreads();
  if (threadIdx.x == 0 && mix_sm<R, WF>().err) atomicOr(b.st + (size_t)kf * ST_N + ST_STATUS, ST_WAIT_TIMEOUT);
}

}  // namespace

template <typename R, int WF>
cudaError_t run_xmatvec_m(const Geo& g, const Bufs& b, int K, int j, int ncols, cudaStream_t st);
template <typename R, int WF>
cudaError_t run_bsolve_m(const Geo& g, const Bufs& b, int K, const cxd* q_dd, cxd* w_dd, cudaStream_t st);

#define DY_CHAIN_VARIANT(R, WF, KERN)                                                                      \
  template <>                                                                                              \
  cudaError_t run_xmatvec_m<R, WF>(const Geo& g, const Bufs& b, int K, int j, int ncols, cudaStream_t st) { \
    const MixPlan mp = mix_plan<R>(g);                                                                     \
    if (mp.rows)                                                                                           \
      return launch_cluster_nt(KERN<WF, true>, dim3(g.p, K * g.nb), g.p, Mix<R, WF>::NT, mp.smem, st, g,   \
                               b, j, ncols);                                                               \
    return launch_cluster_nt(KERN<WF, false>, dim3(g.p, K * g.nb), g.p, Mix<R, WF>::NT, mp.smem, st, g, b, \
                             j, ncols);                                                                    \
  }                                                                                                        \
  template <>                                                                                              \
  cudaError_t run_bsolve_m<R, WF>(const Geo& g, const Bufs& b, int K, const cxd* q_dd, cxd* w_dd,          \
                                  cudaStream_t st) {                                                       \
    const MixPlan mp = mix_plan<R>(g);                                                                     \
    auto kern = mp.rows ? k_bsolve_m<R, WF, true> : k_bsolve_m<R, WF, false>;                              \
    cudaError_t e = raise_smem_limit((const void*)kern, mp.smem);                                          \
    if (e != cudaSuccess) return e;                                                                        \
    kern<<<dim3(g.p, K), Mix<R, WF>::NT, mp.smem, st>>>(g, b, q_dd, w_dd);                                 \
    return cudaGetLastError();                                                                             \
  }

// K1: update + matrix-free residual + norms (Eqs. 3, 1, 19, 2).
//
// Every node first gets the upper-level update of Eq. 3, u += V a (translations,
// gradients and the relaxation modes of the node's own set).  Then each node sums
// the axial forces of its six bars,
//   (K u)_a = sum_b (EA/L)_ab e_ab e_ab^T (u_a - u_b),
// and writes r = p - K u on free DOFs (0 on constrained DOFs), the new u, and
// its share of ||r||_1, ||r||_2^2 and u.(p + r).  The last CTA to finish
// reduces the per-CTA sums in CTA order (deterministic), turns them into the
// relative residuals of Eq. 19 and the energy Pi = 1/2 u.K.u - u.p =
// -1/2 u.(p + r) of Eq. 2, and decides convergence.
//
// The FP64 pipe bounds it (two operations per clock and SM), so the layout is the
// one with the fewest: a warp marches up LatView::rr rows of 32 columns, of which
// the outer two are the neighbours'.  Each bar's force is computed once, by the
// node that owns it, and handed to the other end by a shuffle or, from one row to
// the next, in a register; the update's coefficients of a lane's set are folded
// once per set so that a node's increment is 8 operations.  Per node 18 for r and
// 8 for the sums; with the update 34 in FP64 and 30 in the mixed form, times 32/30
// and the rows below and above a warp's.  One node per thread from a 32 x 8 tile
// with its halo in shared memory took 60 and 42.  Measured: 1024^2 nodes 136 -> 92 us
// in FP64, 117 -> 84 in the mixed form; 1100 x 900 mixed 116 -> 81; below 64 K nodes
// (16 to 20 us) the chain of loads, sums and the last CTA bounds it as before.
//
// In the mixed form (FP32 delta) the increment V a of Eq. 3 is formed in FP32
// and added to the FP64 u: the coefficients of a lane's set are rounded to FP32
// (with the set's representative point as an offset, so that xi and eta are small
// numbers), and a node's increment then costs 4 FP64 operations (two conversions,
// two adds).  The increment carries FP32 rounding errors of about 1e-7 of its
// terms' size, like the FP32 relaxation's delta it multiplies; the residual that
// decides convergence stays FP64, so the iteration still converges to the FP64
// solution (later updates correct what an update got wrong).  The FP64 form, the
// force-controlled modes and sets of only a few nodes keep the FP64 increment.
#include <type_traits>

#include "hms_internal.cuh"
#include "ptx.cuh"

namespace hms {
namespace {

constexpr int TX = 32, TY = 8, NT = TX * TY;  // tiles of the reactions
constexpr int RW = 4, RNT = 32 * RW, RCOLS = 30;  // residual: warps of a CTA, one above the other; columns of a warp

__device__ inline double warp_sum(double v) {
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
  return v;
}

// Deterministic block sum of N values per thread over the TH threads of a
// CTA; the sums land in v of thread 0.  The values go through shared memory:
// warp k adds value k of the warps lane by lane in warp order, then a
// shuffle tree finishes it: a few FP64 adds in N warps instead of a
// shuffle tree in every warp.  sred holds N * (TH + 1) doubles.
template <int N, int TH>
__device__ inline void block_sum(double (&v)[N], double* sred) {
  static_assert(N <= TH / 32, "one warp per value");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll
  for (int k = 0; k < N; ++k) sred[k * TH + tid] = v[k];
  __syncthreads();
  if (warp < N) {
    const double* c = sred + warp * TH + lane;
    double t = c[0];
#pragma unroll
    for (int w = 1; w < TH / 32; ++w) t += c[32 * w];
    t = warp_sum(t);
    if (lane == 0) sred[N * TH + warp] = t;
  }
  __syncthreads();
  if (tid == 0)
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = sred[N * TH + k];
}

template <typename DT>
__device__ inline double2 load_delta(const DT* d, size_t n);
template <>
__device__ inline double2 load_delta<double2>(const double2* d, size_t n) { return d[n]; }
template <>
__device__ inline double2 load_delta<float2>(const float2* d, size_t n) {
  float2 f = d[n];
  return make_double2((double)f.x, (double)f.y);
}

// Whether the mixed form's increment is FP32 (sets of at least a few nodes).
__host__ __device__ inline bool f32_increment_fits(int sx, int sy) {
  return ((TX + 2 + sx - 1) / sx + 1) * ((TY + 2 + sy - 1) / sy + 1) <= 32;
}

__device__ inline double shfl(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ inline double2 shfl(double2 v, int src) { return make_double2(shfl(v.x, src), shfl(v.y, src)); }

// Eq. 3 down one column of nodes: u += sum_m a_m^(I) uhat_m^(I) with the modes of
// Eqs. 9, 10, 13, 14 (zero on constrained DOFs), and with RF the force-
// controlled modes of Eqs. 17-18 (delta^RF and its gradient-weighted copies).
// Rows come in order; enter() takes the coefficients of the set that row j is in.
// In row jr of the set, eta = e0 + h jr, so with xi of even and of odd rows
//   V_x a = (a_0 + a_2 xi + a_3 e0) + (a_3 h) jr + c delta_x,
//   c     = (a_6 + a_7 xi + a_8 e0) + (a_8 h) jr.
template <bool RF>
struct Increment64 {
  double tx[2], ty[2], c[2], cf[2], sx, sy, sc, sf, jr;
  __device__ void enter(const LatView& lv, const double* __restrict__ a, int I, int i, int j, int j0s) {
    const double* aI = a + (size_t)lv.q * I;
    const double2 rep = lv.rep[I];
    const double hh = lv.L * SQ3_2, e0 = fma(hh, (double)j0s, -rep.y);
    const double a2 = __ldg(aI + 2), a3 = __ldg(aI + 3), a4 = __ldg(aI + 4), a5 = __ldg(aI + 5), a7 = __ldg(aI + 7),
                 a8 = __ldg(aI + 8);
    const double x0 = fma(a3, e0, __ldg(aI + 0)), y0 = fma(a5, e0, __ldg(aI + 1)), c0 = fma(a8, e0, __ldg(aI + 6));
    const double xi0 = fma(lv.L, (double)i, -rep.x), xi1 = fma(lv.L, (double)i + 0.5, -rep.x);
    tx[0] = fma(a2, xi0, x0), tx[1] = fma(a2, xi1, x0);
    ty[0] = fma(a4, xi0, y0), ty[1] = fma(a4, xi1, y0);
    c[0] = fma(a7, xi0, c0), c[1] = fma(a7, xi1, c0);
    sx = a3 * hh, sy = a5 * hh, sc = a8 * hh;
    if constexpr (RF) {
      const double a10 = __ldg(aI + 10), a11 = __ldg(aI + 11), f0 = fma(a11, e0, __ldg(aI + 9));
      cf[0] = fma(a10, xi0, f0), cf[1] = fma(a10, xi1, f0);
      sf = a11 * hh;
    }
    jr = (double)(j - j0s);
  }
  // the next row's increment added to v; fm: constrained components
  __device__ double2 add(double2 v, double2 d, double2 f, unsigned fm, int odd) {
    const double cd = fma(sc, jr, odd ? c[1] : c[0]);
    double vx = v.x + fma(cd, d.x, fma(sx, jr, odd ? tx[1] : tx[0]));
    double vy = v.y + fma(cd, d.y, fma(sy, jr, odd ? ty[1] : ty[0]));
    if constexpr (RF) {
      const double g = fma(sf, jr, odd ? cf[1] : cf[0]);
      vx = fma(g, f.x, vx);
      vy = fma(g, f.y, vy);
    }
    jr += 1.0;
    if (!(fm & 1u)) v.x = vx;
    if (!(fm & 2u)) v.y = vy;
    return v;
  }
};
// The same in FP32: xi = L (i - i0s + (j odd ? 1/2 : 0)) + ox, eta = L sqrt3/2
// (j - j0s) + oy with ox = L i0s - x^(I), oy = L sqrt3/2 j0s - y^(I) rounded to FP32.
struct Increment32 {
  float f[NMODES], ox, oy, L, di;
  int jr;
  __device__ void enter(const LatView& lv, const double* __restrict__ a, int I, int i, int j, int j0s) {
    const double* aI = a + (size_t)lv.q * I;
    const double2 rep = lv.rep[I];
    const int i0s = (i / lv.sx) * lv.sx;
#pragma unroll
    for (int m = 0; m < NMODES; ++m) f[m] = (float)__ldg(aI + m);
    ox = (float)fma(lv.L, (double)i0s, -rep.x);
    oy = (float)fma(lv.L * SQ3_2, (double)j0s, -rep.y);
    L = (float)lv.L;
    di = (float)(i - i0s);
    jr = j - j0s;
  }
  __device__ double2 add(double2 v, float2 d, float2, unsigned fm, int odd) {
    const float xi = fmaf(L, di + (odd ? 0.5f : 0.0f), ox);
    const float eta = fmaf(L * (float)SQ3_2, (float)jr, oy);
    const float cd = fmaf(f[8], eta, fmaf(f[7], xi, f[6]));
    ++jr;
    if (!(fm & 1u)) v.x += (double)fmaf(cd, d.x, fmaf(f[3], eta, fmaf(f[2], xi, f[0])));
    if (!(fm & 2u)) v.y += (double)fmaf(cd, d.y, fmaf(f[5], eta, fmaf(f[4], xi, f[1])));
    return v;
  }
};

// A node's loads for the update.
template <typename ET>
struct NodeIn {
  double2 u;
  ET d, f;
  unsigned fm;
};

// The kernel body for CTA (bx, by) of a gx x gy grid (the whole lattice): warp w
// takes rows (RW by + w) rr .. + rr, lane l column RCOLS bx + l - 1.  u is read as
// zero on constrained DOFs.  u_out may be nullptr.
template <typename DT, bool RF, bool F32>
__device__ __forceinline__ void update_residual_rows(
    const LatView& lv, const double2* __restrict__ u_in, double2* __restrict__ u_out, const double2* __restrict__ p,
    const DT* __restrict__ delta, const DT* __restrict__ delta_rf, const double* __restrict__ a,
    double2* __restrict__ r, int bx, int by, double (&s)[3]) {
  using ET = typename std::conditional<F32, float2, double2>::type;
  const bool upd = a != nullptr;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = bx * RCOLS + lane - 1;
  const int jb = (by * RW + warp) * lv.rr, je = min(jb + lv.rr, lv.ny);
  if (jb >= lv.ny) return;
  const bool col = i >= 0 && i < lv.nx, own = col && lane > 0 && lane <= RCOLS;
  const int Ix = col ? i / lv.sx : 0;

  auto load = [&](int j) {
    NodeIn<ET> v;
    v.u = make_double2(0.0, 0.0);
    v.d = v.f = ET{0, 0};
    v.fm = 3u;
    if (!col || j < 0 || j >= lv.ny) return v;
    const size_t n = (size_t)j * lv.nx + i;
    v.u = u_in[n];
    v.fm = lv.fix[n];
    if (upd) {
      if constexpr (F32) v.d = delta[n];
      else v.d = load_delta(delta, n);
      if constexpr (RF) v.f = load_delta(delta_rf, n);
    }
    return v;
  };
  struct Bars {
    double e, ne, nw;
    double2 p;
  };
  auto load_bars = [&](int j) {  // row j's owned bars and, with j its row, the load
    Bars k;
    k.e = bar_k(lv, i, j, 0);
    k.ne = bar_k(lv, i, j, 1);
    k.nw = bar_k(lv, i, j, 2);
    k.p = make_double2(0.0, 0.0);
    if (own) k.p = p[(size_t)j * lv.nx + i];
    return k;
  };
  typename std::conditional<F32, Increment32, Increment64<RF>>::type inc;
  int jset = -1;  // first row of the next set
  auto updated = [&](int j, const NodeIn<ET>& w) {
    double2 v = w.u;
    if (w.fm & 1u) v.x = 0.0;
    if (w.fm & 2u) v.y = 0.0;
    if (upd && j >= 0 && j < lv.ny) {
      if (j >= jset) {
        const int Iy = j / lv.sy;
        inc.enter(lv, a, Iy * lv.Mx + Ix, col ? i : 0, j, Iy * lv.sy);
        jset = (Iy + 1) * lv.sy;
      }
      v = inc.add(v, w.d, w.f, w.fm, j & 1);
    }
    return v;
  };
  // forces of the bars from row j (at v) to row j + 1 (at vn): NE, e = (1/2, sqrt3/2),
  // f1 = k (dx + sqrt3 dy), and NW, e = (-1/2, sqrt3/2), f2 = k (sqrt3 dy - dx); the
  // node's share is (f1 - f2) / 4 in x and sqrt3 / 4 (f1 + f2) in y
  constexpr double SQ3 = 2.0 * SQ3_2;
  auto bars_up = [&](int odd, double kne, double knw, const double2& v, const double2& vn, double& f1, double& f2) {
    const double2 vo = shfl(vn, lane + (odd ? 1 : -1));
    const double2 ne = odd ? vo : vn, nw = odd ? vn : vo;
    f1 = kne * fma(SQ3, v.y - ne.y, v.x - ne.x);
    f2 = knw * fma(SQ3, v.y - nw.y, nw.x - v.x);
  };

  NodeIn<ET> w = load(jb - 1), w1 = load(jb), w2 = load(jb + 1);
  Bars k = load_bars(jb);
  const double kne = bar_k(lv, i, jb - 1, 1), knw = bar_k(lv, i, jb - 1, 2);
  double2 v = updated(jb - 1, w), vn = updated(jb, w1);
  double f1p, f2p;  // forces of the bars from the row below
  bars_up((jb - 1) & 1, kne, knw, v, vn, f1p, f2p);
#pragma unroll 1
  for (int j = jb; j < je; ++j) {
    v = vn;
    w = w2;
    const Bars kc = k;
    if (j + 1 < je) {  // the next row's loads
      w2 = load(j + 2);
      k = load_bars(j + 1);
    }
    vn = updated(j + 1, w);
    const int odd = j & 1;
    const double fe = kc.e * (v.x - shfl(v.x, lane + 1)), fw = shfl(fe, lane - 1);
    double f1, f2;
    bars_up(odd, kc.ne, kc.nw, v, vn, f1, f2);
    const double fo = shfl(odd ? f2p : f1p, lane + (odd ? 1 : -1));
    const double s1 = f1 - (odd ? f1p : fo), s2 = f2 - (odd ? fo : f2p);
    f1p = f1;
    f2p = f2;
    if (own) {
      const size_t n = (size_t)j * lv.nx + i;
      const unsigned fm = w1.fm;
      double2 rn;
      rn.x = fma(-0.25, s1 - s2, kc.p.x - (fe - fw));
      rn.y = fma(-0.5 * SQ3_2, s1 + s2, kc.p.y);
      if (fm & 1u) rn.x = 0.0;
      if (fm & 2u) rn.y = 0.0;
      r[n] = rn;
      if (u_out) u_out[n] = v;
      s[0] += fabs(rn.x);
      s[0] += fabs(rn.y);
      s[1] = fma(rn.x, rn.x, fma(rn.y, rn.y, s[1]));
      s[2] = fma(v.x, kc.p.x + rn.x, fma(v.y, kc.p.y + rn.y, s[2]));
    }
    w1.fm = w.fm;
  }
}

template <typename DT, bool RF = false>
__device__ __forceinline__ void update_residual_body(
    const LatView lv, const double2* __restrict__ u_in, double2* __restrict__ u_out,
    const double2* __restrict__ p, const DT* __restrict__ delta, const DT* __restrict__ delta_rf,
    const double* __restrict__ a,
    double2* __restrict__ r, double* __restrict__ partials, unsigned* ticket, double* norms_out,
    IterCtl* ctl, double* hist, int hist_cap, int bx, int by, int gx, int gy) {
  __shared__ double sred[3 * (RNT + 1)];
  __shared__ bool last;
  int t = 0;
  if (ctl) {
    if (*(volatile int*)&ctl->done) return;
    t = *(volatile int*)&ctl->t;
    if (t == 0) a = nullptr;  // no increment before the first update
  }
  const int tid = threadIdx.x;
  double s[3] = {0.0, 0.0, 0.0};
  constexpr bool MIXED = std::is_same<DT, float2>::value && !RF;
  if (MIXED && f32_increment_fits(lv.sx, lv.sy))
    update_residual_rows<DT, RF, MIXED>(lv, u_in, u_out, p, delta, delta_rf, a, r, bx, by, s);
  else
    update_residual_rows<DT, RF, false>(lv, u_in, u_out, p, delta, delta_rf, a, r, bx, by, s);
  block_sum<3, RNT>(s, sred);
  const unsigned nblocks = (unsigned)(gx * gy);
  const unsigned bid = (unsigned)(by * gx + bx);
  if (tid == 0) {
    partials[3 * (size_t)bid + 0] = s[0];
    partials[3 * (size_t)bid + 1] = s[1];
    partials[3 * (size_t)bid + 2] = s[2];
    __threadfence();
    last = (atomicAdd(ticket, 1u) == nblocks - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double v[3] = {0.0, 0.0, 0.0};
#pragma unroll 4
  for (unsigned b = tid; b < nblocks; b += RNT) {
    v[0] += __ldcg(partials + 3 * (size_t)b + 0);
    v[1] += __ldcg(partials + 3 * (size_t)b + 1);
    v[2] += __ldcg(partials + 3 * (size_t)b + 2);
  }
  __syncthreads();
  block_sum<3, RNT>(v, sred);
  if (tid == 0) {
    *ticket = 0u;  // ready for the next launch
    if (norms_out) {
      norms_out[0] = v[0];
      norms_out[1] = v[1];
      norms_out[2] = v[2];
    }
    if (ctl) {
      const double R1 = ctl->p1 > 0.0 ? v[0] / ctl->p1 : 0.0;
      const double R2 = ctl->p2 > 0.0 ? sqrt(v[1]) / ctl->p2 : 0.0;
      const double Pi = -0.5 * v[2];
      if (t < hist_cap && hist) {
        hist[3 * t + 0] = R1;
        hist[3 * t + 1] = R2;
        hist[3 * t + 2] = Pi;
      }
      if (!isfinite(R1) || !isfinite(R2) || !isfinite(Pi)) {
        ctl->status = 3;
        ctl->err |= DEVERR_NONFINITE;
        ctl->done = 1;
      } else if (R1 < ctl->tol) {
        ctl->status = 1;
        ctl->done = 1;
      } else if (t >= ctl->max_iter || ctl->err != 0) {
        ctl->status = 2;
        ctl->done = 1;
      }
      ctl->t = t + 1;
    }
  }
}

template <typename DT, bool RF>
__global__ void __launch_bounds__(RNT) k_update_residual(
    LatView lv, const double2* __restrict__ u_in, double2* __restrict__ u_out,
    const double2* __restrict__ p, const DT* __restrict__ delta, const DT* __restrict__ delta_rf,
    const double* __restrict__ a, double2* __restrict__ r, double* __restrict__ partials, unsigned* ticket,
    double* norms_out, IterCtl* ctl, double* hist, int hist_cap) {
  dep_wait();
  update_residual_body<DT, RF>(lv, u_in, u_out, p, delta, delta_rf, a, r, partials, ticket, norms_out, ctl, hist,
                               hist_cap, blockIdx.x, blockIdx.y, gridDim.x, gridDim.y);
}

// Batched: update k of a CUDA-graph round (u ping-pongs between u[k & 1] and
// u[(k + 1) & 1]) for the tiles of every problem of a batch.
template <typename DT>
__global__ void __launch_bounds__(RNT) kb_update_residual(const BatchProb* __restrict__ P,
                                                         const BatchItem* __restrict__ items, int k) {
  const BatchItem it = items[blockIdx.x];
  const BatchProb& q = P[it.prob];
  update_residual_body<DT>(q.lv, q.u[k & 1], q.u[(k + 1) & 1], q.p, (const DT*)q.delta, nullptr, q.a, q.r,
                           q.partials, q.ticket, nullptr, q.ctl, q.hist, q.hist_cap, it.bx, it.by, it.gx, it.gy);
}

// Masks the loads on constrained DOFs and computes ||p||_1, ||p||_2 into ctl.
__global__ void __launch_bounds__(NT) k_load_norms(LatView lv, double2* __restrict__ p,
                                                    double* __restrict__ partials, unsigned* ticket,
                                                    IterCtl* ctl) {
  __shared__ double sred[2 * (NT + 1)];
  __shared__ bool last;
  const size_t nn = (size_t)lv.nx * lv.ny;
  double s[2] = {0.0, 0.0};
  for (size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x; n < nn;
       n += (size_t)gridDim.x * blockDim.x) {
    double2 v = p[n];
    const unsigned fm = lv.fix[n];
    if (fm & 1u) v.x = 0.0;
    if (fm & 2u) v.y = 0.0;
    p[n] = v;
    s[0] += fabs(v.x) + fabs(v.y);
    s[1] += fma(v.x, v.x, v.y * v.y);
  }
  block_sum<2, NT>(s, sred);
  if (threadIdx.x == 0) {
    partials[2 * blockIdx.x + 0] = s[0];
    partials[2 * blockIdx.x + 1] = s[1];
    __threadfence();
    last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double v[2] = {0.0, 0.0};
  for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
    v[0] += __ldcg(partials + 2 * b + 0);
    v[1] += __ldcg(partials + 2 * b + 1);
  }
  __syncthreads();
  block_sum<2, NT>(v, sred);
  if (threadIdx.x == 0) {
    *ticket = 0u;
    ctl->p1 = v[0];
    ctl->p2 = sqrt(v[1]);
  }
}

// K u at every DOF (constrained ones included): the nodal forces of the bars,
// with u read as 0 on constrained DOFs.  One CTA per 32 x 8 node tile and its
// one-node halo in shared memory, the six bars of each node summed as in the
// residual above.
__global__ void __launch_bounds__(NT) k_reactions(LatView lv, const double2* __restrict__ u,
                                                  double2* __restrict__ f) {
  __shared__ double2 U[TY + 2][TX + 2];
  const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY;
  const int tid = threadIdx.x;
  for (int idx = tid; idx < (TX + 2) * (TY + 2); idx += NT) {
    const int lx = idx % (TX + 2), ly = idx / (TX + 2);
    const int i = i0 + lx - 1, j = j0 + ly - 1;
    double2 v = make_double2(0.0, 0.0);
    if (i >= 0 && i < lv.nx && j >= 0 && j < lv.ny) {
      const size_t n = (size_t)j * lv.nx + i;
      v = u[n];
      const unsigned fm = lv.fix[n];
      if (fm & 1u) v.x = 0.0;
      if (fm & 2u) v.y = 0.0;
    }
    U[ly][lx] = v;
  }
  __syncthreads();
  const int tx = tid % TX, ty = tid / TX;
  const int i = i0 + tx, j = j0 + ty;
  if (i >= lv.nx || j >= lv.ny) return;
  const int lx = tx + 1, ly = ty + 1, off = j & 1;
  const double2 uc = U[ly][lx];
  const double kE = bar_k(lv, i, j, 0), kW = bar_k(lv, i - 1, j, 0);
  double fx = kE * (uc.x - U[ly][lx + 1].x) + kW * (uc.x - U[ly][lx - 1].x);
  const double kNE = bar_k(lv, i, j, 1), kSW = bar_k(lv, i - 1 + off, j - 1, 1);
  const double2 une = U[ly + 1][lx + off], usw = U[ly - 1][lx - 1 + off];
  const double d1x = kNE * (uc.x - une.x) + kSW * (uc.x - usw.x);
  const double d1y = kNE * (uc.y - une.y) + kSW * (uc.y - usw.y);
  const double p1 = fma(SQ3_2, d1y, 0.5 * d1x);
  const double kNW = bar_k(lv, i, j, 2), kSE = bar_k(lv, i + off, j - 1, 2);
  const double2 unw = U[ly + 1][lx - 1 + off], use = U[ly - 1][lx + off];
  const double d2x = kNW * (uc.x - unw.x) + kSE * (uc.x - use.x);
  const double d2y = kNW * (uc.y - unw.y) + kSE * (uc.y - use.y);
  const double p2 = fma(SQ3_2, d2y, -0.5 * d2x);
  fx = fma(0.5, p1 - p2, fx);
  f[(size_t)j * lv.nx + i] = make_double2(fx, SQ3_2 * (p1 + p2));
}

}  // namespace

cudaError_t launch_reactions(cudaStream_t s, const LatView& lv, const double2* u, double2* f) {
  dim3 grid((lv.nx + TX - 1) / TX, (lv.ny + TY - 1) / TY);
  k_reactions<<<grid, NT, 0, s>>>(lv, u, f);
  return cudaGetLastError();
}

// Rows of a warp: the count (up to 32) that costs the busiest SM the
// fewest FP64 operations, with 34 per row of a warp and 26 for its two outer rows.
// Small lattices get one or two rows (64 x 64 nodes: 1), 1024 x 1024 nodes 10.
int update_residual_rr(const LatView& lv) {
  const long long strips = (lv.nx + RCOLS - 1) / RCOLS;
  long long best = -1;
  int rr = 1;
  for (int h = 1; h <= 32; ++h) {
    const long long ctas = strips * ((lv.ny + RW * h - 1) / (RW * h)), cost = (ctas + lv.nsm - 1) / lv.nsm * (34 * h + 26);
    if (best < 0 || cost <= best) best = cost, rr = h;
  }
  return rr;
}
int update_residual_grid_x(const LatView& lv) { return (lv.nx + RCOLS - 1) / RCOLS; }
int update_residual_grid_y(const LatView& lv) {
  const int rows = RW * update_residual_rr(lv);
  return (lv.ny + rows - 1) / rows;
}
int update_residual_blocks(const LatView& lv) { return update_residual_grid_x(lv) * update_residual_grid_y(lv); }

cudaError_t launch_batch_update_residual(cudaStream_t s, bool fp32, const BatchProb* P, const BatchItem* it, int n,
                                         int k) {
  if (n <= 0) return cudaSuccess;
  if (fp32) kb_update_residual<float2><<<n, RNT, 0, s>>>(P, it, k);
  else kb_update_residual<double2><<<n, RNT, 0, s>>>(P, it, k);
  return cudaGetLastError();
}

cudaError_t launch_update_residual(cudaStream_t s, const LatView& lv, const double2* u_in,
                                   double2* u_out, const double2* p, const void* delta,
                                   bool delta_fp32, const double* a, double2* r, double* partials,
                                   unsigned* ticket, double* norms_out, IterCtl* ctl, double* hist,
                                   int hist_cap, const void* delta_rf) {
  const dim3 grid(update_residual_grid_x(lv), (lv.ny + RW * lv.rr - 1) / (RW * lv.rr));
  const bool rf = lv.q == NMODES_RF;
  auto go = [&](auto k, auto* d) {
    using DT = std::remove_pointer_t<decltype(d)>;
    return launch_dep(k, s, grid, RNT, 0, 0, lv, u_in, u_out, p, (const DT*)delta, rf ? (const DT*)delta_rf : nullptr, a,
                      r, partials, ticket, norms_out, ctl, hist, hist_cap);
  };
  if (delta_fp32)
    return rf ? go(k_update_residual<float2, true>, (float2*)nullptr)
              : go(k_update_residual<float2, false>, (float2*)nullptr);
  return rf ? go(k_update_residual<double2, true>, (double2*)nullptr)
            : go(k_update_residual<double2, false>, (double2*)nullptr);
}

cudaError_t launch_load_norms(cudaStream_t s, const LatView& lv, double2* p, double* partials,
                              unsigned* ticket, IterCtl* ctl) {
  const size_t nn = (size_t)lv.nx * lv.ny;
  int grid = (int)((nn + 255) / 256);
  if (grid > 1024) grid = 1024;
  k_load_norms<<<grid, NT, 0, s>>>(lv, p, partials, ticket, ctl);
  return cudaGetLastError();
}

}  // namespace hms

// K3: the upper-level matrix K_aa = V^T K V of Eq. 6, and its band storage.
//
// K = sum over bars of (EA/L) g g^T with g = e at the owner's DOFs and -e at
// the other end's, so a bar adds (EA/L) s s^T to K_aa, where s_m = e . (V_m(a)
// - V_m(b)) over the modes of the (at most two) sets the bar touches.  A bar
// inside set I touches only I's nine modes; a bar crossing to a neighbour set
// J touches 18 (I's at the owner a, J's at b with a minus sign).
//
// The bars owned by set I's nodes are summed into six 2 q x 2 q slots:
// SELF (bars inside I, upper-left q x q used) and E, W, N, NE, NW (bars to the
// neighbour set in that direction; rows/cols 0..q-1 = I's modes, q.. = J's).
// The translation/gradient entries (modes 1-6) do not depend on delta: they
// are summed once at setup into a base copy, and every iteration only the
// entries that involve the increment modes (7-9, and 10-12 with the force-
// controlled modes of Eqs. 17-18) are summed.  For bars inside I with all four
// DOFs free the translation terms vanish and the gradient terms are constants of
// the bar direction, so those bars only accumulate e.delta sums per direction;
// bars touching a constrained DOF use the general form.  All sums run in a fixed
// order, so the result is the same on every run.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "coarse_blocks.cuh"
#include "hms_internal.cuh"
#include "ptx.cuh"

namespace cg = cooperative_groups;

namespace hms {
namespace {

constexpr int NT = 256, NW = NT / 32;
constexpr int RED_CHUNK = NW;     // accumulators per shared-memory reduction pass

__device__ inline double warp_sum(double v) {
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
  return v;
}

template <typename DT>
__device__ inline double2 ld_delta(const DT* d, size_t n);
template <>
__device__ inline double2 ld_delta<double2>(const double2* d, size_t n) { return d[n]; }
template <>
__device__ inline double2 ld_delta<float2>(const float2* d, size_t n) {
  const float2 f = d[n];
  return make_double2((double)f.x, (double)f.y);
}

// e . V_m at a node, modes m = 0..8 (Eqs. 9, 10, 13, 14), zero on constrained DOFs.
__device__ inline void mode_proj(double ex, double ey, double xi, double eta, unsigned fm, double2 dl,
                                 double* s) {
  const double fx = (fm & 1u) ? 0.0 : 1.0, fy = (fm & 2u) ? 0.0 : 1.0;
  const double ed = ex * dl.x + ey * dl.y;  // delta is 0 on constrained DOFs
  s[0] = ex * fx;
  s[1] = ey * fy;
  s[2] = ex * xi * fx;
  s[3] = ex * eta * fx;
  s[4] = ey * xi * fy;
  s[5] = ey * eta * fy;
  s[6] = ed;
  s[7] = xi * ed;
  s[8] = eta * ed;
}

// mode_proj in the arithmetic AT of the per-bar products (the same formula)
template <typename AT>
__device__ inline void mode_proj_t(AT ex, AT ey, AT xi, AT eta, unsigned fm, AT dx, AT dy, AT* s) {
  const AT fx = (fm & 1u) ? AT(0) : AT(1), fy = (fm & 2u) ? AT(0) : AT(1);
  const AT ed = ex * dx + ey * dy;
  s[0] = ex * fx;
  s[1] = ey * fy;
  s[2] = ex * xi * fx;
  s[3] = ex * eta * fx;
  s[4] = ey * xi * fy;
  s[5] = ey * eta * fy;
  s[6] = ed;
  s[7] = xi * ed;
  s[8] = eta * ed;
}
struct ListCaps {
  int cap[6], off[6], total;
};
__host__ __device__ inline ListCaps list_caps(int w, int h) {
  ListCaps c;
  c.cap[SLOT_SELF] = 0;
  c.cap[SLOT_E] = 2 * h;
  c.cap[SLOT_W] = h;
  c.cap[SLOT_N] = 2 * w;
  c.cap[SLOT_NE] = 2;
  c.cap[SLOT_NW] = 2;
  int o = 0;
  for (int k = 0; k < 6; ++k) {
    c.off[k] = o;
    o += c.cap[k];
  }
  c.total = o;
  return c;
}

// The slot of an interface bar of direction d at node (il, jl) of the set, whose far
// end lies in the set (dxs, dys) away, and its place in the slot's list.
__device__ inline void slot_place(int d, int il, int jl, int dxs, int dys, int& slot, int& idx) {
  if (dys == 0) {
    slot = dxs > 0 ? SLOT_E : SLOT_W;
    idx = dxs > 0 ? 2 * jl + (d == 1 ? 1 : 0) : jl;
  } else if (dxs == 0) {
    slot = SLOT_N;
    idx = 2 * il + (d == 2 ? 1 : 0);
  } else {
    slot = dxs > 0 ? SLOT_NE : SLOT_NW;
    idx = (dxs > 0) == (d == 1) ? 0 : 1;
  }
}

// ---- setup: the entries of modes 1-6 ----
// One CTA per set, FP64: the bars inside the set per thread, then a fixed-shape
// tree; the interface bars' lists slot by slot, in index order.
constexpr int QB = 6, NBASE = QB * (QB + 1) / 2;
constexpr int LSTRIDE = 4 * QB;  // s_a, -s_b, k s_a, -k s_b
__global__ void __launch_bounds__(NT) k_coarse_base(LatView lv, double* __restrict__ slots) {
  extern __shared__ double lists[];
  const int I = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int SD = 2 * lv.q, SZ = SD * SD;
  const int Ix = I % lv.Mx, Iy = I / lv.Mx;
  const int i0 = Ix * lv.sx, j0 = Iy * lv.sy;
  const int w = min(lv.sx, lv.nx - i0), h = min(lv.sy, lv.ny - j0);
  const ListCaps LC = list_caps(w, h);
  double* out = slots + (size_t)I * NSLOTS * SZ;
  for (int q = tid; q < LC.total * LSTRIDE; q += NT) lists[q] = 0.0;
  for (int q = tid; q < NSLOTS * SZ; q += NT) out[q] = 0.0;
  __syncthreads();

  const double2 repI = lv.rep[I], none = make_double2(0.0, 0.0);
  double gen[NBASE];
#pragma unroll
  for (int k = 0; k < NBASE; ++k) gen[k] = 0.0;
  for (int t = tid; t < 3 * w * h; t += NT) {
    const int q = t / 3, d = t - 3 * q;
    const int il = q % w, jl = q / w, i = i0 + il, j = j0 + jl, off = j & 1;
    const double k = bar_k(lv, i, j, d);
    if (__double_as_longlong(k) == 0) continue;  // no bar (bar_k returns +0.0; EA > 0): an integer test
    const int ib = (d == 0) ? i + 1 : (d == 1 ? i + off : i - 1 + off);
    const int jb = (d == 0) ? j : j + 1;
    const int dxs = (ib >= i0 + w) ? 1 : (ib < i0 ? -1 : 0);
    const int dys = (jb >= j0 + h) ? 1 : 0;
    const unsigned fa = lv.fix[(size_t)j * lv.nx + i], fb = lv.fix[(size_t)jb * lv.nx + ib];
    const double ex = (d == 0) ? 1.0 : (d == 1 ? 0.5 : -0.5), ey = (d == 0) ? 0.0 : SQ3_2;
    const double2 repJ = lv.rep[(Iy + dys) * lv.Mx + Ix + dxs];
    double sa[NMODES], sb[NMODES];
    mode_proj(ex, ey, node_x(lv, i, j) - repI.x, node_y(lv, j) - repI.y, fa, none, sa);
    mode_proj(ex, ey, node_x(lv, ib, jb) - repJ.x, node_y(lv, jb) - repJ.y, fb, none, sb);
    if (dxs == 0 && dys == 0) {
#pragma unroll
      for (int m = 0; m < QB; ++m) sa[m] -= sb[m];
#pragma unroll
      for (int m = 0; m < QB; ++m)
#pragma unroll
        for (int l = 0; l <= m; ++l) gen[m * (m + 1) / 2 + l] = fma(k * sa[m], sa[l], gen[m * (m + 1) / 2 + l]);
      continue;
    }
    int slot, idx;
    slot_place(d, il, jl, dxs, dys, slot, idx);
    double* e = lists + (size_t)(LC.off[slot] + idx) * LSTRIDE;
#pragma unroll
    for (int m = 0; m < QB; ++m) {
      e[m] = sa[m];
      e[QB + m] = -sb[m];
      e[2 * QB + m] = k * sa[m];
      e[3 * QB + m] = -(k * sb[m]);
    }
  }
  // deterministic block sums of the per-thread accumulators, RED_CHUNK at a time
  double* red = lists + (size_t)LC.total * LSTRIDE;  // RED_CHUNK x NT
  double* tot = red + RED_CHUNK * NT;                // NBASE CTA totals
#pragma unroll
  for (int c0 = 0; c0 < NBASE; c0 += RED_CHUNK) {
#pragma unroll
    for (int q = 0; q < RED_CHUNK; ++q)
      if (c0 + q < NBASE) red[q * NT + tid] = gen[c0 + q];
    __syncthreads();
    if (c0 + warp < NBASE) {
      const double* q = red + warp * NT + lane;
      double v = q[0];
#pragma unroll
      for (int ww = 1; ww < NW; ++ww) v += q[32 * ww];
      v = warp_sum(v);
      if (lane == 0) tot[c0 + warp] = v;
    }
    __syncthreads();
  }
  if (tid < QB * QB) {
    const int m = tid / QB, l = tid % QB;
    const int mm = m > l ? m : l, ll = m > l ? l : m;
    out[SLOT_SELF * SZ + m * SD + l] = tot[mm * (mm + 1) / 2 + ll];
  }
  // entries (p, c) of I's modes (0..5) and the neighbour's (6..11)
  for (int q = tid; q < 5 * 4 * QB * QB; q += NT) {
    const int slot = 1 + q / (4 * QB * QB), r = q % (4 * QB * QB), p = r / (2 * QB), c = r % (2 * QB);
    if (c < p) continue;
    const double* e = lists + (size_t)LC.off[slot] * LSTRIDE;
    double v = 0.0;
    for (int b = 0; b < LC.cap[slot]; ++b, e += LSTRIDE) v = fma(e[2 * QB + p], e[c], v);
    const int pp = p < QB ? p : lv.q + p - QB, cc = c < QB ? c : lv.q + c - QB;
    out[slot * SZ + pp * SD + cc] = v;
    out[slot * SZ + cc * SD + pp] = v;
  }
}

// mode_proj with the force-controlled modes 10-12 of Eqs. 17-18: s_9 = e.delta^RF,
// s_10 = xi s_9, s_11 = eta s_9
__device__ inline void mode_proj12(double ex, double ey, double xi, double eta, unsigned fm, double2 dl,
                                   double2 df, double* s) {
  mode_proj(ex, ey, xi, eta, fm, dl, s);
  const double ef = ex * df.x + ey * df.y;  // delta^RF is 0 on constrained DOFs
  s[9] = ef;
  s[10] = xi * ef;
  s[11] = eta * ef;
}
// ---- every update: the entries that involve the increment modes ----
// The bars inside a set in SP fixed parts of its nodes, a warp each (32 nodes, then
// every 32 SP-th), summed part by part; the bars to the neighbours slot by slot in
// list order.  Neither depends on how many CTAs (of one cluster) share a set's parts
// and slots, so C = 1 to 4 CTAs give the same bits: four where 152 SMs leave room
// for four per set.  A warp of each SM quarter is all that the FP64 pipe can use.
//
// Q = 9 or 12 modes; NS = 3 or 6 projections s_6.. of a bar.  A regular bar (all
// four DOFs free) adds k s_m to its direction's sum (s_2..s_5 are constants of the
// direction) and k s_m s_l to the products', 50 FP64 operations per node for Q = 9
// and 8 for its three bars' projections; bars at constrained DOFs take the general
// form in a second pass of the warps that have any.  PT: arithmetic of the
// projections, AT: of the products and of a lane's sums, ST: of the sums over lanes (the
// mixed form's: PT and ST FP64 with the force-controlled modes, else FP32).
//
// Measured (us, before: one CTA of 256 threads per set, with Q = 12 every bar in
// the general form): FP64, 16 sets of 16 x 16 nodes 28 -> 23, 256 of 64 x 64 250
// -> 190; mixed 52 -> 43; Q = 12, 48 of 32 x 32 115 -> 65, mixed 98 -> 62 (48 with the
// sums over lanes in FP32).
constexpr int SP = 16;
template <int Q>
struct SlotSums {
  static constexpr int NS = Q == NMODES_RF ? 6 : 3;
  static constexpr int NLIN = 3 * NS, NQUAD = NS * (NS + 1) / 2;
  static constexpr int NGEN = NS * (NS + 1) / 2 + 6 * NS;  // (m, l), 6 <= m < Q, l <= m
  static constexpr int NACC = NLIN + NQUAD + NGEN;
  static constexpr int NPAIR = 2 * Q * (2 * Q + 1) / 2 - 78;  // p <= c of a slot, one of them >= 6
};
// the pairs of a slot's entries that involve an increment mode
template <int Q>
struct SlotPairs {
  unsigned char p[SlotSums<Q>::NPAIR], c[SlotSums<Q>::NPAIR];
};
template <int Q>
constexpr SlotPairs<Q> slot_pairs() {
  SlotPairs<Q> t{};
  int n = 0;
  for (int p = 0; p < 2 * Q; ++p)
    for (int c = p; c < 2 * Q; ++c)
      if (p % Q >= 6 || c % Q >= 6) {
        t.p[n] = (unsigned char)p;
        t.c[n++] = (unsigned char)c;
      }
  return t;
}
__device__ const SlotPairs<NMODES> PAIRS9 = slot_pairs<NMODES>();
__device__ const SlotPairs<NMODES_RF> PAIRS12 = slot_pairs<NMODES_RF>();

// Sums over a warp of N values per lane, N adds and a few, in ST: value k's sum ends
// in lane k (k < 32) and, of values 32.., in lane k - 32, and is stored at dst[k].
template <typename ST, int N, typename AT>
__device__ __forceinline__ void warp_sums(AT (&v)[N], double* dst) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int b = 0; b < N; b += 32) {
    ST x[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) x[k] = b + k < N ? (ST)v[b + k < N ? b + k : 0] : ST(0);
    // halve the values, not the lanes: after step m a lane holds those whose number
    // agrees with its own in the bits seen
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
      const bool up = lane & m;
#pragma unroll
      for (int k = 0; k < m; ++k) {
        if (b + k >= N) continue;  // neither half holds a value
        const ST give = up ? x[k] : x[k + m], keep = up ? x[k + m] : x[k];
        x[k] = keep + __shfl_xor_sync(0xffffffffu, give, m);
      }
    }
    if (b + lane < N) dst[b + lane] = (double)x[0];
  }
}

template <int Q, typename LT>
__host__ __device__ inline size_t slots_it_smem(const ListCaps& LC) {
  // the lists (s_a, -s_b, k s_a, -k s_b), then the parts' sums
  return (size_t)LC.total * 4 * Q * sizeof(LT) + (size_t)SP * SlotSums<Q>::NACC * sizeof(double);
}

template <typename DT, int Q, typename AT>
__device__ __forceinline__ void slots_it_body(const LatView& lv, const DT* __restrict__ delta,
                                              const DT* __restrict__ delta_rf, double* __restrict__ slots, int I) {
  using SS = SlotSums<Q>;
  using LT = typename std::conditional<Q == NMODES_RF, double, AT>::type;  // of the lists
  using PT = LT;
  using ST = LT;
  constexpr int NS = SS::NS, NF = NS / 3, LST = 4 * Q, SD = 2 * Q, SZ = SD * SD;
  extern __shared__ double lists[];
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x;
  if (C > 1) cluster_arrive();
  const int Ix = I % lv.Mx, Iy = I / lv.Mx;
  const int i0 = Ix * lv.sx, j0 = Iy * lv.sy;
  const int w = min(lv.sx, lv.nx - i0), h = min(lv.sy, lv.ny - j0);
  const ListCaps LC = list_caps(w, h);
  double* out = slots + (size_t)I * NSLOTS * SZ;
  double* part = lists;  // SP x NACC (rank 0's holds the cluster's)
  LT* la = reinterpret_cast<LT*>(lists + SP * SS::NACC);
  auto mine = [&](int slot) { return (slot - 1) % C == rank; };  // slots E, W, N, NE, NW
  for (int sl = 1; sl < NSLOTS; ++sl)
    if (mine(sl))
      for (int q = tid; q < LC.cap[sl] * LST; q += nt) la[(size_t)LC.off[sl] * LST + q] = LT(0);
  __syncthreads();

  // Interface bars (the far end in a neighbour set): the right column's E and NE
  // bars, the left column's NW bars, the top row's NE and NW bars.  Each list entry
  // is written by one item.
  const double2 repI = lv.rep[I];
  for (int t = tid; t < 3 * h + 2 * w; t += nt) {
    int il, jl, d;
    if (t < 2 * h) {
      il = w - 1, jl = t >> 1, d = t & 1;
    } else if (t < 3 * h) {
      il = 0, jl = t - 2 * h, d = 2;
    } else {
      const int u = t - 3 * h;
      il = u >> 1, jl = h - 1, d = 1 + (u & 1);
      if ((d == 1 && il == w - 1) || (d == 2 && il == 0)) continue;  // in the column groups
    }
    const int i = i0 + il, j = j0 + jl, off = j & 1;
    const int ib = (d == 0) ? i + 1 : (d == 1 ? i + off : i - 1 + off);
    const int jb = (d == 0) ? j : j + 1;
    const int dxs = (ib >= i0 + w) ? 1 : (ib < i0 ? -1 : 0);
    const int dys = (jb >= j0 + h) ? 1 : 0;
    if (dxs == 0 && dys == 0) continue;  // an inner bar (below)
    int slot, idx;
    slot_place(d, il, jl, dxs, dys, slot, idx);
    if (!mine(slot)) continue;
    const double k = bar_k(lv, i, j, d);
    if (__double_as_longlong(k) == 0) continue;  // no bar (bar_k returns +0.0; EA > 0): an integer test
    const size_t na = (size_t)j * lv.nx + i, nbn = (size_t)jb * lv.nx + ib;
    const unsigned fa = lv.fix[na], fb = lv.fix[nbn];
    const double ex = (d == 0) ? 1.0 : (d == 1 ? 0.5 : -0.5), ey = (d == 0) ? 0.0 : SQ3_2;
    const double2 repJ = lv.rep[(Iy + dys) * lv.Mx + Ix + dxs];
    const double xa = node_x(lv, i, j), ya = node_y(lv, j), xb = node_x(lv, ib, jb), yb = node_y(lv, jb);
    const double2 da = ld_delta(delta, na), db = ld_delta(delta, nbn);
    LT sa[Q], sb[Q];
    if constexpr (Q == NMODES_RF) {
      mode_proj12(ex, ey, xa - repI.x, ya - repI.y, fa, da, ld_delta(delta_rf, na), sa);
      mode_proj12(ex, ey, xb - repJ.x, yb - repJ.y, fb, db, ld_delta(delta_rf, nbn), sb);
    } else {
      mode_proj_t<LT>((LT)ex, (LT)ey, (LT)(xa - repI.x), (LT)(ya - repI.y), fa, (LT)da.x, (LT)da.y, sa);
      mode_proj_t<LT>((LT)ex, (LT)ey, (LT)(xb - repJ.x), (LT)(yb - repJ.y), fb, (LT)db.x, (LT)db.y, sb);
    }
    LT* e = la + (size_t)(LC.off[slot] + idx) * LST;
    const LT kL = (LT)k;
#pragma unroll
    for (int m = 0; m < Q; ++m) {
      e[m] = sa[m];
      e[Q + m] = -sb[m];
      e[2 * Q + m] = kL * sa[m];
      e[3 * Q + m] = -(kL * sb[m]);
    }
  }

  // ---- bars inside the set ----
  if (C > 1) cluster_wait();  // rank 0 runs: its shared memory may be written
  double* part0 = cluster.map_shared_rank(part, 0);
  const PT LA = (PT)lv.L, LyA = (PT)(lv.L * SQ3_2);
  const PT c0x = (PT)fma(lv.L, (double)i0, -repI.x), c0y = (PT)fma(lv.L * SQ3_2, (double)j0, -repI.y);
  for (int pt = rank + C * warp; pt < SP; pt += C * (nt >> 5)) {
    AT acc[SS::NLIN + SS::NQUAD];
#pragma unroll
    for (int k = 0; k < SS::NLIN + SS::NQUAD; ++k) acc[k] = AT(0);
    bool special = false;  // a bar at a constrained DOF
#pragma unroll 1
    for (int q = 32 * pt + lane; q < w * h; q += 32 * SP) {
      const int jl = q / w, il = q - jl * w;
      const int i = i0 + il, j = j0 + jl, off = j & 1;
      const size_t na = (size_t)j * lv.nx + i;
      const unsigned fa = lv.fix[na];
      DT da[NF], db[NF];
      da[0] = delta[na];
      if constexpr (NF == 2) da[1] = delta_rf[na];
      const PT xi = fma(LA, (PT)il + (off ? PT(0.5) : PT(0)), c0x), eta = fma(LyA, (PT)jl, c0y);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int ib = (d == 0) ? i + 1 : (d == 1 ? i + off : i - 1 + off);
        const int jb = (d == 0) ? j : j + 1;
        if (ib >= i0 + w || ib < i0 || jb >= j0 + h) continue;
        const double k = bar_k(lv, i, j, d);
        if (__double_as_longlong(k) == 0) continue;
        const size_t nbn = (size_t)jb * lv.nx + ib;
        if ((fa | lv.fix[nbn]) != 0u) {
          special = true;
          continue;
        }
        db[0] = delta[nbn];
        if constexpr (NF == 2) db[1] = delta_rf[nbn];
        // e = (1, 0), (1/2, sqrt3/2), (-1/2, sqrt3/2); the far end at (xi, eta) + L e:
        // s_6 = e.da - e.db, s_7 = xi s_6 - L e_x e.db, s_8 = eta s_6 - L e_y e.db
        const PT hx = d == 1 ? PT(0.5) : PT(-0.5), kP = (PT)k;
        PT s[NS];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
          const PT ea = d == 0 ? (PT)da[f].x : fma(hx, (PT)da[f].x, (PT)SQ3_2 * (PT)da[f].y);
          const PT eb = d == 0 ? (PT)db[f].x : fma(hx, (PT)db[f].x, (PT)SQ3_2 * (PT)db[f].y);
          s[3 * f] = ea - eb;
          s[3 * f + 1] = fma(xi, s[3 * f], (d == 0 ? -LA : -(hx * LA)) * eb);
          s[3 * f + 2] = d == 0 ? eta * s[3 * f] : fma(eta, s[3 * f], -LyA * eb);
        }
#pragma unroll
        for (int m = 0; m < NS; ++m) {
          const AT km = (AT)(kP * s[m]);
          acc[NS * d + m] += km;
#pragma unroll
          for (int l = 0; l <= m; ++l)
            acc[SS::NLIN + m * (m + 1) / 2 + l] = fma(km, (AT)s[l], acc[SS::NLIN + m * (m + 1) / 2 + l]);
        }
      }
    }
    double* dst = part0 + (size_t)pt * SS::NACC;
    warp_sums<ST>(acc, dst);
    dst += SS::NLIN + SS::NQUAD;
    if (!__any_sync(0xffffffffu, special)) {
      for (int k = lane; k < SS::NGEN; k += 32) dst[k] = 0.0;
      continue;
    }
    AT gen[SS::NGEN];
#pragma unroll
    for (int k = 0; k < SS::NGEN; ++k) gen[k] = AT(0);
#pragma unroll 1
    for (int q = 32 * pt + lane; q < w * h; q += 32 * SP) {
      const int jl = q / w, il = q - jl * w;
      const int i = i0 + il, j = j0 + jl, off = j & 1;
      const size_t na = (size_t)j * lv.nx + i;
      const unsigned fa = lv.fix[na];
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {
        const int ib = (d == 0) ? i + 1 : (d == 1 ? i + off : i - 1 + off);
        const int jb = (d == 0) ? j : j + 1;
        if (ib >= i0 + w || ib < i0 || jb >= j0 + h) continue;
        const double k = bar_k(lv, i, j, d);
        if (__double_as_longlong(k) == 0) continue;
        const size_t nbn = (size_t)jb * lv.nx + ib;
        const unsigned fb = lv.fix[nbn];
        if ((fa | fb) == 0u) continue;
        const double ex = (d == 0) ? 1.0 : (d == 1 ? 0.5 : -0.5), ey = (d == 0) ? 0.0 : SQ3_2;
        const double xa = node_x(lv, i, j) - repI.x, ya = node_y(lv, j) - repI.y;
        const double xb = node_x(lv, ib, jb) - repI.x, yb = node_y(lv, jb) - repI.y;
        double sa[Q], sb[Q];
        if constexpr (Q == NMODES_RF) {
          mode_proj12(ex, ey, xa, ya, fa, ld_delta(delta, na), ld_delta(delta_rf, na), sa);
          mode_proj12(ex, ey, xb, yb, fb, ld_delta(delta, nbn), ld_delta(delta_rf, nbn), sb);
        } else {
          mode_proj(ex, ey, xa, ya, fa, ld_delta(delta, na), sa);
          mode_proj(ex, ey, xb, yb, fb, ld_delta(delta, nbn), sb);
        }
#pragma unroll
        for (int m = 0; m < Q; ++m) sa[m] -= sb[m];
#pragma unroll
        for (int m = 6; m < Q; ++m)
#pragma unroll
          for (int l = 0; l <= m; ++l) {
            const int g = m * (m + 1) / 2 - 21 + l;
            gen[g] = fma((AT)(k * sa[m]), (AT)sa[l], gen[g]);
          }
      }
    }
    warp_sums<ST>(gen, dst);
  }
  __syncthreads();

  // the slots' sums over their lists
  for (int sl = 1; sl < NSLOTS; ++sl) {
    if (!mine(sl)) continue;
    const LT* e0 = la + (size_t)LC.off[sl] * LST;
    // one slot's entries after another's on the same threads would leave most idle:
    // slot sl starts at its own place in the CTA
    for (int q = (tid + nt - (sl - 1) / C * SS::NPAIR % nt) % nt; q < SS::NPAIR; q += nt) {
      const SlotPairs<Q>& T = *[]() {
        if constexpr (Q == NMODES_RF) return &PAIRS12;
        else return &PAIRS9;
      }();
      const int p = T.p[q], c = T.c[q];
      const LT* e = e0;
      double v = 0.0;
      if constexpr (sizeof(LT) == 8) {
        for (int b = 0; b < LC.cap[sl]; ++b, e += LST) v = fma(e[2 * Q + p], e[c], v);
      } else {
        for (int b0 = 0; b0 < LC.cap[sl]; b0 += 16) {
          LT sum = LT(0);
          for (int b = b0; b < b0 + 16 && b < LC.cap[sl]; ++b, e += LST) sum = fma(e[2 * Q + p], e[c], sum);
          v += (double)sum;
        }
      }
      out[sl * SZ + p * SD + c] = v;
      out[sl * SZ + c * SD + p] = v;
    }
  }
  if (C > 1) cluster.sync();  // the parts are in rank 0's memory
  if (rank > 0) return;
  // SELF slot (upper-left Q x Q): the parts in order
  for (int k = tid; k < SS::NACC; k += nt) {
    double v = part[k];
    for (int q = 1; q < SP; ++q) v += part[(size_t)q * SS::NACC + k];
    part[k] = v;  // only this thread reads or writes column k
  }
  __syncthreads();
  for (int t = tid; t < Q * Q; t += nt) {
    const int m = t / Q, l = t % Q;
    const int mm = m > l ? m : l, ll = m > l ? l : m;
    if (mm < 6) continue;
    double v = part[SS::NLIN + SS::NQUAD + mm * (mm + 1) / 2 - 21 + ll];
    // constants s_2..s_5 of a regular bar of direction d: -L e_x^2, -L e_x e_y, -L e_y e_x, -L e_y^2
    if (ll >= 2 && ll <= 5) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double ex = (d == 0) ? 1.0 : (d == 1 ? 0.5 : -0.5), ey = (d == 0) ? 0.0 : SQ3_2;
        const double c = (ll == 2) ? -lv.L * ex * ex : (ll == 5 ? -lv.L * ey * ey : -lv.L * ex * ey);
        v = fma(c, part[NS * d + mm - 6], v);
      }
    } else if (ll >= 6) {
      v += part[SS::NLIN + (mm - 6) * (mm - 5) / 2 + ll - 6];
    }
    out[SLOT_SELF * SZ + m * SD + l] = v;
  }
}

template <typename DT, int Q, typename AT>
__global__ void __launch_bounds__(32 * SP) k_slots_it(LatView lv, const DT* __restrict__ delta,
                                                      const DT* __restrict__ delta_rf, double* __restrict__ slots,
                                                      const IterCtl* ctl) {
  dep_wait();
  if (ctl && *(volatile const int*)&ctl->done) return;  // the same in every CTA of a cluster
  const int C = (int)cg::this_cluster().num_blocks();
  slots_it_body<DT, Q, AT>(lv, delta, delta_rf, slots, blockIdx.x / C);
}

// Batched: the sets of every problem, a CTA each.
template <typename DT, typename AT>
__global__ void __launch_bounds__(32 * SP) kb_coarse_slots(const BatchProb* __restrict__ P,
                                                           const BatchItem* __restrict__ items) {
  const BatchItem it = items[blockIdx.x];
  const BatchProb& q = P[it.prob];
  if (q.ctl && *(volatile const int*)&q.ctl->done) return;
  slots_it_body<DT, NMODES, AT>(q.lv, (const DT*)q.delta, nullptr, q.slots_it, it.bx);
}

// Band (lower, column-major: band[c*(bw+1) + k] = A[c+k][c]) of K_aa from the
// base (modes 1-6) and per-iteration (modes 7-q) slots; q modes per set, slots
// of 2q x 2q.
__device__ inline double slot_entry(const double* base, const double* it, int q, int I, int slot, int p, int c) {
  const size_t o = ((size_t)I * NSLOTS + slot) * slot_size(q) + (size_t)p * slot_dim(q) + c;
  return base[o] + it[o];
}

__device__ __forceinline__ void band_from_slots_body(const LatView lv, const double* __restrict__ base,
                                                     const double* __restrict__ it, double* __restrict__ band,
                                                     int bw, const IterCtl* ctl, int bx, int gx) {
  if (ctl && *(volatile const int*)&ctl->done) return;
  const int nm = lv.q;
  const int n = nm * lv.M;
  const size_t total = (size_t)n * (bw + 1);
  for (size_t q = bx * (size_t)blockDim.x + threadIdx.x; q < total;
       q += (size_t)gx * blockDim.x) {
    const int col = (int)(q / (bw + 1)), k = (int)(q % (bw + 1));
    const int row = col + k;
    double v = 0.0;
    if (row < n) {
      const int I = col / nm, m = col % nm;
      const int J = row / nm, l = row % nm;
      const int Ix = I % lv.Mx, Iy = I / lv.Mx, Jx = J % lv.Mx, Jy = J / lv.Mx;
      if (J == I) {
        v = slot_entry(base, it, nm, I, SLOT_SELF, l, m);
        for (int s = SLOT_E; s < NSLOTS; ++s) v += slot_entry(base, it, nm, I, s, l, m);
        // contributions of neighbours that own bars into I
        const int kx[5] = {-1, 1, 0, -1, 1};   // owner offset for E, W, N, NE, NW
        const int ky[5] = {0, 0, -1, -1, -1};
        for (int s = 0; s < 5; ++s) {
          const int Kx = Ix + kx[s], Ky = Iy + ky[s];
          if (Kx < 0 || Kx >= lv.Mx || Ky < 0 || Ky >= lv.My) continue;
          v += slot_entry(base, it, nm, Ky * lv.Mx + Kx, SLOT_E + s, nm + l, nm + m);
        }
      } else {
        const int dx = Jx - Ix, dy = Jy - Iy;
        if (dy == 0 && dx == 1) {
          v = slot_entry(base, it, nm, I, SLOT_E, nm + l, m) + slot_entry(base, it, nm, J, SLOT_W, l, nm + m);
        } else if (dy == 1 && dx == 0) {
          v = slot_entry(base, it, nm, I, SLOT_N, nm + l, m);
        } else if (dy == 1 && dx == 1) {
          v = slot_entry(base, it, nm, I, SLOT_NE, nm + l, m);
        } else if (dy == 1 && dx == -1) {
          v = slot_entry(base, it, nm, I, SLOT_NW, nm + l, m);
        }
      }
    }
    band[q] = v;
  }
}

__global__ void k_band_from_slots(LatView lv, const double* __restrict__ base,
                                  const double* __restrict__ it, double* __restrict__ band, int bw,
                                  const IterCtl* ctl) {
  band_from_slots_body(lv, base, it, band, bw, ctl, blockIdx.x, gridDim.x);
}
__global__ void kb_band_from_slots(const BatchProb* __restrict__ P, const BatchItem* __restrict__ items) {
  const BatchItem it = items[blockIdx.x];
  const BatchProb& q = P[it.prob];
  band_from_slots_body(q.lv, q.slots_base, q.slots_it, q.band, q.bw, q.ctl, it.bx, it.gx);
}

__global__ void k_band_from_dense(int n, int bw, const double* __restrict__ dense,
                                  double* __restrict__ band) {
  const size_t total = (size_t)n * (bw + 1);
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < total;
       q += (size_t)gridDim.x * blockDim.x) {
    const int col = (int)(q / (bw + 1)), k = (int)(q % (bw + 1));
    const int row = col + k;
    band[q] = row < n ? dense[(size_t)row * n + col] : 0.0;
  }
}

__global__ void k_dense_from_band(int n, int bw, const double* __restrict__ band,
                                  double* __restrict__ dense) {
  const size_t total = (size_t)n * n;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < total;
       q += (size_t)gridDim.x * blockDim.x) {
    const int r = (int)(q / n), c = (int)(q % n);
    const int hi = r > c ? r : c, lo = r > c ? c : r;
    dense[q] = (hi - lo <= bw) ? band[(size_t)lo * (bw + 1) + (hi - lo)] : 0.0;
  }
}

// Jacobi scaling (s_i = D_ii^-1/2), right-hand side b = s P, the solution
// accumulator x = 0, and the modes that take no part: those left out by the
// mode mask (bit m keeps mode m of every set) and those that vanish, D_ii <=
// 1e-300 or <= 1e-28 times the largest diagonal of the set's modes that are
// kept (zero up to rounding).
__device__ __forceinline__ void coarse_diag_body(int n, int bw, const double* __restrict__ band,
                                                 const double* __restrict__ P, double* __restrict__ scale,
                                                 double* __restrict__ b, double* __restrict__ x,
                                                 int* __restrict__ dropped, unsigned mode_mask, int nm,
                                                 const IterCtl* ctl, int bx, int gx) {
  if (ctl && *(volatile const int*)&ctl->done) return;
  for (int i = bx * blockDim.x + threadIdx.x; i < n; i += gx * blockDim.x) {
    const double D = band[(size_t)i * (bw + 1)];
    const int g0 = i - i % nm;
    double dmax = 0.0;
    for (int m = 0; m < nm && g0 + m < n; ++m)
      if ((mode_mask >> m) & 1u) dmax = fmax(dmax, band[(size_t)(g0 + m) * (bw + 1)]);
    const bool drop = !((mode_mask >> (i % nm)) & 1u) || !(D > 1e-300) || !(D > 1e-28 * dmax);
    const double s = drop ? 0.0 : 1.0 / sqrt(D);
    scale[i] = s;
    b[i] = s * P[i];
    x[i] = 0.0;
    dropped[i] = drop ? 1 : 0;
  }
}

__global__ void k_coarse_diag(int n, int bw, const double* __restrict__ band,
                              const double* __restrict__ P, double* __restrict__ scale,
                              double* __restrict__ b, double* __restrict__ x, int* __restrict__ dropped,
                              unsigned mode_mask, int nm, const IterCtl* ctl) {
  coarse_diag_body(n, bw, band, P, scale, b, x, dropped, mode_mask, nm, ctl, blockIdx.x, gridDim.x);
}
__global__ void kb_coarse_diag(const BatchProb* __restrict__ Pb, const BatchItem* __restrict__ items) {
  const BatchItem it = items[blockIdx.x];
  const BatchProb& q = Pb[it.prob];
  coarse_diag_body(q.n_c, q.bw, q.band, q.P, q.scale, q.b, q.x, q.dropped, q.mode_mask, NMODES, q.ctl, it.bx, it.gx);
}

// Modes that depend on earlier modes of the same set get a = 0.  Sets have
// disjoint supports, so the columns of V can only be dependent within a set:
// the Jacobi-scaled 9 x 9 diagonal block of every set is eliminated in FP64 in
// mode order, and a mode whose pivot is <= 1e-14 is dropped (the rule of the
// full upper-level system, decided where FP64 resolves it).
template <int Q = NMODES>
__device__ __forceinline__ void set_drops_body(int nsets, int bw, const double* __restrict__ band,
                                               const double* __restrict__ scale, int* __restrict__ dropped,
                                               const IterCtl* ctl, int bx, int gx) {
  if (ctl && *(volatile const int*)&ctl->done) return;
  const int I = bx * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (I >= nsets) return;
  const int row = lane < Q ? lane : Q - 1;
  double A[Q];
#pragma unroll
  for (int l = 0; l < Q; ++l) {
    const int lo = l < row ? l : row, hi = l < row ? row : l;
    A[l] = scale[Q * I + row] * band[(size_t)(Q * I + lo) * (bw + 1) + (hi - lo)] * scale[Q * I + l];
  }
  const bool dr = drop_pivots<Q>(A, dropped[Q * I + row] != 0, lane);
  if (lane < Q) dropped[Q * I + lane] = dr ? 1 : 0;
}

template <int Q>
__global__ void k_coarse_set_drops(int nsets, int bw, const double* __restrict__ band,
                                   const double* __restrict__ scale, int* __restrict__ dropped,
                                   const IterCtl* ctl) {
  set_drops_body<Q>(nsets, bw, band, scale, dropped, ctl, blockIdx.x, gridDim.x);
}
__global__ void kb_coarse_set_drops(const BatchProb* __restrict__ P, const BatchItem* __restrict__ items) {
  const BatchItem it = items[blockIdx.x];
  const BatchProb& q = P[it.prob];
  set_drops_body(q.lv.M, q.bw, q.band, q.scale, q.dropped, q.ctl, it.bx, it.gx);
}

// Scaled band in FP64 (column layout for the residual's upper part and row
// layout for its lower part) and the factor's input in row layout, in T.
template <typename T>
__device__ __forceinline__ void scale_band_body(int n, int bw, const double* __restrict__ band,
                                                const double* __restrict__ scale, const int* __restrict__ dropped,
                                                double* __restrict__ sband, double* __restrict__ sbandR,
                                                T* __restrict__ frow, double* __restrict__ b, const IterCtl* ctl,
                                                int bx, int gx) {
  if (ctl && *(volatile const int*)&ctl->done) return;
  const size_t total = (size_t)n * (bw + 1);
  for (size_t q = bx * (size_t)blockDim.x + threadIdx.x; q < total;
       q += (size_t)gx * blockDim.x) {
    const int col = (int)(q / (bw + 1)), k = (int)(q % (bw + 1));
    const int row = col + k;
    double v = 0.0;
    if (row < n) {
      if (k == 0) {
        v = 1.0;
      } else if (!dropped[row] && !dropped[col]) {
        v = scale[row] * band[q] * scale[col];
      }
    }
    sband[q] = v;
    if (row < n) {
      sbandR[(size_t)row * (bw + 1) + k] = v;
      frow[(size_t)row * (bw + 1) + k] = (T)v;
    }
    if (k == 0 && dropped[col]) b[col] = 0.0;
  }
}

template <typename T>
__global__ void k_coarse_scale_band(int n, int bw, const double* __restrict__ band,
                                    const double* __restrict__ scale, const int* __restrict__ dropped,
                                    double* __restrict__ sband, double* __restrict__ sbandR,
                                    T* __restrict__ frow, double* __restrict__ b, const IterCtl* ctl) {
  scale_band_body<T>(n, bw, band, scale, dropped, sband, sbandR, frow, b, ctl, blockIdx.x, gridDim.x);
}
// Batched: the FP32 factor's input (the batched path factors in FP32).
__global__ void kb_coarse_scale_band(const BatchProb* __restrict__ P, const BatchItem* __restrict__ items) {
  const BatchItem it = items[blockIdx.x];
  const BatchProb& q = P[it.prob];
  scale_band_body<float>(q.n_c, q.bw, q.band, q.scale, q.dropped, q.sband, q.sband + (size_t)q.n_c * (q.bw + 1),
                         q.lrow, q.b, q.ctl, it.bx, it.gx);
}

}  // namespace

int coarse_bw(const LatView& lv) {
  // set I couples to I + Mx + 1 at most (NE neighbour)
  const int reach = (lv.M > 1) ? (lv.Mx + 1 < lv.M - 1 ? lv.Mx + 1 : lv.M - 1) : 0;
  return lv.q * (reach + 1) - 1;
}

size_t coarse_slots_smem(const LatView& lv) {
  const int w = lv.sx < lv.nx ? lv.sx : lv.nx;
  const int h = lv.sy < lv.ny ? lv.sy : lv.ny;
  // lists of all modes and 2 K of sums: the limit of a set's size; more than the
  // base's kernel or an update's takes
  return ((size_t)list_caps(w, h).total * 4 * lv.q + RED_CHUNK * NT + (lv.q == NMODES_RF ? 57 : 60)) * sizeof(double);
}

size_t coarse_slots_it_smem(const LatView& lv, bool fp32) {
  const ListCaps LC = list_caps(lv.sx < lv.nx ? lv.sx : lv.nx, lv.sy < lv.ny ? lv.sy : lv.ny);
  if (lv.q == NMODES_RF) return slots_it_smem<NMODES_RF, double>(LC);
  return fp32 ? slots_it_smem<NMODES, float>(LC) : slots_it_smem<NMODES, double>(LC);
}

cudaError_t launch_coarse_slots(cudaStream_t s, const LatView& lv, const void* delta, bool delta_fp32,
                                bool full, double* slots, const IterCtl* ctl, const void* delta_rf) {
  const bool rf = lv.q == NMODES_RF;
  float2* const f2 = nullptr;
  double2* const d2 = nullptr;
  if (!full) {
    const int cl = std::max(1, std::min(4, lv.nsm / lv.M));  // CTAs per set while SMs are free
    auto go = [&](auto k, auto* d) {
      using DT = std::remove_pointer_t<decltype(d)>;
      return launch_dep(k, s, lv.M * cl, 32 * ((SP + cl - 1) / cl), coarse_slots_it_smem(lv, delta_fp32),
                        cl > 1 ? cl : 0, lv, (const DT*)delta, (const DT*)delta_rf, slots, ctl);
    };
    if (rf)
      return delta_fp32 ? go(k_slots_it<float2, NMODES_RF, float>, f2) : go(k_slots_it<double2, NMODES_RF, double>, d2);
    return delta_fp32 ? go(k_slots_it<float2, NMODES, float>, f2) : go(k_slots_it<double2, NMODES, double>, d2);
  }
  k_coarse_base<<<lv.M, NT, coarse_slots_smem(lv), s>>>(lv, slots);
  return cudaGetLastError();
}

cudaError_t configure_coarse_assemble(int max_smem) {
  cudaError_t e = set_max_dynamic_smem(k_coarse_base, max_smem);
  if (e == cudaSuccess) e = set_max_dynamic_smem(k_slots_it<float2, NMODES_RF, float>, max_smem);
  if (e == cudaSuccess) e = set_max_dynamic_smem(k_slots_it<double2, NMODES_RF, double>, max_smem);
  if (e == cudaSuccess) e = set_max_dynamic_smem(k_slots_it<float2, NMODES, float>, max_smem);
  if (e == cudaSuccess) e = set_max_dynamic_smem(k_slots_it<double2, NMODES, double>, max_smem);
  if (e == cudaSuccess) e = set_max_dynamic_smem(kb_coarse_slots<float2, float>, max_smem);
  if (e == cudaSuccess) e = set_max_dynamic_smem(kb_coarse_slots<double2, double>, max_smem);
  return e;
}

static int grid_for(size_t total) {
  size_t g = (total + 255) / 256;
  if (g > 4096) g = 4096;
  if (g < 1) g = 1;
  return (int)g;
}

int coarse_grid_for(size_t n) { return grid_for(n); }
int set_drops_blocks(int nsets) { return (nsets + 3) / 4; }  // a warp per set

cudaError_t launch_batch_slots(cudaStream_t s, bool fp32, size_t smem, const BatchProb* P, const BatchItem* it,
                               int n) {
  if (n <= 0) return cudaSuccess;
  if (fp32) kb_coarse_slots<float2, float><<<n, 32 * SP, smem, s>>>(P, it);
  else kb_coarse_slots<double2, double><<<n, 32 * SP, smem, s>>>(P, it);
  return cudaGetLastError();
}
cudaError_t launch_batch_band(cudaStream_t s, const BatchProb* P, const BatchItem* it, int n) {
  if (n <= 0) return cudaSuccess;
  kb_band_from_slots<<<n, 256, 0, s>>>(P, it);
  return cudaGetLastError();
}
cudaError_t launch_batch_diag(cudaStream_t s, const BatchProb* P, const BatchItem* it, int n) {
  if (n <= 0) return cudaSuccess;
  kb_coarse_diag<<<n, 256, 0, s>>>(P, it);
  return cudaGetLastError();
}
cudaError_t launch_batch_set_drops(cudaStream_t s, const BatchProb* P, const BatchItem* it, int n) {
  if (n <= 0) return cudaSuccess;
  kb_coarse_set_drops<<<n, 128, 0, s>>>(P, it);
  return cudaGetLastError();
}
cudaError_t launch_batch_scale_band(cudaStream_t s, const BatchProb* P, const BatchItem* it, int n) {
  if (n <= 0) return cudaSuccess;
  kb_coarse_scale_band<<<n, 256, 0, s>>>(P, it);
  return cudaGetLastError();
}

cudaError_t launch_coarse_band_from_slots(cudaStream_t s, const LatView& lv, const double* base,
                                          const double* slots, double* band, const IterCtl* ctl) {
  const int bw = coarse_bw(lv);
  const size_t total = (size_t)NMODES * lv.M * (bw + 1);
  k_band_from_slots<<<grid_for(total), 256, 0, s>>>(lv, base, slots, band, bw, ctl);
  return cudaGetLastError();
}

cudaError_t launch_coarse_band_from_dense(cudaStream_t s, int n, int bw, const double* dense,
                                          double* band) {
  k_band_from_dense<<<grid_for((size_t)n * (bw + 1)), 256, 0, s>>>(n, bw, dense, band);
  return cudaGetLastError();
}

cudaError_t launch_coarse_dense_from_band(cudaStream_t s, int n, int bw, const double* band,
                                          double* dense) {
  k_dense_from_band<<<grid_for((size_t)n * n), 256, 0, s>>>(n, bw, band, dense);
  return cudaGetLastError();
}

cudaError_t launch_coarse_scale(cudaStream_t s, int n, int bw, bool fp64, const double* band, const double* P,
                                double* sband, void* frow, double* scale, double* b, double* x, int* dropped,
                                unsigned mode_mask, int nm, const IterCtl* ctl) {
  k_coarse_diag<<<grid_for(n), 256, 0, s>>>(n, bw, band, P, scale, b, x, dropped, mode_mask, nm, ctl);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int nsets = n / nm;
  if (nm == NMODES_RF)
    k_coarse_set_drops<NMODES_RF><<<set_drops_blocks(nsets), 128, 0, s>>>(nsets, bw, band, scale, dropped, ctl);
  else
    k_coarse_set_drops<NMODES><<<set_drops_blocks(nsets), 128, 0, s>>>(nsets, bw, band, scale, dropped, ctl);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  double* sbandR = sband + (size_t)n * (bw + 1);
  const int g = grid_for((size_t)n * (bw + 1));
  if (fp64)
    k_coarse_scale_band<double><<<g, 256, 0, s>>>(n, bw, band, scale, dropped, sband, sbandR, (double*)frow, b, ctl);
  else
    k_coarse_scale_band<float><<<g, 256, 0, s>>>(n, bw, band, scale, dropped, sband, sbandR, (float*)frow, b, ctl);
  return cudaGetLastError();
}

}  // namespace hms

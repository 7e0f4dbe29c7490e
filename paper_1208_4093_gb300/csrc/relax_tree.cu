// K2 by nested dissection of every set: the displacement-controlled relaxation
// delta_I = (k^Inner_I)^-1 r_I (Eqs. 11-13) with P = V^T r (Eq. 7).
//
// relax.cu substitutes row by row of the lattice: 2 (2 h - 1) dependent steps
// over a factor of h (2 w)^2 entries per pass.  Here a set's nodes (its extended
// region's with overlap) are ordered by nested dissection: a box of nodes is cut
// by its middle column or row (a small one by both), the parts are eliminated
// independently and the separator last.  Per tree node with own unknowns S and
// the unknowns B around its box the factor holds D = A_SS^-1 and G = A_BS D, so
// that one pass up and one down the tree solve the system:
//   up    z_B -= G z_S           (leaves first; z starts as r)
//   down  x_S = D z_S - G^T x_B  (root first)
// A set of 64 x 64 nodes takes 0.9 M products (the substitution: 2.1 M) in 13
// steps instead of 254.  Rounding the explicit inverses to FP32 gives a
// smaller error than the FP32 substitution (1.1e-7 to 1.6e-7 against 1.3e-7 to
// 1.8e-7 of delta on random loads): each unknown passes through fewer products.
//
// Layout.  A phase (one level, up or down) is a list of independent dot
// products, one per unknown it changes; 32 of them, one per lane, are a panel:
// its matrix is stored by columns, lane after lane, so a warp streams it without
// gaps.  (Both unknowns of a lattice node in one lane would share the loads of
// the inputs but fill fewer lanes: 1473 K stored entries of a 64 x 64 set against
// 1203 K; measured 851 us against 706 in FP64 on the 1024^2 lattice, 300 against
// 261 in FP32.)  On the way up an unknown gathers from all nodes of the level
// around it (up to four segments), so no two products write the same unknown and
// no update vectors are kept.  The panels of a phase are dealt to eight streams;
// a stream's panels lie one after another in device memory in the order they are
// used.  Every lane fetches its own words ahead into a ring of shared-memory
// slots, across panels and phases: the stream never waits for a barrier.  The
// vector stays in shared memory, each panel's inputs are gathered into a short
// contiguous buffer first.  All lists depend on the region's width and height
// only.
//
// Measured per launch, row substitution -> this (FP64, FP32; us): 16 sets of
// 16 x 16 nodes 73 -> 28 and 61 -> 22; 70 of 32 x 32 (4 nodes overlap) 390 -> 271
// and 195 -> 105; 72 of 64 x 64 726 -> 394 and 343 -> 156; 256 of 64 x 64 (1024^2
// lattice) 1191 (its balanced schedule) -> 710 and 448 -> 263.  Bound by: FP64,
// the FP64 units of the SMs that hold sets (1203 K fused multiply-adds of a set
// take 300 us at two per clock and SM, and 104 SMs hold two of the 256); FP32, the
// latency of the dot products' chains in eight warps per set (1.28 GB from HBM in
// 254 us: 5.0 TB/s; issue slots 31 %, shared-memory pipe 27 % busy); on few or small sets, the chain of phases, 1 to 2 us each.  A deeper
// ring, bulk copies by one elected lane and prefetches into the L2 measured the
// same.  Panels of phases too short for eight streams are split by columns: FP64
// 16 x 16 nodes 34 -> 28, 32 x 32 110 -> 94, 24 x 20 87 -> 82 (whole panels left
// the longest stream 1.5 to 2.5 times the mean).
#include <algorithm>
#include <array>
#include <cmath>
#include <type_traits>

#include "hms_internal.cuh"
#include "ptx.cuh"

namespace hms {
namespace {

constexpr int NV = RT_STREAMS;   // streams of a set
// A group is four columns of a panel (one 16-byte word per lane in FP32, two in
// FP64); groups fetched at once (2 KB FP32, 1 KB FP64: small FP64 rings let two
// CTAs of 64 x 64 nodes share an SM)
template <typename T>
constexpr int GROUPS = sizeof(T) == 4 ? 4 : 1;
constexpr int STG = 256;         // gathered inputs of a panel, at most (RtShape::stg of a shape)
constexpr int VL = 256;          // virtual lanes of the P sums

template <typename T> struct Vec2;
template <> struct Vec2<double> { using type = double2; };
template <> struct Vec2<float> { using type = float2; };

// Element (stream column R, lane) of a factor: a lane reads 16 bytes (four or two
// columns) at once.
template <typename T>
__host__ __device__ inline long long rt_elem(long long R, int lane) {
  constexpr int G = 16 / sizeof(T);
  return (R / G) * (32 * G) + lane * G + (int)(R % G);
}

struct RtSmem {
  size_t z, stg, xs, ring, total;  // elements of T (ring slots 16-byte aligned); the panel lists lie behind
};
template <typename T>
__host__ __device__ inline RtSmem rt_smem(int nn, int stg, int xs, int nslot) {
  RtSmem L;
  auto up = [](size_t n) { return (n + 7) / 8 * 8; };
  L.z = 0;
  L.stg = up(2 * (size_t)nn + 4);
  L.xs = L.stg + (size_t)NV * stg;
  L.ring = up(L.xs + (size_t)xs);
  L.total = L.ring + (size_t)NV * nslot * GROUPS<T> * 128;
  return L;
}

// four consecutive values, and a lane's four columns (16-byte words 512 bytes
// apart), from shared-memory addresses
template <typename T>
struct Four {
  T x, y, z, w;
};
__device__ inline Four<float> lds4(uint32_t a, float) {
  Four<float> v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
template <int HALF>
__device__ inline Four<double> lds22(uint32_t a) {
  Four<double> v;
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a));
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2 + %3];" : "=d"(v.z), "=d"(v.w) : "r"(a), "n"(HALF));
  return v;
}
__device__ inline Four<double> lds4(uint32_t a, double) { return lds22<16>(a); }
__device__ inline Four<float> ldm4(uint32_t a, float) { return lds4(a, 0.f); }
__device__ inline Four<double> ldm4(uint32_t a, double) { return lds22<512>(a); }

__device__ inline int u16_of(const int4& v, int k) {
  const int w = k < 2 ? v.x : (k < 4 ? v.y : (k < 6 ? v.z : v.w));
  return (k & 1) ? (int)((unsigned)w >> 16) : (w & 0xffff);
}

// The kernel body for set I: NT compute threads, NS ring slots per stream.
template <typename T, int NT, int NS>
__device__ __forceinline__ void rtree_body(const LatView& lv, const RtView& rt, const T* __restrict__ fac,
                                           const double2* __restrict__ r, T* __restrict__ delta,
                                           double* __restrict__ P, const IterCtl* ctl, int* err, int I, int wait0) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ uint64_t bar;
  __shared__ int posv[NV], vrow[NV + 1];
  using T2 = typename Vec2<T>::type;
  constexpr int NW = NT / 32, PER = NV / NW;  // streams per warp
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const RtShape& sh = rt.shapes[rt.sid[I]];
  const int nn = sh.nn, nup = sh.nup, nphase = sh.nphase;
  const unsigned short *inv = sh.inv, *dlist = sh.dlist;
  const int4* lanes = sh.lane;
  const int2* defer = sh.defer;
  const Region RG = relax_region(lv, I);
  const int i0 = (I % lv.Mx) * lv.sx, j0 = (I / lv.Mx) * lv.sy;
  const int w = min(lv.sx, lv.nx - i0), h = min(lv.sy, lv.ny - j0);
  const int stgn = sh.stg;
  const RtSmem LY = rt_smem<T>(nn, stgn, sh.xs, NS);
  T* sm = reinterpret_cast<T*>(smraw);
  T* z = sm + LY.z;
  T* xs = sm + LY.xs;
  const T* fset = fac + rt.off[I];

  constexpr int GC = GROUPS<T>;                         // groups fetched at once (a chunk)
  constexpr int WV = sizeof(T) / 4;                     // 16-byte words of a lane in a group
  constexpr uint32_t GB = 512 * WV, CB = GC * GB;       // bytes of a group, of a chunk
  // Every lane fetches the words of the matrix that it multiplies itself, so a
  // ring slot needs no barrier: chunk c of a stream goes to slot c mod NS.  The
  // last NS - 1 fetches run past the stream's end, into the next one's (or the
  // padding behind the last set's) elements, and are never used.
  auto fetch = [&](uint32_t dst, const char* src) {
#pragma unroll
    for (int t = 0; t < GC * WV; ++t) cp_async16(dst + 512 * t, src + 512 * t);
    cp_async_commit();
  };
  const uint32_t ring0 = smem_u32(sm + LY.ring) + 16 * lane;
  const char* const fac0 = reinterpret_cast<const char*>(fset) + 16 * lane;
  if (tid == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  if (tid < NV) posv[tid] = 0;
  if (tid <= NV) vrow[tid] = sh.vrow[tid];
  __syncthreads();
  // the panels' descriptors and the streams' panel numbers by one bulk copy
  const int2* desc = reinterpret_cast<const int2*>(sm + LY.total);
  const int* vp = reinterpret_cast<const int*>(desc + sh.npanel);
  if (tid == 0) {
    mbar_arrive_expect_tx(&bar, (uint32_t)sh.lbytes);
    bulk_g2s(sm + LY.total, sh.desc, (uint32_t)sh.lbytes, &bar);
  }
  for (int c = 0; c < NS - 1; ++c)
    for (int q = 0; q < PER; ++q) {
      const int v = warp + q * NW;
      fetch(ring0 + (v * NS + c) * CB, fac0 + (size_t)vrow[v] * (32 * sizeof(T)) + (size_t)c * CB);
    }
  // the lists and the factor are the plan's: fetched while the kernel before runs
  dep_wait();
  if (ctl && *(volatile const int*)&ctl->done) {  // the copies in flight land before the CTA exits
    cp_async_wait<0>();
    mbar_wait_bounded(&bar, 0u);
    return;
  }
  // z = r in the tree's order (four nodes in flight per thread)
  {
    const double2* rg = r + (size_t)RG.j0 * lv.nx + RG.i0;
    for (int n0 = tid; n0 < nn; n0 += 4 * NT) {
      double2 v[4];
      int at[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int n = min(n0 + t * NT, nn - 1), y = n / RG.w;
        v[t] = rg[(size_t)y * lv.nx + (n - y * RG.w)];
        at[t] = inv[n];
      }
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (n0 + t * NT < nn) *reinterpret_cast<T2*>(z + 2 * at[t]) = T2{(T)v[t].x, (T)v[t].y};
    }
  }
  if (tid < 4) z[2 * nn + tid] = T(0);
  // a lane may read past its own inputs, against zero columns: never garbage
  for (int k = tid; k < NV * stgn; k += NT) sm[LY.stg + k] = T(0);
  __syncthreads();

  // the only wait that depends on another agent, bounded (wait0: a shorter bound, tests)
  const bool late = !mbar_wait_bounded(&bar, 0u, wait0 >= 0 ? (uint32_t)wait0 : MBAR_WAIT_TRIES);
  if (__syncthreads_or(late)) {
    cp_async_wait<0>();
    if (tid == 0) {
      mbar_wait_bounded(&bar, 0u);  // the copy in flight lands before the CTA exits
      atomicOr(err, (int)DEVERR_TIMEOUT);
    }
    return;
  }
  for (int ph = 0; ph < nphase; ++ph) {
    const bool down = ph >= nup;
    const int2 df = defer[ph];  // deferred outputs of the phase: first entry of dlist; count, parts of each
    for (int q = 0; q < PER; ++q) {
      const int v = warp + q * NW;
      const int p0 = vp[ph * NV + v], p1 = vp[ph * NV + v + 1];
      if (p0 >= p1) continue;
      T* stg = sm + LY.stg + (size_t)v * stgn;
      const uint32_t stga = smem_u32(stg), rbeg = ring0 + v * NS * CB, rend = rbeg + NS * CB;
      // the stream's place: chunk and group; where the next chunk goes and comes from
      const int c0 = posv[v] / GC;
      int g = posv[v] % GC, used = c0;
      uint32_t ma = rbeg + (c0 % NS) * CB + g * GB;
      const int cn = g == 0 ? c0 + NS - 1 : c0 + NS;
      uint32_t sd = rbeg + (cn % NS) * CB;
      const char* src = fac0 + (size_t)vrow[v] * (32 * sizeof(T)) + (size_t)cn * CB;
      const int4* lp = lanes + (size_t)p0 * 64 + lane;
      int4 ln = lp[0], gn = lp[32];
      for (int p = p0; p < p1; ++p) {
        const int2 d = desc[p];  // segments' groups, 8 bits each; inputs (0: those of the panel before), segments
        const int4 li = ln, gi = gn;
        const int nin = d.y & 0xffff, nseg = d.y >> 16;
        lp += 64;  // (one panel of padding behind the last)
        ln = lp[0];
        gn = lp[32];
#pragma unroll
        for (int t = 0; t < STG / 32; ++t)
          if (32 * t < nin) stg[lane + 32 * t] = z[u16_of(gi, t)];
        __syncwarp();
        T a0 = T(0), a1 = T(0), a2 = T(0), a3 = T(0);
        auto add = [&](const Four<T>& m, const Four<T>& f) {
          a0 = fma(m.x, f.x, a0);
          a1 = fma(m.y, f.y, a1);
          a2 = fma(m.z, f.z, a2);
          a3 = fma(m.w, f.w, a3);
        };
        unsigned long long bases = ((unsigned long long)(unsigned)li.y << 32) | (unsigned)li.x;
        unsigned lens = (unsigned)d.x;
#pragma unroll 1
        for (int sgm = 0; sgm < nseg; ++sgm) {
          int left = lens & 0xff;  // groups
          uint32_t fa = stga + (uint32_t)(bases & 0xffff) * sizeof(T);
          bases >>= 16;
          lens >>= 8;
#pragma unroll 1
          while (left > 0) {
            if (g == 0) {
              fetch(sd, src);
              src += CB;
              sd += CB;
              if (sd == rend) sd = rbeg;
              cp_async_wait<NS - 1>();
              if (GC > 1 && left >= GC) {
                Four<T> m4[GC], f4[GC];
#pragma unroll
                for (int t = 0; t < GC; ++t) {
                  m4[t] = ldm4(ma + t * GB, T(0));
                  f4[t] = lds4(fa + t * (uint32_t)(4 * sizeof(T)), T(0));
                }
#pragma unroll
                for (int t = 0; t < GC; ++t) add(m4[t], f4[t]);
                fa += GC * 4 * sizeof(T);
                left -= GC;
                ma += CB;
                if (ma == rend) ma = rbeg;
                ++used;
                continue;
              }
            }
            add(ldm4(ma, T(0)), lds4(fa, T(0)));
            fa += 4 * sizeof(T);
            --left;
            ma += GB;
            if (++g == GC) {
              g = 0;
              ++used;
              if (ma == rend) ma = rbeg;
            }
          }
        }
        const T s = (a0 + a1) + (a2 + a3);
        const int out = u16_of(li, 4);
        if (out != 0xffff) {
          if (df.y > 0) xs[u16_of(li, 5)] = s;
          else if (down) z[out] = s;
          else z[out] += s;
        }
        __syncwarp();
      }
      if (lane == 0) posv[v] = used * GC + g;
    }
    __syncthreads();
    if (df.y > 0) {
      const int cnt = df.y & 0xffff, parts = df.y >> 16;
      for (int k = tid; k < cnt; k += NT) {
        T s = xs[k];
        for (int j = 1; j < parts; ++j) s += xs[j * cnt + k];
        T* o = z + dlist[df.x + k];
        *o = down ? s : *o + s;
      }
      __syncthreads();
    }
  }
  // delta out, and P = V^T r (Eq. 7) from r and delta: virtual lane v takes
  // column v mod w and every (VL / w)-th row; its xi is that of the column, plus
  // half a bar on odd rows, so a node costs eight FP64 operations.  Modes 1-9 of
  // set I at P[q I + m]; no P (the force-controlled relaxation) with P = nullptr.
  cp_async_wait<0>();
  __syncthreads();
  double* red = reinterpret_cast<double*>(smraw + (LY.stg * sizeof(T)));  // 9 x VL doubles, over staging and ring
  const int grp = VL / w;
  const int ox = i0 - RG.i0, oy = j0 - RG.j0;
  const double2 rep = lv.rep[I];
  for (int vl = tid; vl < VL; vl += NT) {
    const int il = vl % w, g = vl / w;
    // sums of r_x, r_y, d.r on even and odd rows, and weighted with eta
    double s[2][3], e[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) s[0][k] = s[1][k] = e[k] = 0.0;
    if (g < grp) {
      double eta = fma(lv.L * SQ3_2, (double)(j0 + g), -rep.y);
      const double deta = lv.L * SQ3_2 * (double)grp;
      // four rows in flight
      for (int j4 = g; j4 < h; j4 += 4 * grp) {
        double2 rv[4];
        int zi[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int jj = min(j4 + t * grp, h - 1);
          zi[t] = inv[(oy + jj) * RG.w + ox + il];
          if (P != nullptr) rv[t] = r[(size_t)(j0 + jj) * lv.nx + i0 + il];
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int jj = j4 + t * grp;
          if (jj >= h) break;
          const T2 dv = *reinterpret_cast<const T2*>(z + 2 * zi[t]);
          reinterpret_cast<T2*>(delta)[(size_t)(j0 + jj) * lv.nx + i0 + il] = dv;
          if (P == nullptr) continue;
          const double dr = fma((double)dv.x, rv[t].x, (double)dv.y * rv[t].y);
          const double v[3] = {rv[t].x, rv[t].y, dr};
          if ((j0 + jj) & 1) {
#pragma unroll
            for (int k = 0; k < 3; ++k) s[1][k] += v[k];
          } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) s[0][k] += v[k];
          }
#pragma unroll
          for (int k = 0; k < 3; ++k) e[k] = fma(eta, v[k], e[k]);
          eta += deta;
        }
      }
    }
    if (P != nullptr) {
      const double xi = fma(lv.L, (double)(i0 + il), -rep.x), xo = xi + 0.5 * lv.L;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double sx = fma(xi, s[0][k], xo * s[1][k]);
        // modes: 0, 1 = sums; 2, 3 = xi, eta of r_x; 4, 5 of r_y; 6, 7, 8 of d.r
        red[(k < 2 ? k : 6) * VL + vl] = s[0][k] + s[1][k];
        red[(k < 2 ? 2 + 2 * k : 7) * VL + vl] = sx;
        red[(k < 2 ? 3 + 2 * k : 8) * VL + vl] = e[k];
      }
    }
  }
  if (P == nullptr) return;
  __syncthreads();
  // 9 x 256 values: thread (mode, part) adds every sixteenth of a mode's, then the
  // sixteen parts in order
  constexpr int PARTS = 16;
  for (int k = tid; k < NMODES * PARTS; k += NT) {
    const double* c = red + (k / PARTS) * VL + k % PARTS;
    double a = 0.0, b = 0.0;
#pragma unroll
    for (int t = 0; t < VL / PARTS; t += 2) a += c[t * PARTS], b += c[(t + 1) * PARTS];
    red[NMODES * VL + k] = a + b;
  }
  __syncthreads();
  if (tid < NMODES) {
    double sum = 0.0;
    for (int k = 0; k < PARTS; ++k) sum += red[NMODES * VL + PARTS * tid + k];
    P[(size_t)lv.q * I + tid] = sum;
  }
}

// The sets' relaxation and, with fac2, the cut-free sets' of the force-controlled
// modes beside it (CTAs M to 2 M: their own factor, right-hand side and result,
// no P): 256 x 192 nodes, 2 x 48 sets on 152 SMs, projections included, FP64 224 ->
// 136 us, mixed 120 -> 77.
template <typename T, int NT, int NS>
__global__ void __launch_bounds__(NT) k_rtree(LatView lv, RtView rt, const T* __restrict__ fac,
                                              const double2* __restrict__ r, T* __restrict__ delta,
                                              double* __restrict__ P, const IterCtl* ctl, int* err, int wait0,
                                              const T* __restrict__ fac2, const double2* __restrict__ r2,
                                              T* __restrict__ delta2) {
  const bool cut = (int)blockIdx.x >= lv.M;
  rtree_body<T, NT, NS>(lv, rt, cut ? fac2 : fac, cut ? r2 : r, cut ? delta2 : delta, cut ? nullptr : P, ctl, err,
                        cut ? (int)blockIdx.x - lv.M : (int)blockIdx.x, wait0);
}
template <typename T, int NT, int NS>
__global__ void __launch_bounds__(NT) kb_rtree(const BatchProb* __restrict__ Pb, const BatchItem* __restrict__ items) {
  const BatchItem it = items[blockIdx.x];
  const BatchProb& q = Pb[it.prob];
  const T* fac;
  if constexpr (sizeof(T) == 4) fac = q.f32;
  else fac = q.f64;
  rtree_body<T, NT, NS>(q.lv, q.rt, fac, q.r, (T*)q.delta, q.P, q.ctl, q.err, it.bx, -1);
}

// ---------------------------------------------------------------- setup
constexpr int FTH = 256;  // threads of a factor CTA
constexpr double SQ3_4 = 0.43301270189221932338;  // sqrt(3)/4

__device__ inline int pk(int r, int c) { return r * (r + 1) / 2 + c; }

// Entry (component ca of node a, cb of node b) of k^Inner (a, b: region node
// numbers), constrained DOFs as unit rows.  CUT: only bars inside the region
// (Eq. 15, see setup.cu).
template <bool CUT>
__device__ inline double inner_entry(const LatView& lv, const Region& R, int a, int b, int ca, int cb) {
  const int ya = a / R.w, xa = a - ya * R.w, yb = b / R.w, xb = b - yb * R.w;
  if (abs(xa - xb) > 1 || abs(ya - yb) > 1) return 0.0;
  const int ia = R.i0 + xa, ja = R.j0 + ya, ib = R.i0 + xb, jb = R.j0 + yb;
  const unsigned fa = lv.fix[(size_t)ja * lv.nx + ia], fb = lv.fix[(size_t)jb * lv.nx + ib];
  if (((fa >> ca) & 1u) || ((fb >> cb) & 1u)) return a == b && ca == cb ? 1.0 : 0.0;
  if (a == b) {
    const int off = ja & 1;
    auto in = [&](int ii, int jj) {
      return !CUT || (ii >= R.i0 && ii < R.i0 + R.w && jj >= R.j0 && jj < R.j0 + R.h);
    };
    const double kE = in(ia + 1, ja) ? bar_k(lv, ia, ja, 0) : 0.0;
    const double kW = in(ia - 1, ja) ? bar_k(lv, ia - 1, ja, 0) : 0.0;
    const double kNE = in(ia + off, ja + 1) ? bar_k(lv, ia, ja, 1) : 0.0;
    const double kSW = in(ia - 1 + off, ja - 1) ? bar_k(lv, ia - 1 + off, ja - 1, 1) : 0.0;
    const double kNW = in(ia - 1 + off, ja + 1) ? bar_k(lv, ia, ja, 2) : 0.0;
    const double kSE = in(ia + off, ja - 1) ? bar_k(lv, ia + off, ja - 1, 2) : 0.0;
    const double sne = kNE + kSW, snw = kNW + kSE;
    if (ca == cb) return ca == 0 ? kE + kW + 0.25 * (sne + snw) : 0.75 * (sne + snw);
    return SQ3_4 * (sne - snw);
  }
  if (ja == jb) return ca == 0 && cb == 0 ? -bar_k(lv, min(ia, ib), ja, 0) : 0.0;
  // a bar between neighbouring rows, owned by the lower node
  const int il = ja < jb ? ia : ib, jl = min(ja, jb), iu = ja < jb ? ib : ia, off = jl & 1;
  double ex, k;
  if (iu == il + off) ex = 0.5, k = bar_k(lv, il, jl, 1);
  else if (iu == il - 1 + off) ex = -0.5, k = bar_k(lv, il, jl, 2);
  else return 0.0;
  return -k * (ca ? SQ3_2 : ex) * (cb ? SQ3_2 : ex);
}

// One CTA per set (grid-stride over all sets, or over the n sets of a list), FP64: the tree's fronts one after another,
// children first.  Per front: A_SS gathered into shared memory, A_BS and A_BB into
// a work space of the CTA's (original entries plus the children's updates), A_SS swept pivot by
// pivot to -D, G = A_BS D, the update A_BB - G A_BS^T for the parent; D, G and G^T
// go to the panels' places, rounded to FP32 on the mixed path.  A pivot below
// 1e-12 of the unknown's own stiffness means k^Inner is singular to working
// precision.
template <bool CUT>
__global__ void __launch_bounds__(FTH) k_rtree_factor(LatView lv, RtView rt, double* __restrict__ f64,
                                                      float* __restrict__ f32, double* __restrict__ scratch,
                                                      int first, double* __restrict__ work, long long stride,
                                                      int* err, const int* __restrict__ sets, int n) {
  extern __shared__ double S[];  // packed lower triangle of A_SS, then the pivot column
  __shared__ int bad;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* X = (int)blockIdx.x < first ? scratch + (size_t)blockIdx.x * stride
                                      : work + (size_t)((int)blockIdx.x - first) * stride;
  for (int k0 = blockIdx.x; k0 < n; k0 += gridDim.x) {
    const int I = sets ? sets[k0] : k0;
    const RtShape& sh = rt.shapes[rt.sid[I]];
    const Region R = relax_region(lv, I);
    const long long base = rt.off[I];
    auto put = [&](int row, int k, double v) {  // column k of a row; row: its first entry in place
      const int place = sh.place[row + (k >> 2)];
      const long long rr = (place >> 5) + (k & 3);
      if (f64) f64[base + rt_elem<double>(rr, place & 31)] = v;
      if (f32) f32[base + rt_elem<float>(rr, place & 31)] = (float)v;
    };
    if (tid == 0) bad = 0;
    for (int q = 0; q < sh.nnode; ++q) {
      const RtNode nd = sh.nodes[q];
      const int ns = 2 * nd.ns, nb = 2 * nd.nb, nf = ns + nb;
      const int gu = (ns + 3) >> 2, gd = gu + ((nb + 3) >> 2);  // groups of an up row, of a down row
      const unsigned short* fr = sh.front + nd.f_off;  // region nodes of S, then B
      double* col = S + pk(ns - 1, ns - 1) + 1;        // pivot column, and A_SS's own diagonal
      double* dia = col + ns;
      double* A = X + sh.u_max;                        // A_BS [nb][ns]
      double* G = A + sh.bs_max;                       // G [nb][ns]
      double* U = X + nd.u_off;                        // A_BB [nb][nb], lower
      __syncthreads();
      // gather: one thread per entry (i, j), j <= i
      for (int e = warp; e < nf; e += FTH / 32) {
        const int ni = fr[e >> 1], ci = e & 1;
        for (int j = lane; j <= e; j += 32) {
          double v = 0.0;
          const int nj = fr[j >> 1], cj = j & 1;
          if (j < ns) {
            v = inner_entry<CUT>(lv, R, ni, nj, ci, cj);
            if (e == j) dia[j] = v;
          }
          for (int c = 0; c < nd.nchild; ++c) {
            const short* mp = sh.cmap + nd.c_map[c];
            const int a = mp[e >> 1], b = mp[j >> 1];
            if (a >= 0 && b >= 0) {
              const int ra = 2 * a + ci, rb = 2 * b + cj, hi = max(ra, rb), lo = min(ra, rb);
              v += X[nd.c_u[c] + (size_t)hi * nd.c_nb[c] + lo];
            }
          }
          if (e < ns) S[pk(e, j)] = v;
          else if (j < ns) A[(size_t)(e - ns) * ns + j] = v;
          else U[(size_t)(e - ns) * nb + j - ns] = v;
        }
      }
      __syncthreads();
      // sweep A_SS: S becomes -D
      for (int k = 0; k < ns; ++k) {
        for (int i = tid; i < ns; i += FTH) col[i] = i >= k ? S[pk(i, k)] : S[pk(k, i)];
        __syncthreads();
        double piv = col[k];
        if (!(piv > 1e-12 * dia[k])) {
          if (tid == 0) bad = 1;
          piv = 1.0;
        }
        const double inv = 1.0 / piv;
        for (int i = warp; i < ns; i += FTH / 32) {
          const double ci = col[i] * inv;
          for (int j = lane; j <= i; j += 32) {
            const double v = S[pk(i, j)];
            S[pk(i, j)] = i == k ? (j == k ? -inv : col[j] * inv) : (j == k ? ci : fma(-ci, col[j], v));
          }
        }
        __syncthreads();
      }
      // G = A_BS D, a row per warp
      for (int i = warp; i < nb; i += FTH / 32) {
        const double* ar = A + (size_t)i * ns;
        for (int j = lane; j < ns; j += 32) {
          double acc = 0.0;
          for (int k = 0; k < j; ++k) acc = fma(-ar[k], S[pk(j, k)], acc);
          for (int k = j; k < ns; ++k) acc = fma(-ar[k], S[pk(k, j)], acc);
          G[(size_t)i * ns + j] = acc;
          put(nd.p_off + ns * gd + i * gu, j, -acc);
          put(nd.p_off + j * gd, 4 * gu + i, -acc);
        }
      }
      for (int i = warp; i < ns; i += FTH / 32)
        for (int j = lane; j < ns; j += 32)
          put(nd.p_off + i * gd, j, j <= i ? -S[pk(i, j)] : -S[pk(j, i)]);
      __syncthreads();
      // the parent's update A_BB - G A_BS^T
      for (int i = warp; i < nb; i += FTH / 32) {
        const double* gr = G + (size_t)i * ns;
        for (int j = lane; j <= i; j += 32) {
          const double* ar = A + (size_t)j * ns;
          double acc = U[(size_t)i * nb + j];
          for (int k = 0; k < ns; ++k) acc = fma(-gr[k], ar[k], acc);
          U[(size_t)i * nb + j] = acc;
        }
      }
    }
    __syncthreads();
    if (tid == 0 && bad) atomicOr(err, (int)DEVERR_NOT_SPD);
  }
}

// ---------------------------------------------------------------- host plan
struct HNode {
  std::vector<int> S, B;  // region nodes
  std::vector<int> child;
  int height = 0;
};
// Boxes of at most 2 x 2 nodes are not cut; those of at most RT_CROSS nodes a
// side are cut by column and row at once.
constexpr int RT_LEAF = 2, RT_CROSS = 16;
int rt_cut(std::vector<HNode>& out, int W, int H, int x0, int y0, int w, int h) {
  HNode nd;
  const bool whole = w <= RT_LEAF && h <= RT_LEAF;
  int c = -1, r = -1;
  if (!whole) {
    const bool both = w > RT_LEAF && h > RT_LEAF && std::max(w, h) <= RT_CROSS && w <= 2 * h && h <= 2 * w;
    if (both || w >= h) c = x0 + w / 2;
    if (both || w < h) r = y0 + h / 2;
    const int xs[2] = {x0, c + 1}, xe[2] = {c >= 0 ? c : x0 + w, c >= 0 ? x0 + w : 0};
    const int ys[2] = {y0, r + 1}, ye[2] = {r >= 0 ? r : y0 + h, r >= 0 ? y0 + h : 0};
    for (int b = 0; b < 2; ++b)
      for (int a = 0; a < 2; ++a)
        if (xe[a] > xs[a] && ye[b] > ys[b])
          nd.child.push_back(rt_cut(out, W, H, xs[a], ys[b], xe[a] - xs[a], ye[b] - ys[b]));
  }
  for (int y = y0; y < y0 + h; ++y)
    for (int x = x0; x < x0 + w; ++x)
      if (whole || x == c || y == r) nd.S.push_back(y * W + x);
  for (int y = std::max(y0 - 1, 0); y <= std::min(y0 + h, H - 1); ++y)
    for (int x = std::max(x0 - 1, 0); x <= std::min(x0 + w, W - 1); ++x)
      if (x < x0 || x >= x0 + w || y < y0 || y >= y0 + h) nd.B.push_back(y * W + x);
  for (int k : nd.child) nd.height = std::max(nd.height, out[k].height + 1);
  out.push_back(std::move(nd));
  return (int)out.size() - 1;
}

// A panel while it is built: per lane its segments (start in the inputs) and
// its unknown; the inputs; the places to note (front row -> stream row, lane).
struct Panel {
  int seg4[4] = {0, 0, 0, 0}, maxb[4] = {0, 0, 0, 0}, nseg = 0, nlane = 0;
  bool more = false, cont = false;  // its node's panels stay together; not the first of them
  int base[32][4] = {}, out[32] = {}, xs[32] = {};
  std::vector<int> in;  // none: the panel before's (of the same node)
  std::vector<std::array<int, 5>> note;  // row's first entry in place, segment, lane, its first group here, groups in all
};

}  // namespace

int rt_slots(bool fp32, int copies) { return fp32 ? 4 : (copies == 2 ? 2 : 3); }
// the bulk copy of a CTA's lists: descriptors, then panel numbers
size_t rt_list_bytes(const RtShapeHost& P) { return P.desc.size() * 4; }

bool rt_shape_build(int W, int H, RtShapeHost* P) {
  *P = RtShapeHost();
  const int nn = W * H;
  if (2 * nn + 4 > 0xffff) return false;  // and fewer than 2^15 tree nodes
  P->w = W, P->h = H, P->nn = nn;
  std::vector<HNode> hn;
  rt_cut(hn, W, H, 0, 0, W, H);
  const int nnode = (int)hn.size(), top = hn[nnode - 1].height;
  // the tree's order of the region's nodes
  P->inv.assign(nn, 0);
  int zc = 0;
  for (const HNode& v : hn)
    for (int s : v.S) P->inv[s] = (unsigned short)zc++;
  auto zdof = [&](const std::vector<int>& nodes, int d) { return 2 * (int)P->inv[nodes[d >> 1]] + (d & 1); };
  // nodes for the factor, and the scratch their updates take (each given back
  // once the parent has read it)
  struct Span {
    long long off, len;
  };
  std::vector<Span> freed;
  long long u_end = 0;
  auto take = [&](long long len) {
    for (size_t k = 0; k < freed.size(); ++k)
      if (freed[k].len >= len) {
        const long long o = freed[k].off;
        freed[k].off += len;
        freed[k].len -= len;
        if (freed[k].len == 0) freed.erase(freed.begin() + k);
        return o;
      }
    const long long o = u_end;
    u_end += len;
    return o;
  };
  auto give = [&](long long off, long long len) {
    if (len == 0) return;
    size_t k = std::lower_bound(freed.begin(), freed.end(), off,
                                [](const Span& a, long long o) { return a.off < o; }) - freed.begin();
    freed.insert(freed.begin() + k, Span{off, len});
    if (k + 1 < freed.size() && freed[k].off + freed[k].len == freed[k + 1].off) {
      freed[k].len += freed[k + 1].len;
      freed.erase(freed.begin() + k + 1);
    }
    if (k > 0 && freed[k - 1].off + freed[k - 1].len == freed[k].off) {
      freed[k - 1].len += freed[k].len;
      freed.erase(freed.begin() + k);
    }
  };
  int places = 0;
  P->smax = 0;
  std::vector<int> where(nn, -1);
  for (int k = 0; k < nnode; ++k) {
    const HNode& v = hn[k];
    RtNode d{};
    d.ns = (int)v.S.size();
    d.nb = (int)v.B.size();
    const int ns4 = (2 * d.ns + 3) & ~3, nb4 = (2 * d.nb + 3) & ~3;
    if (ns4 + nb4 > STG || v.child.size() > 4) return false;
    d.f_off = (int)P->front.size();
    for (int s : v.S) P->front.push_back((unsigned short)s);
    for (int s : v.B) P->front.push_back((unsigned short)s);
    d.p_off = places;
    places += 2 * d.ns * (ns4 + nb4) / 4 + 2 * d.nb * (ns4 / 4);
    d.u_off = (int)take(4LL * d.nb * d.nb);
    d.nchild = (int)v.child.size();
    for (int c = 0; c < d.nchild; ++c) {
      const HNode& ch = hn[v.child[c]];
      d.c_u[c] = P->nodes[v.child[c]].u_off;
      d.c_nb[c] = 2 * (int)ch.B.size();
      d.c_map[c] = (int)P->cmap.size();
      for (size_t q = 0; q < ch.B.size(); ++q) where[ch.B[q]] = (int)q;
      for (int s : v.S) P->cmap.push_back((short)where[s]);
      for (int s : v.B) P->cmap.push_back((short)where[s]);
      for (int s : ch.B) where[s] = -1;
    }
    for (int c = 0; c < d.nchild; ++c) {
      const long long nb = 2 * (long long)hn[v.child[c]].B.size();
      give(P->nodes[v.child[c]].u_off, nb * nb);
    }
    P->smax = std::max(P->smax, 2 * d.ns);
    P->bs_max = std::max(P->bs_max, 4 * d.ns * d.nb);
    P->nodes.push_back(d);
  }
  P->u_max = (int)u_end;
  P->place.assign(places, 0);
  // ---- panels, phase by phase ----
  std::vector<std::vector<int>> byh(top + 1);
  for (int k = 0; k < nnode; ++k) byh[hn[k].height].push_back(k);
  std::vector<int> vrows(NV, 0);  // columns dealt to each stream so far
  std::vector<std::vector<Panel>> phases;
  std::vector<std::vector<int>> dls;
  // up: every unknown of the level's boundaries, with the tree nodes around it
  // (at most four: boxes of one level are at least two nodes apart)
  struct Around {
    int n = 0, node[4], row[4];
  };
  std::vector<Around> around(2 * (size_t)nn);
  std::vector<int> at(nnode, -1), open;  // start of a node's z_S in the open panel's inputs
  auto groups = [&](int k, bool down) {  // of a row of node k
    const int gu = (2 * (int)hn[k].S.size() + 3) / 4;
    return down ? gu + (2 * (int)hn[k].B.size() + 3) / 4 : gu;
  };
  auto up_row = [&](int k, int b) {
    return P->nodes[k].p_off + 2 * (int)hn[k].S.size() * groups(k, true) + b * groups(k, false);
  };
  for (int hgt = 0; hgt < top; ++hgt) {
    std::vector<int> order;
    for (int k : byh[hgt])
      for (int b = 0; b < 2 * (int)hn[k].B.size(); ++b) {
        const int zi = zdof(hn[k].B, b);
        Around& a = around[zi];
        if (a.n == 0) order.push_back(zi);
        if (a.n == 4) return false;
        a.node[a.n] = k;
        a.row[a.n++] = b;
      }
    // rows with the same nodes side by side, most segments first
    std::vector<std::pair<unsigned long long, int>> keyed(order.size());
    for (size_t k = 0; k < order.size(); ++k) {
      const Around& a = around[order[k]];
      unsigned long long key = 4 - a.n;
      for (int q = 0; q < 4; ++q) key = (key << 15) | (unsigned long long)(q < a.n ? a.node[q] : 0);
      keyed[k] = {key, order[k]};
    }
    std::sort(keyed.begin(), keyed.end());
    for (size_t k = 0; k < order.size(); ++k) order[k] = keyed[k].second;
    std::vector<Panel> ps;
    auto ns4_of = [&](int k) { return (2 * (int)hn[k].S.size() + 3) & ~3; };
    for (int zi : order) {
      Around& rw = around[zi];
      for (bool fresh = ps.empty();; fresh = true) {
        if (fresh) {
          ps.emplace_back();
          for (int k : open) at[k] = -1;
          open.clear();
        }
        Panel& p = ps.back();
        // the row's inputs, and every lane's reads to the length of the panel's
        // segments (zero columns beyond its own), stay within the buffer
        int size = (int)p.in.size();
        bool fits = true;
        for (int q = 0; q < rw.n; ++q) {
          const int k = rw.node[q], b = at[k] >= 0 ? at[k] : size;
          if (at[k] < 0) size += ns4_of(k);
          const int len = std::max(4 * p.seg4[q], ns4_of(k));
          fits = fits && std::max(b, p.maxb[q]) + len <= STG;
        }
        fits = fits && size <= STG;
        if (!fits && fresh) return false;
        if (p.nlane == 32 || !fits) continue;
        for (int q = 0; q < rw.n; ++q) {
          const int k = rw.node[q];
          if (at[k] >= 0) continue;
          at[k] = (int)p.in.size();
          open.push_back(k);
          const int ns = 2 * (int)hn[k].S.size();
          for (int s = 0; s < ns4_of(k); ++s) p.in.push_back(s < ns ? zdof(hn[k].S, s) : 2 * nn);
        }
        const int l = p.nlane++;
        p.out[l] = zi;
        p.nseg = std::max(p.nseg, rw.n);
        for (int q = 0; q < rw.n; ++q) {
          const int k = rw.node[q];
          p.base[l][q] = at[k];
          p.maxb[q] = std::max(p.maxb[q], at[k]);
          p.seg4[q] = std::max(p.seg4[q], ns4_of(k) / 4);
          p.note.push_back({up_row(k, rw.row[q]), q, l, 0, ns4_of(k) / 4});
        }
        break;
      }
      rw.n = 0;
    }
    for (int k : open) at[k] = -1;
    open.clear();
    phases.push_back(std::move(ps));
    dls.emplace_back();
  }
  P->nup = (int)phases.size();
  // down: the level's own unknowns.  A node of more than 32 spans panels: with
  // enough such nodes for all streams, its panels follow one another in one
  // stream and share the inputs gathered for the first; else they run in
  // several streams and the phase's results are held back until all of them
  // have read their inputs
  for (int hgt = top; hgt >= 0; --hgt) {
    std::vector<int> nodes = byh[hgt];
    int wide = 0;  // nodes that span panels
    for (int k : nodes) wide += 2 * (int)hn[k].S.size() > 32;
    const bool defer = wide > 0 && wide < NV;
    auto len4 = [&](int k) {
      return (((2 * (int)hn[k].S.size() + 3) & ~3) + ((2 * (int)hn[k].B.size() + 3) & ~3)) / 4;
    };
    std::stable_sort(nodes.begin(), nodes.end(), [&](int a, int b) { return len4(a) > len4(b); });
    std::vector<Panel> ps;
    std::vector<int> dl;
    for (int k : nodes) {
      const HNode& v = hn[k];
      const int ns = 2 * (int)v.S.size(), nb = 2 * (int)v.B.size();
      for (int s0 = 0; s0 < ns; s0 += 32) {
        const int cnt = std::min(32, ns - s0);
        if (ps.empty() || ns > 32 || ps.back().nlane + cnt > 32 || ps.back().more ||
            (int)ps.back().in.size() + 4 * std::max(len4(k), ps.back().seg4[0]) > STG)
          ps.emplace_back();
        Panel& p = ps.back();
        const bool cont = ns > 32 && !defer && s0 > 0;
        p.more = ns > 32 && !defer;
        p.cont = cont;
        const int at = cont ? 0 : (int)p.in.size();
        if (!cont) {
          for (int s = 0; s < ((ns + 3) & ~3); ++s) p.in.push_back(s < ns ? zdof(v.S, s) : 2 * nn);
          for (int s = 0; s < ((nb + 3) & ~3); ++s) p.in.push_back(s < nb ? zdof(v.B, s) : 2 * nn);
        }
        p.nseg = 1;
        p.seg4[0] = std::max(p.seg4[0], len4(k));
        for (int s = s0; s < s0 + cnt; ++s) {
          const int l = p.nlane++;
          p.out[l] = zdof(v.S, s);
          p.base[l][0] = at;
          p.maxb[0] = std::max(p.maxb[0], at);
          if (defer) {
            p.xs[l] = (int)dl.size();
            dl.push_back(p.out[l]);
          }
          p.note.push_back({P->nodes[k].p_off + s * groups(k, true), 0, l, 0, groups(k, true)});
        }
      }
    }
    phases.push_back(std::move(ps));
    dls.push_back(std::move(dl));
  }
  P->nphase = (int)phases.size();
  // ---- deal the panels to the streams: longest first, to the least loaded
  // stream of the phase.  Phases with few panels for eight streams (the top of the
  // tree, all of a small set's) have each panel's columns split in two or four
  // parts, dealt apart, their sums added when the phase ends ----
  using Deal = std::array<std::vector<int>, NV>;
  constexpr int FIXED = 12, HELD = 10;  // a panel's and a deferred phase's fixed parts, in columns
  auto rows_of = [](const Panel& p) { return 4 * (p.seg4[0] + p.seg4[1] + p.seg4[2] + p.seg4[3]); };
  auto deal_out = [&](const std::vector<Panel>& ps, Deal* out) {  // the longest stream's load
    std::vector<std::vector<int>> units;  // panels that stay together
    for (int q = 0; q < (int)ps.size(); ++q) {
      if (!ps[q].cont) units.emplace_back();
      units.back().push_back(q);
    }
    auto rows_of_unit = [&](const std::vector<int>& u) {
      int t = 0;
      for (int q : u) t += rows_of(ps[q]);
      return t;
    };
    std::stable_sort(units.begin(), units.end(), [&](const std::vector<int>& a, const std::vector<int>& b) {
      return rows_of_unit(a) > rows_of_unit(b);
    });
    std::array<int, NV> load{};
    for (const std::vector<int>& u : units) {
      int best = 0;
      for (int v = 1; v < NV; ++v)
        if (load[v] < load[best]) best = v;
      for (int q : u) {
        load[best] += rows_of(ps[q]) + FIXED;
        (*out)[best].push_back(q);
      }
    }
    return *std::max_element(load.begin(), load.end());
  };
  // part j of np of every panel; outs: the phase's outputs in the order of their places
  auto split = [&](const std::vector<Panel>& ps, int np, std::vector<int>* outs) {
    std::vector<Panel> r;
    outs->clear();
    const std::vector<int>* in = nullptr;
    for (const Panel& p : ps) {
      if (!p.cont) in = &p.in;
      const int g = rows_of(p) / 4, first = (int)outs->size();
      for (int l = 0; l < p.nlane; ++l) outs->push_back(p.out[l]);
      for (int j = 0; j < np; ++j) {
        const int ga = g * j / np, gb = g * (j + 1) / np;
        Panel n;
        n.nlane = p.nlane;
        for (int l = 0; l < p.nlane; ++l) {
          n.out[l] = p.out[l];
          n.xs[l] = (j << 16) | (first + l);
        }
        int at = 0;
        std::array<int, 4> seg{-1, -1, -1, -1}, skip{};
        for (int q = 0; q < p.nseg; ++q) {
          const int a = std::max(ga - at, 0), b = std::min(gb - at, p.seg4[q]);
          at += p.seg4[q];
          if (b <= a) continue;
          seg[q] = n.nseg;
          skip[q] = a;
          n.seg4[n.nseg] = b - a;
          n.maxb[n.nseg] = p.maxb[q] + 4 * a;
          for (int l = 0; l < p.nlane; ++l) n.base[l][n.nseg] = p.base[l][q] + 4 * a;
          ++n.nseg;
        }
        n.note.reserve(p.note.size());
        for (const auto& t : p.note)
          if (seg[t[1]] >= 0) n.note.push_back({t[0], seg[t[1]], t[2], t[3] + skip[t[1]], t[4]});
        if (n.nseg > 0) n.in = *in;
        bool one = n.nseg == 1;  // one input range for all lanes: gather no more than that
        for (int l = 1; l < p.nlane; ++l) one = one && n.base[l][0] == n.base[0][0];
        if (one) {
          const int b0 = n.base[0][0], e0 = std::min(b0 + 4 * n.seg4[0], (int)n.in.size());
          n.in = std::vector<int>(n.in.begin() + b0, n.in.begin() + e0);
          n.maxb[0] = 0;
          for (int l = 0; l < p.nlane; ++l) n.base[l][0] = 0;
        }
        r.push_back(std::move(n));
      }
    }
    const int cnt = (int)outs->size();
    for (Panel& n : r)
      for (int l = 0; l < n.nlane; ++l) n.xs[l] = (n.xs[l] >> 16) * cnt + (n.xs[l] & 0xffff);
    return r;
  };
  std::vector<Deal> deal(P->nphase);
  std::vector<int> parts(P->nphase, 1);
  for (int ph = 0; ph < P->nphase; ++ph) {
    int best = deal_out(phases[ph], &deal[ph]) + (dls[ph].empty() ? 0 : HELD);
    int total = 0;
    for (const Panel& p : phases[ph]) total += rows_of(p) + FIXED;
    if (best * NV <= total + total / 10) continue;  // dealt evenly as they are
    const std::vector<Panel> whole = phases[ph];
    for (int np = 2; np <= 4; np += 2) {
      std::vector<int> outs;
      std::vector<Panel> ps = split(whole, np, &outs);
      if (np * (int)outs.size() > 256) continue;
      Deal d;
      const int cost = deal_out(ps, &d) + HELD;
      if (100 * cost > 92 * best) continue;
      best = cost;
      phases[ph] = std::move(ps);
      dls[ph] = std::move(outs);
      deal[ph] = std::move(d);
      parts[ph] = np;
    }
  }
  for (int ph = 0; ph < P->nphase; ++ph)
    for (int v = 0; v < NV; ++v)
      for (int q : deal[ph][v]) vrows[v] += rows_of(phases[ph][q]);
  P->vrow[0] = 0;
  for (int v = 0; v < NV; ++v) P->vrow[v + 1] = P->vrow[v] + (vrows[v] + 15) / 16 * 16;  // whole chunks
  if ((long long)P->vrow[NV] * 32 > 0x3fffffffLL) return false;
  P->elems = 32LL * P->vrow[NV];
  std::vector<int> row(NV);
  for (int v = 0; v < NV; ++v) row[v] = P->vrow[v];
  int xsmax = 0;
  for (int ph = 0; ph < P->nphase; ++ph) {
    for (int v = 0; v < NV; ++v) {
      P->vp.push_back((int)P->desc.size() / 2);
      for (int q : deal[ph][v]) {
        const Panel& p = phases[ph][q];
        int start[4], r0 = row[v], packed = 0;
        for (int s = 0; s < 4; ++s) {
          start[s] = r0;
          r0 += 4 * p.seg4[s];
          if (p.seg4[s] > 255) return false;
          packed |= p.seg4[s] << (8 * s);
        }
        for (auto& nt : p.note)
          for (int t = 0; t < p.seg4[nt[1]] && nt[3] + t < nt[4]; ++t)
            P->place[nt[0] + nt[3] + t] = (start[nt[1]] + 4 * t) * 32 + nt[2];
        row[v] = r0;
        P->desc.push_back(packed);
        P->desc.push_back((int)p.in.size() | (p.nseg << 16));
        for (int t = 0; t < 4; ++t) P->stg = std::max(P->stg, p.maxb[t] + 4 * p.seg4[t]);
        P->stg = std::max(P->stg, ((int)p.in.size() + 31) / 32 * 32);
        const size_t at = P->lane.size();
        P->lane.resize(at + 512, (unsigned short)(2 * nn));
        unsigned short* u = P->lane.data() + at;
        for (int l = 0; l < 32; ++l, u += 8) {
          for (int s = 0; s < 4; ++s) u[s] = (unsigned short)(l < p.nlane ? p.base[l][s] : 0);
          u[4] = (unsigned short)(l < p.nlane ? p.out[l] : 0xffff);
          u[5] = (unsigned short)(l < p.nlane ? p.xs[l] : 0);
          u[6] = u[7] = 0;
        }
        for (int e = 0; e < (int)p.in.size(); ++e) u[8 * (e & 31) + (e >> 5)] = (unsigned short)p.in[e];
      }
    }
    P->defer.push_back((int)P->dlist.size());
    P->defer.push_back((int)dls[ph].size() | (parts[ph] << 16));
    if (dls[ph].empty()) P->defer.back() = 0;
    for (int zi : dls[ph]) P->dlist.push_back((unsigned short)zi);
    xsmax = std::max(xsmax, parts[ph] * (int)dls[ph].size());
  }
  P->vp.push_back((int)P->desc.size() / 2);
  P->npanel = (int)P->desc.size() / 2;
  P->lane.resize(P->lane.size() + 512, 0);  // read one panel ahead
  P->desc.insert(P->desc.end(), P->vp.begin(), P->vp.end());  // one list, whole 16 bytes
  P->desc.resize((P->desc.size() + 3) / 4 * 4, 0);
  if (P->dlist.empty()) P->dlist.push_back(0);
  if (P->cmap.empty()) P->cmap.push_back(0);
  P->xs = xsmax;
  return true;
}

size_t rt_shape_bytes(const RtShapeHost& P) {
  return P.inv.size() * 2 + P.desc.size() * 4 + P.lane.size() * 2 +
         P.defer.size() * 4 + P.dlist.size() * 2 + P.nodes.size() * sizeof(RtNode) + P.front.size() * 2 +
         P.cmap.size() * 2 + P.place.size() * 4;
}

size_t rt_smem_bytes(const RtShapeHost& P, bool fp32, int copies) {
  const int ns = rt_slots(fp32, copies);
  const size_t b = rt_list_bytes(P) + (fp32 ? rt_smem<float>(P.nn, P.stg, P.xs, ns).total * sizeof(float)
                        : rt_smem<double>(P.nn, P.stg, P.xs, ns).total * sizeof(double));
  // the P sums' buffer lies over the inputs' and the ring
  const size_t zb = fp32 ? rt_smem<float>(P.nn, P.stg, P.xs, ns).stg * sizeof(float)
                         : rt_smem<double>(P.nn, P.stg, P.xs, ns).stg * sizeof(double);
  return std::max(b, zb + (NMODES * (size_t)VL + 16 * NMODES) * sizeof(double));
}
size_t rt_factor_smem_bytes(int smax) { return ((size_t)smax * (smax + 1) / 2 + 2 * (size_t)smax) * sizeof(double); }

cudaError_t launch_rtree_factor(cudaStream_t s, const LatView& lv, const RtView& rt, double* f64, float* f32,
                                double* scratch, int first, double* work, long long stride, int grid, int smax,
                                int* err, bool cut, const int* sets, int n) {
  const size_t smem = rt_factor_smem_bytes(smax);
  if (!sets) n = lv.M;
  if (cut) k_rtree_factor<true><<<grid, FTH, smem, s>>>(lv, rt, f64, f32, scratch, first, work, stride, err, sets, n);
  else k_rtree_factor<false><<<grid, FTH, smem, s>>>(lv, rt, f64, f32, scratch, first, work, stride, err, sets, n);
  return cudaGetLastError();
}

namespace {
template <class F>
cudaError_t rt_dispatch(bool fp32, int threads, int copies, F go) {
  auto nt = [&](auto t, auto ns) {
    if (threads == 64) go(t, std::integral_constant<int, 64>(), ns);
    else if (threads == 128) go(t, std::integral_constant<int, 128>(), ns);
    else if (threads == 256) go(t, std::integral_constant<int, 256>(), ns);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
  };
  if (fp32) return nt(float(), std::integral_constant<int, 4>());
  if (copies == 2) return nt(double(), std::integral_constant<int, 2>());
  return nt(double(), std::integral_constant<int, 3>());
}
}  // namespace

cudaError_t launch_rtree(cudaStream_t s, const LatView& lv, const RtView& rt, const void* fac, bool fp32,
                         const double2* r, void* delta, double* P, const IterCtl* ctl, int* err, int threads,
                         int copies, size_t smem, int wait0, const void* fac2, const double2* r2, void* delta2) {
  return rt_dispatch(fp32, threads, copies, [&](auto t, auto nt, auto ns) {
    using T = decltype(t);
    (void)launch_dep(k_rtree<T, decltype(nt)::value, decltype(ns)::value>, s, fac2 ? 2 * lv.M : lv.M,
                     decltype(nt)::value, smem, 0, lv, rt, (const T*)fac, r, (T*)delta, P, ctl, err, wait0,
                     (const T*)fac2, r2, (T*)delta2);  // rt_dispatch returns its error
  });
}

cudaError_t launch_batch_rtree(cudaStream_t s, bool fp32, int threads, int copies, size_t smem, const BatchProb* P,
                               const BatchItem* it, int n) {
  if (n <= 0) return cudaSuccess;
  return rt_dispatch(fp32, threads, copies, [&](auto t, auto nt, auto ns) {
    kb_rtree<decltype(t), decltype(nt)::value, decltype(ns)::value>
        <<<n, decltype(nt)::value, smem, s>>>(P, it);
  });
}

cudaError_t configure_relax_tree(int max_smem) {
  cudaError_t e = set_max_dynamic_smem(k_rtree_factor<false>, max_smem);
  if (e == cudaSuccess) e = set_max_dynamic_smem(k_rtree_factor<true>, max_smem);
#define HMS_RT_ATTR(K) \
  if (e == cudaSuccess) e = set_max_dynamic_smem(K, max_smem);
  HMS_RT_ATTR((k_rtree<float, 64, 4>))
  HMS_RT_ATTR((k_rtree<float, 128, 4>))
  HMS_RT_ATTR((k_rtree<float, 256, 4>))
  HMS_RT_ATTR((k_rtree<double, 64, 2>))
  HMS_RT_ATTR((k_rtree<double, 128, 2>))
  HMS_RT_ATTR((k_rtree<double, 256, 2>))
  HMS_RT_ATTR((k_rtree<double, 64, 3>))
  HMS_RT_ATTR((k_rtree<double, 128, 3>))
  HMS_RT_ATTR((k_rtree<double, 256, 3>))
  HMS_RT_ATTR((kb_rtree<float, 64, 4>))
  HMS_RT_ATTR((kb_rtree<float, 128, 4>))
  HMS_RT_ATTR((kb_rtree<float, 256, 4>))
  HMS_RT_ATTR((kb_rtree<double, 64, 2>))
  HMS_RT_ATTR((kb_rtree<double, 128, 2>))
  HMS_RT_ATTR((kb_rtree<double, 256, 2>))
  HMS_RT_ATTR((kb_rtree<double, 64, 3>))
  HMS_RT_ATTR((kb_rtree<double, 128, 3>))
  HMS_RT_ATTR((kb_rtree<double, 256, 3>))
#undef HMS_RT_ATTR
  return e;
}

}  // namespace hms

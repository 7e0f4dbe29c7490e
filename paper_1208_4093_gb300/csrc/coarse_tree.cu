// K4 by a tree of dense fronts: the upper-level solve of Eq. 8 for set grids
// whose fronts fit the shared memory of one thread-block cluster (coarse_nd.cu
// takes the larger ones, panel by panel from device memory).
//
// The unknowns are ordered by nested dissection of the set grid: a box of sets
// is cut by its middle column and row of sets (a long box by one of them), the
// parts are eliminated independently and the separator last.  A tree node is a dense symmetric front
// over its own unknowns S and the unknowns B of the sets around its box.
//
// Factor (one launch per tree level, leaves first; one cluster per front).  The
// front F = [A_SS .; A_BS 0] + the children's update matrices is gathered into
// 32 x 32 tiles spread over the cluster's shared memory and its S part is
// *swept* (Gauss-Jordan on a symmetric matrix) 32 pivots at a time:
//   P = F_kk^-1, C_I = F_Ik P, F_IJ -= C_I F_Jk^T, F_Ik = C_I, F_kk = -P,
// which leaves -A_SS^-1 in SS, A_BS A_SS^-1 in BS and the Schur complement in
// BB.  A Cholesky factor would need half the products, but its solves need a
// chain of triangular steps per front; with the swept front both directions
// of a solve are one dense product per front:
//   forward   w_B = (children's w)_B - G f_S        (G = A_BS A_SS^-1)
//   backward  x_S = A_SS^-1 f_S - G^T x_B,
// f_S being the right-hand side plus the children's w.
//
// Solve (one cluster for the whole system).  All solves of an update and the
// FP64 refinement residuals between them run in one launch, level by level
// with a cluster barrier after each.  The work of a level is laid out on the
// host as plain lists per CTA: which values to gather into shared memory and
// which matrix rows to multiply them by (eight lanes per row).
//
// Bound by latency: per 32 pivots of the tree's longest path about 13 K cycles
// (reading the pivot column from L2, two products, the sweep's pivots, a cluster
// barrier), per level the launch, the gather and the output (about 7 us), per
// phase of a solve two trips to L2 and a cluster barrier.  16 x 16 sets of nine modes
// (2304 unknowns): factor 170 us, five solves 129 us; the two-sided band factor
// took 521 and 279 us, the panel-by-panel fronts of coarse_nd.cu 629 and 870 us.
//
// Every sum runs in an order that does not depend on the cluster sizes.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "coarse_blocks.cuh"
#include "hms_internal.cuh"
#include "ptx.cuh"

namespace hms {
namespace {

namespace cg = cooperative_groups;
constexpr int FT = 512;           // threads of a factor CTA
constexpr int FW = FT / 32;
constexpr int ST = 512;           // threads of a solve CTA
constexpr float TREE_TAU = 1e-6f; // FP32 pivot below which a mode is dropped (as the band factors)
constexpr int TS = 32 * 32;       // floats of a tile

__device__ inline bool tree_done(const IterCtl* ctl) { return ctl && *(volatile const int*)&ctl->done; }

// ---------------------------------------------------------------- scaled system
// Work item: a problem of the launch and one of its sets or nodes; the only
// problem's sets in order without a list.
__device__ inline TreeItem item_of(const TreeItem* items, int k) {
  if (items) return items[k];
  return TreeItem{0, k};
}

// One CTA per set: its five blocks of K_aa from the slots (SLOTS; else the
// blocks are there), then, in one warp with lane = mode, the scale s_i =
// D_ii^-1/2, b = s P, x = 0 and the modes that take no part (mode mask,
// vanishing diagonal, a pivot <= 1e-14 in the FP64 elimination of the scaled
// diagonal block in mode order): the rules of k_blk_diag, whose dependent pivots in
// one thread per set took 40 us.  Bound by the chain of FP64 operations, 64 clocks
// each for one warp of an SM: one entry per thread, the pivots' reciprocals by two
// Newton steps from FP32, and L D L^T instead of square roots and divisions take
// 14 us where 128 threads and the Cholesky form took 23 (16 to 256 sets; q = 12: 15
// and 34).  Beyond two sets per SM the entries' loads and sums of one set hide the
// others' chains, and CTAs of 128 threads all fit at once (1015 sets: 12 us less per
// update than one entry per thread).
template <int Q>
constexpr int DIAG_T = (NBLK * Q * Q + 31) / 32 * 32;
template <int Q, bool SLOTS>
__global__ void __launch_bounds__(DIAG_T<Q>) k_tree_diag(const TreeProb* __restrict__ probs,
                                                         const TreeItem* __restrict__ items, int use_ctl) {
  const TreeItem it = item_of(items, blockIdx.x);
  const TreeProb& pb = probs[it.prob];
  constexpr unsigned FULL = 0xffffffffu;
  const int I = it.node, lane = threadIdx.x & 31, tid = threadIdx.x;
  __shared__ double S[Q * Q];
  const LatView lv = pb.lv;
  const double *base = pb.slots_base, *now = pb.slots_it, *Pv = pb.P;
  double *blk = pb.blk, *scale = pb.scale, *bv = pb.b, *xv = pb.x;
  int* dropped = pb.dropped;
  const IterCtl* ctl = pb.ctl;
  const unsigned mask = pb.mode_mask;
  dep_wait();
  dep_launch();
  if (use_ctl && tree_done(ctl)) return;
  const double rhs = tid < Q ? Pv[Q * I + tid] : 0.0;
  double* B = blk + (size_t)I * NBLK * Q * Q;
  for (int e = tid; e < (SLOTS ? NBLK : 1) * Q * Q; e += blockDim.x) {
    double v;
    if constexpr (SLOTS) {
      v = blk_entry(lv, base, now, I, e / (Q * Q), e % (Q * Q) / Q, e % Q);
      B[e] = v;
    } else {
      v = B[e];
    }
    if (e < Q * Q) S[e] = v;
  }
  __syncthreads();
  if (tid >= 32) return;
  const int row = lane < Q ? lane : Q - 1;
  const double D = S[row * Q + row];
  const bool in = lane < Q && ((mask >> row) & 1u);
  // the largest positive diagonal (positive doubles order as their bits do)
  long long top = in && D > 0.0 ? __double_as_longlong(D) : 0;
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) {
    const long long o = __shfl_xor_sync(FULL, top, m);
    top = o > top ? o : top;
  }
  bool dr = !in || !(D > 1e-300) || !(D > 1e-28 * __longlong_as_double(top));
  const double sc = dr ? 0.0 : rsqrt(D);
  double A[Q];
#pragma unroll
  for (int l = 0; l < Q; ++l) {
    const int lo = l < row ? l : row, hi = l < row ? row : l;
    A[l] = sc * S[hi * Q + lo] * __shfl_sync(FULL, sc, l);
  }
  dr = drop_pivots<Q>(A, dr, lane);
  if (lane < Q) {
    const int i = Q * I + lane;
    scale[i] = sc;
    bv[i] = dr ? 0.0 : sc * rhs;
    xv[i] = 0.0;
    dropped[i] = dr ? 1 : 0;
  }
}

// The scaled rows of a set (one CTA): A_ij = s_hi K_ij s_lo (the larger index's
// scale first), 1 on the diagonal, 0 in the rows and columns of dropped modes
// and outside the set grid: row i holds its nine neighbour sets' entries, set
// (dx, dy) at ((dy + 1) 3 + dx + 1) q.  The factor and every refinement residual
// read these; scaling once per update leaves one FP64 operation per entry to
// the residuals instead of three.
__global__ void __launch_bounds__(256) k_tree_rows(const TreeProb* __restrict__ probs,
                                                   const TreeItem* __restrict__ items, int use_ctl) {
  const TreeItem it = item_of(items, blockIdx.x);
  const TreeProb& pb = probs[it.prob];
  dep_wait();
  dep_launch();
  if (use_ctl && tree_done(pb.ctl)) return;
  const int nm = pb.nm, bs = nm * nm, R = 9 * nm, Mx = pb.Mx, My = pb.My, I = it.node;
  const double *blk = pb.blk, *scale = pb.scale;
  const int* dropped = pb.dropped;
  double* arow = pb.arow + (size_t)I * nm * R;
  for (int e = threadIdx.x; e < nm * R; e += 256) {
    const int l = e / R, c = e % R, nb = c / nm, m = c % nm, i = nm * I + l;
    const int dx = nb % 3 - 1, dy = nb / 3 - 1;
    const int Jx = I % Mx + dx, Jy = I / Mx + dy;
    double v = 0.0;
    if (Jx >= 0 && Jx < Mx && Jy >= 0 && Jy < My) {
      const int J = Jy * Mx + Jx, j = nm * J + m;
      if (i == j) {
        v = 1.0;
      } else if (!dropped[i] && !dropped[j]) {
        double k;
        if (J == I) k = blk[(size_t)I * NBLK * bs + (size_t)(l > m ? l : m) * nm + (l > m ? m : l)];
        else if (J > I) k = blk[((size_t)I * NBLK + blk_of(dx, dy)) * bs + (size_t)m * nm + l];
        else k = blk[((size_t)J * NBLK + blk_of(-dx, -dy)) * bs + (size_t)l * nm + m];
        v = i > j ? scale[i] * k * scale[j] : scale[j] * k * scale[i];
      }
    }
    arow[e] = v;
  }
}

// ---------------------------------------------------------------- factor
// element (r, c) of a tile: rows of 32 floats, their eight 16-byte words
// permuted by the row, so that both a thread's own row (lane = row) and 4 x 4
// blocks are read without bank conflicts
__device__ inline int tsw(int r, int c) { return r * 32 + ((((c >> 2) ^ (r & 7)) << 2) | (c & 3)); }

// acc[u][v] = sum_k A[k][4 rg + u] B[k][col(v)], rg = lane / 4, columns
// 4 cg .. + 3 and 16 + 4 cg .. + 3 (cg = lane % 4); A, B rows of lda, ldb floats
__device__ __forceinline__ void mm32(const float* A, int lda, const float* B, int ldb, int kb, int lane,
                                     float (&acc)[4][8]) {
  const float* pa = A + 4 * (lane >> 2);
  const float* pb = B + 4 * (lane & 3);
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 8; ++v) acc[u][v] = 0.f;
#pragma unroll 4
  for (int k = 0; k < kb; ++k) {
    const float4 a4 = *reinterpret_cast<const float4*>(pa + k * lda);
    const float4 b0 = *reinterpret_cast<const float4*>(pb + k * ldb);
    const float4 b1 = *reinterpret_cast<const float4*>(pb + k * ldb + 16);
    const float a[4] = {a4.x, a4.y, a4.z, a4.w};
    const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 8; ++v) acc[u][v] = fmaf(a[u], b[v], acc[u][v]);
  }
}

// A symmetric 32 x 32 block swept on its first kb pivots by four warps: warp w
// holds the columns 8 w .. 8 w + 7, lane = row, a[c] = entry (lane, 8 w + c); on
// return a = -inverse.  A pivot at or below TREE_TAU drops its mode: its row
// and column become zero.  Returns the dropped pivots (every thread).  buf: 128
// floats.  kb is rounded up to a multiple of eight (the block is padded with
// unit pivots).
//
// Bound by the pivots' chain.  Two pivots share a trip through shared memory
// and a barrier (the second one's column, row and pivot are corrected for the
// first in registers): about 100 cycles a pivot, against 170 with one.  One warp
// holding the block needs eight 16-byte loads a pivot and 230 cycles; with its
// 32 pivots written out it is 60 KB of code run once, whose fetching takes 690
// cycles a pivot.  A Newton step on the pivots' reciprocals (1 ulp as they are) does
// not help the refinement: 217 of 12060 updates used every solve with it, 194 without
// and 97 with the two-sided band factor; the explicit inverse is what costs it.
__device__ __forceinline__ unsigned sweep32(float (&a)[8], int kb, int w, int lane, float* buf) {
  unsigned dm = 0u;
#pragma unroll 1
  for (int wo = 0; 8 * wo < kb; ++wo) {
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      const int k = 8 * wo + i;
      float* b1 = buf + 32 * (i & 2);
      float* b2 = b1 + 32;
      if (w == wo) b1[lane] = a[i], b2[lane] = a[i + 1];
      asm volatile("bar.sync 1, 128;" ::: "memory");
      const float p1 = b1[k], x = b1[k + 1], q2 = b2[k + 1], ck1 = b1[lane], cl2 = b2[lane];
      float r1[8], r2[8];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 f = *reinterpret_cast<const float4*>(b1 + 8 * w + 4 * h);
        const float4 g = *reinterpret_cast<const float4*>(b2 + 8 * w + 4 * h);
        r1[4 * h] = f.x, r1[4 * h + 1] = f.y, r1[4 * h + 2] = f.z, r1[4 * h + 3] = f.w;
        r2[4 * h] = g.x, r2[4 * h + 1] = g.y, r2[4 * h + 2] = g.z, r2[4 * h + 3] = g.w;
      }
      // first pivot: other rows lose c times the pivot row; the pivot's own row,
      // equal to its column, becomes inv times it (1 / inv <= 1: nothing cancels)
      const bool d1 = !(p1 > TREE_TAU), mine1 = lane == k, mine2 = lane == k + 1;
      float inv1;
      asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv1) : "f"(p1));
      if (d1) inv1 = 0.f, dm |= 1u << k;
      const float c1 = ck1 * inv1, xi = x * inv1;
      float m1 = mine1 ? inv1 - 1.f : -c1;
      if (d1 && mine1) m1 = 0.f;
      // second pivot, corrected for the first
      const float p2 = fmaf(-xi, x, q2);
      const bool d2 = !(p2 > TREE_TAU);
      float inv2;
      asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv2) : "f"(p2));
      if (d2) inv2 = 0.f, dm |= 2u << k;
      float ck2 = fmaf(m1, x, cl2);
      if (d1 && mine1) ck2 = 0.f;
      const float c2 = ck2 * inv2;
      float m2 = mine2 ? inv2 - 1.f : -c2;
      if (d2 && mine2) m2 = 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        r2[j] = fmaf(-xi, r1[j], r2[j]);
        a[j] = fmaf(m1, r1[j], a[j]);
      }
      if (w == wo) {
        r2[i] = xi;
        a[i] = mine1 ? -inv1 : c1;
      }
      if (d1 && mine1) {  // a dropped mode (rare): its row exactly zero
#pragma unroll
        for (int j = 0; j < 8; ++j) a[j] = 0.f;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) a[j] = fmaf(m2, r2[j], a[j]);
      if (w == wo) a[i + 1] = mine2 ? -inv2 : c2;
      if (d2 && mine2) {
#pragma unroll
        for (int j = 0; j < 8; ++j) a[j] = 0.f;
      }
    }
  }
  return dm;
}

struct TreeFrontSmem {
  int nown, ntile, ldr, ldc;       // own block rows and tiles; row strides of R and C
  size_t r_off, c_off, p_off, buf_off, tab_off, list_off, total;  // floats
};
// shared memory of CTA `rank` of a cluster of `cl` for a front of T block rows
__host__ __device__ inline TreeFrontSmem front_smem(int T, int cl, int rank, int nbuf) {
  TreeFrontSmem L;
  L.nown = rank < T ? (T - rank + cl - 1) / cl : 0;
  L.ntile = 0;
  for (int q = 0; q < L.nown; ++q) L.ntile += rank + q * cl + 1;
  L.ldr = 32 * T;
  L.ldc = 32 * L.nown;
  L.r_off = (size_t)L.ntile * TS;
  L.c_off = L.r_off + (size_t)nbuf * 32 * L.ldr;
  L.p_off = L.c_off + (size_t)32 * L.ldc;
  L.buf_off = L.p_off + 2 * TS;
  L.tab_off = L.buf_off + 128;
  L.list_off = L.tab_off + 6 * (size_t)(32 * T);
  L.total = L.list_off + (size_t)L.ntile;
  return L;
}

// One cluster per front of a level.  CTA r of the cluster owns the block rows
// r, r + cl, ...; tile (I, J), J <= I, lies with its block row.  Per 32 pivots
// every CTA needs the whole pivot column R_I = F_Ik and P.  Their tiles are
// written to a buffer in device memory when they get their last update, and
// after the step's one cluster barrier every CTA reads the buffer from L2 into
// its shared memory (writing each tile into eight CTAs' shared memory instead
// took 6 K cycles a tile).  A step is then: C_I = R_I P for the own rows; the
// own tiles' updates, four warps of the next pivot block's owner updating and
// sweeping that block meanwhile; the barrier.
__global__ void __launch_bounds__(FT, 1) k_tree_factor(const TreeProb* __restrict__ probs,
                                                       const TreeItem* __restrict__ items, int nbuf, int use_ctl) {
  extern __shared__ __align__(16) float fsm[];
  cg::cluster_group cluster = cg::this_cluster();
  const int cl = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const TreeItem it = items[blockIdx.x / cl];
  const TreeProb pb = probs[it.prob];
  const TreeNode nd = pb.nodes[it.node];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nm = pb.nm;
  const int nS = nm * nd.ns, nB = nm * nd.nb, KS = (nS + 31) / 32, nSp = 32 * KS;
  const int T = KS + (nB + 31) / 32;
  const TreeFrontSmem L = front_smem(T, cl, rank, nbuf);
  float* R0 = fsm + L.r_off;
  float* C = fsm + L.c_off;
  float* P0 = fsm + L.p_off;
  int* gpos = reinterpret_cast<int*>(fsm + L.tab_off);  // unknown of a front position, -1: padding
  int* gxy = gpos + 32 * T;                             // its set's row and column and its mode
  int* inc = gxy + 32 * T;                              // its place in each child's boundary, or -1
  int* list = reinterpret_cast<int*>(fsm + L.list_off);  // own tiles
  __shared__ int qhead;
  const int ldr = L.ldr, ldc = L.ldc;
  auto own_of = [&](int I) { return I % cl; };
  // first tile of own block row I = rank + q cl
  auto row_tile = [&](int q) { return q * (rank + 1) + cl * (q * (q - 1) / 2); };
  auto tile = [&](int I, int J) { return fsm + (size_t)(row_tile(I / cl) + J) * TS; };
  auto barrier = [&]() {
    if (cl > 1) cluster.sync();
    else __syncthreads();
  };

  // ---- tables ----
  const int* st = pb.sets + nd.s_off;
  for (int p = tid; p < 32 * T; p += FT) {
    const int u = p < nSp ? p : p - nSp + nS;  // unpadded position
    const bool ok = p < nSp ? p < nS : u < nS + nB;
    int g = -1, xy = 0, ca[4] = {-1, -1, -1, -1};
    if (ok) {
      const int s = u / nm, m = u - s * nm, set = st[s];
      g = set * nm + m;
      xy = ((set / pb.Mx) << 18) | ((set % pb.Mx) << 4) | m;
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (c < nd.nchild) {
          const int t = pb.inv[nd.inv_off[c] + s];
          ca[c] = t < 0 ? -1 : nm * t + m;
        }
    }
    gpos[p] = g;
    gxy[p] = xy;
#pragma unroll
    for (int c = 0; c < 4; ++c) inc[32 * T * c + p] = ca[c];
  }
  for (int q = warp; q < L.nown; q += FW) {
    const int I = rank + q * cl;
    for (int J = lane; J <= I; J += 32) list[row_tile(q) + J] = (I << 16) | J;
  }
  if (tid == 0) qhead = 0;
  // the tables hold nothing but the plan: built while the kernel before runs
  dep_wait();
  dep_launch();
  if (use_ctl && tree_done(pb.ctl)) return;  // the same in every CTA of the cluster
  __syncthreads();

  // ---- assemble: original entries of the S columns and the children's updates,
  // each entry gathered by one thread (the children in order) ----
  // (8 rows of a tile per warp, their loads first: an absent source reads element 0)
  const int Rw = 9 * nm;
  for (int h = warp; h < 4 * L.ntile; h += FW) {
    const int q = h >> 2, r0 = 8 * (h & 3);
    const int I = list[q] >> 16, J = list[q] & 0xffff;
    float* t = fsm + (size_t)q * TS;
    const int jj = 32 * J + lane;
    const int gjj = gpos[jj], xyj = gxy[jj];
    constexpr int AU = 8;
    double v[AU];
    float u[4][AU];
#pragma unroll
    for (int z = 0; z < AU; ++z) {
      const int ii = 32 * I + r0 + z;
      v[z] = (gpos[ii] < 0 || gjj < 0) && ii == jj ? 1.0 : 0.0;
      u[0][z] = u[1][z] = u[2][z] = u[3][z] = 0.f;
    }
    if (J < KS) {
#pragma unroll
      for (int z = 0; z < AU; ++z) {
        const int ii = 32 * I + r0 + z;
        const int gii = gpos[ii], xyi = gxy[ii];
        const bool lower = ii >= jj;
        const int gi = lower ? gii : gjj, xi = lower ? xyi : xyj, xj = lower ? xyj : xyi;
        const int dx = ((xj >> 4) & 0x3fff) - ((xi >> 4) & 0x3fff), dy = (xj >> 18) - (xi >> 18);
        if (gii >= 0 && gjj >= 0 && dx >= -1 && dx <= 1 && dy >= -1 && dy <= 1)
          v[z] = pb.arow[gi * Rw + ((dy + 1) * 3 + dx + 1) * nm + (xj & 15)];
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (c < nd.nchild) {
        const int* in = inc + 32 * T * c;
        const int aj = in[jj], nbc = nd.cnb[c];
        const float* Uc = pb.U + nd.cu_off[c];
#pragma unroll
        for (int z = 0; z < AU; ++z) {
          const int ai = in[32 * I + r0 + z];
          if (ai >= 0 && aj >= 0) u[c][z] = Uc[max(ai, aj) * nbc + min(ai, aj)];
        }
      }
#pragma unroll
    for (int z = 0; z < AU; ++z)
      t[tsw(r0 + z, lane)] = ((((float)v[z] + u[0][z]) + u[1][z]) + u[2][z]) + u[3][z];
  }
  __syncthreads();

  // R and P of step k: a cluster's in device memory, two of each; one CTA
  // writes its shared memory directly (two R there with nbuf = 2, else the
  // column is copied between two barriers)
  float* Gx = pb.X + nd.x_off;
  auto Rout = [&](int k) { return cl > 1 ? Gx + (size_t)(k & 1) * (32 * ldr + TS) : R0 + (nbuf == 2 ? (size_t)(k & 1) * 32 * ldr : 0); };
  auto Pout = [&](int k) { return cl > 1 ? Gx + (size_t)(k & 1) * (32 * ldr + TS) + 32 * ldr : P0 + (size_t)(k & 1) * TS; };
  const bool early = cl > 1 || nbuf == 2;
  // tile (I, J) of the column (or row) of pivot block k into R (k-major:
  // R[kk][32 I + row]); values in the mm32 layout
  auto send = [&](int I, int J, int k, const float (&v)[4][8]) {
    const int rg = 4 * (lane >> 2), cgp = 4 * (lane & 3);
    float* R = Rout(k);
    if (J == k) {  // I > k: rows of I, columns are pivots
#pragma unroll
      for (int w = 0; w < 8; ++w) {
        const int c = (w < 4 ? cgp : 12 + cgp) + w;
        *reinterpret_cast<float4*>(R + (size_t)c * ldr + 32 * I + rg) =
            make_float4(v[0][w], v[1][w], v[2][w], v[3][w]);
      }
    } else {  // I == k: rows are pivots, columns are block J's rows
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float* d = R + (size_t)(rg + u) * ldr + 32 * J + cgp;
        *reinterpret_cast<float4*>(d) = make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
        *reinterpret_cast<float4*>(d + 16) = make_float4(v[u][4], v[u][5], v[u][6], v[u][7]);
      }
    }
  };
  auto load_tile = [&](const float* t, float (&v)[4][8]) {
    const int rg = 4 * (lane >> 2), cgp = 4 * (lane & 3);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float4 a = *reinterpret_cast<const float4*>(t + tsw(rg + u, cgp));
      const float4 b = *reinterpret_cast<const float4*>(t + tsw(rg + u, 16 + cgp));
      v[u][0] = a.x, v[u][1] = a.y, v[u][2] = a.z, v[u][3] = a.w;
      v[u][4] = b.x, v[u][5] = b.y, v[u][6] = b.z, v[u][7] = b.w;
    }
  };
  auto store_tile = [&](float* t, const float (&v)[4][8]) {
    const int rg = 4 * (lane >> 2), cgp = 4 * (lane & 3);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      *reinterpret_cast<float4*>(t + tsw(rg + u, cgp)) = make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
      *reinterpret_cast<float4*>(t + tsw(rg + u, 16 + cgp)) = make_float4(v[u][4], v[u][5], v[u][6], v[u][7]);
    }
  };
  // the column of block k from the tiles as they stand, by all warps
  auto send_column = [&](int k) {
    for (int q = warp; q < L.ntile; q += FW) {
      const int I = list[q] >> 16, J = list[q] & 0xffff;
      if ((I == k) == (J == k)) continue;  // neither, or the pivot block itself
      float v[4][8];
      load_tile(fsm + (size_t)q * TS, v);
      send(I, J, k, v);
    }
  };
  // Step k: the 32 pivots of block k; step -1 only brings in the first pivot
  // block and column.
#pragma unroll 1
  for (int k = -1; k < KS; ++k) {
    const int kb4 = k < 0 ? 0 : (min(32, nS - 32 * k) + 3) & ~3;
    const float* R = R0 + (nbuf == 2 && cl == 1 ? (size_t)(k & 1) * 32 * ldr : 0);
    const float* P = P0 + (size_t)(k & 1) * TS;
    const bool have_k = k >= 0 && own_of(k) == rank, have_n = k + 1 < KS && own_of(k + 1) == rank;
    if (tid == 0) qhead = 0;
    if (cl > 1 && k >= 0) {
      const float4* g = reinterpret_cast<const float4*>(Rout(k));
      float4* d = reinterpret_cast<float4*>(R0);
#pragma unroll 8
      for (int e = tid; e < kb4 * ldr / 4; e += FT) d[e] = __ldcg(g + e);
      const float4* gp = reinterpret_cast<const float4*>(Pout(k));
      if (tid < TS / 4) reinterpret_cast<float4*>(P0 + (size_t)(k & 1) * TS)[tid] = __ldcg(gp + tid);
      __syncthreads();
    }
    // C_I^T = P R_I^T (k-major); tile (I, k) = C_I, and in block row k tile
    // (k, I) = C_I^T.  Eight columns of a C_I^T per warp, so that every warp has a share.
    const int ntask = k < 0 ? 0 : L.nown + (have_k ? k : 0);
    for (int h = warp; h < 4 * ntask; h += FW) {
      const int t = h >> 2;
      const bool own = t < L.nown;
      const int I = own ? rank + t * cl : t - L.nown;
      const int rg = 4 * (lane >> 2), c = 8 * (h & 3) + 2 * (lane & 3);
      float acc[4][2];
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u][0] = acc[u][1] = 0.f;
      if (I == k) {
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u][0] = -P[(rg + u) * 32 + c], acc[u][1] = -P[(rg + u) * 32 + c + 1];
      } else {
        const float* pr = R + 32 * I + c;
#pragma unroll 4
        for (int kk = 0; kk < kb4; ++kk) {
          const float4 p4 = *reinterpret_cast<const float4*>(P + 32 * kk + rg);
          const float2 r2 = *reinterpret_cast<const float2*>(pr + (size_t)kk * ldr);
          const float pv[4] = {p4.x, p4.y, p4.z, p4.w};
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            acc[u][0] = fmaf(pv[u], r2.x, acc[u][0]);
            acc[u][1] = fmaf(pv[u], r2.y, acc[u][1]);
          }
        }
      }
      if (own && I != k) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          *reinterpret_cast<float2*>(C + (size_t)(rg + u) * ldc + 32 * t + c) = make_float2(acc[u][0], acc[u][1]);
      }
      if (I > k) {
        float* tl = tile(I, k);
#pragma unroll
        for (int w = 0; w < 2; ++w)
          *reinterpret_cast<float4*>(tl + tsw(c + w, rg)) = make_float4(acc[0][w], acc[1][w], acc[2][w], acc[3][w]);
      } else if (!own || I == k) {
        float* tl = tile(k, I);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          *reinterpret_cast<float2*>(tl + tsw(rg + u, c)) = make_float2(acc[u][0], acc[u][1]);
      }
    }
    __syncthreads();
    if (have_n) {
      if (warp < 4) {
        // the next pivot block: its update (lane = row, columns 8 w .. + 7), its
        // sweep, P to every CTA, the dropped modes flagged
        const int kr = min(32, nS - 32 * (k + 1));
        const float* t = tile(k + 1, k + 1);
        const float4 f0 = *reinterpret_cast<const float4*>(t + tsw(lane, 8 * warp));
        const float4 f1 = *reinterpret_cast<const float4*>(t + tsw(lane, 8 * warp + 4));
        float a[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
        const float* pc = C + 32 * ((k + 1) / cl) + lane;
        const float* pr = R + 32 * (k + 1) + 8 * warp;
        float u[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) u[j] = 0.f;
#pragma unroll 8
        for (int kk = 0; kk < kb4; ++kk) {
          const float cv = pc[(size_t)kk * ldc];
          const float4 r0 = *reinterpret_cast<const float4*>(pr + (size_t)kk * ldr);
          const float4 r1 = *reinterpret_cast<const float4*>(pr + (size_t)kk * ldr + 4);
          const float r[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
#pragma unroll
          for (int j = 0; j < 8; ++j) u[j] = fmaf(cv, r[j], u[j]);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) a[j] -= u[j];
        const unsigned dm = sweep32(a, kr, warp, lane, fsm + L.buf_off);
        if (warp == 0 && ((dm >> lane) & 1u)) pb.dropped[gpos[32 * (k + 1) + lane]] = 1;
        // symmetric: by columns, without bank conflicts
        float* Pq = Pout(k + 1) + 256 * warp + lane;
#pragma unroll
        for (int j = 0; j < 8; ++j) Pq[32 * j] = (lane < kr && 8 * warp + j < kr) ? -a[j] : 0.f;
      } else if (warp == FW - 1 && early && k >= 0) {
        // C_{k+1}, the new tile (k + 1, k), belongs to the next pivot row
        float v[4][8];
        load_tile(tile(k + 1, k), v);
        send(k + 1, k, k + 1, v);
      }
      // the other warps of this CTA leave the issue slots and the shared-memory
      // pipe to the sweep: beside tile updates its pivots take twice as long
      if (L.ntile > FW) __syncthreads();
    }
    if (k < 0) {
      send_column(0);
    } else {
      // the other own tiles: F_IJ -= C_I R_J^T
      for (;;) {
        int q = 0;
        if (lane == 0) q = atomicAdd(&qhead, 1);
        q = __shfl_sync(0xffffffffu, q, 0);
        if (q >= L.ntile) break;
        const int I = list[q] >> 16, J = list[q] & 0xffff;
        if (I == k || J == k || (I == k + 1 && J == k + 1 && k + 1 < KS)) continue;
        float acc[4][8], v[4][8];
        mm32(C + 32 * (I / cl), ldc, R + 32 * J, ldr, kb4, lane, acc);
        float* t = fsm + (size_t)q * TS;
        load_tile(t, v);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int w = 0; w < 8; ++w) v[u][w] -= acc[u][w];
        store_tile(t, v);
        if (early && k + 1 < KS && ((I == k + 1) != (J == k + 1))) send(I, J, k + 1, v);
      }
    }
    barrier();
    if (!early && k >= 0 && k + 1 < KS) {
      send_column(k + 1);
      __syncthreads();
    }
  }

  // ---- out: -F_SS and -F_SB for the solves, the Schur complement for the parent ----
  const int s4 = (nS + 3) & ~3;
  const int ldb = s4 + ((nB + 3) & ~3);
  float* mf = pb.M + nd.mf_off;
  float* mb = pb.M + nd.mb_off;
  float* U = pb.U + nd.u_off;
  for (int h = warp; h < 2 * L.ntile; h += FW) {
    const int q = h >> 1, r0 = 16 * (h & 1);
    const int I = list[q] >> 16, J = list[q] & 0xffff;
    const float* t = fsm + (size_t)q * TS;
    const int i0 = 32 * I + r0, j = 32 * J + lane;   // 16 rows, lane = column
    const int il = 32 * I + lane, j0 = 32 * J + r0;  // 16 columns, lane = row
    if (J < KS && I < KS) {
      // -F_SS: lower entries by rows, their mirror images by columns
      float* d = mb + (size_t)i0 * ldb + j;
      float* e = mb + (size_t)j0 * ldb + il;
#pragma unroll 4
      for (int r = 0; r < 16; ++r) {
        if (i0 + r < nS && j <= i0 + r) d[r * ldb] = -t[tsw(r0 + r, lane)];
        if (il < nS && j0 + r < il) e[r * ldb] = -t[tsw(lane, r0 + r)];
      }
    } else if (J < KS) {
      float* d = mf + (size_t)(i0 - nSp) * s4 + j;
      float* e = mb + (size_t)j0 * ldb + s4 + il - nSp;
#pragma unroll 4
      for (int r = 0; r < 16; ++r) {
        if (i0 + r - nSp < nB && j < nS) d[r * s4] = -t[tsw(r0 + r, lane)];
        if (il - nSp < nB && j0 + r < nS) e[r * ldb] = -t[tsw(lane, r0 + r)];
      }
    } else {
      float* d = U + (size_t)(i0 - nSp) * nB + j - nSp;
#pragma unroll 4
      for (int r = 0; r < 16; ++r)
        if (i0 + r - nSp < nB && j <= i0 + r) d[r * nB] = t[tsw(r0 + r, lane)];
    }
  }
}

// ---------------------------------------------------------------- solve
// max over the cluster of a value per thread; every thread gets it
__device__ inline double cluster_max(cg::cluster_group& cluster, double v, double* wred, double* cred) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, m));
  if (lane == 0) wred[warp] = v;
  __syncthreads();
  if (warp == 0) {
    double w = lane < ST / 32 ? wred[lane] : 0.0;
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) w = fmax(w, __shfl_xor_sync(0xffffffffu, w, m));
    if (lane < (int)cluster.num_blocks()) *cluster.map_shared_rank(cred + cluster.block_rank(), lane) = w;
  }
  cluster.sync();
  double r = 0.0;
  for (int q = 0; q < (int)cluster.num_blocks(); ++q) r = fmax(r, cred[q]);
  return r;
}

// All solves of one update: x = 0; for q = 0 .. nsolve - 1: x += A_T^-1 res,
// res = b - A x in FP64, until max |res| <= 1e-14 max |b| (the test of the band
// path; cstat[3] counts the updates whose last allowed solve still ran).
//
// A phase waits for nothing but the vector values the phase before wrote: its
// lists and the first PM words of each group's matrix row are loaded ahead of
// the barrier (every one of these loads is a trip to L2 of about 0.4 us).
constexpr int PM = 4;
constexpr int TREE_MAXPH = 64;
template <int Q>
__global__ void __launch_bounds__(ST, 1) k_tree_solve(const TreeProb* __restrict__ probs,
                                                      const int* __restrict__ which, int use_ctl) {
  extern __shared__ __align__(16) float ssm[];
  __shared__ double wred[ST / 32];
  __shared__ double cred[2][16];
  __shared__ int4 span[TREE_MAXPH];
  cg::cluster_group cluster = cg::this_cluster();
  const int cl = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const TreeProb pb = probs[which[blockIdx.x / cl]];
  const int tid = threadIdx.x;
  const int n = pb.n, Mx = pb.Mx, My = pb.My;
  constexpr int Rw = 9 * Q;
  float* V = pb.V;
  double* x = pb.x;
  const int gl = tid & 7;  // lane of a row group
  const int grp = tid >> 3;
  constexpr int ngrp = ST / 8;
  cluster_arrive();
  const int nphase = pb.nphase;
  const int4 *gath = pb.gath, *rows = pb.rows, *phase = pb.phase;
  const float4* M4 = reinterpret_cast<const float4*>(pb.M);
  // this CTA's share of the unknowns
  const int ub = (int)((long long)n * rank / cl), ue = (int)((long long)n * (rank + 1) / cl);
  for (int ph = tid; ph < nphase; ph += ST) span[ph] = phase[ph * cl + rank];
  dep_wait();
  cluster_wait();  // the other CTAs run: their cred may be written
  if (use_ctl && tree_done(pb.ctl)) return;
  double bm = 0.0;
  for (int i = ub + tid; i < ue; i += ST) {
    const double v = pb.dropped[i] ? 0.0 : pb.b[i];
    bm = fmax(bm, fabs(v));
    V[pb.v_rhs + i] = (float)v;
  }
  // the lists of a phase and the head of this group's first row
  // (re: row start, vector start, length, place; ro: the children's entries;
  // n: the ones being fetched)
  int4 ge, gf, re, ro, gen, gfn, ren, ron;
  float4 mh[PM];
  __syncthreads();
  auto load_row = [&](int r, int end) {
    ren = make_int4(0, 0, 0, 0), ron = make_int4(0, 0, 0, 0);
    if (r < end) {
      ren = rows[2 * r];
      ron = rows[2 * r + 1];
    }
  };
  auto load_lists = [&](int ph) {
    const int4 p = span[ph];
    gen = gfn = make_int4(0, 0, 0, 0);
    if (p.x + tid < p.y) {
      gen = gath[2 * (p.x + tid)];
      gfn = gath[2 * (p.x + tid) + 1];
    }
    load_row(p.z + grp, p.w);
  };
  auto load_head = [&]() {
    re = ren, ro = ron;
#pragma unroll
    for (int t = 0; t < PM; ++t)
      mh[t] = gl + 8 * t < re.z ? M4[re.x + gl + 8 * t] : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  auto val = [&](int k) { return __ldcg(V + k); };
  load_lists(0);
  load_head();
  ge = gen, gf = gfn;
  bm = cluster_max(cluster, bm, wred, cred[0]);
  for (int q = 0; q < pb.nsolve; ++q) {
    if (q > 0) {
      // FP64 residual: eight lanes per row over its nine neighbour sets
      double rm = 0.0;
      for (int i0 = ub; i0 < ue; i0 += ngrp) {
        const int i = i0 + grp;
        const int ic = i < ue ? i : ue - 1;
        const int I = ic / Q, Ix = I % Mx, Iy = I / Mx;
        const double* ar = pb.arow + (size_t)ic * Rw;
        constexpr int NC = (Rw + 7) / 8;
        double av[NC], xv[NC];
#pragma unroll
        for (int t = 0; t < NC; ++t) {
          const int c = gl + 8 * t, nb = c / Q, m = c - nb * Q;
          const int dx = nb % 3 - 1, dy = nb / 3 - 1;
          const bool in = c < Rw && Ix + dx >= 0 && Ix + dx < Mx && Iy + dy >= 0 && Iy + dy < My;
          av[t] = ar[in ? c : 0];
          xv[t] = __ldcg(x + (in ? Q * (I + dy * Mx + dx) + m : ic));
          if (!in) av[t] = 0.0;
        }
        const bool live = i < ue && !pb.dropped[ic];
        const double bv = pb.b[ic];
        double a0 = 0.0, a1 = 0.0;
#pragma unroll
        for (int t = 0; t < NC; t += 2) {
          a0 = fma(av[t], xv[t], a0);
          if (t + 1 < NC) a1 = fma(av[t + 1], xv[t + 1], a1);
        }
        double acc = a0 + a1;
#pragma unroll
        for (int s = 4; s > 0; s >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
        if (i < ue && gl == 0) {
          const double r = live ? bv - acc : 0.0;
          rm = fmax(rm, fabs(r));
          V[pb.v_rhs + i] = (float)r;
        }
      }
      rm = cluster_max(cluster, rm, wred, cred[q & 1]);
      if (!(rm > 1e-14 * bm)) break;
      if (q == pb.nsolve - 1 && rank == 0 && tid == 0) atomicAdd(&pb.cstat[3], 1ull);
    }
    for (int ph = 0; ph < nphase; ++ph) {
      // gather entries [ps.x, ps.y), rows [ps.z, ps.w)
      const int4 ps = span[ph];
      const bool more = ps.x + tid < ps.y;
      const float g0 = val(ge.x), g1 = val(ge.y), g2 = val(ge.z), g3 = val(ge.w), g4 = val(gf.x);
      float iv = ((val(ro.x) + val(ro.y)) + val(ro.z)) + val(ro.w);  // (0 for a solution row)
      double xo = re.w < 0 ? __ldcg(x + ~re.w) : 0.0;
      if (more) ssm[tid] = (((g0 + g1) + g2) + g3) + g4;
      // the lists of the next phase and of this group's next row come in beside
      // this phase's work, the head of the next phase's matrix row at its end
      const bool rest = ps.z + ngrp < ps.w;  // more rows than groups in this phase
      if (rest) load_row(ps.z + grp + ngrp, ps.w);
      else load_lists(ph + 1 < nphase ? ph + 1 : 0);
      for (int k = ps.x + ST + tid; k < ps.y; k += ST) {
        const int4 g = gath[2 * k];
        const int g4i = gath[2 * k + 1].x;
        ssm[k - ps.x] = (((val(g.x) + val(g.y)) + val(g.z)) + val(g.w)) + val(g4i);
      }
      __syncthreads();
      for (int r = ps.z + grp; r - grp < ps.w; r += ngrp) {
        const int4 e = re;
        const bool in = r < ps.w;
        const float4* m4 = M4 + e.x;
        const float4* f4 = reinterpret_cast<const float4*>(ssm) + e.y;
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
        auto add = [&](const float4& m, const float4& f) {
          a0 = fmaf(m.x, f.x, a0);
          a1 = fmaf(m.y, f.y, a1);
          a2 = fmaf(m.z, f.z, a2);
          a3 = fmaf(m.w, f.w, a3);
        };
#pragma unroll
        for (int t = 0; t < PM; ++t)
          if (gl + 8 * t < e.z) add(mh[t], f4[gl + 8 * t]);
#pragma unroll 4
        for (int t = gl + 8 * PM; t < e.z; t += 8) add(m4[t], f4[t]);
        const float ivc = iv;
        const double xoc = xo;
        // the group's next row of this phase
        if (r - grp + ngrp < ps.w) {
          load_head();
          iv = ((val(ro.x) + val(ro.y)) + val(ro.z)) + val(ro.w);
          if (re.w < 0) xo = __ldcg(x + ~re.w);
          if (r - grp + 2 * ngrp < ps.w) load_row(r + 2 * ngrp, ps.w);
          else load_lists(ph + 1 < nphase ? ph + 1 : 0);
        }
        float s = (a0 + a1) + (a2 + a3);
#pragma unroll
        for (int m = 4; m > 0; m >>= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
        if (in && gl == 0) {
          if (e.w < 0) {
            // a solution row (dropped modes: their rows of the swept front are zero)
            V[pb.v_x + ~e.w] = s;
            x[~e.w] = xoc + (double)s;
          } else {
            V[e.w] = ivc + s;
          }
        }
      }
      load_head();
      ge = gen, gf = gfn;
      cluster.sync();
    }
  }
  for (int i = ub + tid; i < ue; i += ST) pb.a[i] = pb.scale[i] * __ldcg(x + i);
}

}  // namespace

// ---------------------------------------------------------------- host plan
namespace {
struct HNode {
  std::vector<int> S, B;
  int child[4] = {-1, -1, -1, -1};
  int nchild = 0, height = 0;
};
// The box [x0, x0 + w) x [y0, y0 + h) of sets and its parts.  Boxes of at most
// leaf x leaf sets are not cut.  Cutting a box by its middle column and row at
// once halves the levels (each a launch of the factor and two phases of every
// solve) against cutting by the two in turn, for the same chain of pivots: the
// two arms of the second cut are eliminated one after the other instead of
// side by side, but a level's fixed cost is that of 60 pivots and more.  Only
// where the larger front still fits (tcap block rows of 32 unknowns, nm per set).
int build(std::vector<HNode>& out, int Mx, int My, int x0, int y0, int w, int h, int leaf, int nm, int tcap) {
  HNode nd;
  int kids[4], nk = 0;
  const bool whole = w <= leaf && h <= leaf;
  // cut at column c and / or row r (-1: not)
  int c = -1, r = -1;
  if (!whole) {
    const int ring = (std::min(x0 + w + 1, Mx) - std::max(x0 - 1, 0)) * (std::min(y0 + h + 1, My) - std::max(y0 - 1, 0)) -
                     w * h;
    const bool both = w > leaf && h > leaf && w <= 2 * h && h <= 2 * w &&
                      (nm * (w + h - 1) + 31) / 32 + (nm * ring + 31) / 32 <= tcap;
    if (both || w >= h) c = x0 + w / 2;
    if (both || w < h) r = y0 + h / 2;
  }
  for (int y = y0; y < y0 + h; ++y)
    for (int x = x0; x < x0 + w; ++x)
      if (whole || x == c || y == r) nd.S.push_back(y * Mx + x);
  if (!whole) {
    const int xs[3] = {x0, c >= 0 ? c + 1 : x0 + w, x0 + w}, xe[2] = {c >= 0 ? c : x0 + w, x0 + w};
    const int ys[3] = {y0, r >= 0 ? r + 1 : y0 + h, y0 + h}, ye[2] = {r >= 0 ? r : y0 + h, y0 + h};
    for (int b = 0; b < 2; ++b)
      for (int a = 0; a < 2; ++a)
        if (xe[a] > xs[a] && ye[b] > ys[b])
          kids[nk++] = build(out, Mx, My, xs[a], ys[b], xe[a] - xs[a], ye[b] - ys[b], leaf, nm, tcap);
  }
  for (int y = y0 - 1; y <= y0 + h; ++y)
    for (int x = x0 - 1; x <= x0 + w; ++x) {
      if (x < 0 || y < 0 || x >= Mx || y >= My) continue;
      if (x >= x0 && x < x0 + w && y >= y0 && y < y0 + h) continue;
      nd.B.push_back(y * Mx + x);
    }
  nd.nchild = nk;
  for (int k = 0; k < nk; ++k) {
    nd.child[k] = kids[k];
    nd.height = std::max(nd.height, out[kids[k]].height + 1);
  }
  out.push_back(nd);
  return (int)out.size() - 1;
}
int pad4i(int n) { return (n + 3) & ~3; }
}  // namespace

namespace {
// Leaves of at most 4 x 4 sets, and one dense front for a grid of at most 256
// unknowns: the sum of a factor and five solves on 16 x 16 sets of nine modes
// took 273 us with leaves of 4 x 4, 312 with 3 x 3, 289 with 2 x 2 and 345 with 1 x 1
// (35 x 29 sets: 637, 652, 710, 725).
constexpr int TREE_LEAF = 4, TREE_ROOT = 256;
constexpr int TREE_FREE = 4;    // SMs left over when a level is spread over CTAs
constexpr int TREE_SROWS = 16;  // unknowns of a CTA of a solve, at least
constexpr int TREE_PORTABLE = 8;  // a cluster size that every part can place
}  // namespace

// bytes of shared memory of the largest CTA of a front of T block rows
static size_t front_need(int T, int cl, int nbuf) {
  size_t m = 0;
  for (int r = 0; r < cl; ++r) m = std::max(m, front_smem(T, cl, r, nbuf).total * sizeof(float));
  return m;
}
// Cluster size and shared memory of a launch of n fronts of at most T block rows:
// the smallest cluster that holds the largest front, then more CTAs per front
// while the launch leaves SMs idle and each CTA keeps a block row; two buffers
// of the pivot column where a single CTA has room for them.
TreeLaunch tree_level_launch(int n, int T, int max_smem, int nsm) {
  const size_t cap = (size_t)max_smem - 2048;
  auto need = [&](int cl, int nbuf) {
    size_t m = 0;
    for (int t = 1; t <= T; ++t) m = std::max(m, front_need(t, cl, nbuf));
    return m;
  };
  TreeLaunch L;
  L.cl = 1;
  while (L.cl < 8 && need(L.cl, 1) > cap) ++L.cl;
  while (L.cl < 8 && (long long)n * (L.cl + 1) <= nsm - TREE_FREE && L.cl + 1 <= T) ++L.cl;
  L.nbuf = L.cl == 1 && need(1, 2) <= cap ? 2 : 1;
  L.smem = need(L.cl, L.nbuf);
  return L;
}

// Whether the device can place a cluster of scl CTAs of the solves: above the
// portable size that depends on the part (its SMs per processing cluster).
static bool tree_solve_fits(int q, int scl, size_t smem) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)scl);
  cfg.blockDim = dim3(ST);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)scl;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int n = 0;
  const cudaError_t e = q == NMODES_RF ? cudaOccupancyMaxActiveClusters(&n, k_tree_solve<NMODES_RF>, &cfg)
                                       : cudaOccupancyMaxActiveClusters(&n, k_tree_solve<NMODES>, &cfg);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return n >= 1;
}

bool tree_plan_build(const LatView& lv, int max_smem, int max_cl, TreePlanHost* P) {
  *P = TreePlanHost();
  if (max_cl < 1) return false;
  const int nm = lv.q, n = nm * lv.M;
  if (n > (1 << 20) || std::max(lv.Mx, lv.My) > 8000) return false;
  const size_t cap = (size_t)max_smem - 2048;
  int tcap = 1;
  while (tcap < 64 && front_need(tcap + 1, 8, 1) <= cap) ++tcap;
  std::vector<HNode> hn;
  build(hn, lv.Mx, lv.My, 0, 0, lv.Mx, lv.My, n <= TREE_ROOT ? std::max(lv.Mx, lv.My) : TREE_LEAF, nm, tcap);
  const int nn = (int)hn.size();
  int H = 0;
  for (const HNode& h : hn) H = std::max(H, h.height);
  P->n = n;
  P->nm = nm;
  P->nlev = H + 1;
  P->nodes.assign(nn, TreeNode{});
  auto blocks = [&](const HNode& h) {
    return (nm * (int)h.S.size() + 31) / 32 + (nm * (int)h.B.size() + 31) / 32;
  };
  for (const HNode& h : hn)
    if (blocks(h) > tcap) return false;
  long long mo = 0, uo = 0, wo = 0, xo = 0;
  std::vector<int> w_off(nn), where(lv.M, -1);
  for (int k = 0; k < nn; ++k) {
    TreeNode& d = P->nodes[k];
    const HNode& h = hn[k];
    d.ns = (int)h.S.size();
    d.nb = (int)h.B.size();
    d.s_off = (int)P->sets.size();
    P->sets.insert(P->sets.end(), h.S.begin(), h.S.end());
    P->sets.insert(P->sets.end(), h.B.begin(), h.B.end());
    const int nS = nm * d.ns, nB = nm * d.nb, s4 = pad4i(nS), b4 = pad4i(nB);
    d.mf_off = mo;
    mo += (long long)nB * s4;
    d.mb_off = mo;
    mo += (long long)nS * (s4 + b4);
    d.u_off = uo;
    uo += (long long)nB * nB;
    d.x_off = xo;
    xo += 2LL * (32 * 32 * blocks(h) + TS);
    w_off[k] = (int)wo;
    wo += nB;
    d.nchild = h.nchild;
    for (int c = 0; c < h.nchild; ++c) {
      const int ch = h.child[c];
      d.cu_off[c] = P->nodes[ch].u_off;
      d.cnb[c] = nm * P->nodes[ch].nb;
      d.inv_off[c] = (int)P->inv.size();
      // place of each set of this front in the child's boundary list
      for (size_t q = 0; q < hn[ch].B.size(); ++q) where[hn[ch].B[q]] = (int)q;
      for (int J : h.S) P->inv.push_back(where[J]);
      for (int J : h.B) P->inv.push_back(where[J]);
      for (int J : hn[ch].B) where[J] = -1;
    }
  }
  if (mo / 4 > 0x7fffffffLL || wo > 0x3fffffffLL) return false;
  P->m_elems = (size_t)std::max(mo, 4LL);
  P->u_elems = (size_t)std::max(uo, 4LL);
  P->x_elems = (size_t)xo;
  P->v_rhs = 4;  // V[0..3] = 0
  const int v_w = P->v_rhs + n;
  P->v_x = v_w + (int)wo;
  P->v_elems = (size_t)P->v_x + n;
  // ---- factor launches: per level the nodes and the cluster size ----
  std::vector<std::vector<int>> byh(H + 1);
  for (int k = 0; k < nn; ++k) byh[hn[k].height].push_back(k);
  P->level_begin.assign(H + 2, 0);
  P->level_cl.assign(H + 1, 1);
  P->level_nbuf.assign(H + 1, 2);
  P->level_T.assign(H + 1, 1);
  P->level_smem.assign(H + 1, 0);
  for (int h = 0; h <= H; ++h) {
    P->level_begin[h] = (int)P->items.size();
    int Tmax = 1;
    for (int k : byh[h]) {
      P->items.push_back(TreeItem{0, k});
      Tmax = std::max(Tmax, blocks(hn[k]));
    }
    const TreeLaunch tl = tree_level_launch((int)byh[h].size(), Tmax, max_smem, lv.nsm);
    P->level_cl[h] = tl.cl;
    P->level_nbuf[h] = tl.nbuf;
    P->level_T[h] = Tmax;
    P->level_smem[h] = tl.smem;
  }
  P->level_begin[H + 1] = (int)P->items.size();
  // ---- solve schedule ----
  int scl = max_cl;
  while (scl > 1 && n < TREE_SROWS * scl) scl /= 2;
  P->scl = scl;
  P->nphase = 0;
  int smax = 4;
  for (int dir = 0; dir < 2; ++dir)
    for (int q = 0; q <= H; ++q) {
      const int h = dir == 0 ? q : H - q;
      auto rows_of = [&](int k) { return dir == 0 ? nm * P->nodes[k].nb : nm * P->nodes[k].ns; };
      auto len_of = [&](int k) {
        const int s4 = pad4i(nm * P->nodes[k].ns) / 4;
        return dir == 0 ? s4 : s4 + pad4i(nm * P->nodes[k].nb) / 4;
      };
      // cost: a row's 16-byte words in units of eight lanes, plus a row's fixed part
      auto cost_of = [&](int k) { return 2.0 + (len_of(k) + 7) / 8; };
      double total = 0.0;
      for (int k : byh[h]) total += cost_of(k) * rows_of(k);
      if (total == 0.0) continue;
      std::vector<TreeSpan> ph(scl);
      size_t node = 0;
      int row = 0;
      double done = 0.0;
      for (int c = 0; c < scl; ++c) {
        TreeSpan& sp = ph[c];
        sp.g0 = (int)P->gath.size() / 8;
        sp.r0 = (int)P->rows.size() / 8;
        const double upto = total * (c + 1) / scl;
        while (node < byh[h].size() && (c + 1 == scl || done < upto - 1e-9)) {
          const int k = byh[h][node];
          const int R = rows_of(k);
          if (row >= R) {
            ++node;
            row = 0;
            continue;
          }
          int take = R - row;
          if (c + 1 < scl) take = std::min(take, std::max(1, (int)std::ceil((upto - done) / cost_of(k))));
          const TreeNode& d = P->nodes[k];
          const HNode& hk = hn[k];
          const int nS = nm * d.ns, nB = nm * d.nb, s4 = pad4i(nS), b4 = pad4i(nB);
          // a front position's children's W entries (0: none)
          auto wsrc = [&](int s, int m, int child) {
            if (child >= d.nchild) return 0;
            const int t = P->inv[d.inv_off[child] + s];
            return t < 0 ? 0 : v_w + w_off[hk.child[child]] + nm * t + m;
          };
          const int f0 = (int)P->gath.size() / 8 - sp.g0;  // this front's vector in shared memory
          for (int p = 0; p < s4; ++p) {
            const bool ok = p < nS;
            const int s = ok ? p / nm : 0, m = p % nm;
            int v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
            if (ok) {
              v[0] = P->v_rhs + nm * hk.S[s] + m;
              for (int c4 = 0; c4 < 4; ++c4) v[1 + c4] = wsrc(s, m, c4);
            }
            P->gath.insert(P->gath.end(), v, v + 8);
          }
          if (dir == 1)
            for (int p = 0; p < b4; ++p) {
              const int v[8] = {p < nB ? P->v_x + nm * hk.B[p / nm] + p % nm : 0, 0, 0, 0, 0, 0, 0, 0};
              P->gath.insert(P->gath.end(), v, v + 8);
            }
          for (int r = row; r < row + take; ++r) {
            const long long off = dir == 0 ? d.mf_off + (long long)r * s4 : d.mb_off + (long long)r * (s4 + b4);
            int v[8] = {(int)(off / 4), f0 / 4, len_of(k),
                        dir == 0 ? v_w + w_off[k] + r : ~(nm * hk.S[r / nm] + r % nm), 0, 0, 0, 0};
            if (dir == 0)
              for (int c4 = 0; c4 < 4; ++c4) v[4 + c4] = wsrc(d.ns + r / nm, r % nm, c4);
            P->rows.insert(P->rows.end(), v, v + 8);
          }
          done += cost_of(k) * take;
          row += take;
        }
        sp.g1 = (int)P->gath.size() / 8;
        sp.r1 = (int)P->rows.size() / 8;
        smax = std::max(smax, sp.g1 - sp.g0);
      }
      for (const TreeSpan& sp : ph) P->phase.push_back(sp);
      ++P->nphase;
    }
  P->solve_smem = (size_t)smax * sizeof(float);
  if (P->nphase > TREE_MAXPH || P->solve_smem + 4096 > (size_t)max_smem) return false;
  if (scl <= TREE_PORTABLE || tree_solve_fits(nm, scl, P->solve_smem)) return true;
  return tree_plan_build(lv, max_smem, scl / 2, P);
}

size_t tree_arow_elems(const LatView& lv) { return (size_t)lv.q * lv.M * 9 * lv.q; }

cudaError_t launch_tree_system(cudaStream_t s, int q, bool slots, const TreeProb* probs, const TreeItem* sets, int n,
                               bool use_ctl, int nsm) {
  if (n <= 0) return cudaSuccess;
  const int c = (int)use_ctl;
  const auto diag = q == NMODES_RF ? (slots ? k_tree_diag<NMODES_RF, true> : k_tree_diag<NMODES_RF, false>)
                                   : (slots ? k_tree_diag<NMODES, true> : k_tree_diag<NMODES, false>);
  const int dt = n > 2 * nsm ? 128 : (q == NMODES_RF ? DIAG_T<NMODES_RF> : DIAG_T<NMODES>);
  const cudaError_t e = launch_dep(diag, s, n, dt, 0, 0, probs, sets, c);
  if (e != cudaSuccess) return e;
  return launch_dep(k_tree_rows, s, n, 256, 0, 0, probs, sets, c);
}

cudaError_t launch_tree_level(cudaStream_t s, const TreeLaunch& L, const TreeProb* probs, const TreeItem* nodes, int n,
                              bool use_ctl) {
  if (n <= 0) return cudaSuccess;
  return launch_dep(k_tree_factor, s, n * L.cl, FT, L.smem, L.cl, probs, nodes, L.nbuf, (int)use_ctl);
}

cudaError_t launch_tree_factor(cudaStream_t s, const TreePlanHost& P, const TreeProb* prob, const TreeItem* items,
                               bool use_ctl) {
  for (int h = 0; h < P.nlev; ++h) {
    const TreeLaunch L{P.level_cl[h], P.level_nbuf[h], P.level_smem[h]};
    const cudaError_t e =
        launch_tree_level(s, L, prob, items + P.level_begin[h], P.level_begin[h + 1] - P.level_begin[h], use_ctl);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_tree_solve(cudaStream_t s, int q, int scl, size_t smem, const TreeProb* probs, const int* which,
                              int n, bool use_ctl) {
  if (n <= 0) return cudaSuccess;
  return launch_dep(q == NMODES_RF ? k_tree_solve<NMODES_RF> : k_tree_solve<NMODES>, s, n * scl, ST, smem, scl, probs, which,
                    (int)use_ctl);
}

cudaError_t configure_coarse_tree(int max_smem) {
  cudaError_t e = set_max_dynamic_smem(k_tree_factor, max_smem);
  if (e != cudaSuccess) return e;
  if ((e = set_max_dynamic_smem(k_tree_solve<NMODES>, max_smem)) != cudaSuccess) return e;
  if ((e = set_max_dynamic_smem(k_tree_solve<NMODES_RF>, max_smem)) != cudaSuccess) return e;
  e = cudaFuncSetAttribute((const void*)k_tree_solve<NMODES>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute((const void*)k_tree_solve<NMODES_RF>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

}  // namespace hms

// Entries of K_aa from the slots of coarse_assemble.cu, shared by the blocks of
// coarse_blocks.cu and the scaled system of coarse_tree.cu.
#pragma once
#include "hms_internal.cuh"

namespace hms {

__device__ inline double slot_val(const double* base, const double* it, int nm, int I, int slot, int p, int c) {
  const size_t o = ((size_t)I * NSLOTS + slot) * slot_size(nm) + (size_t)p * slot_dim(nm) + c;
  return base[o] + it[o];
}

// entry (J mode l, I mode m) of K_aa, J the neighbour b of I (b = 0: J = I);
// 0 if J lies outside the set grid
__device__ inline double blk_entry(const LatView& lv, const double* base, const double* it, int I, int b, int l,
                                   int m) {
  const int nm = lv.q;
  const int Ix = I % lv.Mx, Iy = I / lv.Mx;
  if (b == BLK_SELF) {
    double v = slot_val(base, it, nm, I, SLOT_SELF, l, m);
    for (int s = SLOT_E; s < NSLOTS; ++s) v += slot_val(base, it, nm, I, s, l, m);
    // neighbours that own bars into I
    const int kx[5] = {-1, 1, 0, -1, 1};  // owner offset for E, W, N, NE, NW
    const int ky[5] = {0, 0, -1, -1, -1};
    for (int s = 0; s < 5; ++s) {
      const int Kx = Ix + kx[s], Ky = Iy + ky[s];
      if (Kx < 0 || Kx >= lv.Mx || Ky < 0 || Ky >= lv.My) continue;
      v += slot_val(base, it, nm, Ky * lv.Mx + Kx, SLOT_E + s, nm + l, nm + m);
    }
    return v;
  }
  const int dx = blk_dx(b), dy = blk_dy(b);
  const int Jx = Ix + dx, Jy = Iy + dy;
  if (Jx < 0 || Jx >= lv.Mx || Jy >= lv.My) return 0.0;
  const int J = Jy * lv.Mx + Jx;
  if (b == BLK_E) return slot_val(base, it, nm, I, SLOT_E, nm + l, m) + slot_val(base, it, nm, J, SLOT_W, l, nm + m);
  if (b == BLK_N) return slot_val(base, it, nm, I, SLOT_N, nm + l, m);
  if (b == BLK_NE) return slot_val(base, it, nm, I, SLOT_NE, nm + l, m);
  return slot_val(base, it, nm, I, SLOT_NW, nm + l, m);
}

// The modes of a set left out by the FP64 elimination of its scaled diagonal block in
// mode order, by one warp: lane = row, A[l] = entry (row, l), dr = left out
// beforehand.  A pivot <= 1e-14 leaves its mode out.  L D L^T with 1 / piv by two
// Newton steps from FP32: an FP64 operation of one warp takes 64 clocks, a square
// root or a division a dozen of them.
template <int Q>
__device__ __forceinline__ bool drop_pivots(double (&A)[Q], bool dr, int lane) {
  constexpr unsigned FULL = 0xffffffffu;
  const unsigned dr0 = __ballot_sync(FULL, dr);
#pragma unroll
  for (int m = 0; m < Q; ++m) {
    const double piv = __shfl_sync(FULL, A[m], m);
    const bool out = (dr0 >> m) & 1u;  // its row and column count as zero
    const bool low = !out && !(piv > 1e-14);
    if (low && lane == m) dr = true;
    // FP32, then 24 -> 48 -> 53 bits (piv <= 1 but for rounding, > 1e-14)
    double ri = (double)__frcp_rn((float)piv);
    ri = fma(ri, fma(-piv, ri, 1.0), ri);
    ri = fma(ri, fma(-piv, ri, 1.0), ri);
    const double t = out || low ? 0.0 : A[m] * ri;
#pragma unroll
    for (int l = m + 1; l < Q; ++l) {
      const double al = __shfl_sync(FULL, A[m], l);
      A[l] = out || low ? A[l] : fma(-t, al, A[l]);
    }
  }
  return dr;
}

}  // namespace hms

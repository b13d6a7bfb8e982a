// Per-thread and per-tile bodies of the colour passes of the Vanka smoother
// (the setup of the local inverses is in vnode.cuh).
//
// Tiled colour pass: a block owns kTCX x kTCY cells of the colour, i.e. the
// (2 kTCX) x (2 kTCY) nodes they cover.  It stages the masked iterate, vbar
// and the flags of those nodes plus a two-node halo in shared memory,
// computes the 12 rows of every cell touching the tile and the 9 LPS rows of
// every patch touching it once, sums them per node, exchanges each cell's 12
// defects among the cell's four threads by warp shuffles and applies the
// 12x12 inverse.  Cells of one colour share no node; nodes outside the
// colour's fluid cells are copied, so x_out is complete and the next colour
// reads it without races.
#pragma once
#include "kernels.h"

namespace dnnmg {

// 16-byte vectors of T
template <typename T>
struct Vec16;
template <>
struct Vec16<float> {
  using type = float4;
};
template <>
struct Vec16<double> {
  using type = double2;
};
__device__ __forceinline__ void vec_unpack(const float4& v, float* o) {
  o[0] = v.x, o[1] = v.y, o[2] = v.z, o[3] = v.w;
}
__device__ __forceinline__ void vec_unpack(const double2& v, double* o) { o[0] = v.x, o[1] = v.y; }
__device__ __forceinline__ float4 vec_pack(const float* o) {
  return make_float4(o[0], o[1], o[2], o[3]);
}
__device__ __forceinline__ double2 vec_pack(const double* o) { return make_double2(o[0], o[1]); }

// 36 entries stored as 16-byte vectors `stride` vectors apart, read only
// during the kernel
template <typename T>
__device__ __forceinline__ void load36(const T* base, size_t first, size_t stride, T out[36]) {
  using V = typename Vec16<T>::type;
  const V* p = reinterpret_cast<const V*>(base) + first;
#pragma unroll
  for (int v = 0; v < 36 / kVec16<T>; ++v) vec_unpack(__ldg(p + v * stride), out + v * kVec16<T>);
}
// the rows c * 4 + a of the inverse of the cell of `slot` (see vanka_inv_index)
template <typename T>
__device__ __forceinline__ void load_inv_rows(const T* inv, int nslots, int colour, int slot, int a,
                                              T iv[36]) {
  load36<T>(inv, ((size_t)colour * (36 / kVec16<T>) * nslots + slot) * 4 + a, (size_t)nslots * 4,
            iv);
}

// Resident blocks per SM the pass kernels ask the compiler for: FP32 passes
// are held to 128 registers per thread so that 512 threads per SM fit.
template <typename T>
constexpr int pass_min_blocks(int threads) {
  return sizeof(T) == 4 ? (512 / threads > 0 ? 512 / threads : 1) : 1;
}

template <typename T, int kTCX, int kTCY>
struct PassSmem {
  T w[3][2 * kTCY + 4][2 * kTCX + 4];
  T vb[2][2 * kTCY + 4][2 * kTCX + 4];
  uint8_t fl[2 * kTCY + 4][2 * kTCX + 4];
  uint8_t sol[2 * kTCY + 4][2 * kTCX + 4];  // solid flag of the cell whose lower-left node this is
  T cres[(2 * kTCY + 1) * (2 * kTCX + 1)][12];
  T pres[(kTCY + 2) * (kTCX + 2)][9];
  int8_t cvalid[(2 * kTCY + 1) * (2 * kTCX + 1)];
  int8_t pvalid[(kTCY + 2) * (kTCX + 2)];
};

// Stage the tile whose first node is (i0, j0) -- nodes [i0-2, i0-2+kSX) x
// [j0-2, j0-2+kSY) with the masked iterate, vbar, flags and the solid flag
// of the cell whose lower-left node each one is -- then compute the 12 rows
// of every cell touching the tile and the 9 LPS rows of every patch touching
// it, once each.  Thread t of NTT; ends with the rows visible to all
// threads of the group (two block barriers).
template <typename T, int kTCX, int kTCY, int NTT>
__device__ __forceinline__ void pass_stage_rows(const Grid& g, const Sten<T>& s,
                                                const T* __restrict__ xin,
                                                const T* __restrict__ vb, int i0, int j0, int t,
                                                PassSmem<T, kTCX, kTCY>& S) {
  constexpr int kSX = 2 * kTCX + 4;
  constexpr int kCX = 2 * kTCX + 1, kCY = 2 * kTCY + 1;
  constexpr int kPX = kTCX + 2, kPY = kTCY + 2;
  constexpr int kSY = 2 * kTCY + 4;
  const int nn = g.nn;
  for (int e = t; e < kSX * kSY; e += NTT) {
    const int li = e % kSX, lj = e / kSX;
    const int i = i0 - 2 + li, j = j0 - 2 + lj;
    T xu1 = 0, xv1 = 0, xp1 = 0, bu = 0, bvv = 0;
    uint8_t f = 0xFF, so = 1;
    if (i >= 0 && j >= 0 && i <= g.nx && j <= g.ny) {
      const int n = j * g.nnx + i;
      f = g.flags[n];
      xu1 = xin[n];
      xv1 = xin[nn + n];
      xp1 = xin[2 * nn + n];
      bu = vb[n];
      bvv = vb[nn + n];
      if (i < g.nx && j < g.ny) so = g.solid[j * g.nx + i];
    }
    S.w[0][lj][li] = (f & kVDir) ? T(0) : xu1;
    S.w[1][lj][li] = (f & kVDir) ? T(0) : xv1;
    S.w[2][lj][li] = (f & kPFix) ? T(0) : xp1;
    S.vb[0][lj][li] = bu;
    S.vb[1][lj][li] = bvv;
    S.fl[lj][li] = f;
    S.sol[lj][li] = so;
  }
  __syncthreads();
  // ---- cells [i0-1, i0-1+kCX) x [j0-1, j0-1+kCY): 12 rows each, then the
  // patches touching the tile: 9 LPS rows each; these are the patches from
  // ceil((i0 - 2) / 2) (also for negative i0) to floor((i0 + 2 kTCX - 1) / 2),
  // likewise in y
  const int PI0 = (i0 - 1) >> 1, PJ0 = (j0 - 1) >> 1;
  const int PI1 = (i0 + 2 * kTCX - 1) >> 1, PJ1 = (j0 + 2 * kTCY - 1) >> 1;
  for (int e = t; e < kCX * kCY; e += NTT) {
    const int lc = e % kCX, lr = e / kCX;
    const int ci = i0 - 1 + lc, cj = j0 - 1 + lr;
    const bool ok = ci >= 0 && cj >= 0 && ci < g.nx && cj < g.ny && !S.sol[lr + 1][lc + 1];
    S.cvalid[e] = ok;
    if (!ok) continue;
    T wu[4], wv[4], wp[4], bu[4], bv[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int li = lc + 1 + (a & 1), lj = lr + 1 + (a >> 1);  // staged coords of the node
      wu[a] = S.w[0][lj][li];
      wv[a] = S.w[1][lj][li];
      wp[a] = S.w[2][lj][li];
      bu[a] = S.vb[0][lj][li];
      bv[a] = S.vb[1][lj][li];
    }
    T r[12];
    cell_all_rows<T, false>(s, wu, wv, wp, bu, bv, r);
#pragma unroll
    for (int k = 0; k < 12; ++k) S.cres[e][k] = r[k];
  }
  // the patches start where the cells left off, on the threads that the
  // cell loop leaves idle (a rotation of the thread index)
  constexpr int kOff = (kCX * kCY) % NTT;
  for (int e = (t + NTT - kOff) % NTT; e < kPX * kPY; e += NTT) {
    const int pi = PI0 + e % kPX, pj = PJ0 + e / kPX;
    const bool ok = pi <= PI1 && pj <= PJ1 && pi >= 0 && pj >= 0 && pi < g.nx / 2 &&
                    pj < g.ny / 2 && !S.sol[2 * pj - j0 + 2][2 * pi - i0 + 2];
    S.pvalid[e] = ok;
    if (!ok) continue;
    T p[9];
#pragma unroll
    for (int m = 0; m < 9; ++m) {
      const int li = 2 * pi + m % 3 - (i0 - 2), lj = 2 * pj + m / 3 - (j0 - 2);
      p[m] = S.w[2][lj][li];
    }
#pragma unroll
    for (int mn = 0; mn < 9; ++mn) {
      T acc = 0;
#pragma unroll
      for (int m = 0; m < 9; ++m) acc += s.S9[mn * 9 + m] * p[m];
      S.pres[e][mn] = acc;
    }
  }
  __syncthreads();
}

// Defect b - A x at node (i, j) of the staged tile with first node (i0, j0)
// from the staged rows (constrained rows: b - x), for a node of a fluid
// colour cell; xu.. and bu0.. are the node's unmasked iterate and
// right-hand side.
template <typename T, int kTCX, int kTCY>
__device__ __forceinline__ void pass_node_defect(int i, int j, int i0, int j0, T xu, T xv, T xp,
                                                 T bu0, T bv0, T bp0,
                                                 const PassSmem<T, kTCX, kTCY>& S, T& du, T& dv,
                                                 T& dp) {
  constexpr int kCX = 2 * kTCX + 1, kPX = kTCX + 2;
  const int PI0 = (i0 - 1) >> 1, PJ0 = (j0 - 1) >> 1;
  T ru = 0, rv = 0, rp = 0;
#pragma unroll
  for (int dyy = 0; dyy < 2; ++dyy)
#pragma unroll
    for (int dxx = 0; dxx < 2; ++dxx) {
      const int lc = i - 1 + dxx - (i0 - 1), lr = j - 1 + dyy - (j0 - 1);
      const int e = lr * kCX + lc;
      if (!S.cvalid[e]) continue;
      const int al = (1 - dxx) + 2 * (1 - dyy);
      ru += S.cres[e][al];
      rv += S.cres[e][4 + al];
      rp += S.cres[e][8 + al];
    }
#pragma unroll
  for (int dJ = 0; dJ < 2; ++dJ) {
    const int PJ = (j >> 1) - dJ;
    if (j - 2 * PJ > 2) continue;
#pragma unroll
    for (int dI = 0; dI < 2; ++dI) {
      const int PI = (i >> 1) - dI;
      if (i - 2 * PI > 2) continue;
      const int e = (PJ - PJ0) * kPX + (PI - PI0);
      if (!S.pvalid[e]) continue;
      rp += S.pres[e][(i - 2 * PI) + 3 * (j - 2 * PJ)];
    }
  }
  const uint8_t f = S.fl[j - (j0 - 2)][i - (i0 - 2)];
  du = bu0 - ((f & kVDir) ? xu : ru);
  dv = bv0 - ((f & kVDir) ? xv : rv);
  dp = bp0 - ((f & kPFix) ? xp : rp);
}

// Tile (bx, by) of the colour pass, computed by a group of NTT consecutive
// threads of the block (a block may hold several such groups, each with its
// own S; every thread of the block must call this together because of the
// block barriers).  The first 4 kTCX kTCY threads own one node of a colour
// cell each; with NTT larger, the other threads help stage the tile and
// compute the cell and patch rows, so that those take one round instead of
// two.  A group with active = false takes part in the barriers only and
// writes nothing.
template <typename T, int kTCX, int kTCY, int NTT = 4 * kTCX * kTCY>
__device__ __forceinline__ void vanka_pass_tile(const Grid& g, const Sten<T>& s, int colour,
                                                const T* __restrict__ b, const T* __restrict__ xin,
                                                const T* __restrict__ vb, const T* __restrict__ inv,
                                                T omega, T* __restrict__ xout, int bx, int by,
                                                PassSmem<T, kTCX, kTCY>& S, bool active = true) {
  if (!active) bx = by = 0;
  constexpr int kTileThreads = 4 * kTCX * kTCY;
  static_assert(NTT >= kTileThreads && NTT % 32 == 0 && kTileThreads % 32 == 0, "tile group");
  const int cx = colour & 1, cy = colour >> 1;
  const int sx = g.nx / 2 + 1, sy = g.ny / 2 + 1;
  const int pitch = vanka_pitch(g), nslots = vanka_slots(g);
  const int nn = g.nn;
  const int tx0 = bx * kTCX, ty0 = by * kTCY;
  const int i0 = 2 * tx0 - cx, j0 = 2 * ty0 - cy;  // first node of the tile
  const int t = threadIdx.x % NTT;
  const bool owner = t < kTileThreads;  // owns a node of a colour cell
  // ---- this thread's node (quad q, local node a) and its loads that do not
  // depend on the defect: b, x_in and its three rows of the cell's inverse,
  // issued first so that their latency overlaps the stencil work below
  const int q = t >> 2, a = t & 3;
  const int ti = tx0 + (q % kTCX), tj = ty0 + (q / kTCX);
  const bool slot_ok = owner && ti < sx && tj < sy;
  const int slot = tj * pitch + ti;
  const int ci = 2 * ti - cx, cj = 2 * tj - cy;
  const int i = ci + (a & 1), j = cj + (a >> 1);
  const bool node_ok = slot_ok && i >= 0 && j >= 0 && i <= g.nx && j <= g.ny;
  const int n = node_ok ? j * g.nnx + i : 0;
  // every global load of the tile is issued before the first barrier, none
  // depends on another: the thread's b, x_in and three inverse rows (read
  // even for a solid cell, whose rows are then not used), and the staged
  // nodes' flags, iterate, vbar and cell solid flags
  T xu = 0, xv = 0, xp = 0, bu0 = 0, bv0 = 0, bp0 = 0;
  T iv[36];
  if (node_ok) {
    xu = xin[n], xv = xin[nn + n], xp = xin[2 * nn + n];
    bu0 = b[n], bv0 = b[nn + n], bp0 = b[2 * nn + n];
    load_inv_rows<T>(inv, nslots, colour, slot, a, iv);
  }
  pass_stage_rows<T, kTCX, kTCY, NTT>(g, s, xin, vb, i0, j0, t, S);
  // own cell (ci, cj) sits at staged index (ci - i0 + 2, cj - j0 + 2)
  const bool cell_ok = slot_ok && ci >= 0 && cj >= 0 && ci < g.nx && cj < g.ny &&
                       !S.sol[cj - j0 + 2][ci - i0 + 2];
  if (!owner) return;  // helpers are whole warps past the owners
  T du = 0, dv = 0, dp = 0;
  if (node_ok && cell_ok)
    pass_node_defect<T, kTCX, kTCY>(i, j, i0, j0, xu, xv, xp, bu0, bv0, bp0, S, du, dv, dp);
  const int lane = t & 31, base = lane & ~3;
  T d[12];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    d[k] = __shfl_sync(0xffffffffu, du, base + k);
    d[4 + k] = __shfl_sync(0xffffffffu, dv, base + k);
    d[8 + k] = __shfl_sync(0xffffffffu, dp, base + k);
  }
  if (!node_ok || !active) return;
  if (cell_ok) {
    T acc[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      acc[c] = 0;
#pragma unroll
      for (int k = 0; k < 12; ++k) acc[c] += iv[c * 12 + k] * d[k];
    }
    xout[n] = xu + omega * acc[0];
    xout[nn + n] = xv + omega * acc[1];
    xout[2 * nn + n] = xp + omega * acc[2];
  } else {
    xout[n] = xu;
    xout[nn + n] = xv;
    xout[2 * nn + n] = xp;
  }
}

}  // namespace dnnmg

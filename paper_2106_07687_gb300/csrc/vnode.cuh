// Node-wise evaluation of the linearised operator from assembled
// coefficients, and the colour pass and defect of the persistent V-cycle
// built on it.
//
// The operator A'(vbar) of a level does not change during its cycles, while
// every colour pass and defect applies it once (17 times per level and
// cycle).  Evaluated cell by cell, with its Gauss points, a row costs about
// 370 multiply-adds per node and three dependent stages with two block
// barriers.  Here the 2x2 velocity blocks between a node and its 3x3
// neighbours, which are all that depends on vbar, are assembled once per
// linearisation (36 coefficients per node); the gradient, divergence and
// stabilisation stencils depend only on which of the cells and patches around
// the node are fluid, so their coefficients come from a small table in shared
// memory.  A row is then 36 + 36 + 25 multiply-adds, and one warp does a tile
// of 8 x 4 nodes by itself: no block barrier, and a level of few nodes still
// spreads over all SMs.
#pragma once
#include "recip.cuh"
#include "vanka_body.cuh"

namespace dnnmg {

// ---- node patterns ---------------------------------------------------------------
// Bits of the pattern of node (i, j): the four cells around it that are fluid
// (bit cx + 2 cy, cell (i - 1 + cx, j - 1 + cy)), the four stabilisation
// patches that hold it and are fluid (bit dI + 2 dJ, patch ((i >> 1) - dI,
// (j >> 1) - dJ)), and its constrained unknowns.
constexpr int kPatPatch = 4, kPatVDir = 1 << 8, kPatPFix = 1 << 9;

// ---- coefficient tables -----------------------------------------------------------
// For a mesh of width 1 (a level scales them by h and h^2, powers of two):
//   gd[cell mask][neighbour (di + 1) + 3 (dj + 1)] = coefficients of the
//     neighbour's pressure in the u and v rows, and of its u and v in the
//     pressure row;
//   lps[patch mask][(i & 1) + 2 (j & 1)][(di + 2) + 5 (dj + 2)] = coefficients of
//     the pressures around the node in its pressure row;
//   gc[cell mask] = the node's own entries of gd, in whose place gd holds the
//     row's sums in FP32 (see assemble_node; the sums of lps are zero).
template <typename T>
struct OpTable {
  T gd[16][9][4];
  T lps[16][4][25];
  T gc[16][4];
};

// Fill a table from the constants s of a mesh of width 1 (host).
template <typename T>
void fill_op_table(const Sten<double>& s, OpTable<T>& t) {
  for (int m = 0; m < 16; ++m) {
    double gd[9][4] = {};
    for (int c = 0; c < 4; ++c) {
      if (!(m & (1 << c))) continue;
      const int cx = c & 1, cy = c >> 1, a = (1 - cx) + 2 * (1 - cy);
      for (int b = 0; b < 4; ++b) {
        double* g = gd[(cx + (b & 1)) + 3 * (cy + (b >> 1))];
        g[0] -= s.Dx[b * 4 + a];
        g[1] -= s.Dy[b * 4 + a];
        g[2] += s.Dx[a * 4 + b];
        g[3] += s.Dy[a * 4 + b];
      }
    }
    for (int e = 0; e < 9; ++e)
      for (int k = 0; k < 4; ++k) t.gd[m][e][k] = (T)gd[e][k];
    for (int k = 0; k < 4; ++k) t.gc[m][k] = (T)gd[4][k];
    if (sizeof(T) == 4)  // applied to differences (see assemble_node): the row's sum
      for (int k = 0; k < 4; ++k) {
        double sum = 0.0;
        for (int e = 0; e < 9; ++e) sum += gd[e][k];
        t.gd[m][4][k] = (T)(std::abs(sum) < 1e-12 ? 0.0 : sum);
      }
    for (int cls = 0; cls < 4; ++cls) {
      double l[25] = {};
      for (int d = 0; d < 4; ++d) {
        const int s0 = (cls & 1) + 2 * (d & 1), t0 = (cls >> 1) + 2 * (d >> 1);  // in the patch
        if (!(m & (1 << d)) || s0 > 2 || t0 > 2) continue;
        for (int q = 0; q < 9; ++q)
          l[(q % 3 - s0 + 2) + 5 * (q / 3 - t0 + 2)] += s.S9[(s0 + 3 * t0) * 9 + q];
      }
      for (int e = 0; e < 25; ++e) t.lps[m][cls][e] = (T)l[e];
    }
  }
}

// ---- assembled velocity blocks -----------------------------------------------------
// Coefficients of node (i, j): c[4 e + {0, 1, 2, 3}] = the uu, uv, vu and vv
// entries towards neighbour e = (di + 1) + 3 (dj + 1), summed over the fluid
// cells (rows of cells first).  Stored as 16-byte vectors of all nodes,
// vector v of node n at v * nn + n.
// In FP32 block 4, the node's own, holds the sums of the row's entries, formed
// from the shape functions' sums (1 and 0) instead of the rounded entries, and
// the rows are applied to differences, sum_e c_e (x_e - x_4) + c_4 x_4 (so are
// the rows of OpTable): rounded entries then act on the iterate's variation
// only.  One FP32 cycle against FP64, nu and dt over 0.001 .. 0.02 and 0.002 ..
// 0.05: 1e-6 .. 8e-6 -> 6e-8 .. 7e-7, at the same time (185 us on 512x128
// cells).  The node's own entries, which the setup needs, follow as block 9.
template <typename T>
constexpr int kCoefs = sizeof(T) == 4 ? 40 : 36;

template <typename T>
__device__ __forceinline__ void assemble_node(const Grid& g, const Sten<T>& s,
                                              const T* __restrict__ vb, T* __restrict__ cf, int n) {
  const int i = n % g.nnx, j = n / g.nnx;
  T c[kCoefs<T>];
#pragma unroll
  for (int k = 0; k < kCoefs<T>; ++k) c[k] = T(0);
#pragma unroll
  for (int cy = 0; cy < 2; ++cy)
#pragma unroll
    for (int cx = 0; cx < 2; ++cx) {
      const int ci = i - 1 + cx, cj = j - 1 + cy;
      if (ci < 0 || cj < 0 || ci >= g.nx || cj >= g.ny || g.solid[cj * g.nx + ci]) continue;
      T bu[4], bv[4];
      load_cell<T, false>(g, vb, ci, cj, 0, bu);
      load_cell<T, false>(g, vb + g.nn, ci, cj, 0, bv);
      GaussData<T> gd;
      if constexpr (sizeof(T) == 8)
        gauss_data_shared<T>(bu, bv, gd);
      else
        gauss_data<T>(bu, bv, gd);
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        T J[3][3];
        elem_pair<T>(s, gd, (1 - cx) + 2 * (1 - cy), b, J);
        const int e = (cx + (b & 1)) + 3 * (cy + (b >> 1));
        T* q = c + (sizeof(T) == 4 && e == 4 ? 36 : 4 * e);
        q[0] += J[0][0], q[1] += J[0][1], q[2] += J[1][0], q[3] += J[1][1];
      }
      if constexpr (sizeof(T) == 4) {
        T R[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          T pa, dxa, dya;
          shape_one<T>(q, (1 - cx) + 2 * (1 - cy), pa, dxa, dya);
          R[0] += pa * gd.Bux[q], R[1] += pa * gd.Buy[q];
          R[2] += pa * gd.Bvx[q], R[3] += pa * gd.Bvy[q];
        }
        const T sc = s.wq * s.ih;
        c[16] += s.Es + sc * R[0], c[17] += sc * R[1];
        c[18] += sc * R[2], c[19] += s.Es + sc * R[3];
      }
    }
  using V = typename Vec16<T>::type;
  V* o = reinterpret_cast<V*>(cf) + n;
#pragma unroll
  for (int v = 0; v < kCoefs<T> / kVec16<T>; ++v) o[(size_t)v * g.nn] = vec_pack(c + v * kVec16<T>);
}

// ---- setup of the local inverses -------------------------------------------------------
__device__ __forceinline__ float pivot_recip(float d) { return 1.0f / d; }
__device__ __forceinline__ double pivot_recip(double d) { return recip64_any(d); }

// Inverse of the restriction of the level's Jacobian to the 12 unknowns of
// the fluid cell of `slot` in `colour` (its 4 nodes x u, v, p), with identity
// rows and columns on constrained unknowns, by a group of 16 consecutive lanes
// (a half-warp; every lane of it calls this with the same cell).  Lane r < 12
// gathers row r = (component c, node a) from the assembled blocks of node a
// and the coefficient table and keeps it in registers.  Gauss-Jordan
// elimination with partial pivoting then runs across the lanes, in place: at
// step k the unused lane with the largest |A[.][k]| (lowest lane on ties) is
// the pivot row p, and every lane adds a multiple of it,
//   A[.][j] = m A[p][j] + (0 on the pivot row, A[.][j] elsewhere),
// m = 1 / A[p][k] there and -A[.][k] / A[p][k] elsewhere, which column k then
// holds.  Rows are never swapped; the lane that pivoted on column k ends with
// row k of the inverse, whose column pcol[j] sits in column j.
// Assembling the 12 x 12 matrix cell by cell took most of the former setup
// (Gauss-point data of nine cells and 36 element blocks per cell): per launch,
// mean over levels 2 .. 5 in FP32 48.7 -> 28.1 us, levels 2 and 3 in FP64 137
// -> 44 us.
template <typename T>
__device__ __forceinline__ void vanka_setup_cell(const Grid& g, const uint16_t* pat, const T* cf,
                                                 const OpTable<T>& tab, T h, T h2,
                                                 T* __restrict__ inv, int* status, int colour,
                                                 int slot) {
  const int cx = colour & 1, cy = colour >> 1;
  const int sx = g.nx / 2 + 1, pitch = vanka_pitch(g);
  const int nslots = vanka_slots(g);
  if (slot >= nslots || slot % pitch >= sx) return;
  const int ci = 2 * (slot % pitch) - cx, cj = 2 * (slot / pitch) - cy;
  if (ci < 0 || cj < 0 || ci >= g.nx || cj >= g.ny || g.solid[cj * g.nx + ci]) return;
  const int lane = threadIdx.x & 15;
  const unsigned mask = 0xFFFFu << (threadIdx.x & 16);  // this half-warp
  const int r = lane < 12 ? lane : 0;                   // lanes 12..15 shadow row 0
  const int c = r >> 2, ax = r & 1, ay = (r >> 1) & 1;
  const int n0 = cj * g.nnx + ci, na = n0 + ay * g.nnx + ax;
  int pt[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) pt[b] = __ldg(pat + n0 + (b >> 1) * g.nnx + (b & 1));
  const int pa = __ldg(pat + na);
  const int cls = ((ci + ax) & 1) + 2 * ((cj + ay) & 1);
  T A[12];
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int di = (b & 1) - ax, dj = (b >> 1) - ay, e = (di + 1) + 3 * (dj + 1);
    const T* gd = e == 4 ? tab.gc[pa & 15] : tab.gd[pa & 15][e];
    if (c < 2) {
      // the uu, uv (c = 0) or vu, vv (c = 1) entries of the block
      const int k = (sizeof(T) == 4 && e == 4 ? 36 : 4 * e) + 2 * c;
      constexpr int V = kVec16<T>;
      const T* q = cf + ((size_t)(k / V) * g.nn + na) * V + k % V;
      A[b] = __ldg(q);
      A[4 + b] = __ldg(q + 1);
      A[8 + b] = h * __ldg(gd + c);
    } else {
      A[b] = h * __ldg(gd + 2);
      A[4 + b] = h * __ldg(gd + 3);
      A[8 + b] = h2 * __ldg(tab.lps[(pa >> kPatPatch) & 15][cls] + (di + 2) + 5 * (dj + 2));
    }
  }
  // identity rows and zero columns on constrained unknowns
  const bool own_cons = pa & (c < 2 ? kPatVDir : kPatPFix);
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const bool col_cons = pt[k & 3] & (k < 8 ? kPatVDir : kPatPFix);
    if (own_cons) A[k] = k == r ? T(1) : T(0);
    else if (col_cons) A[k] = T(0);
  }
  bool used = lane >= 12, ok = true;
  int my_col = 0;
  int pcol[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    // the bit patterns of non-negative numbers order like the numbers: one
    // maximum over the half-warp (FP64: of the high words, then of the low words
    // beside the largest), then the lowest unused lane that holds it
    unsigned key, low = 0u, mlow = 0u;
    if constexpr (sizeof(T) == 4)
      key = __float_as_uint(A[k]) & 0x7FFFFFFFu;
    else
      key = (unsigned)__double2hiint(A[k]) & 0x7FFFFFFFu;
    if (used) key = 0u;
    const unsigned mx = __reduce_max_sync(mask, key);
    if constexpr (sizeof(T) == 8) {
      low = key == mx && !used ? (unsigned)__double2loint(A[k]) : 0u;
      mlow = __reduce_max_sync(mask, low);
    }
    const int p = (__ffs(__ballot_sync(mask, key == mx && low == mlow && !used) & mask) - 1) & 15;
    pcol[k] = p;
    // a pivot that is neither zero nor NaN (whose bits lie above infinity's; the
    // same in every lane of the group)
    constexpr unsigned kInf = sizeof(T) == 4 ? 0x7F800000u : 0x7FF00000u;
    ok = ok && (mx | mlow) != 0u && mx <= kInf;
    if (ok) {
      const bool piv = lane == p;
      const T ip = pivot_recip(__shfl_sync(mask, A[k], p, 16));
      const T m = piv ? ip : -A[k] * ip;
#pragma unroll
      for (int cc = 0; cc < 12; ++cc) {
        if (cc == k) continue;
        const T ap = __shfl_sync(mask, A[cc], p, 16);
        A[cc] = m * ap + (piv ? T(0) : A[cc]);
      }
      A[k] = m;
      if (piv) used = true, my_col = k;
    }
  }
  if (!ok) {
    if (lane == 0) atomicOr(status, 1);
  }
  if (lane >= 12) return;
#pragma unroll
  for (int j = 0; j < 12; ++j)
    inv[vanka_inv_index<T>(nslots, colour, slot, my_col & 3, (my_col >> 2) * 12 + pcol[j])] =
        ok ? A[j] : T(0);
}

// ---- persistent kernels -----------------------------------------------------------------
// Threads per block, one block per SM: a pass holds 36 coefficients and 36
// inverse entries per thread, so FP32 takes 16 warps of 128 registers and FP64
// 8 warps of 255.
template <typename T>
constexpr int walk_threads() {
  return sizeof(T) == 4 ? 512 : 256;
}
// count records from global to shared memory, by the whole block
template <class S>
__device__ __forceinline__ void copy_ints(S* dst, const S* src, int count) {
  static_assert(sizeof(S) % sizeof(int) == 0, "record size");
  const int* s = reinterpret_cast<const int*>(src);
  int* d = reinterpret_cast<int*>(dst);
  for (int e = threadIdx.x; e < (int)(count * sizeof(S) / sizeof(int)); e += blockDim.x) d[e] = s[e];
}

// ---- one warp, 8 x 4 nodes -----------------------------------------------------------
// Masked iterate of the warp's nodes plus a two-node halo: 12 x 8 nodes, rows
// of 24 so that the four rows of a tile fall on different banks.
constexpr int kWX = 8, kWY = 4, kWSX = kWX + 4, kWSY = kWY + 4, kWPitch = 24;
template <typename T>
struct WarpTile {
  T w[3][kWSY][kWPitch];
};

// Level data of the node-wise kernels.  With SPLIT the stabilisation's scale is a
// sum of two (a batch's FP32 levels, whose table is scaled by alpha0 / nu).
template <typename T, bool SPLIT = false>
struct NodeLevel {
  static constexpr bool kSplit = SPLIT;
  int nx, ny, nnx, nn;
  const uint16_t* pat;  // node patterns
  const T* cf;          // assembled velocity blocks
  T h, h2;              // mesh width and the scale of the stabilisation's table
  T h2lo = T(0);        // what h2 lacks of the exact scale
};

// ---- the iterate of a level ------------------------------------------------------------
// PlanarX: [3][nn] arrays (the coarsest level's solution); a barrier lies between
// the phases that write and read it.
// TaggedX: every node's values carry the number of the update that wrote them,
// in the same 16-byte word (FP32: u, v, p, tag; FP64: three words of a value and
// a tag), which is stored and loaded as one access.  A reader waits until the
// tag is the one it needs, so that consecutive phases need no grid-wide barrier:
// the barrier's chain (stores acknowledged, an atomic, a poll) and the load
// behind it become one store and one polled load.  Two buffers suffice: the
// tile that overwrites a node has waited for the values of every tile that read
// the node's previous ones (they lie within its own two-node halo).  The numbers
// run on from cycle to cycle (vcycle_numbers per cycle, whatever its sweeps), in a
// word on the device: they come round after 2^32 updates, 238 million V(2,2)
// cycles, in which every word that a cycle reads is rewritten.  The wait is
// bounded (a warp's rounds over a single problem's cycle of at most 160 phases, or
// between two barriers of a batch's, by kTagPolls unless the caller sets another
// bound; then bit 8 of *status is set and the warp waits no more).  All lanes of the warp call load; other_loads
// is run once, behind the first round's loads, to issue what the tile reads
// besides the iterate: the tags are then mostly there when it is through.
constexpr int kTagPolls = 1 << 21;  // over a second

template <typename T>
struct PlanarX {
  const T* in;
  int nn;
  template <int N, class F>
  __device__ __forceinline__ void load(const int (&n)[N], const bool (&)[N], T (&u)[N], T (&v)[N],
                                       T (&p)[N], int&, F other_loads) const {
#pragma unroll
    for (int r = 0; r < N; ++r)
      u[r] = __ldcg(in + n[r]), v[r] = __ldcg(in + nn + n[r]), p[r] = __ldcg(in + 2 * nn + n[r]);
    other_loads();
  }
};

// (no clobber of memory: nothing but these two touches a tagged buffer, and a
// tag vouches for the values beside it only)
__device__ __forceinline__ void ld_pair(const ulonglong2* p, unsigned long long& a,
                                        unsigned long long& b) {
  asm volatile("{ .reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t; }"
               : "=l"(a), "=l"(b)
               : "l"(p));
}
__device__ __forceinline__ void st_pair(ulonglong2* p, unsigned long long a, unsigned long long b) {
  asm volatile("{ .reg .b128 t; mov.b128 t, {%1, %2}; st.relaxed.gpu.global.b128 [%0], t; }" ::"l"(p),
               "l"(a), "l"(b));
}

// words of a node in a tagged buffer
template <typename T>
constexpr int kTagWords = sizeof(T) == 4 ? 1 : 3;

template <typename T>
struct TaggedX {
  const ulonglong2* in;
  ulonglong2* out;
  T* planar;  // when set, the values go there instead (the cycle's result)
  int nn;
  unsigned tin, tout;
  int* status;
  template <int N, class F>
  __device__ __forceinline__ void load(const int (&n)[N], const bool (&need)[N], T (&u)[N],
                                       T (&v)[N], T (&p)[N], int& budget, F other_loads) const {
    unsigned long long q[N][sizeof(T) == 4 ? 2 : 6];
    if constexpr (sizeof(T) == 8) other_loads();  // FP64 has no registers to spare for the tags
    round(n, q);
    if constexpr (sizeof(T) == 4) other_loads();
    // the warp stays together: lanes that left one by one would run what
    // follows in turn (FP64 tiles 13.6 k instead of 5.9 k cycles)
    while (!__all_sync(0xffffffffu, ready(need, q)) && --budget > 0) round(n, q);
    if (budget <= 0) {
      budget = 0;
      atomicOr(status, 8);
    }
#pragma unroll
    for (int r = 0; r < N; ++r) {
      if constexpr (sizeof(T) == 4) {
        u[r] = __uint_as_float((unsigned)q[r][0]);
        v[r] = __uint_as_float((unsigned)(q[r][0] >> 32));
        p[r] = __uint_as_float((unsigned)q[r][1]);
      } else {
        u[r] = __longlong_as_double((long long)q[r][0]);
        v[r] = __longlong_as_double((long long)q[r][2]);
        p[r] = __longlong_as_double((long long)q[r][4]);
      }
    }
  }
  template <int N, int W>
  __device__ __forceinline__ void round(const int (&n)[N], unsigned long long (&q)[N][W]) const {
#pragma unroll
    for (int r = 0; r < N; ++r)
#pragma unroll
      for (int c = 0; c < W / 2; ++c) ld_pair(in + c * nn + n[r], q[r][2 * c], q[r][2 * c + 1]);
  }
  template <int N, int W>
  __device__ __forceinline__ bool ready(const bool (&need)[N],
                                        const unsigned long long (&q)[N][W]) const {
    bool ok = true;
#pragma unroll
    for (int r = 0; r < N; ++r)
#pragma unroll
      for (int c = 0; c < W / 2; ++c) {
        const unsigned tag =
            sizeof(T) == 4 ? (unsigned)(q[r][2 * c + 1] >> 32) : (unsigned)q[r][2 * c + 1];
        ok = ok && (!need[r] || tag == tin);
      }
    return ok;
  }
  __device__ __forceinline__ void store(int n, T u, T v, T p) const {
    if (planar) {
      planar[n] = u, planar[nn + n] = v, planar[2 * nn + n] = p;
    } else if constexpr (sizeof(T) == 4) {
      st_pair(out + n,
              (unsigned long long)__float_as_uint(u) |
                  ((unsigned long long)__float_as_uint(v) << 32),
              (unsigned long long)__float_as_uint(p) | ((unsigned long long)tout << 32));
    } else {
      store_one(n, 0, u), store_one(n, 1, v), store_one(n, 2, p);
    }
  }
  __device__ __forceinline__ void store_one(int n, int c, T v) const {  // FP64
    if (planar)
      planar[c * nn + n] = v;
    else
      st_pair(out + c * nn + n, (unsigned long long)__double_as_longlong((double)v), tout);
  }
};

// Stage the nodes around tile (i0, j0), three per lane, and load this lane's own
// node `own` (its unmasked values; -1: none).
template <typename T, bool OWN, class NL, class X, class F>
__device__ __forceinline__ void stage_warp_tile(const NL& L, const X& x, int i0, int j0,
                                                int lane, int own, WarpTile<T>& S, T& xu, T& xv,
                                                T& xp, int& budget, F other_loads) {
  static_assert(kWSX * kWSY == 96, "three nodes per lane");
  constexpr int N = OWN ? 4 : 3;
  T u[N], v[N], p[N];
  int pt[3], n[N];
  bool in[N];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const int e = lane + 32 * r, i = i0 - 2 + e % kWSX, j = j0 - 2 + e / kWSX;
    in[r] = i >= 0 && j >= 0 && i <= L.nx && j <= L.ny;
    n[r] = in[r] ? j * L.nnx + i : 0;
  }
  if constexpr (OWN) in[3] = own >= 0, n[3] = in[3] ? own : 0;
  x.template load<N>(n, in, u, v, p, budget, [&] {
    other_loads();
#pragma unroll
    for (int r = 0; r < 3; ++r)
      pt[r] = in[r] ? (int)__ldg(L.pat + n[r]) : (kPatVDir | kPatPFix);
  });
  if constexpr (OWN) xu = u[3], xv = v[3], xp = p[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const int e = lane + 32 * r, li = e % kWSX, lj = e / kWSX;
    S.w[0][lj][li] = (pt[r] & kPatVDir) ? T(0) : u[r];
    S.w[1][lj][li] = (pt[r] & kPatVDir) ? T(0) : v[r];
    S.w[2][lj][li] = (pt[r] & kPatPFix) ? T(0) : p[r];
  }
}

// Rows of A'(vbar) at the staged node (li, lj) with pattern pt, coefficients c
// and class cls = (i & 1) + 2 (j & 1); constrained rows are the caller's.
template <typename T, class NL>
__device__ __forceinline__ void node_rows_assembled(const NL& L, const OpTable<T>& tab,
                                                    const WarpTile<T>& S, const T c[36], int li,
                                                    int lj, int pt, int cls, T& ru, T& rv, T& rp) {
  const T(*gd)[4] = tab.gd[pt & 15];
  T u0 = 0, v0 = 0, u1 = 0, v1 = 0, d0 = 0, d1 = 0;
  const T uc = S.w[0][lj][li], vc = S.w[1][lj][li], pc = S.w[2][lj][li];
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const T u = S.w[0][lj - 1 + e / 3][li - 1 + e % 3];
    const T v = S.w[1][lj - 1 + e / 3][li - 1 + e % 3];
    const T p = S.w[2][lj - 1 + e / 3][li - 1 + e % 3];
    const bool diff = sizeof(T) == 4 && e != 4;
    const T du = diff ? u - uc : u, dv = diff ? v - vc : v, dp = diff ? p - pc : p;
    u0 += c[4 * e] * du + c[4 * e + 1] * dv;
    v0 += c[4 * e + 2] * du + c[4 * e + 3] * dv;
    u1 += gd[e][0] * dp;
    v1 += gd[e][1] * dp;
    d0 += gd[e][2] * du;
    d1 += gd[e][3] * dv;
  }
  const T* ls = tab.lps[(pt >> kPatPatch) & 15][cls];
  T s[5];
#pragma unroll
  for (int dj = 0; dj < 5; ++dj) {
    s[dj] = T(0);
#pragma unroll
    for (int di = 0; di < 5; ++di) {
      const T p = S.w[2][lj - 2 + dj][li - 2 + di];
      if constexpr (sizeof(T) == 4) {
        if (dj != 2 || di != 2) s[dj] += ls[5 * dj + di] * (p - pc);
      } else {
        s[dj] += ls[5 * dj + di] * p;
      }
    }
  }
  ru = u0 + L.h * u1;
  rv = v0 + L.h * v1;
  const T sum = ((s[0] + s[1]) + (s[3] + s[4])) + s[2];
  rp = L.h * (d0 + d1) + L.h2 * sum;
  if constexpr (NL::kSplit) rp += L.h2lo * sum;
}

// One colour pass (see vanka_body.cuh) on the warp's 4 x 2 colour cells (bx,
// by).  Lane 4 q + a owns node a of cell q.
template <typename T, class NL, class X>
__device__ __forceinline__ void warp_pass_tile(const NL& L, const OpTable<T>& tab,
                                               int colour, const T* b, const X& x, const T* inv,
                                               int pitch, int nslots, T omega, int bx, int by,
                                               int lane, WarpTile<T>& S, int& budget) {
  const int cx = colour & 1, cy = colour >> 1;
  const int i0 = kWX * bx - cx, j0 = kWY * by - cy;
  const int q = lane >> 2, a = lane & 3;
  const int li = 2 * (q & 3) + (a & 1), lj = 2 * (q >> 2) + (a >> 1);
  const int i = i0 + li, j = j0 + lj;
  const bool node_ok = i >= 0 && j >= 0 && i <= L.nx && j <= L.ny;
  const int n = node_ok ? j * L.nnx + i : 0;
  const int slot = node_ok ? (2 * by + (q >> 2)) * pitch + 4 * bx + (q & 3) : 0;
  // every load of the tile is issued before the first is used, the iterate's
  // (behind which the others' latency hides) first
  T c[36], iv[36], xu, xv, xp, bu, bv, bp;
  int pt;
  stage_warp_tile<T, true>(L, x, i0, j0, lane, node_ok ? n : -1, S, xu, xv, xp, budget, [&] {
    load36<T>(L.cf, n, L.nn, c);
    pt = node_ok ? (int)__ldg(L.pat + n) : 0;
    bu = __ldcg(b + n), bv = __ldcg(b + L.nn + n), bp = __ldcg(b + 2 * L.nn + n);
    load_inv_rows<T>(inv, nslots, colour, slot, a, iv);
  });
  __syncwarp();
  // the cell is fluid: its bit in the node's pattern
  const bool cell_ok = node_ok && ((pt >> ((1 - (a & 1)) + 2 * (1 - (a >> 1)))) & 1);
  T ru, rv, rp;
  node_rows_assembled<T>(L, tab, S, c, li + 2, lj + 2, pt, (i & 1) + 2 * (j & 1), ru, rv, rp);
  T du = bu - ((pt & kPatVDir) ? xu : ru), dv = bv - ((pt & kPatVDir) ? xv : rv),
    dp = bp - ((pt & kPatPFix) ? xp : rp);
  T d[12];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    d[k] = __shfl_sync(0xffffffffu, du, (lane & ~3) + k);
    d[4 + k] = __shfl_sync(0xffffffffu, dv, (lane & ~3) + k);
    d[8 + k] = __shfl_sync(0xffffffffu, dp, (lane & ~3) + k);
  }
  if (node_ok) {
    T acc[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      acc[r] = 0;
#pragma unroll
      for (int k = 0; k < 12; ++k) acc[r] += iv[r * 12 + k] * d[k];
    }
    x.store(n, cell_ok ? xu + omega * acc[0] : xu, cell_ok ? xv + omega * acc[1] : xv,
            cell_ok ? xp + omega * acc[2] : xp);
  }
  __syncwarp();  // the tile's shared memory is reused
}

// The first colour pass of a smoothing sweep that starts from x = 0, for
// item e = 4 * slot + a (node a of the colour cell of `slot`): the defect is
// then b on every row (b - A 0 = b, and b - x = b on constrained rows), so
// the pass needs neither the iterate nor any operator rows:
// x_out = omega A_c^-1 b on the colour's fluid cells and 0 on every other
// node, bitwise what the tiled pass computes from x = 0, and every node of the
// level is written.  The four items of a cell are consecutive lanes of one
// warp; all 32 lanes call this (valid = false for padding items).
template <typename T, class X>
__device__ __forceinline__ void zero_pass_node(const Grid& g, int colour, const T* b, const X& x,
                                               const T* inv, T omega, int e, bool valid) {
  const int cx = colour & 1, cy = colour >> 1;
  const int sx = g.nx / 2 + 1, pitch = vanka_pitch(g), nslots = vanka_slots(g), nn = g.nn;
  const int slot = e >> 2, a = e & 3;
  const bool slot_ok = valid && slot < nslots && slot % pitch < sx;
  const int ci = 2 * (slot % pitch) - cx, cj = 2 * (slot / pitch) - cy;
  const int i = ci + (a & 1), j = cj + (a >> 1);
  const bool node_ok = slot_ok && i >= 0 && j >= 0 && i <= g.nx && j <= g.ny;
  const bool cell_ok = slot_ok && ci >= 0 && cj >= 0 && ci < g.nx && cj < g.ny &&
                       !g.solid[cj * g.nx + ci];
  const int n = node_ok ? j * g.nnx + i : 0;
  T du = 0, dv = 0, dp = 0;
  if (node_ok) du = __ldcg(b + n), dv = __ldcg(b + nn + n), dp = __ldcg(b + 2 * nn + n);
  const int base = (threadIdx.x & 31) & ~3;
  T d[12];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    d[k] = __shfl_sync(0xffffffffu, du, base + k);
    d[4 + k] = __shfl_sync(0xffffffffu, dv, base + k);
    d[8 + k] = __shfl_sync(0xffffffffu, dp, base + k);
  }
  if (!node_ok) return;
  T acc[3] = {T(0), T(0), T(0)};
  if (cell_ok) {
    T iv[36];
    load_inv_rows<T>(inv, nslots, colour, slot, a, iv);
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int k = 0; k < 12; ++k) acc[c] += iv[c * 12 + k] * d[k];
  }
  x.store(n, omega * acc[0], omega * acc[1], omega * acc[2]);
}

// x += P xc at fine node (i, j) on free unknowns (prolong_add_node of vbody.cuh).
// All lanes of a warp call it.
template <typename T, class XC, class XF>
__device__ __forceinline__ void prolong_node(const Grid& f, const Grid& c, const XC& xc,
                                             const XF& x, int i, int j, bool valid, int& budget) {
  const int I0 = i >> 1, J0 = j >> 1, nI = (i & 1) ? 2 : 1, nJ = (j & 1) ? 2 : 1;
  int m[4], n[1] = {j * f.nnx + i};
  bool use[4], one[1] = {valid};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    use[e] = valid && (e & 1) < nI && (e >> 1) < nJ;
    m[e] = use[e] ? (J0 + (e >> 1)) * c.nnx + I0 + (e & 1) : J0 * c.nnx + I0;
  }
  uint8_t fl, cfl[4];
  T xv[3][1], cv[3][4];
  xc.template load<4>(m, use, cv[0], cv[1], cv[2], budget, [&] {
    x.template load<1>(n, one, xv[0], xv[1], xv[2], budget, [&] {
      fl = f.flags[n[0]];
#pragma unroll
      for (int e = 0; e < 4; ++e) cfl[e] = use[e] ? c.flags[m[e]] : uint8_t(0xFF);
    });
  });
  const T w = T(1) / T(nI * nJ);
#pragma unroll
  for (int comp = 0; comp < 3; ++comp) {
    const uint8_t bit = comp < 2 ? kVDir : kPFix;
    T acc = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (!(cfl[e] & bit)) acc += cv[comp][e];
    if (!(fl & bit)) xv[comp][0] += w * acc;
  }
  if (valid) x.store(n[0], xv[0][0], xv[1][0], xv[2][0]);
}

// ---- one warp, 4 x 2 nodes: four lanes per node -----------------------------------------
// On a level with few tiles a warp's chain is all that a phase lasts, and in
// FP64 every instruction of a warp takes 64 cycles of its scheduler.  Here lanes
// 4 m + s, s = 0..3, share node m: each takes every fourth neighbour and every
// fourth pressure of the stabilisation, then the columns of the inverse that
// belong to node s of the cell; two butterfly sums join them.  A lane issues
// about 60 instead of 180 multiply-adds, all lanes together a third more.
constexpr int kSX = 4, kSY = 2, kSSX = kSX + 4, kSSY = kSY + 4;

template <typename T>
__device__ __forceinline__ T quad_sum(T v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// Stage the 8 x 6 nodes around tile (i0, j0) and load this lane's own node.
template <typename T, bool OWN, class NL, class X, class F>
__device__ __forceinline__ void stage_split_tile(const NL& L, const X& x, int i0, int j0,
                                                 int lane, int own, WarpTile<T>& S, T& xu, T& xv,
                                                 T& xp, int& budget, F other_loads) {
  constexpr int N = OWN ? 3 : 2;
  T u[N], v[N], p[N];
  int pt[2], n[N];
  bool in[N];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int e = lane + 32 * r, i = i0 - 2 + e % kSSX, j = j0 - 2 + e / kSSX;
    in[r] = e < kSSX * kSSY && i >= 0 && j >= 0 && i <= L.nx && j <= L.ny;
    n[r] = in[r] ? j * L.nnx + i : 0;
  }
  if constexpr (OWN) in[2] = own >= 0, n[2] = in[2] ? own : 0;
  x.template load<N>(n, in, u, v, p, budget, [&] {
    other_loads();
#pragma unroll
    for (int r = 0; r < 2; ++r)
      pt[r] = in[r] ? (int)__ldg(L.pat + n[r]) : (kPatVDir | kPatPFix);
  });
  if constexpr (OWN) xu = u[2], xv = v[2], xp = p[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int e = lane + 32 * r, li = e % kSSX, lj = e / kSSX;
    if (e >= kSSX * kSSY) break;
    S.w[0][lj][li] = (pt[r] & kPatVDir) ? T(0) : u[r];
    S.w[1][lj][li] = (pt[r] & kPatVDir) ? T(0) : v[r];
    S.w[2][lj][li] = (pt[r] & kPatPFix) ? T(0) : p[r];
  }
}

// this lane's coefficients: neighbours s, s + 4 and (s = 0) 8
template <typename T, class NL>
__device__ __forceinline__ void load_split_blocks(const NL& L, int n, int s, T c[12]) {
  using V = typename Vec16<T>::type;
  constexpr int NV = 4 / kVec16<T>;
  const V* p = reinterpret_cast<const V*>(L.cf);
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const int e = s + 4 * r < 9 ? s + 4 * r : 8;
#pragma unroll
    for (int h = 0; h < NV; ++h)
      vec_unpack(__ldg(p + (size_t)(e * NV + h) * L.nn + n), c + 4 * r + h * kVec16<T>);
  }
}

template <typename T, class NL>
__device__ __forceinline__ void node_rows_split(const NL& L, const OpTable<T>& tab,
                                                const WarpTile<T>& S, const T c[12], int li, int lj,
                                                int pt, int cls, int s, T& ru, T& rv, T& rp) {
  T u0 = 0, v0 = 0, u1 = 0, v1 = 0, d0 = 0, ls = 0;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const int e = s + 4 * r;
    if (e >= 9) break;
    const int dj = e / 3, di = e - 3 * dj;
    const T* g = tab.gd[pt & 15][e];
    const T u = S.w[0][lj - 1 + dj][li - 1 + di], v = S.w[1][lj - 1 + dj][li - 1 + di],
            p = S.w[2][lj - 1 + dj][li - 1 + di];
    u0 += c[4 * r] * u + c[4 * r + 1] * v;
    v0 += c[4 * r + 2] * u + c[4 * r + 3] * v;
    u1 += g[0] * p;
    v1 += g[1] * p;
    d0 += g[2] * u + g[3] * v;
  }
  const T* l = tab.lps[(pt >> kPatPatch) & 15][cls];
#pragma unroll
  for (int r = 0; r < 7; ++r) {
    const int e = s + 4 * r;
    if (e >= 25) break;
    const int dj = e / 5, di = e - 5 * dj;
    ls += l[e] * S.w[2][lj - 2 + dj][li - 2 + di];
  }
  ru = quad_sum(u0 + L.h * u1);
  rv = quad_sum(v0 + L.h * v1);
  rp = quad_sum(L.h * d0 + L.h2 * ls);
}

// One colour pass on the warp's 2 x 1 colour cells (bx, by).
template <typename T, class NL, class X>
__device__ __forceinline__ void split_pass_tile(const NL& L, const OpTable<T>& tab,
                                                int colour, const T* b, const X& x, const T* inv,
                                                int pitch, int nslots, T omega, int bx, int by,
                                                int lane, WarpTile<T>& S, int& budget) {
  const int cx = colour & 1, cy = colour >> 1;
  const int i0 = kSX * bx - cx, j0 = kSY * by - cy;
  const int q = lane >> 4, a = (lane >> 2) & 3, s = lane & 3;
  const int li = 2 * q + (a & 1), lj = a >> 1, i = i0 + li, j = j0 + lj;
  const bool node_ok = i >= 0 && j >= 0 && i <= L.nx && j <= L.ny;
  const int n = node_ok ? j * L.nnx + i : 0;
  const int slot = node_ok ? by * pitch + 2 * bx + q : 0;
  T c[12], iv[3][3], bu, bv, bp, xu, xv, xp;
  int pt;
  stage_split_tile<T, true>(L, x, i0, j0, lane, node_ok ? n : -1, S, xu, xv, xp, budget, [&] {
    load_split_blocks<T>(L, n, s, c);
    pt = node_ok ? (int)__ldg(L.pat + n) : 0;
    bu = __ldcg(b + n), bv = __ldcg(b + L.nn + n), bp = __ldcg(b + 2 * L.nn + n);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int k = 0; k < 3; ++k)
        iv[r][k] = __ldg(inv + vanka_inv_index<T>(nslots, colour, slot, a, r * 12 + 4 * k + s));
  });
  __syncwarp();
  const bool cell_ok = node_ok && ((pt >> ((1 - (a & 1)) + 2 * (1 - (a >> 1)))) & 1);
  T ru, rv, rp;
  node_rows_split<T>(L, tab, S, c, li + 2, lj + 2, pt, (i & 1) + 2 * (j & 1), s, ru, rv, rp);
  const T du = bu - ((pt & kPatVDir) ? xu : ru), dv = bv - ((pt & kPatVDir) ? xv : rv),
          dp = bp - ((pt & kPatPFix) ? xp : rp);
  const int src = (lane & 16) + 4 * s;  // node s of the cell
  const T d0 = __shfl_sync(0xffffffffu, du, src), d1 = __shfl_sync(0xffffffffu, dv, src),
          d2 = __shfl_sync(0xffffffffu, dp, src);
  T acc[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) acc[r] = quad_sum(iv[r][0] * d0 + iv[r][1] * d1 + iv[r][2] * d2);
  if (node_ok && s < 3) {  // lane s writes component s
    const T o = s == 0 ? xu : (s == 1 ? xv : xp), y = s == 0 ? acc[0] : (s == 1 ? acc[1] : acc[2]);
    x.store_one(n, s, cell_ok ? o + omega * y : o);
  }
  __syncwarp();
}

// d = b - A'(vbar) x, zero on constrained unknowns, on the warp's 4 x 2 nodes.
template <typename T, class NL, class X>
__device__ __forceinline__ void split_defect_tile(const NL& L, const OpTable<T>& tab,
                                                  const T* b, const X& x, T* d, int bx, int by,
                                                  int lane, WarpTile<T>& S, int& budget) {
  const int i0 = kSX * bx, j0 = kSY * by, m = lane >> 2, s = lane & 3;
  const int li = m % kSX, lj = m / kSX, i = i0 + li, j = j0 + lj;
  const bool ok = i <= L.nx && j <= L.ny;
  const int n = ok ? j * L.nnx + i : 0;
  T c[12], bb, xu, xv, xp;
  int pt;
  stage_split_tile<T, false>(L, x, i0, j0, lane, -1, S, xu, xv, xp, budget, [&] {
    load_split_blocks<T>(L, n, s, c);
    pt = ok ? (int)__ldg(L.pat + n) : 0;
    bb = __ldcg(b + (s < 3 ? s : 0) * L.nn + n);
  });
  __syncwarp();
  T ru, rv, rp;
  node_rows_split<T>(L, tab, S, c, li + 2, lj + 2, pt, (i & 1) + 2 * (j & 1), s, ru, rv, rp);
  if (ok && s < 3) {
    const bool cons = pt & (s < 2 ? kPatVDir : kPatPFix);
    d[s * L.nn + n] = cons ? T(0) : bb - (s == 0 ? ru : (s == 1 ? rv : rp));
  }
  __syncwarp();
}

// d = b - A'(vbar) x, zero on constrained unknowns, on the warp's 8 x 4 nodes.
template <typename T, class NL, class X>
__device__ __forceinline__ void warp_defect_tile(const NL& L, const OpTable<T>& tab,
                                                 const T* b, const X& x, T* d, int bx, int by,
                                                 int lane, WarpTile<T>& S, int& budget) {
  const int i0 = kWX * bx, j0 = kWY * by, li = lane % kWX, lj = lane / kWX;
  const int i = i0 + li, j = j0 + lj;
  const bool ok = i <= L.nx && j <= L.ny;
  const int n = ok ? j * L.nnx + i : 0;
  T c[36], bu, bv, bp, xu, xv, xp;
  int pt;
  stage_warp_tile<T, false>(L, x, i0, j0, lane, -1, S, xu, xv, xp, budget, [&] {
    load36<T>(L.cf, n, L.nn, c);
    pt = ok ? (int)__ldg(L.pat + n) : 0;
    bu = __ldcg(b + n), bv = __ldcg(b + L.nn + n), bp = __ldcg(b + 2 * L.nn + n);
  });
  __syncwarp();
  T ru, rv, rp;
  node_rows_assembled<T>(L, tab, S, c, li + 2, lj + 2, pt, (i & 1) + 2 * (j & 1), ru, rv, rp);
  if (ok) {
    d[n] = (pt & kPatVDir) ? T(0) : bu - ru;
    d[L.nn + n] = (pt & kPatVDir) ? T(0) : bv - rv;
    d[2 * L.nn + n] = (pt & kPatPFix) ? T(0) : bp - rp;
  }
  __syncwarp();
}

}  // namespace dnnmg

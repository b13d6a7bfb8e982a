// Direct solve on the coarsest multigrid level: launchers of the assembly,
// banded LU, explicit inverse and the dense solve (bodies in coarse_body.cuh).
#include <cooperative_groups.h>
#include <cstdio>
#include <type_traits>

#include "coarse_body.cuh"
#include "kernels.h"
#include "recip.cuh"

namespace cg = cooperative_groups;

namespace dnnmg {

namespace {

// 61 us per assembly with one thread per row (7 of the 152 SMs had a block).
__global__ void __launch_bounds__(128)
    assemble_kernel(Grid g, Sten<double> s, const double* __restrict__ vb, double* __restrict__ ab,
                    const __grid_constant__ PatchPieces pp, int use_pieces) {
  assemble_entry(g, s, vb, ab, blockIdx.x * blockDim.x + threadIdx.x, use_pieces ? &pp : nullptr);
}

void launch_assemble(const Grid& g, const Sten<double>& s, const double* vb, double* ab,
                     const PatchPieces* pp, cudaStream_t st) {
  static const PatchPieces none{};
  const Band bd = band_of(g);
  cudaMemsetAsync(ab, 0, sizeof(double) * (size_t)bd.n * bd.W, st);
  note_launch();
  assemble_kernel<<<cdiv(bd.n * 100, 128), 128, 0, st>>>(g, s, vb, ab, pp ? *pp : none, pp ? 1 : 0);
}

// ---- inverse by elimination of node columns ---------------------------------------
//
// With the unknowns of one grid column (x = const) as a block of 27, the
// matrix is block tridiagonal after the odd columns are eliminated: an odd
// column couples to its two neighbours only, and the stabilisation reaches from
// an even column to the next even ones.  Eliminating every other remaining
// column leaves a block tridiagonal matrix again, so six levels (strides 1, 2,
// .. 32) reduce the 33 columns to one; going back, each level's blocks of the
// inverse follow from the level above:
//   eliminated column i between i - s and i + s, Z = D_i^-1,
//     P = -Z A(i, i-s), Q = -Z A(i, i+s), RP = -A(i-s, i) Z, RQ = -A(i+s, i) Z,
//   inverse blocks  X(i, j) = P X(i-s, j) + Q X(i+s, j)   (j kept)
//                   X(j, i) = X(j, i-s) RP + X(j, i+s) RQ
//                   X(i, k) = [i = k] Z + X(i, k-s) RP_k + X(i, k+s) RQ_k.
// The 27 x 27 blocks are inverted by Gauss-Jordan elimination with partial
// pivoting, one thread block each.  Every level is a handful of grid-wide
// phases instead of a chain of 891 columns: a banded LU of the whole matrix on
// one cluster takes 1,843 us and its inverse 647 us, both set by dependent
// FP64 operations on few SMs; this takes 369 us, of which the seven levels of
// block inverses 137 and the last level's products 90.  The blocks are regular because the velocity
// part of the Jacobian and the stabilisation are positive on any set of
// columns; a check at the end (componentwise backward error of one product,
// tolerance kInvTol) asks for the banded LU where rounding has grown all the
// same (strong convection at large time steps), and contexts with part-solid
// patches, whose blocks can be singular, take the LU from the start.
// Against the exact inverse both are off by 1e-14 to 8e-13 over nu = 0.004 ..
// 0.02, dt = 0.005 .. 0.02 (means 2.3e-13 LU, 2.2e-13 here).
constexpr int kCB = 27, kCBB = kCB * kCB;
constexpr int kInvThreads = 512;
constexpr int kGjWarps = 8;   // warps that invert a block together
constexpr double kInvTol = 2e-12;
enum { kBlkD, kBlkL, kBlkU, kBlkL2, kBlkU2, kBlkC1, kBlkC2, kBlkZ, kBlkP, kBlkQ, kBlkRP, kBlkRQ, kBlkKinds };

__host__ __device__ inline bool columns_supported(const Grid& g) { return 3 * g.nny == kCB; }
__host__ __device__ inline size_t column_blocks_doubles(const Grid& g) {
  return (size_t)kBlkKinds * g.nnx * kCBB + 2 * (size_t)band_of(g).n;
}

// Invert the 27 x 27 block whose entry (r, c) is load(r, c) into out (row
// stride ldo).  The first kGjWarps warps of the block: lane r of warp w holds
// the entries (r, w), (r, w + kGjWarps), ...  Column k's warp picks the pivot row (largest magnitude by the
// high words, which order like the doubles; rows are never swapped) and
// publishes the multipliers (every FP64 instruction of a warp takes 64 cycles
// of its scheduler, so the reciprocal is formed once).
template <class F>
__device__ __forceinline__ void invert_column_block(F load, double* out, int ldo, int* bad) {
  __shared__ double mult[2][32];
  __shared__ int pc[kCB];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  constexpr int NC = (kCB + kGjWarps - 1) / kGjWarps;
  double a[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q)
    a[q] = lane < kCB && w + kGjWarps * q < kCB ? load(lane, w + kGjWarps * q) : 0.0;
  bool used = lane >= kCB;
  int my = 0;
#pragma unroll
  for (int kq = 0; kq < NC; ++kq)
#pragma unroll 1
    for (int kw = 0; kw < kGjWarps; ++kw) {
      const int k = kGjWarps * kq + kw;
      if (k >= kCB) break;
      if (kw == w) {
        const unsigned key = used ? 0u : (unsigned)(__double2hiint(a[kq]) & 0x7FFFFFFF);
        const unsigned mx = __reduce_max_sync(0xffffffffu, key);
        const int p = max(0, __ffs(__ballot_sync(0xffffffffu, key == mx && !used)) - 1);
        const double ip = recip64(__shfl_sync(0xffffffffu, a[kq], p));
        mult[k & 1][lane] = lane == p ? ip : -a[kq] * ip;
        if (lane == 0) {
          pc[k] = p;
          if (mx == 0u) *bad = 1;
        }
      }
      asm volatile("bar.sync 1, %0;" ::"n"(32 * kGjWarps) : "memory");
      const int p = pc[k];
      const bool piv = lane == p;
      const double m = mult[k & 1][lane];
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        const double ap = __shfl_sync(0xffffffffu, a[q], p);
        if (q != kq || kw != w) a[q] = fma(m, ap, piv ? 0.0 : a[q]);
      }
      if (kw == w) a[kq] = m;
      if (piv) used = true, my = k;
    }
  if (lane >= kCB) return;
#pragma unroll
  for (int q = 0; q < NC; ++q)
    if (w + kGjWarps * q < kCB) out[(size_t)my * ldo + pc[w + kGjWarps * q]] = a[q];
}

// A product of blocks: out = sign (init + M N [+ M2 N2]) with the row strides
// below (M2, init may be null).  One warp forms an 8 x 8 tile of it with FP64
// tensor instructions, whose rate is that of the scalar ones here but which
// take a twentieth of the instructions (with scalar multiply-adds and
// shuffles a product's code did not fit the instruction cache beside the
// rest, and its instructions took longer to arrive than its operands).  All
// loads go out first: another SM has just written the blocks.
struct Prod {
  const double *M, *N, *M2, *N2, *init;
  double* out;
  int ldm, ldn, ldm2, ldn2, ldi, ldo;
  double sign;
};
constexpr int kCT = (kCB + 7) / 8, kTiles = kCT * kCT, kCK = (kCB + 3) / 4;
__device__ __forceinline__ void block_tile(const Prod& P, int tile, int lane) {
  const int r = tile / kCT * 8 + (lane >> 2), c = tile % kCT * 8 + (lane >> 2), q = lane & 3;
  double m[2][kCK], v[2][kCK];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const double *M = h ? P.M2 : P.M, *N = h ? P.N2 : P.N;
    const size_t ldm = h ? P.ldm2 : P.ldm, ldn = h ? P.ldn2 : P.ldn;
#pragma unroll
    for (int k = 0; k < kCK; ++k) {
      const int e = 4 * k + q;
      m[h][k] = M && r < kCB && e < kCB ? M[r * ldm + e] : 0.0;
      v[h][k] = M && c < kCB && e < kCB ? N[e * ldn + c] : 0.0;
    }
  }
  const int co = tile % kCT * 8 + 2 * q;
  double d[2];
#pragma unroll
  for (int e = 0; e < 2; ++e)
    d[e] = P.init && r < kCB && co + e < kCB ? P.init[(size_t)r * P.ldi + co + e] : 0.0;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (h && !P.M2) break;
#pragma unroll
    for (int k = 0; k < kCK; ++k)
      asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                   : "+d"(d[0]), "+d"(d[1])
                   : "d"(m[h][k]), "d"(v[h][k]));
  }
#pragma unroll
  for (int e = 0; e < 2; ++e)
    if (r < kCB && co + e < kCB) P.out[(size_t)r * P.ldo + co + e] = P.sign * d[e];
}

__global__ void __launch_bounds__(kInvThreads, 1)
    column_inverse_kernel(Grid g, const double* __restrict__ ab, double* blk, double* X,
                          int* need_lu) {
  cg::grid_group grid = cg::this_grid();
  const Band bd = band_of(g);
  const int nc = g.nnx, n = bd.n, kl = bd.kl;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kWarps = kInvThreads / 32;
  const int gt = blockIdx.x * kInvThreads + tid, ngt = gridDim.x * kInvThreads;
  auto B = [&](int kind, int i) { return blk + ((size_t)kind * nc + i) * kCBB; };
  auto A = [&](int r, int c) {  // entry of the assembled band
    const int o = c - r + kl;
    return o >= 0 && o <= 2 * kl ? ab[(size_t)r * bd.W + o] : 0.0;
  };
  // items [0, total) in contiguous runs of a block, one warp per item
  auto for_items = [&](int total, auto f) {
    const int per = cdiv(total, gridDim.x), i0 = blockIdx.x * per, i1 = min(total, i0 + per);
    for (int t = i0 + warp; t < i1; t += kWarps) f(t);
  };
  if (gt == 0) *need_lu = 0;
  for (int e = gt; e < nc * kCBB; e += ngt) {
    const int i = e / kCBB, r = e % kCBB / kCB, c = e % kCB;
    B(kBlkD, i)[e % kCBB] = A(kCB * i + r, kCB * i + c);
    if (i > 0) B(kBlkL, i)[e % kCBB] = A(kCB * i + r, kCB * (i - 1) + c);
    if (i + 1 < nc) B(kBlkU, i)[e % kCBB] = A(kCB * i + r, kCB * (i + 1) + c);
    if (i > 1) B(kBlkL2, i)[e % kCBB] = A(kCB * i + r, kCB * (i - 2) + c);
    if (i + 2 < nc) B(kBlkU2, i)[e % kCBB] = A(kCB * i + r, kCB * (i + 2) + c);
  }
  grid.sync();
  // D_i with the contributions of the columns eliminated at stride h on both sides
  auto diag = [&](int i, int h, int e) {
    double v = B(kBlkD, i)[e];
    if (h > 0) {
      if (i > 0) v += B(kBlkC1, i)[e];
      if (i + h < nc) v += B(kBlkC2, i)[e];
    }
    return v;
  };
  int s = 1;
  auto XB = [&](int i, int j) { return X + (size_t)(kCB * i) * n + kCB * j; };
  // The products of a phase of stride s, one 8 x 8 tile per warp:
  //   0: P, Q, RP, RQ of the eliminated columns
  //   1: the kept neighbours' contributions to D and couplings to the next kept
  //   2: X(eliminated, kept), X(kept, eliminated)     3: X(eliminated, eliminated)
  auto run_phase = [&](int phase) {
    const int ne = (nc + s - 1) / (2 * s), nk = (nc + 2 * s - 1) / (2 * s);
    const int total = phase < 2 ? 4 * ne : (phase == 2 ? 2 * ne * nk : ne * ne);
    for_items(total * kTiles, [&](int t) {
      const int u = t / kTiles;
      Prod P{};
      P.sign = 1.0;
      P.ldm = P.ldn = P.ldm2 = P.ldn2 = P.ldi = P.ldo = kCB;
      if (phase < 2) {
        // even kinds towards the left neighbour j, odd kinds towards the right
        const int i = s + 2 * s * (u >> 2), kind = u & 3, side = kind & 1;
        const int j = side ? i + s : i - s;
        if (side && j >= nc) return;
        double *L = B(kBlkL, i), *U = B(kBlkU, i), *C = B(side ? kBlkL : kBlkU, j);
        if (phase == 0) {
          P.sign = -1.0;
          if (kind < 2)
            P.M = B(kBlkZ, i), P.N = side ? U : L, P.out = B(side ? kBlkQ : kBlkP, i);
          else
            P.M = C, P.N = B(kBlkZ, i), P.out = B(side ? kBlkRQ : kBlkRP, i);
        } else {
          P.M = B(side ? kBlkRQ : kBlkRP, i);
          if (kind < 2) {
            P.N = side ? U : L, P.out = B(side ? kBlkC1 : kBlkC2, j);
          } else {
            if (i + s >= nc) return;
            P.N = side ? L : U, P.out = C;
            // the coupling of two even columns that the matrix itself holds
            if (s == 1) P.init = B(side ? kBlkL2 : kBlkU2, j);
          }
        }
      } else {
        P.ldo = n;
        const int j = phase == 2 ? 2 * s * (u % nk) : 0, e = phase == 2 ? u / nk : u;
        const int i = s + 2 * s * (e % ne);
        if (phase == 2 && e < ne) {  // X(i, j)
          P.M = B(kBlkP, i), P.N = XB(i - s, j), P.ldn = n;
          if (i + s < nc) P.M2 = B(kBlkQ, i), P.N2 = XB(i + s, j), P.ldn2 = n;
          P.out = XB(i, j);
        } else {  // X(a, i), a kept or eliminated
          const int a = phase == 2 ? j : s + 2 * s * (e / ne);
          if (a == i) P.init = B(kBlkZ, i);
          P.M = XB(a, i - s), P.N = B(kBlkRP, i), P.ldm = n;
          if (i + s < nc) P.M2 = XB(a, i + s), P.N2 = B(kBlkRQ, i), P.ldm2 = n;
          P.out = XB(a, i);
        }
      }
      block_tile(P, t % kTiles, lane);
    });
    grid.sync();
  };
  // down: levels of stride 1, 2, ..; the last "level" is column 0 alone
  for (;; s *= 2) {
    const bool last = s >= nc;
    const int ne = last ? 1 : (nc + s - 1) / (2 * s);  // columns s, 3 s, ..
    if ((int)blockIdx.x < ne) {
      const int i = last ? 0 : s + 2 * s * (int)blockIdx.x;
      if (tid < 32 * kGjWarps)
        invert_column_block([&](int r, int c) { return diag(i, s / 2, r * kCB + c); },
                            last ? X : B(kBlkZ, i), last ? n : kCB, need_lu);
    } else if (s > 1 && !last) {  // kept columns 0, 2 s, ..: add the contributions
      const int nk = (nc + 2 * s - 1) / (2 * s);
      for (int e = ((int)blockIdx.x - ne) * kInvThreads + tid; e < nk * kCBB;
           e += ((int)gridDim.x - ne) * kInvThreads) {
        const int j = 2 * s * (e / kCBB);
        B(kBlkD, j)[e % kCBB] = diag(j, s / 2, e % kCBB);
      }
    }
    grid.sync();
    if (last) break;
    run_phase(0);
    run_phase(1);
  }
  for (s /= 2; s >= 1; s /= 2) {  // and back
    run_phase(2);
    run_phase(3);
  }
  // y = X b for a vector of signs, then the componentwise backward error of A y = b
  double* y = blk + (size_t)kBlkKinds * nc * kCBB;
  auto sign = [](int k) { return ((unsigned)k * 2654435761u >> 17) & 1u ? 1.0 : -1.0; };
  for_items(n, [&](int r) {
    double acc = 0.0;
    for (int c = lane; c < n; c += 32) acc = fma(X[(size_t)r * n + c], sign(c), acc);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) y[r] = acc;
  });
  grid.sync();
  for_items(n, [&](int r) {
    double res = 0.0, mag = 0.0;
    for (int c = max(0, r - kl) + lane; c <= min(n - 1, r + kl); c += 32) {
      const double v = A(r, c) * y[c];
      res += v;
      mag += fabs(v);
    }
    for (int o = 16; o > 0; o >>= 1) {
      res += __shfl_xor_sync(0xffffffffu, res, o);
      mag += __shfl_xor_sync(0xffffffffu, mag, o);
    }
    if (lane == 0 && !(fabs(res - sign(r)) <= kInvTol * (mag + 1.0))) *need_lu = 1;
  });
}

__global__ void __launch_bounds__(kLUThreads)
    band_lu_kernel(Grid g, double* __restrict__ ab, int* __restrict__ piv, int* status,
                   const int* need) {
  if (need && !*need) return;
  extern __shared__ double win[];  // kWin * W
  band_lu_block(g, ab, piv, status, win);
}

// The same banded LU (dgbtf2 ordering, partial pivoting, lowest row on
// ties, multipliers in place) by a cluster of kLUCluster CTAs.  The columns
// are dealt to the CTAs in panels of two (panel j = columns 2j, 2j + 1 in
// CTA j % kLUCluster) and stay in its shared memory for the whole
// factorisation, entry (r, c) at position r - c + ku + kl of the column (the
// kl subdiagonals, the diagonal and the ku + kl superdiagonals of U with
// fill-in).  Warp 0 of a panel's owner factors it: pivot of the first
// column, its step applied to the second column, pivot of the second; it
// writes both pivots and multiplier columns into every CTA's shared memory
// (double-buffered by panel parity).  After one cluster barrier per panel,
// every CTA applies the panel's two steps (row interchange, rank-1 update) to
// its columns right of the panel, one warp per column; the next panel's
// owner does its own panel columns first (warp 0) and factors them while its
// other warps finish.  Every entry sees the same floating-point operations
// in the same order as in band_lu_block, so the factors are the same.
constexpr int kLUCluster = 8;
constexpr int kLUCThreads = 256;

__host__ __device__ inline int lu_cluster_cols(const Band& b) {
  const int panels = (b.n + 1) / 2;
  return 2 * ((panels + kLUCluster - 1) / kLUCluster);
}
__host__ __device__ inline size_t lu_cluster_smem(const Band& b) {
  return sizeof(double) * ((size_t)lu_cluster_cols(b) * b.W + 4 * (b.kl + 1)) + 4 * sizeof(int);
}

__device__ __forceinline__ void cl_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cl_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

__global__ void __launch_bounds__(kLUCThreads)
    band_lu_cluster_kernel(Grid g, double* __restrict__ ab, int* __restrict__ piv, int* status,
                           const int* need) {
  if (need && !*need) return;  // every block of the cluster reads the same word
  cg::cluster_group cl = cg::this_cluster();
  const Band bd = band_of(g);
  const int q = (int)cl.block_rank();
  const int n = bd.n, kl = bd.kl, KU2 = bd.ku + bd.kl, W = bd.W;
  const int ncl = lu_cluster_cols(bd);
  const int NP = (n + 1) / 2;  // panels
  extern __shared__ __align__(16) double lsm[];
  double* cols = lsm;                                  // [ncl][W]
  double* mult = lsm + (size_t)ncl * W;                // [2 parity][2 step][kl + 1]
  int* pv = reinterpret_cast<int*>(mult + 4 * (kl + 1));  // [2 parity][2 step]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kWarps = kLUCThreads / 32;
  // local slot of (owned) column c: panel c / 2 is the (c / 2 / kLUCluster)-th of this CTA
  auto slot = [&](int c) { return ((c >> 1) / kLUCluster) * 2 + (c & 1); };
  auto A = [&](int r, int c) -> double& { return cols[(size_t)slot(c) * W + (r - c + KU2)]; };
  auto col_of = [&](int lc) { return ((lc >> 1) * kLUCluster + q) * 2 + (lc & 1); };
  // this CTA's columns from the row-major band: (r, c) at ab[r W + c - r + kl]
  for (int e = tid; e < ncl * W; e += kLUCThreads) {
    const int lc = e / W, t = e % W;
    const int c = col_of(lc), r = c - KU2 + t;
    cols[e] = (c < n && r >= 0 && r < n) ? ab[(size_t)r * W + (W - 1 - t)] : 0.0;
  }
  __syncthreads();
  // step k applied to column c (one warp): rows k and p interchanged, then
  // rows k+1 .. k+kl minus multiplier times the new row-k entry
  auto apply = [&](int k, int p, const double* m, int c) {
    const double a = A(k, c), b = A(p, c);
    __syncwarp();
    if (lane == 0 && p != k) {
      A(k, c) = b;
      A(p, c) = a;
    }
    __syncwarp();
    const int rmax = min(n - 1, k + kl);
    for (int r = k + 1 + lane; r <= rmax; r += 32) A(r, c) -= m[r - k - 1] * b;
    __syncwarp();
  };
  // pivot of column k (owned here, up to date): |entries| compared as the
  // bit patterns of non-negative doubles (the same order), lowest row on
  // ties; multipliers in place and into slot `sl` of every CTA.  One warp.
  auto pivot = [&](int k, double* mloc, int sl) {
    const int rmax = min(n - 1, k + kl);
    long long best = -1;
    int bi = k;
    for (int r = k + lane; r <= rmax; r += 32) {
      const long long v = __double_as_longlong(A(r, k)) & 0x7FFFFFFFFFFFFFFFLL;
      if (v > best) best = v, bi = r;
    }
    for (int o = 16; o > 0; o >>= 1) {
      const long long ov = __shfl_down_sync(0xffffffffu, best, o);
      const int oi = __shfl_down_sync(0xffffffffu, bi, o);
      if (ov > best || (ov == best && oi < bi)) best = ov, bi = oi;
    }
    const int p = __shfl_sync(0xffffffffu, bi, 0);
    best = __shfl_sync(0xffffffffu, best, 0);
    const double d = A(p, k), akk = A(k, k);
    const double id = d != 0.0 ? 1.0 / d : 0.0;
    __syncwarp();
    for (int r = k + 1 + lane; r <= rmax; r += 32) {
      const double m = (r == p ? akk : A(r, k)) * id;
      A(r, k) = m;
      mloc[r - k - 1] = m;
      for (int dst = 0; dst < kLUCluster; ++dst)
        if (dst != q) cl.map_shared_rank(mloc, dst)[r - k - 1] = m;
    }
    if (lane == 0) {
      A(k, k) = d;
      piv[k] = p;
      pv[sl] = p;
      for (int dst = 0; dst < kLUCluster; ++dst)
        if (dst != q) cl.map_shared_rank(pv, dst)[sl] = p;
      if (!(best > 0)) atomicOr(status, 2);
    }
    __syncwarp();
    return p;
  };
  // panel j by warp 0 of its owner: columns 2j (and 2j + 1)
  auto factor_panel = [&](int j) {
    const int k = 2 * j, par = j & 1;
    double* m0 = mult + (size_t)(2 * par) * (kl + 1);
    const int p0 = pivot(k, m0, 2 * par);
    if (k + 1 < n) {
      apply(k, p0, m0, k + 1);
      pivot(k + 1, m0 + (kl + 1), 2 * par + 1);
    }
  };
  if (q == 0 && warp == 0) factor_panel(0);
  cl_arrive();
  for (int J = 0; J < NP; ++J) {
    cl_wait();  // pivots and multipliers of panel J are in buffer J & 1
    const int k0 = 2 * J, par = J & 1;
    const double* m0 = mult + (size_t)(2 * par) * (kl + 1);
    const double* m1 = m0 + (kl + 1);
    const int p0 = pv[2 * par], p1 = pv[2 * par + 1];
    const bool two = k0 + 1 < n;
    // columns right of the panel that its steps reach: (k0 + 1, cmax]
    const int cmax = min(n - 1, (two ? k0 + 1 : k0) + KU2);
    auto both = [&](int c) {
      if (c <= k0 + KU2) apply(k0, p0, m0, c);
      if (two) apply(k0 + 1, p1, m1, c);
    };
    // this CTA's panels j in [J + 1, cmax / 2]
    const int j0 = J + 1, j1 = cmax >> 1;
    const int jf = j0 + ((q - j0 % kLUCluster) + kLUCluster) % kLUCluster;  // first owned
    const bool next_owner = J + 1 < NP && jf == J + 1;
    if (next_owner && warp == 0) {  // the next panel first, then factor it
      both(k0 + 2);
      if (k0 + 3 <= cmax) both(k0 + 3);
      factor_panel(J + 1);
    }
    // the other owned columns, one warp each
    const int w0 = next_owner ? 1 : 0;
    int idx = 0;  // running index over the owned columns (next panel excluded)
    for (int j = next_owner ? jf + kLUCluster : jf; j <= j1; j += kLUCluster)
      for (int h = 0; h < 2; ++h, ++idx) {
        const int c = 2 * j + h;
        if (c > cmax) break;
        if (warp >= w0 && idx % (kWarps - w0) == warp - w0) both(c);
      }
    cl_arrive();
  }
  cl_wait();
  // the factored columns back into the row-major band
  for (int e = tid; e < ncl * W; e += kLUCThreads) {
    const int lc = e / W, t = e % W;
    const int c = col_of(lc), r = c - KU2 + t;
    if (c < n && r >= 0 && r < n) ab[(size_t)r * W + (W - 1 - t)] = cols[e];
  }
}

__global__ void diag_recip_kernel(Grid g, const double* __restrict__ ab, double* __restrict__ rd,
                                  const int* need) {
  if (need && !*need) return;
  band_diag_recip(g, ab, rd, blockIdx.x * blockDim.x + threadIdx.x);
}

// Columns [kInvWarps * block, +kInvWarps) of the inverse.
__global__ void __launch_bounds__(32 * kInvWarps)
    band_inverse_kernel(Grid g, const double* __restrict__ ab, const int* __restrict__ piv,
                        const double* __restrict__ rd, double* __restrict__ Ainv,
                        const int* need) {
  if (need && !*need) return;
  extern __shared__ __align__(16) double sm[];
  band_inverse_block(g, ab, piv, rd, Ainv, blockIdx.x * kInvWarps, sm);
}

// x = Ainv b with the band numbering on both sides; one warp per row.
template <typename T>
__global__ void __launch_bounds__(32 * kSolveWarps)
    coarse_solve_kernel(Grid g, const double* __restrict__ Ainv, const T* __restrict__ b,
                        T* __restrict__ x) {
  extern __shared__ double sb[];
  coarse_solve_rows<T>(g, Ainv, b, x, blockIdx.x, sb);
}

// x = (LU)^{-1} b with the factors and pivots of band_lu_kernel; one block,
// b and x in the [3][nn] layout of the level, work in shared memory.
__global__ void __launch_bounds__(1024)
    band_solve_kernel(Grid g, const double* __restrict__ ab, const int* __restrict__ piv,
                      const double* __restrict__ b, double* __restrict__ x) {
  const Band bd = band_of(g);
  extern __shared__ double sx[];
  const int tid = threadIdx.x;
  for (int p = tid; p < bd.n; p += blockDim.x) sx[p] = b[lidx(g, p)];
  __syncthreads();
  for (int k = 0; k < bd.n; ++k) {
    const int p = piv[k];
    if (tid == 0 && p != k) {
      const double t = sx[k];
      sx[k] = sx[p];
      sx[p] = t;
    }
    __syncthreads();
    const double xk = sx[k];
    const int rmax = min(bd.n - 1, k + bd.kl);
    for (int r = k + 1 + tid; r <= rmax; r += blockDim.x)
      sx[r] -= ab[(size_t)r * bd.W + (k - r + bd.kl)] * xk;
    __syncthreads();
  }
  __shared__ double red[32];
  for (int k = bd.n - 1; k >= 0; --k) {
    const int cmax = min(bd.n - 1, k + bd.ku + bd.kl);
    double acc = 0.0;
    for (int c2 = k + 1 + tid; c2 <= cmax; c2 += blockDim.x)
      acc += ab[(size_t)k * bd.W + (c2 - k + bd.kl)] * sx[c2];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((tid & 31) == 0) red[tid >> 5] = acc;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
      sx[k] = (sx[k] - t) / ab[(size_t)k * bd.W + bd.kl];
    }
    __syncthreads();
  }
  for (int p = tid; p < bd.n; p += blockDim.x) x[lidx(g, p)] = sx[p];
}

// Banded LU of the assembled coarse Jacobian: the cluster kernel when a
// cluster of kLUCluster CTAs with its shared memory can be placed, else the
// single-block kernel.
void launch_band_lu(const Grid& g, double* ab, int* piv, int* status, const int* need,
                    cudaStream_t st) {
  const Band bd = band_of(g);
  const size_t csm = lu_cluster_smem(bd);
  // whether the cluster can be placed, checked once per process (thread-safe
  // initialisation of a function-local static)
  static const int cluster_ok = [&] {
    int ok = 0;
    if (csm <= 227 * 1024 &&
        cudaFuncSetAttribute(band_lu_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             227 * 1024) == cudaSuccess) {
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = kLUCluster;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.gridDim = dim3(kLUCluster);
      cfg.blockDim = dim3(kLUCThreads);
      cfg.dynamicSmemBytes = csm;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, (void*)band_lu_cluster_kernel, &cfg) == cudaSuccess &&
          n > 0)
        ok = 1;
    }
    cudaGetLastError();
    return ok;
  }();
  if (cluster_ok == 1 && csm <= 227 * 1024) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kLUCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(kLUCluster);
    cfg.blockDim = dim3(kLUCThreads);
    cfg.dynamicSmemBytes = csm;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    note_launch();
    if (cudaLaunchKernelEx(&cfg, band_lu_cluster_kernel, g, ab, piv, status, need) == cudaSuccess) return;
    cudaGetLastError();
  }
  const size_t win_bytes = sizeof(double) * kWin * bd.W;
  cudaFuncSetAttribute(band_lu_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)win_bytes);
  note_launch();
  band_lu_kernel<<<1, kLUThreads, win_bytes, st>>>(g, ab, piv, status, need);
}

}  // namespace

size_t coarse_band_doubles(const Grid& g) {
  const Band bd = band_of(g);
  return (size_t)bd.n * bd.W;
}

void launch_coarse_lu(const Grid& g, const Sten<double>& s, const double* vb, double* band,
                      int* piv, int* status, cudaStream_t st) {
  launch_assemble(g, s, vb, band, nullptr, st);
  launch_band_lu(g, band, piv, status, nullptr, st);
}

void launch_coarse_lu_solve(const Grid& g, const double* band, const int* piv, const double* b,
                            double* x, cudaStream_t st) {
  const Band bd = band_of(g);
  note_launch();
  band_solve_kernel<<<1, 1024, sizeof(double) * bd.n, st>>>(g, band, piv, b, x);
}

bool coarse_supported(const Grid& g) {
  const Band bd = band_of(g);
  return bd.kl + 2 <= kWin && bd.W <= kLUThreads && sizeof(double) * kWin * bd.W <= 200 * 1024 &&
         bd.kl <= 64 && bd.ku + bd.kl <= 128 &&  // L and U entries of a step per lane
         sizeof(double) * inv_block_smem_doubles(bd.n) <= 200 * 1024;
}

size_t coarse_work_doubles(const Grid& g) {
  const Band bd = band_of(g);
  // band + pivots (as ints, over-allocated) + reciprocals of the U diagonal
  return (size_t)bd.n * bd.W + (size_t)bd.n + (size_t)bd.n;
}

size_t coarse_factor_doubles(const Grid& g) {
  return coarse_work_doubles(g) + (columns_supported(g) ? column_blocks_doubles(g) + 1 : 0);
}

const int* launch_coarse_factor(const Grid& g, const Sten<double>& s, const double* vb,
                                double* work, double* Ainv, int* status, cudaStream_t st,
                                const PatchPieces* pp) {
  const Band bd = band_of(g);
  double* ab = work;
  int* piv = reinterpret_cast<int*>(work + (size_t)bd.n * bd.W);
  launch_assemble(g, s, vb, ab, pp, st);
  // the inverse by node columns where the grid can be resident; the banded LU
  // then runs only when that asks for it
  const int* need = nullptr;
  static const int blocks = [] {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, column_inverse_kernel, kInvThreads,
                                                      0) != cudaSuccess)
      per = 0;
    cudaGetLastError();
    return per > 0 ? sms : 0;
  }();
  if (!pp && columns_supported(g) && blocks > g.nnx) {
    double* blk = work + coarse_work_doubles(g);
    int* flag = reinterpret_cast<int*>(blk + column_blocks_doubles(g));
    Grid gc = g;
    const double* abc = ab;
    void* args[] = {(void*)&gc, (void*)&abc, (void*)&blk, (void*)&Ainv, (void*)&flag};
    note_launch();
    if (cudaLaunchCooperativeKernel((void*)column_inverse_kernel, dim3(blocks), dim3(kInvThreads),
                                    args, 0, st) == cudaSuccess)
      need = flag;
    else
      cudaGetLastError();
  }
  launch_band_lu(g, ab, piv, status, need, st);
  double* rd = work + (size_t)bd.n * bd.W + bd.n;
  note_launch();
  diag_recip_kernel<<<cdiv(bd.n, 128), 128, 0, st>>>(g, ab, rd, need);
  const size_t smem = sizeof(double) * inv_block_smem_doubles(bd.n);
  static const bool inv_attr =
      cudaFuncSetAttribute(band_inverse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem) == cudaSuccess;
  (void)inv_attr;
  note_launch();
  band_inverse_kernel<<<cdiv(bd.n, kInvWarps), 32 * kInvWarps, smem, st>>>(g, ab, piv, rd, Ainv,
                                                                           need);
  return need;
}

template <typename T>
void launch_coarse_solve(const Grid& g, const double* Ainv, const T* b, T* x, cudaStream_t st) {
  const Band bd = band_of(g);
  note_launch();
  coarse_solve_kernel<T><<<cdiv(bd.n, kSolveWarps), 32 * kSolveWarps, sizeof(double) * bd.n, st>>>(
      g, Ainv, b, x);
}

template void launch_coarse_solve<float>(const Grid&, const double*, const float*, float*,
                                         cudaStream_t);
template void launch_coarse_solve<double>(const Grid&, const double*, const double*, double*,
                                          cudaStream_t);

}  // namespace dnnmg

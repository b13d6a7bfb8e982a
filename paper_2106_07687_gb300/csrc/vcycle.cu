// One V(nu1, nu2) cycle in a single persistent launch: a cooperative grid,
// or one thread-block cluster (up to 16 blocks on 16 SMs).
//
// The cycle (Sec. 2.2: multigrid as the GMRES preconditioner) is a fixed
// sequence of phases -- Vanka colour passes, defect, restriction (with the
// coarse iterate zeroed), the coarse direct solve, prolongation -- built once
// per top level on the host.  The kernel walks the phase list; all blocks
// share every phase.
//
// A phase is bound by its dependent chain (barrier, loads from L2, rows,
// products, stores), not by bandwidth, on all but the largest levels.  Colour
// passes and defects therefore work from assembled coefficients, one warp per
// 8 x 4 nodes and without a block barrier, and the iterate's values carry the
// number of their update, so that a tile waits for its own inputs only
// (vnode.cuh).  Barriers (grid-wide, or the hardware cluster barrier) remain
// after the defect, the restriction and the coarse solve, whose outputs are
// plain arrays.  One cycle, barriers after every phase -> numbered updates: FP32
// on levels 3 / 5 / 6 (128x32, 512x128, 1024x256 cells) 92 -> 82, 244 -> 185,
// 528 -> 430 us (72, 168, 407 us since), FP64 on level 3 191 -> 154 us (151).
#include <algorithm>
#include <cooperative_groups.h>

#include "kernels.h"
#include "vbody.cuh"
#include "vcycle.h"

namespace cg = cooperative_groups;

namespace dnnmg {

namespace {

constexpr int kMaxPhases = 160;  // phases of one launch (a V(2,2) cycle from level 8)
constexpr int kMaxVLevels = 10;

// What a colour pass or defect reads of its phase and level, resolved once per
// launch: a phase is a chain of dependent steps, and looking its level up,
// dividing by its tile counts and rounding its mesh width took 700 of its 4,400
// cycles (FP32; one cycle on 512x128 cells 180 -> 168 us).
template <typename T>
struct alignas(16) PassRec {
  int type, colour;
  int nx, ny, nnx, nn, pitch, nslots;
  int tiles, nbx;      // warp tiles, and how many in a row
  unsigned inv_nbx;    // 2^32 / nbx, rounded up (nbx > 1): t / nbx for t nbx < 2^32
  int split;           // four lanes per node
  unsigned tin, tout;
  T h, h2;
  const T *b, *inv, *cf;
  const uint16_t* pat;
  const ulonglong2* in;
  ulonglong2* out;
  T *planar, *d;
};

// Dynamic shared memory of a block: the launch's phase list, level records
// and coefficient table, loaded once so that no phase starts with a dependent
// global load, and a scratch area for the warp tiles or the coarse vector.
template <typename T>
struct WalkSmem {
  OpTable<T> tab;
  VLevel<T> lv[kMaxVLevels];
  Phase ph[kMaxPhases];
  PassRec<T> rec[kMaxPhases];
  alignas(16) WarpTile<T> tile[walk_threads<T>() / 32];
};

// Item n < count of a node-wise phase for every thread of the grid: chunks
// of 32 consecutive items (one warp, coalesced) go round-robin over the
// blocks first, so that a small level still spreads over all of them.
template <int NT, class F>
__device__ __forceinline__ void for_items(int count, F f) {
  constexpr int kWarps = NT / 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nchunks = (count + 31) >> 5;
  for (int c = blockIdx.x + gridDim.x * w; c < nchunks; c += gridDim.x * kWarps) {
    const int n = (c << 5) + lane;
    if (n < count) f(n);
  }
}

// Walk the phase list; `sync` separates the phases whose outputs are plain
// arrays (a grid-wide barrier for the cooperative launch, the cluster barrier for
// the single-cluster launch).  Threads of all blocks split every node-wise
// phase; the warp tiles of a colour pass or defect go round-robin over the
// blocks first.  state: see launch_vcycle_persistent.
template <typename T, class Sync>
__device__ __forceinline__ void walk_phases(const VLevel<T>* glv, const OpTable<T>* gtab,
                                            const Phase* gph, int nph, int top, const T* topb,
                                            T* topx, const double* __restrict__ Ainv, T omega,
                                            int* state, unsigned numbers, int polls,
                                            WalkSmem<T>& S, Sync sync) {
  constexpr int NT = walk_threads<T>();
  double* sbuf = reinterpret_cast<double*>(S.tile);  // the coarse right-hand side
  copy_ints(S.lv, glv, top + 1);
  copy_ints(S.ph, gph, nph);
  copy_ints(&S.tab, gtab, 1);
  const unsigned word = __ldcg(reinterpret_cast<unsigned*>(state) + 1), tag0 = word << 1;
  __syncthreads();
  for (int p = threadIdx.x; p < nph; p += NT) {
    const Phase f = S.ph[p];
    const VLevel<T>& L = S.lv[f.level];
    const Grid& g = L.g;
    PassRec<T> r;
    r.type = f.type, r.colour = f.colour;
    r.nx = g.nx, r.ny = g.ny, r.nnx = g.nnx, r.nn = g.nn;
    r.pitch = vanka_pitch(g), r.nslots = vanka_slots(g);
    // FP64: four lanes per node while that gives every scheduler (four per
    // block) at most little more than one warp.  On 152 blocks that is up to
    // level 3 (612 warps): one cycle with barriers, one -> four lanes per node on
    // levels 2 and 3, 287 -> 191 us on 128x32, 435 -> 339 us on 256x64; with level
    // 4 (2,244 warps) as well 401 us.  In FP32 the same gains 2 us a cycle, but
    // the larger kernel loses 15 (its instructions come through the cache once
    // per phase).
    r.split = sizeof(T) == 8 && 4 * cdiv(g.nnx, kWX) * cdiv(g.nny, kWY) <= 5 * (int)gridDim.x;
    const int sx = r.split ? kSX : kWX, sy = r.split ? kSY : kWY;
    if (f.type == kPhasePass) {
      r.nbx = cdiv(g.nx / 2 + 1, sx / 2);
      r.tiles = r.nbx * cdiv(g.ny / 2 + 1, sy / 2);
    } else {
      r.nbx = cdiv(g.nnx, sx);
      r.tiles = r.nbx * cdiv(g.nny, sy);
    }
    r.inv_nbx = 0xFFFFFFFFu / r.nbx + 1u;
    r.tin = tag0 + f.tin, r.tout = tag0 + f.tout;
    r.h = (T)g.h, r.h2 = (T)(g.h * g.h);
    r.b = f.level == top ? topb : L.b;
    r.inv = L.inv, r.cf = L.cf, r.pat = L.pat;
    const size_t words = (size_t)kTagWords<T> * g.nn;
    r.in = L.xt + f.in * words, r.out = L.xt + f.out * words;
    r.planar = f.last && f.level == top ? topx : nullptr;
    r.d = L.d;
    S.rec[p] = r;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int w0 = blockIdx.x + gridDim.x * w, nw = gridDim.x * (NT / 32);
  int budget = polls;
  for (int p = 0; p < nph; ++p) {
    const PassRec<T>& R = S.rec[p];
    const int type = R.type;
    if (type == kPhasePass || type == kPhaseDefect) {
      const TaggedX<T> x{R.in, R.out, R.planar, R.nn, R.tin, R.tout, state};
      const NodeLevel<T> N{R.nx, R.ny, R.nnx, R.nn, R.pat, R.cf, R.h, R.h2};
      for (int t = w0; t < R.tiles; t += nw) {
        const int by = __umulhi(t, R.inv_nbx), bx = t - by * R.nbx;
        if constexpr (sizeof(T) == 8)
          if (R.split) {
            if (type == kPhasePass)
              split_pass_tile<T>(N, S.tab, R.colour, R.b, x, R.inv, R.pitch, R.nslots, omega, bx,
                                 by, lane, S.tile[w], budget);
            else
              split_defect_tile<T>(N, S.tab, R.b, x, R.d, bx, by, lane, S.tile[w], budget);
            continue;
          }
        if (type == kPhasePass)
          warp_pass_tile<T>(N, S.tab, R.colour, R.b, x, R.inv, R.pitch, R.nslots, omega, bx, by,
                            lane, S.tile[w], budget);
        else
          warp_defect_tile<T>(N, S.tab, R.b, x, R.d, bx, by, lane, S.tile[w], budget);
      }
      if (type == kPhaseDefect) sync();
      continue;
    }
    const Phase f = S.ph[p];
    const int k = f.level;
    const VLevel<T>& L = S.lv[k];
    const Grid& g = L.g;
    const T* b = k == top ? topb : L.b;
    const size_t words = (size_t)kTagWords<T> * g.nn;
    const TaggedX<T> x{L.xt + f.in * words, L.xt + f.out * words, f.last && k == top ? topx : nullptr, g.nn,
                       tag0 + f.tin,        tag0 + f.tout,        state};
    bool barrier = false;
    switch (f.type) {
      case kPhaseRestrict: {
        barrier = true;
        const VLevel<T>& C = S.lv[k - 1];
        const Grid& c = C.g;
        const TaggedX<T> xc{C.xt, C.xt, nullptr, c.nn, tag0, tag0, state};
        for_items<NT>(c.nn, [&](int n) {
          restrict_node<T, true>(g, c, L.d, C.b, 3, n % c.nnx, n / c.nnx);
          if (f.colour == 1 && k > 1) xc.store(n, T(0), T(0), T(0));
        });
        break;
      }
      case kPhasePassZero: {
        // four items per colour cell, warp-sized chunks round-robin over the
        // blocks; every lane of a warp takes part in the cell's shuffles
        const int count = 4 * vanka_slots(g), nchunks = (count + 31) >> 5;
        for (int c = w0; c < nchunks; c += nw) {
          const int e = (c << 5) + lane;
          zero_pass_node<T>(g, f.colour, b, x, L.inv, omega, e, e < count);
        }
        break;
      }
      case kPhaseCoarse: {
        barrier = true;
        T* x0 = k == top ? topx : L.x;
        const int nd = 3 * g.nn;
        for (int q0 = threadIdx.x; q0 < nd; q0 += 4 * NT) {  // four loads in flight
          double v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int q = q0 + u * NT;
            v[u] = q < nd ? (double)b[band_to_level(g, q)] : 0.0;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (q0 + u * NT < nd) sbuf[q0 + u * NT] = v[u];
        }
        __syncthreads();
        // one warp per row, rows round-robin over the blocks first
        for (int r = w0; r < nd; r += nw) {
          const double* row = Ainv + (size_t)r * nd;
          // chunks of 16 entries per lane: every load of a chunk is issued
          // before its products are summed, so that a row of up to 512
          // entries costs one round trip to L2 instead of one per entry
          double acc[4] = {0.0, 0.0, 0.0, 0.0};
          for (int c0 = lane; c0 < nd; c0 += 16 * 32) {
            double rv[16], sv[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) {
              const int c2 = c0 + 32 * u;
              rv[u] = c2 < nd ? row[c2] : 0.0;
              sv[u] = c2 < nd ? sbuf[c2] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < 16; ++u) acc[u & 3] += rv[u] * sv[u];
          }
          double a = (acc[0] + acc[1]) + (acc[2] + acc[3]);
          for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
          if (lane == 0) x0[band_to_level(g, r)] = (T)a;
        }
        break;
      }
      case kPhaseProlong: {
        const VLevel<T>& C = S.lv[k - 1];
        const Grid& c = C.g;
        const TaggedX<T> xc{C.xt + f.cin * (size_t)kTagWords<T> * c.nn, nullptr, nullptr, c.nn,
                            tag0 + f.tcin, 0u, state};
        const int nchunks = (g.nn + 31) >> 5;  // whole warps wait together
        for (int q = w0; q < nchunks; q += nw) {
          const bool valid = (q << 5) + lane < g.nn;
          const int n = valid ? (q << 5) + lane : 0, i = n % g.nnx, j = n / g.nnx;
          if (f.tcin)
            prolong_node<T>(g, c, xc, x, i, j, valid, budget);
          else
            prolong_node<T>(g, c, PlanarX<T>{C.x, c.nn}, x, i, j, valid, budget);
        }
        break;
      }
      case kPhaseZeroTop: {
        if (k > 0) for_items<NT>(g.nn, [&](int n) { x.store(n, T(0), T(0), T(0)); });
        break;
      }
    }
    if (barrier && p + 1 < nph) sync();
  }
  // every block has read the number before its first barrier (a cycle with a
  // phase that uses it has one)
  if (blockIdx.x == 0 && threadIdx.x == 0)
    *(reinterpret_cast<volatile unsigned*>(state) + 1) = word + numbers;
}

template <typename T>
__global__ void __launch_bounds__(walk_threads<T>(), 1)
    vcycle_kernel(const VLevel<T>* lv, const OpTable<T>* tab, const Phase* ph, int nph, int top,
                  const T* topb, T* topx, const double* __restrict__ Ainv, T omega, int* state,
                  unsigned numbers, int polls, const int* skip) {
  // a speculative FGMRES iteration after the cycle stopped: every block
  // reads the same flag (set before this launch) and returns before any barrier
  if (skip && *skip) return;
  extern __shared__ __align__(16) uint8_t dyn[];
  cg::grid_group grid = cg::this_grid();
  walk_phases<T>(lv, tab, ph, nph, top, topb, topx, Ainv, omega, state, numbers, polls,
                 *reinterpret_cast<WalkSmem<T>*>(dyn), [&] { grid.sync(); });
}

// The whole grid is one thread-block cluster; the barriers are the cluster's
// (release / acquire at cluster scope, so the global-memory results of one phase
// are visible to every block of the cluster in the next).
template <typename T>
__global__ void __launch_bounds__(walk_threads<T>(), 1)
    vcycle_cluster_kernel(const VLevel<T>* lv, const OpTable<T>* tab, const Phase* ph, int nph,
                          int top, const T* topb, T* topx, const double* __restrict__ Ainv,
                          T omega, int* state, unsigned numbers, int polls) {
  extern __shared__ __align__(16) uint8_t dyn[];
  cg::cluster_group cl = cg::this_cluster();
  walk_phases<T>(lv, tab, ph, nph, top, topb, topx, Ainv, omega, state, numbers, polls,
                 *reinterpret_cast<WalkSmem<T>*>(dyn), [&] { cl.sync(); });
}

template <typename T>
__global__ void __launch_bounds__(128)
    assemble_blocks_kernel(const AsmLevel<T>* __restrict__ lv, int nlev, int nodes) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nodes) return;
  int k = 0;
  while (k + 1 < nlev && t >= lv[k + 1].first) ++k;
  assemble_node<T>(lv[k].g, lv[k].s, lv[k].vb, lv[k].cf, t - lv[k].first);
}

__global__ void __launch_bounds__(256) node_patterns_kernel(Grid g, uint16_t* __restrict__ pat) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= g.nn) return;
  const int i = n % g.nnx, j = n / g.nnx;
  unsigned p = 0;
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int ci = i - 1 + (b & 1), cj = j - 1 + (b >> 1);
    if (ci >= 0 && cj >= 0 && ci < g.nx && cj < g.ny && !g.solid[cj * g.nx + ci]) p |= 1u << b;
    const int PI = (i >> 1) - (b & 1), PJ = (j >> 1) - (b >> 1);
    if (PI >= 0 && PJ >= 0 && PI < g.nx / 2 && PJ < g.ny / 2 && i - 2 * PI <= 2 &&
        j - 2 * PJ <= 2 && !g.solid[(2 * PJ) * g.nx + 2 * PI])
      p |= 1u << (kPatPatch + b);
  }
  const uint8_t f = g.flags[n];
  if (f & kVDir) p |= kPatVDir;
  if (f & kPFix) p |= kPatPFix;
  pat[n] = (uint16_t)p;
}

// phases of the cycle of level k; returns the buffer and number of its final
// iterate (0: the coarsest level's solution)
std::pair<int, int> build_phases(int k, int nu1, int nu2, std::vector<Phase>& out) {
  if (k == 0) {
    out.push_back({kPhaseCoarse, 0, 0, 0, 0});
    return {0, 0};
  }
  // with pre-smoothing, the first pass starts from the zero iterate and
  // writes every node, so no level needs zeroing beforehand
  int cur = 0, tag = 0;
  auto push = [&](int type, int colour, bool update) {
    Phase f{type, k, colour, cur, update ? 1 - cur : 0};
    f.tin = tag;
    if (update) cur = f.out, ++tag;
    f.tout = tag;
    out.push_back(f);
  };
  for (int s = 0; s < nu1; ++s)
    for (int c = 0; c < 4; ++c) push(s == 0 && c == 0 ? kPhasePassZero : kPhasePass, c, true);
  push(kPhaseDefect, 0, false);
  push(kPhaseRestrict, nu1 > 0 ? 0 : 1, false);
  const std::pair<int, int> coarse = build_phases(k - 1, nu1, nu2, out);
  push(kPhaseProlong, 0, true);
  out.back().cin = coarse.first;
  out.back().tcin = coarse.second;
  for (int s = 0; s < nu2; ++s)
    for (int c = 0; c < 4; ++c) push(kPhasePass, c, true);
  out.back().last = 1;
  return {cur, tag};
}

}  // namespace

namespace {
// shared memory of a block: its tables and the larger of the warp tiles and
// the coarse right-hand side (FP64)
template <typename T>
size_t walk_smem(int coarse_nd) {
  const size_t tiles = sizeof(WarpTile<T>) * (walk_threads<T>() / 32);
  const size_t head = offsetof(WalkSmem<T>, tile);
  return head + std::max(tiles, sizeof(double) * coarse_nd);
}
}  // namespace

void launch_node_patterns(const Grid& g, uint16_t* pat, cudaStream_t st) {
  note_launch();
  node_patterns_kernel<<<cdiv(g.nn, 256), 256, 0, st>>>(g, pat);
}

template <typename T>
void launch_assemble_blocks(const AsmLevel<T>* lv, int nlev, int nodes, cudaStream_t st) {
  if (nodes <= 0) return;
  note_launch();
  assemble_blocks_kernel<T><<<cdiv(nodes, 128), 128, 0, st>>>(lv, nlev, nodes);
}

int vcycle_tile_columns(const Grid& g) { return cdiv(g.nx / 2 + 1, kWX / 2); }

int vcycle_warp_tiles(const Grid& g) {
  return cdiv(g.nx / 2 + 1, kWX / 2) * cdiv(g.ny / 2 + 1, kWY / 2);
}

int vcycle_defect_tiles(const Grid& g) { return cdiv(g.nnx, kWX) * cdiv(g.nny, kWY); }

bool vcycle_fits(int nphases, int nlevels) {
  return nphases <= kMaxPhases && nlevels <= kMaxVLevels;
}

std::vector<Phase> vcycle_phases(int top, int nu1, int nu2) {
  std::vector<Phase> out;
  if (nu1 == 0 || top == 0) out.push_back({kPhaseZeroTop, top, 0, 0, 0});
  build_phases(top, nu1, nu2, out);
  return out;
}

template <typename T>
int vcycle_grid(int coarse_nd) {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const size_t smem = walk_smem<T>(coarse_nd);
  if (cudaFuncSetAttribute(vcycle_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, vcycle_kernel<T>, walk_threads<T>(),
                                                    smem) != cudaSuccess ||
      per <= 0)
    return 0;
  return sms;  // one block per SM
}

template <typename T>
int launch_vcycle_persistent(const VLevel<T>* lv, const OpTable<T>* tab, const Phase* ph, int nph,
                             int top, const T* topb, T* topx, const double* Ainv, T omega,
                             int* state, unsigned numbers, int polls, int grid,
                             int coarse_nd, cudaStream_t st, const int* skip) {
  void* args[] = {(void*)&lv,   (void*)&tab,  (void*)&ph,   (void*)&nph,   (void*)&top,
                  (void*)&topb, (void*)&topx, (void*)&Ainv, (void*)&omega, (void*)&state,
                  (void*)&numbers, (void*)&polls, (void*)&skip};
  note_launch();
  const cudaError_t e =
      cudaLaunchCooperativeKernel((void*)vcycle_kernel<T>, dim3(grid), dim3(walk_threads<T>()),
                                  args, walk_smem<T>(coarse_nd), st);
  return e == cudaSuccess ? 0 : 1;
}

template <typename T>
int vcycle_cluster_size(int coarse_nd) {
  const size_t smem = walk_smem<T>(coarse_nd);
  if (cudaFuncSetAttribute(vcycle_cluster_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  for (int cs : {16, 8}) {
    if (cs > 8 && cudaFuncSetAttribute(vcycle_cluster_kernel<T>,
                                       cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                      cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(walk_threads<T>());
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, (void*)vcycle_cluster_kernel<T>, &cfg) == cudaSuccess &&
        n > 0)
      return cs;
    cudaGetLastError();
  }
  return 0;
}

template <typename T>
int launch_vcycle_cluster(const VLevel<T>* lv, const OpTable<T>* tab, const Phase* ph, int nph,
                          int top, const T* topb, T* topx, const double* Ainv, T omega,
                          int* state, unsigned numbers, int polls, int cluster, int coarse_nd,
                          cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(cluster);
  cfg.blockDim = dim3(walk_threads<T>());
  cfg.dynamicSmemBytes = walk_smem<T>(coarse_nd);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  note_launch();
  const cudaError_t e = cudaLaunchKernelEx(&cfg, vcycle_cluster_kernel<T>, lv, tab, ph, nph, top,
                                           topb, topx, Ainv, omega, state, numbers, polls);
  return e == cudaSuccess ? 0 : 1;
}

#define DNNMG_INST(T)                                                                            \
  template void launch_assemble_blocks<T>(const AsmLevel<T>*, int, int, cudaStream_t);           \
  template int vcycle_grid<T>(int);                                                              \
  template int launch_vcycle_persistent<T>(const VLevel<T>*, const OpTable<T>*, const Phase*,    \
                                           int, int, const T*, T*, const double*, T, int*,       \
                                           unsigned, int, int, int, cudaStream_t, const int*);   \
  template int vcycle_cluster_size<T>(int);                                                      \
  template int launch_vcycle_cluster<T>(const VLevel<T>*, const OpTable<T>*, const Phase*, int,  \
                                        int, const T*, T*, const double*, T, int*, unsigned,     \
                                        int, int, int, cudaStream_t);
DNNMG_INST(float)
DNNMG_INST(double)
#undef DNNMG_INST

}  // namespace dnnmg

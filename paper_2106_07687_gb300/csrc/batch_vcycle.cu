// The V(nu1, nu2) cycle of all problems of a batch as one cooperative launch.
//
// The phases are those of the single problem's cycle (vcycle.cu) from the
// largest level of the batch down: a phase of level k works on every problem
// that has the level, over a list of (problem, tile) or (problem, chunk of 32
// nodes) items, one warp each, with the same warp bodies and the same numbered
// updates of the iterate instead of barriers (vnode.cuh).  One FP32 cycle of
// twelve channels on levels 3 to 5: 77 launches with cell-by-cell tiles 1,338
// us, this with a barrier per phase 704 us, with numbered updates 563 us; a pass
// of the top level moves 80 MB of inverses and blocks (265 k nodes, 12 us).
// Where the grid cannot be resident the same kernel is launched once per phase.
#include <algorithm>
#include <cooperative_groups.h>

#include "batch.h"
#include "coarse_body.cuh"
#include "vbody.cuh"
#include "vcycle.h"

namespace cg = cooperative_groups;

namespace dnnmg {

namespace {

constexpr int kRecBytes = 104 * 1024;  // level records kept in shared memory, at most

template <typename T>
struct BWalkSmem {
  OpTable<T> tab;
  alignas(16) WarpTile<T> tile[walk_threads<T>() / 32];  // or the coarse right-hand side
};

template <typename T>
__global__ void __launch_bounds__(walk_threads<T>(), 1)
    bvcycle_kernel(const __grid_constant__ BWalk<T> W, const Phase* __restrict__ ph, int p0, int p1,
                   const T* topb, T* topx, T omega, const int* act, int bump) {
  constexpr int NT = walk_threads<T>(), NW = NT / 32;
  extern __shared__ __align__(16) uint8_t dyn[];
  BWalkSmem<T>& S = *reinterpret_cast<BWalkSmem<T>*>(dyn);
  BLev<T>* srec = reinterpret_cast<BLev<T>*>(dyn + sizeof(BWalkSmem<T>));
  const int nrec = W.nprob * W.nL;
  const bool in_smem = nrec * (int)sizeof(BLev<T>) <= kRecBytes;
  if (in_smem) copy_ints(srec, W.lev, nrec);
  copy_ints(&S.tab, W.tab + (W.mode >= 0 ? W.mode : 0), 1);
  __syncthreads();
  const BLev<T>* rec = in_smem ? srec : W.lev;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int w0 = blockIdx.x + gridDim.x * w, nw = gridDim.x * NW;
  const unsigned word = __ldcg(reinterpret_cast<unsigned*>(W.state) + 1), tag0 = word << 1;
  int budget = W.polls;
  for (int p = p0; p < p1; ++p) {
    Phase f{};
    f.type = __ldg(&ph[p].type), f.level = __ldg(&ph[p].level), f.colour = __ldg(&ph[p].colour);
    f.in = __ldg(&ph[p].in), f.out = __ldg(&ph[p].out);
    f.tin = __ldg(&ph[p].tin), f.tout = __ldg(&ph[p].tout), f.cin = __ldg(&ph[p].cin);
    f.tcin = __ldg(&ph[p].tcin), f.last = __ldg(&ph[p].last);
    const int k = f.level;
    // item t of a list: its problem's record of level k and its index there
    auto items = [&](const Work& list, auto body) {
      for (int t = w0; t < list.n; t += nw) {
        const int2 it = __ldg(list.d + t);
        if (act && !act[it.x]) continue;
        body(rec[it.x * W.nL + k], it.x, it.y);
      }
    };
    auto table = [&](const BLev<T>& L) -> const OpTable<T>& {
      return W.mode >= 0 ? S.tab : W.tab[L.mode];
    };
    auto node_level = [&](const BLev<T>& L) {
      return NodeLevel<T, sizeof(T) == 4>{L.g.nx, L.g.ny, L.g.nnx, L.g.nn,
                                          L.pat,  L.cf,   L.h,     L.hs,   L.hslo};
    };
    auto iterate = [&](const BLev<T>& L) {
      const size_t words = (size_t)kTagWords<T> * L.g.nn;
      return TaggedX<T>{L.xt + f.in * words, L.xt + f.out * words,
                        f.last && L.top ? topx + L.off : nullptr, L.g.nn, tag0 + f.tin,
                        tag0 + f.tout,       W.state};
    };
    switch (f.type) {
      case kPhasePass:
        items(W.pass[k], [&](const BLev<T>& L, int, int t) {
          warp_pass_tile<T>(node_level(L), table(L), f.colour, L.top ? topb + L.off : L.b,
                            iterate(L), L.inv, vanka_pitch(L.g), vanka_slots(L.g), omega,
                            t & 0xFFFF, t >> 16, lane, S.tile[w], budget);
        });
        break;
      case kPhasePassZero:
        items(W.zero[k], [&](const BLev<T>& L, int, int c) {
          const int e = (c << 5) + lane;
          zero_pass_node<T>(L.g, f.colour, L.top ? topb + L.off : L.b, iterate(L), L.inv, omega, e,
                            e < 4 * vanka_slots(L.g));
        });
        break;
      case kPhaseDefect:
        items(W.defect[k], [&](const BLev<T>& L, int, int t) {
          const int nbx = cdiv(L.g.nnx, kWX);
          warp_defect_tile<T>(node_level(L), table(L), L.top ? topb + L.off : L.b, iterate(L), L.d,
                              t % nbx, t / nbx, lane, S.tile[w], budget);
        });
        break;
      case kPhaseRestrict:
        items(W.restr[k], [&](const BLev<T>& F, int prob, int c) {
          const BLev<T>& C = rec[prob * W.nL + k - 1];
          const int n = (c << 5) + lane;
          if (n >= C.g.nn) return;
          restrict_node<T, true>(F.g, C.g, F.d, C.b, 3, n % C.g.nnx, n / C.g.nnx);
          if (f.colour == 1 && C.xt)
            TaggedX<T>{C.xt, C.xt, nullptr, C.g.nn, tag0, tag0, W.state}.store(n, T(0), T(0), T(0));
        });
        break;
      case kPhaseProlong:
        items(W.prol[k], [&](const BLev<T>& F, int prob, int c) {
          const BLev<T>& C = rec[prob * W.nL + k - 1];
          const bool valid = (c << 5) + lane < F.g.nn;  // whole warps wait together
          const int n = valid ? (c << 5) + lane : 0, i = n % F.g.nnx, j = n / F.g.nnx;
          if (f.tcin)
            prolong_node<T>(F.g, C.g,
                            TaggedX<T>{C.xt + f.cin * (size_t)kTagWords<T> * C.g.nn, nullptr,
                                       nullptr, C.g.nn, tag0 + f.tcin, 0u, W.state},
                            iterate(F), i, j, valid, budget);
          else
            prolong_node<T>(F.g, C.g, PlanarX<T>{C.x, C.g.nn}, iterate(F), i, j, valid,
                            budget);
        });
        break;
      case kPhaseCoarse: {
        // the blocks share the problems out, and a problem's blocks its rows
        double* sb = reinterpret_cast<double*>(S.tile);
        const int per = max(1, (int)gridDim.x / W.nprob);  // blocks per problem
        for (int prob = (int)blockIdx.x / per; prob < W.nprob;
             prob += max(1, (int)gridDim.x / per)) {
          if (act && !act[prob]) continue;  // the same for the whole block
          const BLev<T>& L = rec[prob * W.nL + k];
          const T* b = L.top ? topb + L.off : L.b;
          T* x = L.top ? topx + L.off : L.x;
          const int nd = 3 * L.g.nn;
          __syncthreads();
          for (int q = threadIdx.x; q < nd; q += NT) sb[q] = (double)__ldcg(b + band_to_level(L.g, q));
          __syncthreads();
          for (int r = (int)blockIdx.x % per + per * w; r < nd; r += per * NW) {
            const double* row = W.Ainv + (size_t)prob * W.astride + (size_t)r * nd;
            double acc[4] = {0.0, 0.0, 0.0, 0.0};
            for (int c0 = lane; c0 < nd; c0 += 16 * 32) {
              double rv[16];
#pragma unroll
              for (int u = 0; u < 16; ++u) rv[u] = c0 + 32 * u < nd ? row[c0 + 32 * u] : 0.0;
#pragma unroll
              for (int u = 0; u < 16; ++u)
                if (c0 + 32 * u < nd) acc[u & 3] += rv[u] * sb[c0 + 32 * u];
            }
            double a = (acc[0] + acc[1]) + (acc[2] + acc[3]);
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (lane == 0) x[band_to_level(L.g, r)] = (T)a;
          }
          __syncthreads();
        }
        break;
      }
      case kPhaseZeroTop:  // every problem's own top level
        for (int l = 2; l < W.nL && l < kBLevels; ++l)
          for (int t = w0; t < W.prol[l].n; t += nw) {
            const int2 it = __ldg(W.prol[l].d + t);
            const BLev<T>& L = rec[it.x * W.nL + l];
            const int n = (it.y << 5) + lane;
            if ((!act || act[it.x]) && L.top && n < L.g.nn)
              TaggedX<T>{L.xt, L.xt, nullptr, L.g.nn, tag0, tag0, W.state}.store(n, T(0), T(0),
                                                                              T(0));
          }
        break;
      default: break;
    }
    // the defect, the restricted one and the coarse solution are plain arrays
    const bool plain =
        f.type == kPhaseDefect || f.type == kPhaseRestrict || f.type == kPhaseCoarse;
    if (plain && p + 1 < p1) {
      if (budget > 0) budget = W.polls;  // a batch's size and sweeps have no bound
      cg::this_grid().sync();
    }
  }
  // every block has read the number before its first barrier (a cycle with a
  // phase that uses it has one)
  if (bump && blockIdx.x == 0 && threadIdx.x == 0)
    *(reinterpret_cast<volatile unsigned*>(W.state) + 1) = word + W.numbers;
}

__global__ void next_cycle_kernel(int* state, unsigned numbers) {
  state[1] = (int)((unsigned)state[1] + numbers);
}

template <typename T>
size_t walk_bytes(int nprob, int nL, int n1) {
  const size_t rec = (size_t)nprob * nL * sizeof(BLev<T>);
  const size_t head = std::max(sizeof(BWalkSmem<T>),
                               offsetof(BWalkSmem<T>, tile) + sizeof(double) * n1);
  return std::max(head, sizeof(BWalkSmem<T>)) + (rec <= (size_t)kRecBytes ? rec : 0);
}

}  // namespace

template <typename T>
void bk_vcycle(const BWalk<T>& W, const Phase* ph, int nph, const T* topb, T* topx, T omega,
               const int* act, cudaStream_t st) {
  const size_t smem = walk_bytes<T>(W.nprob, W.nL, W.n1);
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaFuncSetAttribute(bvcycle_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, bvcycle_kernel<T>, walk_threads<T>(),
                                                    smem) != cudaSuccess)
    per = 0;
  if (per > 0) {
    BWalk<T> w = W;
    int p0 = 0, bump = 1;
    void* args[] = {(void*)&w,    (void*)&ph,   (void*)&p0,    (void*)&nph,
                    (void*)&topb, (void*)&topx, (void*)&omega, (void*)&act,
                    (void*)&bump};
    note_launch();
    if (cudaLaunchCooperativeKernel((void*)bvcycle_kernel<T>, dim3(sms), dim3(walk_threads<T>()),
                                    args, smem, st) == cudaSuccess)
      return;
    cudaGetLastError();
  }
  for (int p = 0; p < nph; ++p) {
    note_launch();
    bvcycle_kernel<T><<<sms, walk_threads<T>(), smem, st>>>(W, ph, p, p + 1, topb, topx, omega, act,
                                                     0);
  }
  note_launch();
  next_cycle_kernel<<<1, 1, 0, st>>>(W.state, W.numbers);
}

template void bk_vcycle<float>(const BWalk<float>&, const Phase*, int, const float*, float*, float,
                               const int*, cudaStream_t);
template void bk_vcycle<double>(const BWalk<double>&, const Phase*, int, const double*, double*,
                                double, const int*, cudaStream_t);

}  // namespace dnnmg

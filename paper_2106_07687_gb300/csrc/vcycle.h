// Persistent V-cycle (internal to libdnnmg).
#pragma once
#include <vector>

#include "kernels.h"
#include "vnode.cuh"

namespace dnnmg {

// Everything the cycle needs on one level; an array of these lives in
// device memory (index = level - coarsest level).
template <typename T>
struct VLevel {
  Grid g;
  T *x, *b, *d, *inv;    // x: the coarsest level's solution
  const T* cf;           // assembled velocity blocks (null on the coarsest level)
  const uint16_t* pat;   // node patterns
  ulonglong2* xt;        // the iterate: two tagged buffers of kTagWords nn words (vnode.cuh)
};

// A level's input to the assembly of its velocity blocks; `first` is its
// first node in the concatenation of the levels of one launch.
template <typename T>
struct AsmLevel {
  Grid g;
  Sten<T> s;
  const T* vb;
  T* cf;
  int first;
};
// patterns of a level's nodes (vnode.cuh)
void launch_node_patterns(const Grid& g, uint16_t* pat, cudaStream_t st);
// velocity blocks of the first nlev levels of `lv` (device array), `nodes`
// nodes in all, in one launch
template <typename T>
void launch_assemble_blocks(const AsmLevel<T>* lv, int nlev, int nodes, cudaStream_t st);

enum PhaseType {
  kPhasePass,
  kPhaseDefect,
  kPhaseRestrict,
  kPhaseCoarse,
  kPhaseProlong,
  kPhaseZeroTop,
  kPhasePassZero  // first pass of a sweep from x = 0 (the input is not read)
};

// in / out select the level's iterate (two buffers); a restriction with colour
// = 1 also starts the coarse iterate from zero (needed when no pre-smoothing pass
// does).  tin / tout: number, within the cycle, of the level's update that the
// phase reads and writes; cin / tcin: buffer and number of the coarse level's
// iterate that a prolongation reads (tcin 0: the coarsest level's solution).
// last: the level's final update (on the top level it goes to the result).
struct Phase {
  int type, level, colour, in, out;
  int tin = 0, tout = 0, cin = 0, tcin = 0, last = 0;
};

// Half of what a cycle advances the numbers of the updates by: a level's iterate
// takes the numbers 0 (its start from zero) to 4 (nu1 + nu2) + 1 (every colour pass
// and the prolongation) above the cycle's first, an even number.  (The state word
// holds half of it: with the number itself there the batch's FP64 kernel, at its
// limit of registers, took 2,790 instead of 2,740 us for twelve channels.)
inline unsigned vcycle_numbers(int nu1, int nu2) {
  return 2u * ((unsigned)nu1 + (unsigned)nu2) + 1u;
}

// phase list of one V(nu1, nu2) cycle with top level `top`, x zeroed first
std::vector<Phase> vcycle_phases(int top, int nu1, int nu2);
// whether a launch of nphases phases over nlevels levels fits the kernels'
// shared-memory tables
bool vcycle_fits(int nphases, int nlevels);
// warp tiles of a colour pass on a level
int vcycle_warp_tiles(const Grid& g);
// and how many of them lie side by side
int vcycle_tile_columns(const Grid& g);
// warp tiles of a defect
int vcycle_defect_tiles(const Grid& g);
// co-resident grid size for the cooperative launch (0 if not available)
template <typename T>
int vcycle_grid(int coarse_nd);
// blocks of the largest single-cluster launch that can be resident (16 or
// 8; 0 if none)
template <typename T>
int vcycle_cluster_size(int coarse_nd);
// the same cycle as one thread-block cluster of `cluster` blocks; 0 on success
template <typename T>
int launch_vcycle_cluster(const VLevel<T>* lv, const OpTable<T>* tab, const Phase* ph, int nph,
                          int top, const T* topb, T* topx, const double* Ainv, T omega,
                          int* state, unsigned numbers, int polls, int cluster, int coarse_nd,
                          cudaStream_t st);
// state: two device words, a status word (8: a wait for an update hit its bound)
// and half of the cycle's first number, which the launch advances by `numbers`
// (vcycle_numbers; the word starts above 0).  polls: the bound of a warp's polls
// (kTagPolls).
// returns 0 on success; with skip, nothing runs when *skip != 0 at the
// launch's start
template <typename T>
int launch_vcycle_persistent(const VLevel<T>* lv, const OpTable<T>* tab, const Phase* ph, int nph,
                             int top, const T* topb, T* topx, const double* Ainv, T omega,
                             int* state, unsigned numbers, int polls, int grid,
                             int coarse_nd, cudaStream_t st,
                             const int* skip = nullptr);

}  // namespace dnnmg

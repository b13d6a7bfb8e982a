// Patch network on fifth-generation tensor cores (Sec. 2.2 / Sec. 3.1: GRU
// cells with memory per patch, then dense layers; inputs and outputs per
// patch as in the network evaluation of Algorithm 1).
//
// patchnet_forward_kernel<TRAIN, m, n, G>: persistent, 512 threads in G
// groups that each take one 128-patch tile at a time.  Patch row r of a tile
// is TMEM lane r; warp w serves lanes 32 (w % 4) .. +31, and the 4 / G
// warpgroups of a group split every accumulator's columns in the epilogues
// (m G / 4 hidden units per thread).  All weights live in shared memory as
// BF16 K-major operands (one bulk copy per block); per GRU layer the tensor
// core accumulates in TMEM (4m FP32 columns)
//   [0,2m)   x W_ih[r,z]^T + h W_hh[r,z]^T      (gates r and z)
//   [2m,3m)  x W_ih[n]^T                        (input part of gate n)
//   [3m,4m)  h W_hh[n]^T                        (hidden part of gate n)
// and each thread applies the gate nonlinearities to its units in
// registers, writing the new hidden state (FP32) to HBM and (BF16) to shared
// memory as the next GEMM's operand.  In training the states stay in TMEM
// (columns 256..) from step to step.  The dense head reuses TMEM columns [0,128)
// and [128,128+N2).
//
// A tile is a serial chain (loads, MMA, wait, gates, MMA, ...), so with more
// tiles than SMs two groups run in each block, one computing gates while the
// other waits for loads or MMAs; with at most one tile per SM a single group
// gives the tile all 512 threads, which shortens the chain, and x_t and the
// next layer's previous state are loaded a stage ahead.  The gates are the
// longest part of a tile (3.5 of 16 us per layer): branch-free reciprocals,
// biases in 16-byte loads and paired BF16 conversions took the kernel from 20.2
// to 15.9 us for one tile per SM, from 68.8 to 49.7 us over 61,440 patches and
// the training forward (19,456 x 10, 64 x 2) from 229 to 197 us.
#include "kernels.h"
#include "krylov_body.cuh"
#include "patchnet.cuh"
#include "recip.cuh"
#include "umma.cuh"

namespace dnnmg {

namespace {

using namespace umma;

constexpr uint32_t kWaitPolls = 1u << 22;  // bound of every mbarrier wait
constexpr int kTile = 128;
constexpr int kFwdWG = 4;                      // warpgroups of the forward kernel
constexpr int kFwdThreads = kTile * kFwdWG;
constexpr size_t kSmemMax = kSmemLimit;

__device__ __forceinline__ uint16_t f2bf(float v) {
  return __bfloat16_as_ushort(__float2bfloat16_rn(v));
}

// the compiled division branches, which kept the gates of a thread's units from
// overlapping
__device__ __forceinline__ float sigmoidf_(float x) { return recip_ge1(1.0f + __expf(-x)); }

// two values as BF16, lo in the low half
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&p);
}

// -- packing -----------------------------------------------------------------
// fused biases; a network without biases gets zeros
__device__ __forceinline__ void pack_bias(const float* __restrict__ w, const NetDims& d,
                                          float* __restrict__ bias) {
  const int H = d.hidden;
  const NetOffsets o = d.offsets();
  for (int l = 0; l < d.layers; ++l) {
    for (int j = threadIdx.x; j < H; j += blockDim.x) {
      float* b = bias + (size_t)l * 4 * H;
      if (d.bias) {
        const float* bih = w + o.bih[l];
        const float* bhh = w + o.bhh[l];
        b[j] = bih[j] + bhh[j];
        b[H + j] = bih[H + j] + bhh[H + j];
        b[2 * H + j] = bih[2 * H + j];
        b[3 * H + j] = bhh[2 * H + j];
      } else {
        b[j] = b[H + j] = b[2 * H + j] = b[3 * H + j] = 0.0f;
      }
    }
  }
  float* ob = bias + (size_t)d.layers * 4 * H;
  for (int j = threadIdx.x; j < d.mlp; j += blockDim.x) ob[j] = d.bias ? w[o.b1 + j] : 0.0f;
  for (int j = threadIdx.x; j < d.nout(); j += blockDim.x)
    ob[d.mlp + j] = d.bias && j < d.c_out ? w[o.b2 + j] : 0.0f;
}

// All operands of a network in one launch, a job per blockIdx.y, and the biases
// (bias != null) as one more.  For 2 x 64 units fifteen launches of 1.5 us before;
// with one host wait per call instead of two, a training step of 19,456 sequences
// x 10 steps 689 -> 630 us, a gradient of 32 x 2 units 233 -> 215 us.
struct PackArgs {
  PackJob job[kMaxPackJobs];
  int n;
  const float* w;
  float* bias;
};
__global__ void __launch_bounds__(256)
    pack_kernel(const __grid_constant__ PackArgs a, const NetDims d) {
  if ((int)blockIdx.y == a.n) {
    if (blockIdx.x == 0) pack_bias(a.w, d, a.bias);
    return;
  }
  const PackJob& J = a.job[blockIdx.y];
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < J.R * J.K;
       idx += gridDim.x * blockDim.x) {
    const int r = idx / J.K, k = idx % J.K;
    const float v = r < J.rows && k < J.cols ? J.src[(size_t)r * J.rstride + (size_t)k * J.kstride]
                                             : 0.0f;
    J.dst[kmajor_offset(r, k, J.K) >> 1] = f2bf(v);
  }
}

// -- shared-memory plan of the forward kernel ---------------------------------
// Weights and biases once per block, and an operand area per group.  Operand
// regions are reused as soon as the MMA that reads them has completed:
//   a: x_t (layer 0 input, kx0 columns), then each layer's new state (the
//      next layer's input, m columns; the top layer's is the head's input);
//   b: the previous state of the layer being evaluated (m columns), staged
//      before that layer's MMAs;
//   m: the dense head's hidden layer (128 columns), over a and b.
// With two groups and a wide input (split), x_t lies over a and b too and the
// first layer's previous state is staged after the MMAs of x_t.
struct FwdSmem {
  uint32_t w, bias, area, area_size, b, bar, tmem, total;
  bool split;
  static __host__ __device__ uint32_t up(uint32_t v) { return (v + 127u) & ~127u; }
  static __host__ __device__ FwdSmem of(const NetDims& d, size_t w_elems, int groups) {
    FwdSmem s{};
    uint32_t o = 0;
    s.w = o;    o = up(o + (uint32_t)(w_elems * 2));
    s.bias = o; o = up(o + (uint32_t)((d.layers * 4 * d.hidden + d.mlp + d.nout()) * 4));
    const int ka = d.kx0() > d.hidden ? d.kx0() : d.hidden;
    s.split = groups > 1 && ka + d.hidden > 128;
    s.b = kTile * (s.split ? d.hidden : ka) * 2;
    const uint32_t absz = s.b + kTile * d.hidden * 2, msz = kTile * 128 * 2;
    s.area = o;
    s.area_size = absz > msz ? absz : msz;
    o += groups * s.area_size;
    s.bar = o;  o += 32;
    s.tmem = o; o += 16;
    s.total = o;
    return s;
  }
};

// barrier of one group's threads; group_any: whether p holds in any of them
__device__ __forceinline__ void group_sync(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ bool group_any(int id, int n, bool p) {
  int r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\t"
      "bar.red.or.pred q, %2, %3, p;\n\tselp.b32 %0, 1, 0, q;\n\t}\n"
      : "=r"(r)
      : "r"((int)p), "r"(id), "r"(n)
      : "memory");
  return r != 0;
}

// write U (8 or 16) consecutive values of row r (columns k0..) as BF16 operand
template <int U>
__device__ __forceinline__ void store_row(uint8_t* buf, int r, int k0, int K, const float* v) {
#pragma unroll
  for (int h = 0; h < U / 8; ++h) {
    uint32_t p[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) p[i] = bf16_pair(v[8 * h + 2 * i], v[8 * h + 2 * i + 1]);
    *reinterpret_cast<uint4*>(buf + kmajor_offset(r, k0 + 8 * h, K)) =
        make_uint4(p[0], p[1], p[2], p[3]);
  }
}

// Issue D(+)= A * B^T over K (in 16-wide slices) for one accumulator.
__device__ __forceinline__ void mma_run(uint32_t d_tmem, uint32_t a_addr, int a_K, uint32_t b_addr,
                                        int b_K, int N, int K, bool acc_first) {
  const uint32_t id = idesc_bf16(kTile, N);
  for (int ks = 0; ks < K / 16; ++ks) {
    const uint64_t da = smem_desc(a_addr + ks * 256, 128, (a_K / 8) * 128);
    const uint64_t db = smem_desc(b_addr + ks * 256, 128, (b_K / 8) * 128);
    mma_bf16(d_tmem, da, db, id, (ks > 0 || acc_first) ? 1u : 0u);
  }
}

// U consecutive values as U / 4 groups of 16 bytes, `stride` groups apart
template <int U>
__device__ __forceinline__ void store_f32(float4* dst, size_t stride, const float* v) {
#pragma unroll
  for (int q = 0; q < U / 4; ++q)
    dst[q * stride] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}
template <int U>
__device__ __forceinline__ void load_f32(const float4* src, size_t stride, float* v) {
#pragma unroll
  for (int q = 0; q < U / 4; ++q) {
    const float4 u = src[q * stride];
    v[4 * q] = u.x, v[4 * q + 1] = u.y, v[4 * q + 2] = u.z, v[4 * q + 3] = u.w;
  }
}

// One GRU layer's epilogue for U units [u0, u0 + U) of this thread's row:
// gates from TMEM, new hidden state from hprev into `next` (BF16 operand)
// and `hout` (FP32, HBM, the U units).  With `gsave` the gates r, z, n and
// the hidden part of gate n (incl. bias) are stored for the backward pass
// ([r | z | n | hn], m each); hout and gsave are groups `stride` apart.  With
// `hT` the new state is also written transposed in BF16 (rows `ldT` apart).
template <int H, int U>
__device__ __forceinline__ void gru_epilogue(uint32_t tm, const float* bias, const float* hprev,
                                             float (&hn)[U], uint8_t* next, int row, int u0,
                                             float4* hout, bool valid, float4* gsave,
                                             size_t stride, uint16_t* hT, size_t ldT) {
  float g[4][U];
  tmem_ld4(tm + u0, H, g);
#pragma unroll
  for (int q = 0; q < U / 4; ++q) {
    float b[4][4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      load_f32<4>(reinterpret_cast<const float4*>(bias + k * H + u0 + 4 * q), 1, b[k]);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int i = 4 * q + e;
      const float r = sigmoidf_(g[0][i] + b[0][e]);
      const float z = sigmoidf_(g[1][i] + b[1][e]);
      const float ghn = g[3][i] + b[3][e];
      const float n = tanhf(g[2][i] + b[2][e] + r * ghn);
      hn[i] = (1.0f - z) * n + z * hprev[i];
      g[0][i] = r, g[1][i] = z, g[2][i] = n, g[3][i] = ghn;
    }
  }
  store_row<U>(next, row, u0, H, hn);
  if (!valid) return;
  store_f32<U>(hout, stride, hn);
  if (gsave) {
#pragma unroll
    for (int k = 0; k < 4; ++k) store_f32<U>(gsave + (k * H + u0) / 4 * stride, stride, g[k]);
  }
  if (hT)
#pragma unroll
    for (int i = 0; i < U; ++i) hT[(size_t)(u0 + i) * ldT] = f2bf(hn[i]);
}

// The sum of 16 squares, off by at most 2^-53 of itself as a sum in FP64 is, with
// three FP64 instructions instead of 32 (they run at 1/64 of the FP32 rate here; a
// gradient of 1,040 sequences x 7 steps 216.9 -> 213.5 us): the squares are whole
// numbers of 48 bits times powers of four, added as such in 64 bits relative to the
// largest one's (truncated there: 16 units of at least 2^58).
__device__ __forceinline__ double sum_squares(const float (&e)[16]) {
  unsigned top = 1;  // largest exponent field; 1 for subnormal values, as 2^-149 units
#pragma unroll
  for (int i = 0; i < 16; ++i) top = max(top, (__float_as_uint(e[i]) >> 23) & 255u);
  if (top == 255u) {  // an infinity or a NaN
    double s = 0.0;
#pragma unroll 1
    for (int i = 0; i < 16; ++i) s = fma((double)e[i], (double)e[i], s);
    return s;
  }
  unsigned long long sum = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const unsigned b = __float_as_uint(e[i]) & 0x7FFFFFFFu, ex = max(b >> 23, 1u);
    const unsigned m = b - ((ex - 1u) << 23), down = 2u * (top - ex);
    sum += down < 64u ? ((unsigned long long)m * m << 12) >> down : 0ull;
  }
  // m^2 2^12 counts 2^(2 (top - 150) - 12)
  return (double)sum * __hiloint2double((int)(1023u - 312u + 2u * top) << 20, 0);
}

// Arguments of the forward kernel.  Inference: T = 1, hidden state read from
// h_in and written to h_out, prediction to out.  Training: the hidden state
// starts at zero and the kernel stores, per (t, p), the activations the
// backward pass needs, the output gradients scale * (y - Y) and transposed
// BF16 copies of the GEMM inputs for the weight gradients (column index
// t * P + p), and per block the sum of (y - Y)^2.
struct FwdArgs {
  const uint16_t* x;  // [P][T][C_in]
  int P, T;
  const float* h_in;  // [layers][P][m]
  float* h_out;       // [layers][P][m]
  float* out;         // [P][C_out]
  const float* Y;     // [P][T][C_out]
  bool y_pairs;       // Y can be read in 8-byte pairs
  bool out_pairs;     // out can be written in 8-byte pairs
  float scale;
  float4* act;        // [T][act_groups][P]
  uint16_t* xT;       // [kx0 + 16][T * P]
  uint16_t* hT[kMaxLayers];  // [m + 16][(T + 1) * P], state of step t at column (t + 1) * P + p
  uint16_t* y1T;      // [144][T * P]
  uint16_t* dyT;      // [128][T * P]
  double* loss_partial;
  int* status;
  NetPost post;
};

template <bool TRAIN, int H, int NL, int G>
__global__ void __launch_bounds__(kFwdThreads, 1)
    patchnet_forward_kernel(NetDims d, PackLayout L, const uint16_t* __restrict__ wimg,
                            const float* __restrict__ bias_g, const __grid_constant__ FwdArgs a) {
  constexpr int GT = kFwdThreads / G;     // threads of a group
  constexpr int CQ = GT / kTile;          // column parts of an accumulator
  constexpr int U = H / CQ;               // hidden units of this thread's row
  constexpr int UC = U < 16 ? U : 16;     // of which one epilogue takes UC
  constexpr int KG = act_groups(H, NL);
  constexpr int NX = 4;                   // 16-byte chunks of x_t a thread loads at once
  // one group: x_t and the next layer's previous state are loaded a stage
  // ahead of their use (one epilogue and NX chunks cover a thread's part)
  constexpr bool AHEAD = G == 1;
  static_assert(AHEAD || !TRAIN, "training runs one group");
  // training keeps the states of its sequences in TMEM from step to step
  constexpr int TCOLS = TRAIN ? 512 : 256 * G;
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ double red[kFwdThreads / 32];
  const FwdSmem S = FwdSmem::of(d, L.total, G);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int grp = t / GT, tg = t % GT;
  const int row = (warp & 3) * 32 + lane;  // patch row of the tile = TMEM lane
  const int cq = tg / kTile;               // column part of the epilogues
  uint64_t* wbar = reinterpret_cast<uint64_t*>(sm + S.bar);  // the weights' arrival
  uint64_t* bar = wbar + 1 + grp;                            // this group's MMAs
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + S.tmem);
  float* bias = reinterpret_cast<float*>(sm + S.bias);
  uint8_t* A = sm + S.area + (size_t)grp * S.area_size;      // regions a and m
  uint8_t* Bh = A + S.b;                                     // region b
  const int P = a.P, T = a.T;

  const int kx0 = d.kx0();
  const int u0 = U * cq;  // this thread's hidden units
  const int ntiles = (P + kTile - 1) / kTile;
  const size_t HP = (size_t)P * H;
  const size_t ld = (size_t)T * P, ldh = (size_t)(T + 1) * P;
  // 16-byte chunks of x_t: chunk e of the tile is columns 8 q.. of row r.
  // Inference: a thread's neighbours take the next chunks of the same row
  // (coalesced loads); training: the same chunk of the next rows, so that the
  // transposed copy is written coalesced
  const int nq = kx0 / 8;
  const bool vec = d.c_in % 8 == 0;  // input rows start on 16-byte boundaries
  auto x_chunk = [&](int e, int& r, int& q) {
    r = TRAIN ? e % kTile : e / nq;
    q = TRAIN ? e / kTile : e % nq;
  };
  auto load_x = [&](int tile, int step, int e0, uint4* xr) {
#pragma unroll
    for (int c = 0; c < NX; ++c) {
      const int e = e0 + c * GT;
      int r, q;
      x_chunk(e, r, q);
      const int pr = tile * kTile + r;
      xr[c] = make_uint4(0, 0, 0, 0);
      if (e < kTile * nq && pr < P && q * 8 < d.c_in) {
        const uint16_t* src = a.x + ((size_t)pr * T + step) * d.c_in;
        if (vec) {
          xr[c] = reinterpret_cast<const uint4*>(src)[q];
        } else {  // element by element, zeros past C_in
          uint32_t w[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int k = q * 8 + 2 * i;
            w[i] = (k < d.c_in ? src[k] : 0u) | ((k + 1 < d.c_in ? (uint32_t)src[k + 1] : 0u) << 16);
          }
          xr[c] = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
    }
  };
  auto store_x = [&](int tile, int step, int e0, const uint4* xr) {
#pragma unroll
    for (int c = 0; c < NX; ++c) {
      const int e = e0 + c * GT;
      if (e >= kTile * nq) break;
      int r, q;
      x_chunk(e, r, q);
      *reinterpret_cast<uint4*>(A + kmajor_offset(r, q * 8, kx0)) = xr[c];
      const int pr = tile * kTile + r;
      if (TRAIN && pr < P) {
        const uint32_t w[4] = {xr[c].x, xr[c].y, xr[c].z, xr[c].w};
        uint16_t* o = a.xT + (size_t)(q * 8) * ld + (size_t)step * P + pr;
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (q * 8 + i < d.c_in) o[i * ld] = (uint16_t)(w[i >> 1] >> (16 * (i & 1)));
      }
    }
  };

  // previous state of layer l of the tile's patch p, units u..u + UC (inference)
  auto load_prev = [&](int p, int l, int u, float* hv) {
#pragma unroll
    for (int i = 0; i < UC; ++i) hv[i] = 0.0f;
    if (p < P)
      load_f32<UC>(reinterpret_cast<const float4*>(a.h_in + l * HP + (size_t)p * H + u), 1, hv);
  };
  // the first tile's loads go out before the block is set up
  uint4 xr[NX];
  float hnext[UC];
  if (AHEAD) {
    load_x(blockIdx.x, 0, tg, xr);
    if (!TRAIN) load_prev(blockIdx.x * kTile + row, 0, u0, hnext);
  }
  if (t == 0) {
    for (int q = 0; q <= G; ++q) mbar_init(wbar + q, 1);
    fence_async_smem();
    const uint32_t bytes = (uint32_t)(L.total * 2);
    mbar_expect_tx(wbar, bytes);
    bulk_load(sm + S.w, wimg, bytes, wbar);
  }
  for (int i = t; i < NL * 4 * H + d.mlp + d.nout(); i += kFwdThreads) bias[i] = bias_g[i];
  if (warp == 0) tmem_alloc(tslot, TCOLS);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tbase = *tslot + 256 * grp;
  const uint32_t tm = tbase + ((uint32_t)((warp & 3) * 32) << 16);  // this warp's lanes
  const uint32_t sw = smem_u32(sm + S.w), sa = smem_u32(A), sbh = smem_u32(Bh);
  const uint32_t tstate = tm + 256;  // TMEM columns of the states (training)
  uint32_t phase = 0;
  bool failed = false, weights = false;
  double loss = 0.0;

  // publish the group's operand writes, then one thread issues MMAs and the
  // group waits for them; false when the wait hit its bound
  auto run_mma = [&](auto issue) {
    fence_async_smem();
    fence_before_sync();
    group_sync(1 + grp, GT);
    if (tg == 0) {
      fence_after_sync();
      issue();
      mma_commit(bar);
    }
    const bool late = !mbar_wait(bar, phase, kWaitPolls);
    phase ^= 1;
    failed = group_any(1 + grp, GT, late);
    fence_after_sync();
    return !failed;
  };
  for (int tile = blockIdx.x + grp * gridDim.x; tile < ntiles && !failed;
       tile += gridDim.x * G) {
    const int p = tile * kTile + row;
    const bool valid = p < P;
#pragma unroll 1
    for (int step = 0; step < T && !failed; ++step) {
      const size_t col = (size_t)step * P + p;
      float4* act = TRAIN ? a.act + (size_t)step * KG * P + p : nullptr;  // this step's groups
      float hprev[UC];
      // previous state of layer l into region b: loaded by now, or from TMEM
      // (zero at a sequence's start); with two epilogues per layer it is read
      // here and again there
      auto stage_prev = [&](int l) {
        if (TRAIN) {
#pragma unroll
          for (int i = 0; i < UC; ++i) hprev[i] = 0.0f;
          if (step > 0) tmem_ld<UC>(tstate + l * H + u0, hprev);
          store_row<UC>(Bh, row, u0, H, hprev);
        } else if (AHEAD) {
#pragma unroll
          for (int i = 0; i < UC; ++i) hprev[i] = hnext[i];
          store_row<UC>(Bh, row, u0, H, hprev);
        } else {
#pragma unroll
          for (int c = 0; c < U / UC; ++c) {
            load_prev(p, l, u0 + c * UC, hprev);
            store_row<UC>(Bh, row, u0 + c * UC, H, hprev);
          }
        }
      };
      if (AHEAD) {
        store_x(tile, step, tg, xr);
        stage_prev(0);
        if (step + 1 < T)
          load_x(tile, step + 1, tg, xr);
        else
          load_x(tile + gridDim.x, 0, tg, xr);
      } else {
        for (int e = tg; e < kTile * nq; e += NX * GT) {
          load_x(tile, step, e, xr);
          store_x(tile, step, e, xr);
        }
        if (!S.split) stage_prev(0);
      }
      if (!weights) {  // their copy, once
        if ((failed = group_any(1 + grp, GT, !mbar_wait(wbar, 0, kWaitPolls)))) break;
        weights = true;
      }
      // ---- the GRU layers (unrolled); layer l reads its input from region
      // a and its previous state from region b and writes its new state into
      // region a
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        const int kx = l == 0 ? kx0 : H;
        if (AHEAD && !TRAIN) {  // the next layer's state, or the next tile's first
          if (l + 1 < NL)
            load_prev(p, l + 1, u0, hnext);
          else
            load_prev(p + gridDim.x * kTile, 0, u0, hnext);
        }
        auto mma_x = [&] {
          mma_run(tbase + 0, sa, kx, sw + 2 * L.rz[l], kx, 2 * H, kx, false);
        };
        auto mma_n = [&] {
          mma_run(tbase + 2 * H, sa, kx, sw + 2 * L.in[l], kx, H, kx, false);
        };
        auto mma_h = [&] {
          mma_run(tbase + 0, sbh, H, sw + 2 * L.hrz[l], H, 2 * H, H, true);
        };
        auto mma_hn = [&] {
          mma_run(tbase + 3 * H, sbh, H, sw + 2 * L.hn[l], H, H, H, false);
        };
        if (l == 0 && S.split) {
          if (!run_mma([&] { mma_x(), mma_n(); })) break;
          stage_prev(0);
          if (!run_mma([&] { mma_h(), mma_hn(); })) break;
        } else {
          if (!run_mma([&] { mma_x(), mma_h(), mma_n(), mma_hn(); })) break;
        }
#pragma unroll
        for (int c = 0; c < U / UC; ++c) {
          const int u = u0 + c * UC;
          if (!AHEAD) load_prev(p, l, u, hprev);
          float4* hout = TRAIN ? act + (size_t)(act_h(H, l) + u / 4) * P
                               : reinterpret_cast<float4*>(a.h_out + l * HP + (size_t)p * H + u);
          float hn[UC];
          gru_epilogue<H, UC>(tm, bias + l * 4 * H, hprev, hn, A, row, u, hout, valid,
                              TRAIN ? act + (size_t)act_g(H, NL, l) * P : nullptr, TRAIN ? P : 1,
                              TRAIN ? a.hT[l] + ldh - ld + col : nullptr, ldh);
          if (TRAIN) {
            __syncwarp();
            tmem_st(tstate + l * H + u, hn);
          }
        }
        if (l + 1 < NL) stage_prev(l + 1);  // region b is free
      }
      if (failed) break;
      // ---- dense head: relu(h W1^T + b1) W2^T + b2 on the top layer's state,
      // or h W2^T + b2 without the hidden dense layer
      const float* b1 = bias + NL * 4 * H;
      const int n2 = d.nout();
      float yv[16];  // targets of this thread's 16 outputs, loaded ahead of the head
      if (TRAIN && valid && cq < n2 / 16) {
        const float* Y = a.Y + ((size_t)p * T + step) * d.c_out + cq * 16;
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
          const int left = d.c_out - (cq * 16 + i);
          if (a.y_pairs && left >= 2) {
            const float2 q = *reinterpret_cast<const float2*>(Y + i);
            yv[i] = q.x, yv[i + 1] = q.y;
          } else {
            yv[i] = left > 0 ? Y[i] : 0.0f;
            yv[i + 1] = left > 1 ? Y[i + 1] : 0.0f;
          }
        }
      }
      if (d.mlp) {
        if (!run_mma([&] { mma_run(tbase, sa, H, sw + 2 * L.w1, H, 128, H, false); })) break;
#pragma unroll 1
        for (int c2 = cq * (4 / CQ); c2 < (cq + 1) * (4 / CQ); ++c2) {  // 32 of the 128 units
          uint32_t signs = 0;
#pragma unroll
          for (int c = 2 * c2; c < 2 * c2 + 2; ++c) {
            float v[16];
            tmem_ld16(tm + c * 16, v);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              v[i] += b1[c * 16 + i];
              signs |= (v[i] > 0.0f ? 1u : 0u) << ((c & 1) * 16 + i);
              v[i] = fmaxf(v[i], 0.0f);
            }
            store_row<16>(A, row, c * 16, 128, v);
            if (TRAIN && valid)
#pragma unroll
              for (int i = 0; i < 16; ++i) a.y1T[(size_t)(c * 16 + i) * ld + col] = f2bf(v[i]);
          }
          if (TRAIN && valid)
            reinterpret_cast<uint32_t*>(act + (size_t)act_sign(H, NL) * P)[c2] = signs;
        }
      }
      if (!run_mma([&] {
            if (d.mlp)
              mma_run(tbase + 128, sa, 128, sw + 2 * L.w2, 128, n2, 128, false);
            else  // the single dense layer reads the top state in region a
              mma_run(tbase + 128, sa, H, sw + 2 * L.w2, H, n2, H, false);
          }))
        break;
      const float* b2 = b1 + d.mlp;
      for (int c = cq; c < n2 / 16; c += CQ) {  // 16-column chunks of the output
        float v[16];
        tmem_ld16(tm + 128 + c * 16, v);
        if (!valid) continue;
        if (!TRAIN) {
          float* o = a.out + (size_t)p * d.c_out + c * 16;
          const float* bo = b2 + c * 16;
          const int left = d.c_out - c * 16;
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
            if (a.out_pairs && i + 1 < left) {
              *reinterpret_cast<float2*>(o + i) = make_float2(v[i] + bo[i], v[i + 1] + bo[i + 1]);
            } else {
              if (i < left) o[i] = v[i] + bo[i];
              if (i + 1 < left) o[i + 1] = v[i + 1] + bo[i + 1];
            }
          }
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int j = c * 16 + i;
            v[i] = j < d.c_out ? v[i] + b2[j] - yv[i] : 0.0f;
            if (j < d.c_out) a.dyT[(size_t)j * ld + col] = f2bf(a.scale * v[i]);
          }
          loss += sum_squares(v);
        }
      }
      fence_before_sync();
      group_sync(1 + grp, GT);
      fence_after_sync();
    }
  }
  if (TRAIN) {  // per-block sum of squares (fixed order)
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (lane == 0) red[warp] = loss;
  }
  if (failed) {
    if (tg == 0) atomicOr(a.status, 4);
    // let copies and MMAs still in flight finish before their memory is released
    mbar_wait(wbar, 0, kWaitPolls);
    mbar_wait(bar, phase, kWaitPolls);
  }
  fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    fence_after_sync();
    tmem_dealloc(*tslot, TCOLS);
  }
  if (t != 0) return;
  if (TRAIN) {
    double s = 0.0;
    for (int w = 0; w < kFwdThreads / 32; ++w) s += red[w];
    a.loss_partial[blockIdx.x] = s;
  } else if (a.post.mail) {
    // every block's results are written before it counts itself, and the
    // last one posts
    __threadfence();
    if (atomicAdd(a.post.counter, 1u) == gridDim.x - 1) {
      __threadfence();
      *a.post.counter = 0u;
      a.post.mail->iv[0] = *reinterpret_cast<volatile int*>(a.status);
      mail_post(a.post.mail, a.post.seq);
    }
  }
}

// -- generic GEMM: C = A B^T ----------------------------------------------------
constexpr int kKC = 64;
__global__ void __launch_bounds__(kTile, 1)
    umma_gemm_kernel(const uint16_t* __restrict__ A, const uint16_t* __restrict__ B,
                     float* __restrict__ C, int M, int N, int K, uint32_t ncols, int* status) {
  extern __shared__ __align__(1024) uint8_t sm[];
  uint8_t* sa = sm;                       // 128 x kKC
  uint8_t* sb = sm + kTile * kKC * 2;     // N x kKC
  uint64_t* bar = reinterpret_cast<uint64_t*>(sb + 256 * kKC * 2);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 2);
  const int t = threadIdx.x, warp = t >> 5;
  if (warp == 0) tmem_alloc(tslot, ncols);
  if (t == 0) mbar_init(bar, 1);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tbase = *tslot;
  const int row0 = blockIdx.x * kTile;
  uint32_t phase = 0;
  bool failed = false;
  for (int k0 = 0; k0 < K && !failed; k0 += kKC) {
    const int kc = min(kKC, K - k0);
    for (int e = t; e < kTile * (kc / 8); e += kTile) {
      const int r = e / (kc / 8), q = e % (kc / 8);
      *reinterpret_cast<uint4*>(sa + kmajor_offset(r, q * 8, kc)) =
          *reinterpret_cast<const uint4*>(A + (size_t)(row0 + r) * K + k0 + q * 8);
    }
    for (int e = t; e < N * (kc / 8); e += kTile) {
      const int r = e / (kc / 8), q = e % (kc / 8);
      *reinterpret_cast<uint4*>(sb + kmajor_offset(r, q * 8, kc)) =
          *reinterpret_cast<const uint4*>(B + (size_t)r * K + k0 + q * 8);
    }
    fence_async_smem();
    fence_before_sync();
    __syncthreads();
    if (t == 0) {
      fence_after_sync();
      mma_run(tbase, smem_u32(sa), kc, smem_u32(sb), kc, N, kc, k0 > 0);
      mma_commit(bar);
    }
    if (!mbar_wait(bar, phase, kWaitPolls)) failed = true;
    phase ^= 1;
    failed = __syncthreads_or(failed);
    fence_after_sync();
  }
  if (!failed) {
    const int r = row0 + t;
    for (int c = 0; c < N / 16; ++c) {
      float v[16];
      tmem_ld16(tbase + ((uint32_t)(warp * 32) << 16) + c * 16, v);
      for (int i = 0; i < 16; ++i) C[(size_t)r * N + c * 16 + i] = v[i];
    }
  } else {
    if (t == 0) atomicOr(status, 4);
    mbar_wait(bar, phase, kWaitPolls);
  }
  fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    fence_after_sync();
    tmem_dealloc(tbase, ncols);
  }
}

template <bool TRAIN, int H, int NL, int G>
int launch_forward_groups(const NetDims& d, const PackedNet& pk, const FwdArgs& a, int blocks,
                          cudaStream_t st) {
  const PackLayout L = PackLayout::of(d);
  const FwdSmem S = FwdSmem::of(d, L.total, G);
  cudaFuncSetAttribute(patchnet_forward_kernel<TRAIN, H, NL, G>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                       TRAIN ? kSmemLimit - 1024 : kSmemLimit);  // beside its static part
  note_launch();
  patchnet_forward_kernel<TRAIN, H, NL, G>
      <<<blocks, kFwdThreads, S.total, st>>>(d, L, pk.w, pk.bias, a);
  return blocks;
}

// Two groups per block for inference with more tiles than SMs, where the
// second operand area fits beside the weights (not for 64 x 3), else one.
template <bool TRAIN, int H, int NL>
int launch_forward_shape(const NetDims& d, const PackedNet& pk, const FwdArgs& a, cudaStream_t st) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int ntiles = (a.P + kTile - 1) / kTile;
  if constexpr (!TRAIN)
    if (ntiles > sms && FwdSmem::of(d, PackLayout::of(d).total, 2).total + 256 <= kSmemMax)
      return launch_forward_groups<TRAIN, H, NL, 2>(d, pk, a, sms, st);
  return launch_forward_groups<TRAIN, H, NL, 1>(d, pk, a, ntiles < sms ? ntiles : sms, st);
}

// one instantiation per network size of Table 1; returns the blocks launched
template <bool TRAIN>
int launch_forward_impl(const NetDims& d, const PackedNet& pk, const FwdArgs& a, cudaStream_t st) {
  switch (d.hidden * 10 + d.layers) {
    case 321: return launch_forward_shape<TRAIN, 32, 1>(d, pk, a, st);
    case 322: return launch_forward_shape<TRAIN, 32, 2>(d, pk, a, st);
    case 323: return launch_forward_shape<TRAIN, 32, 3>(d, pk, a, st);
    case 641: return launch_forward_shape<TRAIN, 64, 1>(d, pk, a, st);
    case 642: return launch_forward_shape<TRAIN, 64, 2>(d, pk, a, st);
    case 643: return launch_forward_shape<TRAIN, 64, 3>(d, pk, a, st);
    default: return 0;  // rejected by net_supported
  }
}

}  // namespace

size_t patchnet_forward_smem(const NetDims& d) {
  return FwdSmem::of(d, PackLayout::of(d).total, 1).total + 256;  // and the static part
}

bool net_supported(const NetDims& d) {
  // (the input stream of the first layer's weight gradient, C_in + 1 rows
  // with the ones row, must fit the 144-row operand of that GEMM)
  if ((d.hidden != 32 && d.hidden != 64) || d.layers < 1 || d.layers > kMaxLayers ||
      (d.mlp != 128 && d.mlp != 0) || d.c_in < 1 || d.c_in > 127 || d.c_out < 1 ||
      d.c_out > 64 || d.nout() > 16 * kFwdWG || (d.bias != 0 && d.bias != 1))
    return false;
  return patchnet_forward_smem(d) <= kSmemMax && patchnet_backward_smem(d) <= kSmemMax;
}

void launch_pack(const NetDims& d, const PackJob* jobs, int n, const float* w, float* bias,
                 cudaStream_t st) {
  PackArgs a{};
  for (int q = 0; q < n; ++q) a.job[q] = jobs[q];
  a.n = n;
  a.w = w;
  a.bias = bias;
  note_launch();
  pack_kernel<<<dim3(32, n + (bias ? 1 : 0)), 256, 0, st>>>(a, d);
}

void launch_pack_weights(const NetDims& d, const float* w, PackedNet& pk, cudaStream_t st) {
  const PackLayout L = PackLayout::of(d);
  const NetOffsets o = d.offsets();
  const int H = d.hidden;
  PackJob jobs[kMaxPackJobs];
  int n = 0;
  for (int l = 0; l < d.layers; ++l) {
    const int c = l == 0 ? d.c_in : H, kx = L.kx[l];
    const float* Wih = w + o.wih[l];
    const float* Whh = w + o.whh[l];
    jobs[n++] = {Wih, pk.w + L.rz[l], c, 1, 2 * H, c, 2 * H, kx};
    jobs[n++] = {Wih + (size_t)2 * H * c, pk.w + L.in[l], c, 1, H, c, H, kx};
    jobs[n++] = {Whh, pk.w + L.hrz[l], H, 1, 2 * H, H, 2 * H, H};
    jobs[n++] = {Whh + (size_t)2 * H * H, pk.w + L.hn[l], H, 1, H, H, H, H};
  }
  if (d.mlp) jobs[n++] = {w + o.w1, pk.w + L.w1, H, 1, 128, H, 128, H};
  const int k2 = d.k2();
  jobs[n++] = {w + o.w2, pk.w + L.w2, k2, 1, d.c_out, k2, d.nout(), k2};
  launch_pack(d, jobs, n, w, pk.bias, st);
}

void launch_patchnet_forward(const NetDims& d, const PackedNet& pk, const uint16_t* x,
                             const float* h, float* h_out, float* out, int P, int* status,
                             cudaStream_t st, const NetPost& post) {
  if (P <= 0) return;
  FwdArgs a{};
  a.x = x;
  a.P = P;
  a.T = 1;
  a.h_in = h;
  a.h_out = h_out;
  a.out = out;
  a.out_pairs = d.c_out % 2 == 0 && (reinterpret_cast<uintptr_t>(out) & 7) == 0;
  a.status = status;
  a.post = post;
  launch_forward_impl<false>(d, pk, a, st);
}

int launch_patchnet_train_forward(const NetDims& d, const PackedNet& pk, const uint16_t* x,
                                  const float* Y, int B, int T, float scale, const TrainBufs& tb,
                                  int* status, cudaStream_t st) {
  if (B <= 0 || T <= 0) return 0;
  FwdArgs a{};
  a.x = x;
  a.P = B;
  a.T = T;
  a.Y = Y;
  a.y_pairs = d.c_out % 2 == 0 && (reinterpret_cast<uintptr_t>(Y) & 7) == 0;
  a.scale = scale;
  a.act = tb.act;
  a.xT = tb.xT;
  for (int l = 0; l < kMaxLayers; ++l) a.hT[l] = tb.hT[l];
  a.y1T = tb.y1T;
  a.dyT = tb.dyT;
  a.loss_partial = tb.loss_partial;
  a.status = status;
  return launch_forward_impl<true>(d, pk, a, st);
}

int launch_umma_gemm(const uint16_t* A, const uint16_t* B, float* C, int M, int N, int K,
                     int* status, cudaStream_t st) {
  if (M <= 0 || M % kTile || N < 16 || N > 256 || N % 16 || K < 16 || K % 16) return 1;
  uint32_t ncols = 32;
  while (ncols < (uint32_t)N) ncols <<= 1;
  const size_t smem = (size_t)kTile * kKC * 2 + (size_t)256 * kKC * 2 + 64;
  cudaFuncSetAttribute(umma_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  note_launch();
  umma_gemm_kernel<<<M / kTile, kTile, smem, st>>>(A, B, C, M, N, K, ncols, status);
  return 0;
}

}  // namespace dnnmg

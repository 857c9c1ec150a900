// mlp.cu -- training of the branching network on the GPU: forward on the
// tensor cores, softmax cross-entropy per decision node and backward (dW1^T on
// the tensor cores as dH^T * X) in one kernel, Adam with FP32 master weights, BF16 packing.
//
// Training data are the decision traces of the plain search (scuba_trace):
// node k has rows [node_row[k], node_row[k] + node_nrows[k]) -- one row per
// variable unassigned at that decision -- and per-row targets counting the
// variable's occurrences in falsified clauses of the node's subtree. The loss
// of a node is the cross-entropy between the normalised targets and the
// softmax of the scores over its rows.
//
// Master parameter layout (FP32, NPARAM = 1153): W1[i][j] at i*64 + j
// (i < 16 features, j < 64 hidden), b1[j] at 1024 + j, w2[j] at 1088 + j,
// b2 at 1152.
#include <cuda_runtime.h>

#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <map>
#include <string>

#include "../../include/scuba.h"
#include "learn.cuh"
#include "scuba_internal.h"

namespace scuba {
namespace mlpk {

using learn::mma_add;
using learn::MlpWeights;
using learn::NFEAT;
using learn::NHID;
using learn::NPARAM;
constexpr int OFF_B1 = NFEAT * NHID, OFF_W2 = OFF_B1 + NHID, OFF_B2 = OFF_W2 + NHID;
constexpr uint32_t FULL = 0xffffffffu;

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

// He-style initialisation from a counter-based stream (Box-Muller).
__global__ void k_init(float* master, uint64_t seed) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= NPARAM) return;
  float std = 0.0f;
  if (p < OFF_B1) std = sqrtf(2.0f / NFEAT);
  else if (p >= OFF_W2 && p < OFF_B2) std = sqrtf(1.0f / NHID);
  const uint64_t r1 = mix64(seed * 0x9E3779B97F4A7C15ULL + 2 * (uint64_t)p + 1);
  const uint64_t r2 = mix64(seed * 0x9E3779B97F4A7C15ULL + 2 * (uint64_t)p + 2);
  const float u1 = ((r1 >> 11) + 0.5f) * (1.0f / 9007199254740992.0f);
  const float u2 = (r2 >> 11) * (1.0f / 9007199254740992.0f);
  master[p] = std * sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
}

// Packed weight of parameter p (BF16 matrices transposed as the solver
// reads them, FP32 biases).
__device__ __forceinline__ void pack_one(const float* master, MlpWeights* W, int p) {
  if (p < OFF_B1) {
    const int i = p / NHID, j = p % NHID;
    W->w1t[j * NFEAT + i] = __float2bfloat16(master[p]);
  } else if (p < OFF_W2) {
    W->b1[p - OFF_B1] = master[p];
  } else if (p < OFF_B2) {
    W->w2[p - OFF_W2] = __float2bfloat16(master[p]);
  } else if (p == OFF_B2) {
    W->b2 = master[p];
    W->pad[0] = W->pad[1] = W->pad[2] = 0.0f;
  }
}

__global__ void k_pack(const float* master, MlpWeights* W) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < NPARAM) pack_one(master, W, p);
}

// ---- one 16-row tile on the tensor cores -----------------------------------
//
// The forward pass runs transposed, z^T = W1^T X^T: the weights are the A
// operand (four 16-unit tiles that stay in registers), the rows the B operand,
// so a lane loads its operand straight from a row (8 contiguous bytes) and the
// pre-activations of hidden units g, g + 8 at rows 2t, 2t + 1 land in the layout
// in which the backward pass needs dH^T as an A operand: dW1^T = dH^T X takes
// no trip of dH through shared memory, only X is transposed (movmatrix).
// The 16 features are numbered so that lane t's 8 bytes (features 4t .. 4t+3)
// are the logical columns 2t, 2t+1, 2t+8, 2t+9 of the mma; the sum over them
// does not depend on that numbering.

struct HiddenWeights {
  uint32_t a[4][4];         // W1^T: hidden units 16q .. 16q+15, logical features
  float b1[4][2], w2[4][2];  // units 16q + g, 16q + g + 8
};

__device__ __forceinline__ void load_hidden(const MlpWeights* W, int g, int t, HiddenWeights& H) {
#pragma unroll
  for (int q = 0; q < 4; q++) {
#pragma unroll
    for (int u = 0; u < 2; u++) {
      const int j = 16 * q + g + 8 * u;
      const uint32_t* r = reinterpret_cast<const uint32_t*>(W->w1t + j * NFEAT + 4 * t);
      H.a[q][u] = r[0];
      H.a[q][2 + u] = r[1];
      H.b1[q][u] = W->b1[j];
      H.w2[q][u] = __bfloat162float(W->w2[j]);
    }
  }
}

__device__ __forceinline__ uint32_t transpose8x8(uint32_t m) {
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(r) : "r"(m));
  return r;
}

// Lane (g, t)'s features 4t .. 4t+3 of one row; zeros past the end. WIDE: x is
// 8-byte aligned (rows are 32 bytes); otherwise the elements are read one by one.
template <bool WIDE>
__device__ __forceinline__ uint2 load_row(const __nv_bfloat16* x, int64_t row, int64_t end, int t) {
  uint2 v = make_uint2(0u, 0u);
  if (row < end) {
    const __nv_bfloat16* p = x + row * NFEAT + 4 * t;
    if (WIDE) {
      v = __ldg(reinterpret_cast<const uint2*>(p));
    } else {
      v.x = learn::pack_bf16(p[0], p[1]);
      v.y = learn::pack_bf16(p[2], p[3]);
    }
  }
  return v;
}

// The row of its tile whose score a lane keeps: lanes with g < 4 take one row
// each, lanes with g >= 4 repeat them.
__device__ __forceinline__ int lane_row(int g, int t) {
  return 8 * ((g >> 1) & 1) + 2 * t + (g & 1);
}

// Score (without the output bias) of row lane_row(g, t) of the tile whose
// rows g and g + 8 the lanes hold in x0 and x1.
__device__ __forceinline__ float tile_score(const HiddenWeights& H, uint2 x0, uint2 x1, int g) {
  float p[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
  for (int q = 0; q < 4; q++) {
#pragma unroll
    for (int h = 0; h < 2; h++) {
      float z[4];
      mma_add(z, H.a[q], h ? x1.x : x0.x, h ? x1.y : x0.y, H.b1[q][0], H.b1[q][0], H.b1[q][1],
              H.b1[q][1]);
      p[h][0] += fmaxf(z[0], 0.f) * H.w2[q][0] + fmaxf(z[2], 0.f) * H.w2[q][1];
      p[h][1] += fmaxf(z[1], 0.f) * H.w2[q][0] + fmaxf(z[3], 0.f) * H.w2[q][1];
    }
  }
  // sum over g (8 lanes), each step halving the rows a lane goes on with:
  // rows 8h + 2t + j end at the lanes with g = 2h + j (mod 4)
  const bool h = (g & 2) != 0, j = (g & 1) != 0;
  float r0 = h ? p[1][0] : p[0][0], r1 = h ? p[1][1] : p[0][1];
  r0 += __shfl_xor_sync(FULL, h ? p[0][0] : p[1][0], 8);
  r1 += __shfl_xor_sync(FULL, h ? p[0][1] : p[1][1], 8);
  float s = j ? r1 : r0;
  s += __shfl_xor_sync(FULL, j ? r0 : r1, 4);
  return s + __shfl_xor_sync(FULL, s, 16);
}

// Scores of all rows [0, rows): one warp per 16-row tile (grid-stride), the
// next tile's rows loaded while this one's are multiplied.
template <bool WIDE>
__global__ void __launch_bounds__(256) k_forward(const __nv_bfloat16* x, int64_t rows,
                                                 const MlpWeights* W, float* scores) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  HiddenWeights H;
  load_hidden(W, g, t, H);
  const float b2 = W->b2;
  const int64_t step = 16 * (int64_t)gridDim.x * (blockDim.x >> 5);
  int64_t r = 16 * ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
  uint2 x0 = load_row<WIDE>(x, r + g, rows, t), x1 = load_row<WIDE>(x, r + g + 8, rows, t);
  for (; r < rows; r += step) {
    const uint2 n0 = load_row<WIDE>(x, r + step + g, rows, t);
    const uint2 n1 = load_row<WIDE>(x, r + step + g + 8, rows, t);
    const float s = tile_score(H, x0, x1, g) + b2;
    const int64_t row = r + lane_row(g, t);
    if (g < 4 && row < rows) scores[row] = s;
    x0 = n0;
    x1 = n1;
  }
}

// Softmax statistics of a set of scores: the maximum and the sum of
// exp(score - maximum), with the set's targets summed beside them.
struct SoftStat {
  float m, e, t;
};

// exp(s - m), 0 for s = -inf beside an m that is still -inf.
__device__ __forceinline__ float exp_from(float s, float m) {
  return expf(s - (m == -INFINITY ? 0.0f : m));
}

__device__ __forceinline__ SoftStat merge(const SoftStat& a, const SoftStat& b) {
  const float m = fmaxf(a.m, b.m);
  return SoftStat{m, a.e * exp_from(a.m, m) + b.e * exp_from(b.m, m), a.t + b.t};
}

// Loss and gradients of trace nodes [k0, k1) in one pass per node: scores,
// softmax cross-entropy against the normalised targets, dS = softmax - target
// and the gradients of every parameter (dW1 on the tensor cores from dH in
// BF16). `split` blocks (a cluster) share a node's 16-row tiles and exchange
// their softmax statistics through distributed shared memory; a block takes one
// node, keeps its gradients in registers and adds them to the global sums once.
// (Blocks that stride over the nodes were slower: 101 against 91 us at 1,001
// nodes.) A thread keeps the scores of its own rows in dS between the two passes
// over the node's rows; the rows' features come from L1 or L2 the second time.
//
// Many nodes: about 700 instructions per 16-row tile, the block's reduction
// included (activations, masks and sums of 64 hidden units per row), against 640
// bytes; 1,001 nodes of 300 to 1,500 rows take 79 us, of which their issue is 33 and
// most of the rest the uneven nodes over 3.3 waves of blocks (scores, loss and
// gradient as kernels of their own: 383). A minibatch of 64 nodes has 64,000 rows,
// too few for one warp per node: the split is the one that fills 2 blocks on each
// of the 152 SMs (17 us, was 213).
constexpr int kGradWarps = 8;
constexpr int kGradStride = 17 * NHID + 2 * NHID + 4;  // floats one warp stages for the reduction

template <bool WIDE>
__global__ void __launch_bounds__(32 * kGradWarps, 2)
    k_node_grad(const int64_t* node_row, const int32_t* node_nrows, const int32_t* node_closed,
                int64_t k0, int64_t k1, const __nv_bfloat16* x, const MlpWeights* W,
                const float* target, float* dS, float* grad, int split) {
  __shared__ float stage[kGradWarps][kGradStride];
  __shared__ SoftStat warp_stat[kGradWarps];
  __shared__ SoftStat cta_stat;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int rank = blockIdx.x % split;
  HiddenWeights H;
  load_hidden(W, g, t, H);
  const float b2 = W->b2;
  float cw1[4][2][4], gw2[4][2], gb1[4][2], gb2 = 0.0f, ce = 0.0f;
#pragma unroll
  for (int q = 0; q < 4; q++) {
    gw2[q][0] = gw2[q][1] = gb1[q][0] = gb1[q][1] = 0.0f;
#pragma unroll
    for (int f = 0; f < 2; f++) cw1[q][f][0] = cw1[q][f][1] = cw1[q][f][2] = cw1[q][f][3] = 0.0f;
  }
  const int64_t k = k0 + blockIdx.x / split;
  const int64_t step = 16 * (int64_t)kGradWarps * split;
  const int64_t r0 = node_row[k], end = r0 + node_nrows[k];
  const int64_t first = r0 + 16 * ((int64_t)wib * split + rank);
  // scores and their statistics
  SoftStat st{-INFINITY, 0.0f, 0.0f};
  uint2 x0 = load_row<WIDE>(x, first + g, end, t), x1 = load_row<WIDE>(x, first + g + 8, end, t);
  for (int64_t r = first; r < end; r += step) {
    const uint2 n0 = load_row<WIDE>(x, r + step + g, end, t);
    const uint2 n1 = load_row<WIDE>(x, r + step + g + 8, end, t);
    const int64_t row = r + lane_row(g, t);
    const bool mine = g < 4 && row < end;
    const float tv = mine ? target[row] : 0.0f;
    const float s = tile_score(H, x0, x1, g) + b2;
    if (mine) {
      dS[row] = s;
      st.t += tv;
      if (s > st.m) {
        st.e *= expf(st.m - s);
        st.m = s;
      }
      st.e += exp_from(s, st.m);
    }
    x0 = n0;
    x1 = n1;
  }
  for (int d = 16; d > 0; d >>= 1)
    st = merge(st, SoftStat{__shfl_xor_sync(FULL, st.m, d), __shfl_xor_sync(FULL, st.e, d),
                            __shfl_xor_sync(FULL, st.t, d)});
  if (lane == 0) warp_stat[wib] = st;
  __syncthreads();
  st = warp_stat[0];
  for (int w = 1; w < kGradWarps; w++) st = merge(st, warp_stat[w]);
  if (split > 1) {
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    if (threadIdx.x == 0) cta_stat = st;
    cl.sync();
    st = *cl.map_shared_rank(&cta_stat, 0);
    for (int b = 1; b < split; b++) st = merge(st, *cl.map_shared_rank(&cta_stat, b));
  }
  if (!(node_closed[k] && end - r0 > 1 && st.t > 0.0f)) {  // the node takes no part
    for (int64_t r = first; r < end; r += step) {
      const int64_t row = r + lane_row(g, t);
      if (g < 4 && row < end) dS[row] = 0.0f;
    }
    if (split > 1) cooperative_groups::this_cluster().sync();  // the others have read cta_stat
    return;
  }
  // (probabilities from the sum itself: its logarithm, rounded at the size of the
  // scores, would move all of a node's by up to 2.4e-7 one way)
  const float lse = st.m + logf(st.e), inv_e = 1.0f / st.e;
  for (int64_t r = first; r < end; r += step) {
    x0 = load_row<WIDE>(x, r + g, end, t);
    x1 = load_row<WIDE>(x, r + g + 8, end, t);
    const int64_t row = r + lane_row(g, t);
    float ds_mine = 0.0f;
    if (g < 4 && row < end) {
      const float s = dS[row], tn = target[row] / st.t;
      ds_mine = expf(s - st.m) * inv_e - tn;
      dS[row] = ds_mine;
      ce -= tn * (s - lse);
      gb2 += ds_mine;
    }
    float ds[2][2];  // rows 8h + 2t + j
#pragma unroll
    for (int h = 0; h < 2; h++)
#pragma unroll
      for (int j = 0; j < 2; j++)
        ds[h][j] = __shfl_sync(FULL, ds_mine, 4 * (2 * h + j) + t);
    // X as a B operand (rows x logical features): b[f][h] for rows 8h .. 8h+7
    const uint32_t bx[2][2] = {{transpose8x8(x0.x), transpose8x8(x1.x)},
                               {transpose8x8(x0.y), transpose8x8(x1.y)}};
#pragma unroll
    for (int q = 0; q < 4; q++) {
      uint32_t dh[4];  // dH^T: units 16q .. 16q+15, the tile's rows
#pragma unroll
      for (int h = 0; h < 2; h++) {
        float z[4], d[4];
        mma_add(z, H.a[q], h ? x1.x : x0.x, h ? x1.y : x0.y, H.b1[q][0], H.b1[q][0], H.b1[q][1],
                H.b1[q][1]);
#pragma unroll
        for (int u = 0; u < 4; u++)
          d[u] = z[u] > 0.f ? ds[h][u & 1] * H.w2[q][u >> 1] : 0.f;
#pragma unroll
        for (int u = 0; u < 4; u++) {
          if (z[u] > 0.f) gw2[q][u >> 1] += z[u] * ds[h][u & 1];
          gb1[q][u >> 1] += d[u];
        }
        dh[2 * h] = learn::pack_bf16(__float2bfloat16(d[0]), __float2bfloat16(d[1]));
        dh[2 * h + 1] = learn::pack_bf16(__float2bfloat16(d[2]), __float2bfloat16(d[3]));
      }
#pragma unroll
      for (int f = 0; f < 2; f++)
        mma_add(cw1[q][f], dh, bx[f][0], bx[f][1], cw1[q][f][0], cw1[q][f][1], cw1[q][f][2],
                cw1[q][f][3]);
    }
  }
  if (split > 1) cooperative_groups::this_cluster().sync();  // every remote read is done
  // one sum per parameter over the block's warps, then global
  float* mine = stage[wib];
#pragma unroll
  for (int q = 0; q < 4; q++) {
#pragma unroll
    for (int u = 0; u < 2; u++) {
      const int j = 16 * q + g + 8 * u;
#pragma unroll
      for (int f = 0; f < 2; f++) {  // logical features 2t, 2t+1 (f = 0), 2t+8, 2t+9 (f = 1)
        mine[17 * j + 4 * t + 2 * f] = cw1[q][f][2 * u];
        mine[17 * j + 4 * t + 2 * f + 1] = cw1[q][f][2 * u + 1];
      }
      float a = gb1[q][u], b = gw2[q][u];
      a += __shfl_xor_sync(FULL, a, 1);
      a += __shfl_xor_sync(FULL, a, 2);
      b += __shfl_xor_sync(FULL, b, 1);
      b += __shfl_xor_sync(FULL, b, 2);
      if (t == 0) {
        mine[17 * NHID + j] = a;
        mine[18 * NHID + j] = b;
      }
    }
  }
  for (int d = 16; d > 0; d >>= 1) {
    gb2 += __shfl_xor_sync(FULL, gb2, d);
    ce += __shfl_xor_sync(FULL, ce, d);
  }
  if (lane == 0) {
    mine[19 * NHID] = gb2;
    mine[19 * NHID + 1] = ce;
    mine[19 * NHID + 2] = rank == 0 && wib == 0 ? 1.0f : 0.0f;  // nodes used
  }
  __syncthreads();
  for (int p = threadIdx.x; p < NPARAM + 2; p += blockDim.x) {
    const int at = p < OFF_B1 ? 17 * (p % NHID) + p / NHID : 17 * NHID + (p - OFF_B1);
    float s = 0.0f;
#pragma unroll
    for (int w = 0; w < kGradWarps; w++) s += stage[w][at];
    if (s != 0.0f) atomicAdd(&grad[p], s);
  }
}

// One training step after a minibatch's gradient: Adam (Kingma and Ba,
// Algorithm 1; beta 0.9/0.999, eps 1e-8) on the mean gradient over the
// minibatch's nodes, then the packed weight of each parameter, the epoch's
// loss sums, and the other gradient buffer cleared for the next minibatch
// (the two buffers alternate, so nothing here reads what it clears).
__global__ void k_adam_pack(float* master, float* m, float* v, const float* grad,
                            float* grad_next, MlpWeights* W, float lr, int step,
                            float* epoch_loss) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= NPARAM + 2) return;
  grad_next[p] = 0.0f;
  if (p >= NPARAM) {
    if (epoch_loss) epoch_loss[p - NPARAM] += grad[p];  // summed loss, nodes used
    return;
  }
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float nodes = grad[NPARAM + 1];
  const float s = nodes > 0.0f ? 1.0f / nodes : 0.0f;  // mean over nodes
  const float gr = grad[p] * s;
  m[p] = b1 * m[p] + (1.0f - b1) * gr;
  v[p] = b2 * v[p] + (1.0f - b2) * gr * gr;
  const float mh = m[p] / (1.0f - powf(b1, (float)step));
  const float vh = v[p] / (1.0f - powf(b2, (float)step));
  master[p] -= lr * mh / (sqrtf(vh) + eps);
  pack_one(master, W, p);
}

}  // namespace mlpk

namespace {

struct TrainScratch {
  void* dS = nullptr;
  size_t dS_cap = 0;
  void* grad = nullptr;  // 2 x (NPARAM + 2): gradient, loss sum, nodes used (ping-pong)
};

std::map<int, TrainScratch>& train_scratch() {
  static std::map<int, TrainScratch> m;
  return m;
}

// SMs of the current device (read once per device and process).
int sm_count() {
  static std::atomic<int> known[64];
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 152;
  if (dev < 64 && (sms = known[dev].load(std::memory_order_relaxed)) > 0) return sms;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 152;
  if (dev < 64) known[dev].store(sms, std::memory_order_relaxed);
  return sms;
}

// Whether the feature rows allow 8-byte loads (a caller may pass any 2-byte
// aligned pointer).
bool wide_rows(const void* x) { return (reinterpret_cast<uintptr_t>(x) & 7) == 0; }

int fail(const char* what, cudaError_t e) {
  set_error(std::string(what) + ": " + cudaGetErrorString(e));
  return SCUBA_ERR_CUDA;
}

}  // namespace
}  // namespace scuba

using namespace scuba;

extern "C" int scuba_mlp_layout(int64_t* out) {
  if (!out) return SCUBA_ERR_ARG;
  out[0] = (int64_t)sizeof(learn::MlpWeights);
  out[1] = learn::NPARAM;
  out[2] = learn::NFEAT;
  out[3] = learn::NHID;
  return SCUBA_OK;
}

extern "C" int scuba_mlp_init(float* master, void* weights, uint64_t seed, void* stream) {
  if (!master || !weights) return SCUBA_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  mlpk::k_init<<<(learn::NPARAM + 255) / 256, 256, 0, st>>>(master, seed);
  mlpk::k_pack<<<(learn::NPARAM + 255) / 256, 256, 0, st>>>(
      master, static_cast<learn::MlpWeights*>(weights));
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? SCUBA_OK : fail("scuba_mlp_init", e);
}

extern "C" int scuba_mlp_pack(const float* master, void* weights, void* stream) {
  if (!master || !weights) return SCUBA_ERR_ARG;
  mlpk::k_pack<<<(learn::NPARAM + 255) / 256, 256, 0, (cudaStream_t)stream>>>(
      master, static_cast<learn::MlpWeights*>(weights));
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? SCUBA_OK : fail("scuba_mlp_pack", e);
}

extern "C" int scuba_mlp_forward(const uint16_t* x, int64_t rows, const void* weights,
                                 float* scores, void* stream) {
  if (rows < 0 || (rows > 0 && (!x || !weights || !scores))) return SCUBA_ERR_ARG;
  if (rows == 0) return SCUBA_OK;
  const int64_t tiles = (rows + 15) / 16;
  // 8 tiles per block, at most 8 blocks on each SM: a warp of a large call
  // then loads its next tile while it multiplies this one
  const int grid = (int)std::min<int64_t>((tiles + 7) / 8, (int64_t)sm_count() * 8);
  const __nv_bfloat16* xb = reinterpret_cast<const __nv_bfloat16*>(x);
  const learn::MlpWeights* W = static_cast<const learn::MlpWeights*>(weights);
  if (wide_rows(xb))
    mlpk::k_forward<true><<<grid, 256, 0, (cudaStream_t)stream>>>(xb, rows, W, scores);
  else
    mlpk::k_forward<false><<<grid, 256, 0, (cudaStream_t)stream>>>(xb, rows, W, scores);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? SCUBA_OK : fail("scuba_mlp_forward", e);
}

// The loss and gradients of nodes [k0, k1) into grad (cleared by the caller).
static void grad_kernels(const scuba_trace* tr, int64_t k0, int64_t k1, const void* weights,
                         float* grad, float* dS, cudaStream_t st) {
  const int64_t nodes = k1 - k0;
  if (nodes <= 0) return;
  // blocks per node: as many (1, 2, 4, 8) as still fit two blocks on each SM
  const int64_t slots = 2 * (int64_t)sm_count();
  int split = 1;
  while (split < 8 && 2 * split * nodes <= slots) split *= 2;
  const __nv_bfloat16* x = reinterpret_cast<const __nv_bfloat16*>(tr->x);
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = split;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nodes * split));
  cfg.blockDim = dim3(32 * mlpk::kGradWarps);
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(
      &cfg, wide_rows(x) ? mlpk::k_node_grad<true> : mlpk::k_node_grad<false>, tr->node_row,
      tr->node_nrows, tr->node_closed, k0, k1, x, static_cast<const learn::MlpWeights*>(weights),
      tr->target, dS, grad, split);
}

static int grad_impl(const scuba_trace* tr, int64_t k0, int64_t k1, const void* weights,
                     float* grad, float* dS, cudaStream_t st) {
  cudaMemsetAsync(grad, 0, sizeof(float) * (learn::NPARAM + 2), st);
  grad_kernels(tr, k0, k1, weights, grad, dS, st);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? SCUBA_OK : fail("scuba_mlp_grad", e);
}

extern "C" int scuba_mlp_grad(const scuba_trace* tr, int64_t node_begin, int64_t node_end,
                              const void* weights, float* grad, float* dS, void* stream) {
  if (!tr || !weights || !grad || !dS || node_begin < 0 || node_end < node_begin)
    return SCUBA_ERR_ARG;
  return grad_impl(tr, node_begin, node_end, weights, grad, dS, (cudaStream_t)stream);
}

extern "C" int scuba_mlp_train(const scuba_trace* tr, int64_t nodes, float* master, float* adam_m,
                               float* adam_v, void* weights, int32_t epochs, int32_t batch_nodes,
                               float lr, float* epoch_loss, void* stream) {
  if (!tr || !master || !adam_m || !adam_v || !weights || epochs < 0 || batch_nodes < 1 ||
      nodes < 0 || nodes > tr->max_nodes || !(lr > 0.0f))
    return SCUBA_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  int dev = 0;
  cudaGetDevice(&dev);
  TrainScratch& S = train_scratch()[dev];
  const size_t need = sizeof(float) * (size_t)std::max<int64_t>(tr->max_rows, 1);
  if (S.dS_cap < need) {
    if (S.dS) cudaFree(S.dS);
    S.dS = nullptr;
    S.dS_cap = 0;
    if (cudaMalloc(&S.dS, need) != cudaSuccess) return SCUBA_ERR_NOMEM;
    S.dS_cap = need;
  }
  const size_t gwords = learn::NPARAM + 2;
  if (!S.grad && cudaMalloc(&S.grad, sizeof(float) * 2 * gwords) != cudaSuccess)
    return SCUBA_ERR_NOMEM;
  float* gbuf = static_cast<float*>(S.grad);
  float* dS = static_cast<float*>(S.dS);
  cudaMemsetAsync(adam_m, 0, sizeof(float) * learn::NPARAM, st);
  cudaMemsetAsync(adam_v, 0, sizeof(float) * learn::NPARAM, st);
  cudaMemsetAsync(gbuf, 0, sizeof(float) * 2 * gwords, st);
  if (epoch_loss) cudaMemsetAsync(epoch_loss, 0, sizeof(float) * 2 * (size_t)epochs, st);
  // two launches per minibatch: loss and gradients, Adam + packing (which also
  // clears the other gradient buffer for the next minibatch)
  int step = 0;
  for (int ep = 0; ep < epochs; ep++) {
    for (int64_t k0 = 0; k0 < nodes; k0 += batch_nodes) {
      const int64_t k1 = std::min<int64_t>(nodes, k0 + batch_nodes);
      float* grad = gbuf + (size_t)(step & 1) * gwords;
      float* grad_next = gbuf + (size_t)((step + 1) & 1) * gwords;
      grad_kernels(tr, k0, k1, weights, grad, dS, st);
      step++;
      mlpk::k_adam_pack<<<(learn::NPARAM + 2 + 255) / 256, 256, 0, st>>>(
          master, adam_m, adam_v, grad, grad_next, static_cast<learn::MlpWeights*>(weights),
          lr, step, epoch_loss ? epoch_loss + 2 * ep : nullptr);
    }
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? SCUBA_OK : fail("scuba_mlp_train", e);
}

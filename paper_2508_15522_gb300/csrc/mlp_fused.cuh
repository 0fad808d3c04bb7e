// The proposal network's step in four launches, for networks whose padded
// widths are at most 256: forward of all layers, loss and backward of all
// layers, weight and bias gradients of all layers, and the update (gradient
// sums, Adam, the bfloat16 operands).  Every product, sum and rounding is that of
// the layer-by-layer kernels in mlp.cu, in the same order, so both give the
// same bits; what changes is how often the chip is started and how often an
// activation goes through memory.
//
// A training step of 2048 rows x 80-256-256-256-19 is 1.9 GFLOP, about 2 us of
// tensor time, and took 147 us as 45 dependent launches of 3 to 8 us, the loss
// (one thread per target) alone 25 us.
#pragma once

#include <cuda_bf16.h>

#include "internal.h"

namespace {

constexpr int kFusedMaxL = 8;       // layers
constexpr int kFusedW = 256;        // widest padded layer
constexpr int kFusedLd = kFusedW + 8;

// bfloat16 operands in the order of the tensor-core fragments: for the
// product over k of 32 k values and 8 outputs n, lane (n % 8) 4 + (k / 2) % 4
// holds eight consecutive elements, so a warp reads an n8 x k32 tile as 512
// contiguous bytes.
__host__ __device__ __forceinline__ size_t frag_index(int n, int k, int kp32) {
  const int r = k & 31, kk = r & 15;
  return ((((size_t)(n >> 3) * kp32 + (k >> 5)) * 32 + ((n & 7) * 4 + ((kk & 7) >> 1))) << 3) + (r >> 4) * 4 +
         (kk >> 3) * 2 + (kk & 1);
}
__host__ __device__ __forceinline__ int k32(int k) { return (k + 31) >> 5; }

struct FusedNet {
  int L, rows, Mp;
  int size[kFusedMaxL + 1], pad[kFusedMaxL + 1];
  size_t woff[kFusedMaxL], boff[kFusedMaxL];
  float* P;                           // parameters
  __nv_bfloat16* Wf[kFusedMaxL];      // forward operand: n = output, k = input
  __nv_bfloat16* Wr[kFusedMaxL];      // backward operand: n = input, k = output
  __nv_bfloat16* H[kFusedMaxL];       // layer inputs [Mp][pad[l]] (training)
  float* Gf[kFusedMaxL];              // dL/da [Mp][pad[l + 1]]
  __nv_bfloat16* Gb[kFusedMaxL];      // the same as a bfloat16 operand
  float* part[kFusedMaxL];            // weight-gradient parts [S][pad[l + 1]][pad[l]]
  float* dbp[kFusedMaxL];             // bias-gradient parts [chunks][size[l + 1]]
  int S[kFusedMaxL];                  // parts of the weight gradient
  int rpc, chunks;                    // rows per part of the bias gradient
  float* Y;                           // outputs [rows][size[L]]
  float *Gr, *Am, *Av;                // gradients, Adam moments
};

// Where the input rows come from: X (FP32 rows), or a descriptor followed by
// normal noise from the counter (base + row) * 64 + j hashed with the seed.
struct FusedInput {
  const float* X;
  const float* desc;
  int n_desc;
  unsigned long long seed, base;
};

// Targets of the loss: row b of T, or (n_all > 0) row
// splitmix64(seed ^ splitmix64(base + b)) mod n_all.
struct FusedLoss {
  const float *T, *mask;
  int n_targets, K, n_all;
  unsigned long long seed, base;
  float w_q, w_t, tile_x, tile_y;
  float* loss;
  int* winner;
};

__device__ __forceinline__ void mma_bf16(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void ldsm4(const void* smem, unsigned (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((unsigned)__cvta_generic_to_shared(smem)));
}
__device__ __forceinline__ void ldsm4_t(const void* smem, unsigned (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((unsigned)__cvta_generic_to_shared(smem)));
}

// The four launches of a step overlap: each is started when every block of the
// one before has called next_may_start(), and waits in previous_done() until that
// one has ended and its writes are visible.  next_may_start() always stands
// behind previous_done(), so what runs ahead of the wait sees the end of
// every launch but the one before, and runs beside that one alone: the inputs
// (written where only the gradients read), the weights of the backward pass (the
// forward does not write them), the optimiser's state.  At 2048 rows x
// 80-256-256-256-19 a step took 48 us, about 6 of them between the launches; now 42.
__device__ __forceinline__ void previous_done() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void next_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Weights are written by the launch before: an ordinary load that stays behind
// previous_done() (a read-only load may not be used while another grid writes).
__device__ __forceinline__ uint4 load_weights(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}

// A warp's share of a product: the n8 tiles w + 8 c (c < 4, below nt) of the
// fragment-ordered operand B, k = 0 .. 32 kp - 1.  The whole share of a layer (up
// to 128 registers) is requested at once and one layer ahead: the weights come
// from L2, and a load per step of 32 left the kernels waiting (forward 27 us,
// backward 34 us at 2048 rows, now 15 and 15).
struct RowsB {
  uint4 v[4][kFusedW / 32];
};
// FULL: 256 inputs and 256 outputs, no tile of the share is missing.
template <bool FULL>
__device__ __forceinline__ void rows_load_t(RowsB& B, const __nv_bfloat16* W, int kp, int nt, int w, int lane) {
  const uint4* b = (const uint4*)W + lane;
#pragma unroll
  for (int p = 0; p < kFusedW / 32; ++p)
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (FULL || (p < kp && w + 8 * c < nt)) 
        B.v[c][p] = load_weights(b + ((w + 8 * c) * (FULL ? kFusedW / 32 : kp) + p) * 32);
}
__device__ __forceinline__ bool rows_full(int kp, int nt) { return kp == kFusedW / 32 && nt == kFusedW / 8; }
__device__ __forceinline__ void rows_load(RowsB& B, const __nv_bfloat16* W, int kp, int nt, int w, int lane) {
  if (rows_full(kp, nt)) rows_load_t<true>(B, W, kp, nt, w, lane);
  else rows_load_t<false>(B, W, kp, nt, w, lane);
}
// acc[i][c] += A (16 MT rows of sA) x B
template <int MT, bool FULL>
__device__ __forceinline__ void rows_gemm_t(const __nv_bfloat16 (*sA)[kFusedLd], const RowsB& B, int kp, int nt, int w,
                                            int lane, float (&acc)[MT][4][4]) {
  const __nv_bfloat16* a = &sA[(lane & 7) + ((lane >> 3) & 1) * 8][(lane >> 4) * 8];
#pragma unroll
  for (int p = 0; p < kFusedW / 32; ++p) {
    if (!FULL && p >= kp) break;
#pragma unroll
    for (int i = 0; i < MT; ++i) {
      unsigned a0[4], a1[4];
      ldsm4(a + 16 * i * kFusedLd + 32 * p, a0);
      ldsm4(a + 16 * i * kFusedLd + 32 * p + 16, a1);
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (FULL || w + 8 * c < nt) mma_bf16(acc[i][c], a0, B.v[c][p].x, B.v[c][p].y);
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (FULL || w + 8 * c < nt) mma_bf16(acc[i][c], a1, B.v[c][p].z, B.v[c][p].w);
    }
  }
}
template <int MT>
__device__ __forceinline__ void rows_gemm(const __nv_bfloat16 (*sA)[kFusedLd], const RowsB& B, int kp, int nt, int w,
                                          int lane, float (&acc)[MT][4][4]) {
  if (rows_full(kp, nt)) rows_gemm_t<MT, true>(sA, B, kp, nt, w, lane, acc);
  else rows_gemm_t<MT, false>(sA, B, kp, nt, w, lane, acc);
}

// Forward of 16 MT rows per block of 8 warps, all layers; every warp has the
// outputs of up to four n8 tiles.  The weights come from L2 in fragment order
// (0.35 MB a block); activations stay in shared memory, and are written for
// the backward pass when `train`.  16 rows a block fill the chip at a training
// batch of 2048; from 8192 rows 64 rows a block read the weights a quarter as
// often.
template <int MT>
__global__ void __launch_bounds__(256) fused_forward_kernel(FusedNet net, FusedInput in, int train) {
  extern __shared__ __align__(16) __nv_bfloat16 smem_h[];
  __nv_bfloat16 (*sH[2])[kFusedLd] = {(__nv_bfloat16 (*)[kFusedLd])smem_h,
                                      (__nv_bfloat16 (*)[kFusedLd])(smem_h + (size_t)16 * MT * kFusedLd)};
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int m0 = blockIdx.x * 16 * MT;
  if (in.X) previous_done();          // rows from memory: the launch before may write them
  {
    const int ip = net.pad[0], ip32 = 32 * k32(ip), n_in = net.size[0];
    // 16 threads a row, columns 16 apart: the noise inputs (a logarithm, a square
    // root and a cosine) fall to all threads alike
    for (int r = tid >> 4; r < 16 * MT; r += 16)
      for (int k = tid & 15; k < ip32; k += 16) {
        const int m = m0 + r;
        float v = 0.f;
        if (m < net.rows && k < n_in) {
          if (in.X) v = in.X[(size_t)m * n_in + k];
          else if (k < in.n_desc) v = in.desc[k];
          else v = normal_of(splitmix64(in.seed ^ splitmix64(((in.base + (unsigned long long)m) << 6) + (k - in.n_desc))));
        }
        const __nv_bfloat16 b = __float2bfloat16(v);
        sH[0][r][k] = b;
        if (train && k < ip && m < net.Mp) net.H[0][(size_t)m * ip + k] = b;
      }
  }
  previous_done();
  next_may_start();
  RowsB B;
  rows_load(B, net.Wf[0], k32(net.pad[0]), net.pad[1] >> 3, w, lane);
  __syncthreads();
  for (int l = 0; l < net.L; ++l) {
    const int op = net.pad[l + 1], nt = op >> 3, n_out = net.size[l + 1], cur = l & 1;
    const bool last = l == net.L - 1;
    float acc[MT][4][4];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[i][c][v] = 0.f;
    rows_gemm<MT>(sH[cur], B, k32(net.pad[l]), nt, w, lane, acc);
    if (!last) rows_load(B, net.Wf[l + 1], k32(op), net.pad[l + 2] >> 3, w, lane);
    const float* bias = net.P + net.boff[l];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int j = 8 * (w + 8 * c) + 2 * (lane & 3);
      if (w + 8 * c >= nt) continue;
      const float b0 = j < n_out ? bias[j] : 0.f, b1 = j + 1 < n_out ? bias[j + 1] : 0.f;
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = 16 * i + (lane >> 2) + 8 * h, m = m0 + r;
          const bool live = m < net.rows;
          const float x = live && j < n_out ? acc[i][c][2 * h] + b0 : 0.f;
          const float y = live && j + 1 < n_out ? acc[i][c][2 * h + 1] + b1 : 0.f;
          if (last) {
            if (live && j < n_out) net.Y[(size_t)m * n_out + j] = x;
            if (live && j + 1 < n_out) net.Y[(size_t)m * n_out + j + 1] = y;
          } else {
            const __nv_bfloat162 v = __halves2bfloat162(__float2bfloat16(fmaxf(x, 0.f)), __float2bfloat16(fmaxf(y, 0.f)));
            *(__nv_bfloat162*)&sH[cur ^ 1][r][j] = v;
            if (train && m < net.Mp) *(__nv_bfloat162*)&net.H[l + 1][(size_t)m * op + j] = v;
          }
        }
    }
    if (!last && (op & 31))      // the next product runs over whole steps of 32
      for (int e = tid; e < 16 * MT * 16; e += 256) sH[cur ^ 1][e >> 4][op + (e & 15)] = __float2bfloat16(0.f);
    __syncthreads();
  }
}

// Distance of output o to target t (see gridff.h), from the torsions'
// 1 - cos(theta - theta*) in cs.
__device__ __forceinline__ float pose_loss(const FusedLoss& q, const float* o, const float* t, const float* mk,
                                           const float* cs) {
  float dx = o[0] - t[0], dy = o[1] - t[1], dz = o[2] - t[2];
  dx -= q.tile_x * rintf(dx / q.tile_x);
  dy -= q.tile_y * rintf(dy / q.tile_y);
  float nu = sqrtf(o[3] * o[3] + o[4] * o[4] + o[5] * o[5] + o[6] * o[6]);
  nu = fmaxf(nu, 1e-12f);
  const float s = (o[3] * t[3] + o[4] * t[4] + o[5] * t[5] + o[6] * t[6]) / nu;
  float d = dx * dx + dy * dy + dz * dz + q.w_q * (1.f - s * s);
  if (mk)
    for (int j = 0; j < 12; ++j) d += q.w_t * mk[j] * cs[j];
  return d;
}

__device__ __forceinline__ int target_row(const FusedLoss& q, int b) {
  return q.n_all > 0 ? (int)(splitmix64(q.seed ^ splitmix64(q.base + b)) % (unsigned long long)q.n_all) : b;
}

// Loss and backward of 16 rows per block.  A block evaluates every proposal of
// the targets that touch its rows (one thread each), so rows are split without
// regard to the proposals per target; the block with a target's first row
// writes its loss.  Writes dL/da of every layer in FP32 (bias gradients) and
// as the bfloat16 operand (weight gradients).
constexpr int kLossMax = 512;       // proposals evaluated per block at most: K <= 248
constexpr int kLossTargets = 20;    // targets per block at most (K = 1: 16)
__global__ void __launch_bounds__(256) fused_backward_kernel(FusedNet net, FusedLoss q) {
  __shared__ __align__(16) __nv_bfloat16 sG[2][16][kFusedLd];
  __shared__ float s_cos[kLossMax * 12], s_d[kLossMax];
  __shared__ int s_row[kLossTargets], s_win[kLossTargets];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int m0 = blockIdx.x * 16, L = net.L, K = q.K, n_out = net.size[L], opl = net.pad[L];
  const int ba = m0 / K, bb = min(q.n_targets - 1, (m0 + 15) / K), nb = bb - ba + 1;
  RowsB B;
  if (L > 1) rows_load(B, net.Wr[L - 1], k32(opl), net.pad[L - 1] >> 3, w, lane);
  if (tid < nb) s_row[tid] = target_row(q, ba + tid);
  for (int e = tid; e < 16 * 32 * k32(opl); e += 256) sG[0][e / (32 * k32(opl))][e % (32 * k32(opl))] = __float2bfloat16(0.f);
  previous_done();
  next_may_start();
  __syncthreads();
  const float* Yb = net.Y + (size_t)ba * K * n_out;
  if (q.mask)
    for (int e = tid; e < nb * K * 12; e += 256) {
      const int p = e / 12, j = e % 12;
      s_cos[e] = 1.f - cosf(Yb[(size_t)p * n_out + 7 + j] - q.T[(size_t)s_row[p / K] * 19 + 7 + j]);
    }
  __syncthreads();
  for (int e = tid; e < nb * K; e += 256) {
    const size_t row = s_row[e / K];
    s_d[e] = pose_loss(q, Yb + (size_t)e * n_out, q.T + row * 19, q.mask ? q.mask + row * 12 : nullptr, s_cos + 12 * e);
  }
  __syncthreads();
  if (tid < nb) {
    const int b = ba + tid;
    float best = INFINITY;
    int kb = 0;
    for (int k = 0; k < K; ++k)
      if (s_d[tid * K + k] < best) {
        best = s_d[tid * K + k];
        kb = k;
      }
    s_win[tid] = b * K + kb;
    if (b * K >= m0 && b * K < m0 + 16) {
      q.winner[b] = kb;
      q.loss[b] = best;
    }
  }
  __syncthreads();
  // dL/dY of this block's rows: zero except the winners'
  for (int e = tid; e < 16 * opl; e += 256) {
    const int r = e / opl, j = e % opl, m = m0 + r;
    if (m >= net.Mp) continue;
    float g = 0.f;
    const int b = m / K;
    if (m < net.rows && j < n_out && s_win[b - ba] == m) {
      const int row = s_row[b - ba];
      const float *o = net.Y + (size_t)m * n_out, *t = q.T + (size_t)row * 19;
      const float* mk = q.mask ? q.mask + (size_t)row * 12 : nullptr;
      const float inv_b = 1.f / q.n_targets;
      if (j < 3) {
        float d = o[j] - t[j];
        if (j == 0) d -= q.tile_x * rintf(d / q.tile_x);
        if (j == 1) d -= q.tile_y * rintf(d / q.tile_y);
        g = 2.f * d * inv_b;
      } else if (j < 7) {
        float nu = sqrtf(o[3] * o[3] + o[4] * o[4] + o[5] * o[5] + o[6] * o[6]);
        nu = fmaxf(nu, 1e-12f);
        const float u[4] = {o[3] / nu, o[4] / nu, o[5] / nu, o[6] / nu};
        const float s = u[0] * t[3] + u[1] * t[4] + u[2] * t[5] + u[3] * t[6];
        g = -2.f * q.w_q * s * (t[j] - s * u[j - 3]) / nu * inv_b;
      } else {
        g = mk ? q.w_t * mk[j - 7] * sinf(o[j] - t[j]) * inv_b : 0.f;
      }
    }
    net.Gf[L - 1][(size_t)m * opl + j] = g;
    const __nv_bfloat16 v = __float2bfloat16(g);
    net.Gb[L - 1][(size_t)m * opl + j] = v;
    sG[0][r][j] = v;
  }
  __syncthreads();
  for (int l = L - 1, cur = 0; l > 0; --l, cur ^= 1) {
    // dL/da_{l-1} = (dL/da_l W_l) where the pre-activation was positive
    const int ip = net.pad[l], nt = ip >> 3, n_in = net.size[l];
    float acc[1][4][4];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[0][c][v] = 0.f;
    // the layer's activations (their sign is the mask), requested before the product
    __nv_bfloat162 act[4][2];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int m = m0 + (lane >> 2) + 8 * h;
        if (w + 8 * c < nt && m < net.rows)
          act[c][h] = *(const __nv_bfloat162*)&net.H[l][(size_t)m * ip + 8 * (w + 8 * c) + 2 * (lane & 3)];
      }
    rows_gemm<1>(sG[cur], B, k32(net.pad[l + 1]), nt, w, lane, acc);
    if (l > 1) rows_load(B, net.Wr[l - 1], k32(ip), net.pad[l - 1] >> 3, w, lane);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (w + 8 * c >= nt) continue;
      const int j = 8 * (w + 8 * c) + 2 * (lane & 3);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = (lane >> 2) + 8 * h, m = m0 + r;
        float2 v = make_float2(0.f, 0.f);
        if (m < net.rows) {
          const float2 a = __bfloat1622float2(act[c][h]);
          if (j < n_in && a.x > 0.f) v.x = acc[0][c][2 * h];
          if (j + 1 < n_in && a.y > 0.f) v.y = acc[0][c][2 * h + 1];
        }
        const __nv_bfloat162 b = __halves2bfloat162(__float2bfloat16(v.x), __float2bfloat16(v.y));
        *(__nv_bfloat162*)&sG[cur ^ 1][r][j] = b;
        if (m < net.Mp) {
          *(float2*)&net.Gf[l - 1][(size_t)m * ip + j] = v;
          *(__nv_bfloat162*)&net.Gb[l - 1][(size_t)m * ip + j] = b;
        }
      }
    }
    if (ip & 31)
      for (int e = tid; e < 16 * 16; e += 256) sG[cur ^ 1][e >> 4][ip + (e & 15)] = __float2bfloat16(0.f);
    __syncthreads();
  }
}

// Weight gradients of all layers in one launch: block = a 64 x 64 tile of one
// layer's dW [out][in] over one part of the rows (dW = G^T H, both operands read
// row by row and transposed by ldmatrix), then the blocks of the bias
// gradients: 32 columns x one chunk of rows, eight row groups.
struct GradMap {
  int first[kFusedMaxL + 1];      // first block of layer l's tiles; [L]: first bias block
  int tx[kFusedMaxL];             // tiles along the inputs
  int ty[kFusedMaxL];             // tiles along the outputs
  int db_first[kFusedMaxL + 1];
};

constexpr int kGLd = 72;          // 64 columns + 8: rows 144 B apart, conflict-free ldmatrix

__global__ void __launch_bounds__(128) fused_grad_kernel(FusedNet net, GradMap map) {
  __shared__ __align__(16) __nv_bfloat16 sA[2][32][kGLd], sB[2][32][kGLd];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  previous_done();
  next_may_start();
  if ((int)blockIdx.x >= map.first[net.L]) {
    // part[chunk][j] = sum over the chunk's rows of G[m][j]
    int l = 0;
    const int bx = blockIdx.x - map.first[net.L];
    while (bx >= map.db_first[l + 1]) ++l;
    const int k = bx - map.db_first[l], n_out = net.size[l + 1], op = net.pad[l + 1], cols = (n_out + 31) / 32;
    const int j = (k % cols) * 32 + lane, chunk = k / cols;
    const int r0 = chunk * net.rpc, r1 = min(net.Mp, r0 + net.rpc);
    float* sh = (float*)&sA[0][0][0];         // [8][33]
    for (int y = w; y < 8; y += 4) {
      float s = 0.f;
      if (j < n_out)
        for (int m = r0 + y; m < r1; m += 8) s += net.Gf[l][(size_t)m * op + j];
      sh[y * 33 + lane] = s;
    }
    __syncthreads();
    if (w == 0 && j < n_out) {
      float t = 0.f;
      for (int y = 0; y < 8; ++y) t += sh[y * 33 + lane];
      net.dbp[l][(size_t)chunk * n_out + j] = t;
    }
    return;
  }
  int l = 0;
  while ((int)blockIdx.x >= map.first[l + 1]) ++l;
  const int k = blockIdx.x - map.first[l], op = net.pad[l + 1], ip = net.pad[l];
  const int n0 = (k % map.tx[l]) * 64, o0 = (k / map.tx[l] % map.ty[l]) * 64, part = k / (map.tx[l] * map.ty[l]);
  const int rows = net.Mp / net.S[l], r0 = part * rows;
  const __nv_bfloat16 *G = net.Gb[l] + (size_t)r0 * op, *H = net.H[l] + (size_t)r0 * ip;
  auto load = [&](int stage, int m) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int e = tid + 128 * c, r = e >> 3, col = (e & 7) * 8;
      const bool in = m + r < rows, va = in && o0 + col < op, vb = in && n0 + col < ip;
      const unsigned da = (unsigned)__cvta_generic_to_shared(&sA[stage][r][col]);
      const unsigned db = (unsigned)__cvta_generic_to_shared(&sB[stage][r][col]);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(da),
                   "l"(va ? (const void*)(G + (size_t)(m + r) * op + o0 + col) : (const void*)G), "r"(va ? 16 : 0)
                   : "memory");
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(db),
                   "l"(vb ? (const void*)(H + (size_t)(m + r) * ip + n0 + col) : (const void*)H), "r"(vb ? 16 : 0)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[i][j][v] = 0.f;
  const int wm = (w >> 1) * 32, wn = (w & 1) * 32, n_sl = (rows + 31) / 32;
  const int q = lane >> 3, r8 = lane & 7;
  load(0, 0);
  for (int sl = 0; sl < n_sl; ++sl) {
    const int st = sl & 1;
    if (sl + 1 < n_sl) {
      load(st ^ 1, 32 * (sl + 1));
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 32; kk += 16) {
      unsigned a[2][4], b[2][4];
#pragma unroll
      for (int i = 0; i < 2; ++i)      // 8 x 8 blocks (k 0-7 | 8-15) x (outputs 0-7 | 8-15)
        ldsm4_t(&sA[st][kk + r8 + (q >> 1) * 8][wm + 16 * i + (q & 1) * 8], a[i]);
#pragma unroll
      for (int j = 0; j < 2; ++j)      // (inputs 0-7 | 8-15) x (k 0-7 | 8-15)
        ldsm4_t(&sB[st][kk + r8 + (q & 1) * 8][wn + 16 * j + (q >> 1) * 8], b[j]);
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a[i], b[j >> 1][2 * (j & 1)], b[j >> 1][2 * (j & 1) + 1]);
    }
    __syncthreads();
  }
  float* C = net.part[l] + (size_t)part * op * ip;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int row = o0 + wm + 16 * i + (lane >> 2), col = n0 + wn + 8 * j + 2 * (lane & 3);
      if (row < op && col < ip) {     // op, ip multiples of 16: a fragment is all in or all out
        *(float2*)&C[(size_t)row * ip + col] = make_float2(acc[i][j][0], acc[i][j][1]);
        *(float2*)&C[(size_t)(row + 8) * ip + col] = make_float2(acc[i][j][2], acc[i][j][3]);
      }
    }
}

// bfloat16 operands of one weight.
__device__ __forceinline__ void put_weight(const FusedNet& net, int l, int o, int i, float v) {
  const __nv_bfloat16 b = __float2bfloat16(v);
  net.Wf[l][frag_index(o, i, k32(net.pad[l]))] = b;
  net.Wr[l][frag_index(i, o, k32(net.pad[l + 1]))] = b;
}

struct AdamArgs {
  float b1, b2, eps, c1, c2;
  int update;
};

// Gradient of every parameter (parts added in order), Adam, the operands, and
// (last block) the mean loss of the step.
__global__ void __launch_bounds__(256) fused_update_kernel(FusedNet net, AdamArgs ad, int n_params,
                                                           const float* loss, int n_targets, float* hist) {
  if (blockIdx.x == gridDim.x - 1) {
    previous_done();
    next_may_start();
    if (!hist) return;
    __shared__ float part[256];
    float s = 0.f;
    for (int i = threadIdx.x; i < n_targets; i += 256) s += loss[i];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
      if ((int)threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) hist[0] = part[0] / n_targets;
    return;
  }
  const int p = blockIdx.x * 256 + threadIdx.x;
  float m0 = 0.f, v0 = 0.f, x0 = 0.f;
  if (p < n_params && ad.update) {
    m0 = net.Am[p];
    v0 = net.Av[p];
    x0 = net.P[p];
  }
  previous_done();
  next_may_start();
  if (p >= n_params) return;
  int l = 0;
  while (l + 1 < net.L && (size_t)p >= net.woff[l + 1]) ++l;
  const int n_in = net.size[l], ip = net.pad[l], op = net.pad[l + 1];
  const bool bias = (size_t)p >= net.boff[l];
  int o = 0, i = 0;
  float g = 0.f;
  if (bias) {
    const int j = p - (int)net.boff[l];
    for (int c = 0; c < net.chunks; ++c) g += net.dbp[l][(size_t)c * net.size[l + 1] + j];
  } else {
    const int e = p - (int)net.woff[l];
    o = e / n_in;
    i = e % n_in;
    const size_t at = (size_t)o * ip + i, st = (size_t)op * ip;
    if (net.S[l] == 1) g = net.part[l][at];
    else
      for (int k = 0; k < net.S[l]; ++k) g += net.part[l][k * st + at];
  }
  net.Gr[p] = g;
  if (!ad.update) return;
  // the contractions written out: the bits of adam_kernel
  const float m = fmaf(1.f - ad.b1, g, ad.b1 * m0);
  const float v = fmaf((1.f - ad.b2) * g, g, ad.b2 * v0);
  net.Am[p] = m;
  net.Av[p] = v;
  const float x = x0 - ad.c1 * m / (sqrtf(v * ad.c2) + ad.eps);
  net.P[p] = x;
  if (!bias) put_weight(net, l, o, i, x);
}

// The operands of all weights from the FP32 parameters (padding stays zero).
__global__ void fused_weights_kernel(FusedNet net, int n_params) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n_params) return;
  int l = 0;
  while (l + 1 < net.L && (size_t)p >= net.woff[l + 1]) ++l;
  if ((size_t)p >= net.boff[l]) return;
  const int e = p - (int)net.woff[l];
  put_weight(net, l, e / net.size[l], e % net.size[l], net.P[p]);
}

}  // namespace

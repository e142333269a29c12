// mlp.cu -- the learned screen's network on tensor cores: 12 -> 64 -> 64 -> 1,
// ReLU hidden units, sigmoid output, mean binary cross-entropy.
//
// Every product runs as mma.sync m16n8k16 with BF16 operands and FP32
// accumulators.  A warp owns 16 rows: layer-1 and layer-2 accumulator tiles
// are turned into the next product's A fragments in registers (bias, ReLU,
// BF16 pack).  Training adds the backward pass in the same kernel: the
// activation gradients stay in registers, the weight gradients of a tile of 64
// rows are formed with mma from shared-memory tiles, and the tiles' partial
// gradients are added in tile order, whatever CTA formed them: the sums depend
// on the rows alone, not on the grid (a run of a hundred steps multiplies the
// last bit of a sum: a BF16 copy flips, and Adam divides a gradient by its own
// size).  Then Adam updates the FP32 master weights and refreshes the BF16
// copies.  A training run is one cooperative kernel over all its mini-batches: a
// step is a few microseconds of work, so four launches a step were most of its
// time.
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "common.cuh"

namespace dcd {
namespace {

constexpr int NF = 12, NH = 64, NP = 5057;
constexpr int OFF_W1 = 0, OFF_B1 = 768, OFF_W2 = 832, OFF_B2 = 4928, OFF_W3 = 4992, OFF_B3 = 5056;
constexpr int kRowsPerCta = 64;  // 4 warps x 16 rows

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ float lo_f(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float hi_f(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }
__device__ __forceinline__ uint32_t ld_pair(const __nv_bfloat16* p) { return *reinterpret_cast<const uint32_t*>(p); }

__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// BF16 operand copies: w1t[64][16] (output-major, inputs 12..15 zero),
// w2[64][64] (input-major), w2t[64][64] (output-major), w3[64].
struct Weights {
  const __nv_bfloat16* w1t;
  const __nv_bfloat16* w2;
  const __nv_bfloat16* w2t;
  const __nv_bfloat16* w3;
  const float* P;  // FP32 master (biases are read from here)
};

__global__ void prepare(const float* __restrict__ P, __nv_bfloat16* __restrict__ w1t, __nv_bfloat16* __restrict__ w2,
                        __nv_bfloat16* __restrict__ w2t, __nv_bfloat16* __restrict__ w3) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 64 * 64; i += gridDim.x * blockDim.x) {
    const int a = i / 64, b = i % 64;  // W2[a][b]
    const __nv_bfloat16 v = __float2bfloat16_rn(P[OFF_W2 + i]);
    w2[i] = v;
    w2t[b * 64 + a] = v;
    if (i < 64 * 16) {
      const int o = i / 16, k = i % 16;  // w1t[o][k] = W1[k][o]
      w1t[i] = __float2bfloat16_rn(k < NF ? P[OFF_W1 + k * NH + o] : 0.f);
    }
    if (i < 64) w3[i] = __float2bfloat16_rn(P[OFF_W3 + i]);
  }
}

// Row strides in shared memory (elements): a fragment load reads 8 rows at 4
// consecutive words each, which these strides spread over all 32 banks (the
// natural 64 and 16 put all rows, or every other one, on the same four).
constexpr int SH = 72, SX = 24;

struct __align__(16) Smem {
  __nv_bfloat16 w1t[64 * SX];
  __nv_bfloat16 w2t[64 * SH];
  float w3f[64];
  float b1[64], b2[64];
  float b3;
};

// Rows of `cols` BF16 words (a multiple of 8) into padded rows, 16 bytes a
// load, around L1: another CTA of the same kernel may have written them.
__device__ __forceinline__ void load_rows(__nv_bfloat16* dst, int stride, const __nv_bfloat16* src, int rows, int cols) {
  const int per = cols / 8;
  for (int i = threadIdx.x; i < rows * per; i += blockDim.x) {
    const uint4 v = __ldcg(reinterpret_cast<const uint4*>(src) + i);
    *reinterpret_cast<uint4*>(dst + (i / per) * stride + (i % per) * 8) = v;
  }
}

// The caller synchronises.
__device__ __forceinline__ void load_weights(Smem& s, const Weights& W) {
  load_rows(s.w2t, SH, W.w2t, 64, 64);
  load_rows(s.w1t, SX, W.w1t, 64, 16);
  if (threadIdx.x < 64) {
    const int i = threadIdx.x;
    const unsigned short w3 = __ldcg(reinterpret_cast<const unsigned short*>(W.w3) + i);
    s.w3f[i] = __uint_as_float((uint32_t)w3 << 16);
    s.b1[i] = __ldcg(W.P + OFF_B1 + i);
    s.b2[i] = __ldcg(W.P + OFF_B2 + i);
    if (i == 0) s.b3 = __ldcg(W.P + OFF_B3);
  }
}

// Forward of one 16-row tile.  Outputs: the X fragment, the layer-1
// activations as layer-2 A fragments, h2 (BF16-rounded, C layout) and z.
struct Fwd {
  uint32_t xa[4];
  uint32_t h1a[4][4];
  float h2[8][4];
  float z0, z1;  // logits of rows g and g + 8
};

__device__ __forceinline__ void load_x(const float* __restrict__ X, int64_t r0, int64_t n, uint32_t (&xa)[4]) {
  const int lane = lane_id(), g = lane >> 2, t = lane & 3;
  const int64_t ra = r0 + g, rb = r0 + g + 8;
  auto xv = [&](int64_t r, int c) -> float { return (r < n && c < NF) ? X[r * NF + c] : 0.f; };
  xa[0] = pack_bf16(xv(ra, 2 * t), xv(ra, 2 * t + 1));
  xa[1] = pack_bf16(xv(rb, 2 * t), xv(rb, 2 * t + 1));
  xa[2] = pack_bf16(xv(ra, 2 * t + 8), xv(ra, 2 * t + 9));
  xa[3] = pack_bf16(xv(rb, 2 * t + 8), xv(rb, 2 * t + 9));
}

// f.xa holds the tile's rows.
__device__ __forceinline__ void forward_tile(const Smem& s, float b3, Fwd& f) {
  const int lane = lane_id(), g = lane >> 2, t = lane & 3;
  float c1[8][4];
#pragma unroll
  for (int j = 0; j < 8; j++) {
    c1[j][0] = c1[j][1] = c1[j][2] = c1[j][3] = 0.f;
    const __nv_bfloat16* col = s.w1t + (8 * j + g) * SX;
    mma16816(c1[j], f.xa, ld_pair(col + 2 * t), ld_pair(col + 2 * t + 8));
  }
#pragma unroll
  for (int kk = 0; kk < 4; kk++) {
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const int j = 2 * kk + h, c = 8 * j + 2 * t;
      const float v00 = fmaxf(c1[j][0] + s.b1[c], 0.f), v01 = fmaxf(c1[j][1] + s.b1[c + 1], 0.f);
      const float v10 = fmaxf(c1[j][2] + s.b1[c], 0.f), v11 = fmaxf(c1[j][3] + s.b1[c + 1], 0.f);
      f.h1a[kk][2 * h] = pack_bf16(v00, v01);
      f.h1a[kk][2 * h + 1] = pack_bf16(v10, v11);
    }
  }
  float c2[8][4];
#pragma unroll
  for (int j = 0; j < 8; j++) c2[j][0] = c2[j][1] = c2[j][2] = c2[j][3] = 0.f;
#pragma unroll
  for (int kk = 0; kk < 4; kk++)
#pragma unroll
    for (int j = 0; j < 8; j++) {
      const __nv_bfloat16* col = s.w2t + (8 * j + g) * SH + 16 * kk;
      mma16816(c2[j], f.h1a[kk], ld_pair(col + 2 * t), ld_pair(col + 2 * t + 8));
    }
  float za = 0.f, zb = 0.f;
#pragma unroll
  for (int j = 0; j < 8; j++) {
    const int c = 8 * j + 2 * t;
    f.h2[j][0] = bf16r(fmaxf(c2[j][0] + s.b2[c], 0.f));
    f.h2[j][1] = bf16r(fmaxf(c2[j][1] + s.b2[c + 1], 0.f));
    f.h2[j][2] = bf16r(fmaxf(c2[j][2] + s.b2[c], 0.f));
    f.h2[j][3] = bf16r(fmaxf(c2[j][3] + s.b2[c + 1], 0.f));
    za += f.h2[j][0] * s.w3f[c] + f.h2[j][1] * s.w3f[c + 1];
    zb += f.h2[j][2] * s.w3f[c] + f.h2[j][3] * s.w3f[c + 1];
  }
  za += __shfl_xor_sync(0xffffffffu, za, 1);
  za += __shfl_xor_sync(0xffffffffu, za, 2);
  zb += __shfl_xor_sync(0xffffffffu, zb, 1);
  zb += __shfl_xor_sync(0xffffffffu, zb, 2);
  f.z0 = za + b3;
  f.z1 = zb + b3;
}

__device__ __forceinline__ float sigmoidf_(float z) { return 1.f / (1.f + __expf(-z)); }

__global__ void __launch_bounds__(128) mlp_infer(Weights W, const float* __restrict__ X, int64_t n,
                                                 float* __restrict__ p) {
  __shared__ Smem s;
  load_weights(s, W);
  __syncthreads();
  const float b3 = s.b3;
  const int lane = lane_id(), g = lane >> 2, t = lane & 3;
  const int64_t tiles = cdiv(n, 16);
  for (int64_t tile = blockIdx.x * 4 + (threadIdx.x >> 5); tile < tiles; tile += (int64_t)gridDim.x * 4) {
    Fwd f;
    load_x(X, tile * 16, n, f.xa);
    forward_tile(s, b3, f);
    if (t == 0) {
      const int64_t ra = tile * 16 + g, rb = ra + 8;
      if (ra < n) p[ra] = sigmoidf_(f.z0);
      if (rb < n) p[rb] = sigmoidf_(f.z1);
    }
  }
}

// Four transposed 8 x 8 BF16 tiles from shared memory: lane l gives the row
// address of tile l / 8, row l % 8; register x holds tile x, in the layout of an
// mma operand whose K dimension runs along the stored rows.
__device__ __forceinline__ void ldsm_t(uint32_t (&r)[4], const __nv_bfloat16* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}

// Shared memory of a training CTA: the weights and the activations and
// activation gradients of 64 rows.
struct __align__(16) GradSmem {
  Smem w;
  __nv_bfloat16 w2[64 * SH];
  __nv_bfloat16 h1[kRowsPerCta * SH], dh2[kRowsPerCta * SH], dh1[kRowsPerCta * SH];
  __nv_bfloat16 x[kRowsPerCta * SX];
  float wpart[4][66];  // per warp: dW3[64], db3, loss
};

__device__ __forceinline__ void load_grad_weights(GradSmem& s, const Weights& W) {
  load_weights(s.w, W);
  load_rows(s.w2, SH, W.w2, 64, 64);
}

// A thread's inputs of the 64-row tile at tile0 (of rows [0, n)).
struct TileIn {
  uint32_t xa[4];
  float ya, yb;
};
__device__ __forceinline__ void load_tile(const float* __restrict__ X, const float* __restrict__ Y, int64_t tile0,
                                          int64_t n, TileIn& in) {
  const int64_t r0 = tile0 + (threadIdx.x >> 5) * 16, ra = r0 + (lane_id() >> 2), rb = ra + 8;
  load_x(X, r0, n, in.xa);
  in.ya = ra < n ? Y[ra] : 0.f;
  in.yb = rb < n ? Y[rb] : 0.f;
}

// The gradient sums of the tile at tile0 of [0, n) to its partial vector (128
// threads; the weights are in s, and the caller has synchronised).  Warp w forms
// dW2 rows 16 w .. 16 w + 15 and dW1 columns likewise; thread j < 64 db1[j] and
// dW3[j], thread 64 + j db2[j], thread 0 db3 and thread 1 the loss.
__device__ __forceinline__ void grad_tile(GradSmem& s, const TileIn& in, int64_t tile0, int64_t n, float inv_n,
                                          float* __restrict__ out, double* __restrict__ lout) {
  const int lane = lane_id(), g = lane >> 2, t = lane & 3, wid = threadIdx.x >> 5;
  const int64_t r0 = tile0 + wid * 16;
  Fwd f;
#pragma unroll
  for (int x = 0; x < 4; x++) f.xa[x] = in.xa[x];
  forward_tile(s.w, s.w.b3, f);
  const int64_t ra = r0 + g, rb = r0 + g + 8;
  const float ya = in.ya, yb = in.yb;
  const float pa = sigmoidf_(f.z0), pb = sigmoidf_(f.z1);
  const float dza = ra < n ? (pa - ya) * inv_n : 0.f, dzb = rb < n ? (pb - yb) * inv_n : 0.f;
  float la = 0.f, lb = 0.f;
  if (t == 0) {
    if (ra < n) la = fmaxf(f.z0, 0.f) - f.z0 * ya + log1pf(__expf(-fabsf(f.z0)));
    if (rb < n) lb = fmaxf(f.z1, 0.f) - f.z1 * yb + log1pf(__expf(-fabsf(f.z1)));
  }
  // layer 3: dW3 partial (rows of the warp) and dh2 = (h2 > 0) * dz * w3
  float dw3[8][2];
  uint32_t dh2a[4][4];
#pragma unroll
  for (int j = 0; j < 8; j++) {
    const int c = 8 * j + 2 * t;
    const float w0 = s.w.w3f[c], w1 = s.w.w3f[c + 1];
    dw3[j][0] = f.h2[j][0] * dza + f.h2[j][2] * dzb;
    dw3[j][1] = f.h2[j][1] * dza + f.h2[j][3] * dzb;
    const float d00 = f.h2[j][0] > 0.f ? dza * w0 : 0.f, d01 = f.h2[j][1] > 0.f ? dza * w1 : 0.f;
    const float d10 = f.h2[j][2] > 0.f ? dzb * w0 : 0.f, d11 = f.h2[j][3] > 0.f ? dzb * w1 : 0.f;
    const int kk = j >> 1, h = j & 1;
    dh2a[kk][2 * h] = pack_bf16(d00, d01);
    dh2a[kk][2 * h + 1] = pack_bf16(d10, d11);
  }
  // dh1 = dh2 W2^T, masked by h1 > 0
  float c3[8][4];
#pragma unroll
  for (int j = 0; j < 8; j++) c3[j][0] = c3[j][1] = c3[j][2] = c3[j][3] = 0.f;
#pragma unroll
  for (int kk = 0; kk < 4; kk++)
#pragma unroll
    for (int j = 0; j < 8; j++) {
      const __nv_bfloat16* row = s.w2 + (8 * j + g) * SH + 16 * kk;  // B[k][n] = W2[n][k]
      mma16816(c3[j], dh2a[kk], ld_pair(row + 2 * t), ld_pair(row + 2 * t + 8));
    }
  __syncthreads();  // the previous tile's rows have been read
  // stage x, h1, dh2, dh1 of the warp's 16 rows in shared memory (row-major)
  const int la_ = wid * 16 + g, lb_ = la_ + 8;
  *reinterpret_cast<uint32_t*>(&s.x[la_ * SX + 2 * t]) = f.xa[0];
  *reinterpret_cast<uint32_t*>(&s.x[lb_ * SX + 2 * t]) = f.xa[1];
  *reinterpret_cast<uint32_t*>(&s.x[la_ * SX + 2 * t + 8]) = f.xa[2];
  *reinterpret_cast<uint32_t*>(&s.x[lb_ * SX + 2 * t + 8]) = f.xa[3];
#pragma unroll
  for (int j = 0; j < 8; j++) {
    const int c = 8 * j + 2 * t, kk = j >> 1, h = j & 1;
    const uint32_t h1_a = f.h1a[kk][2 * h], h1_b = f.h1a[kk][2 * h + 1];
    *reinterpret_cast<uint32_t*>(&s.h1[la_ * SH + c]) = h1_a;
    *reinterpret_cast<uint32_t*>(&s.h1[lb_ * SH + c]) = h1_b;
    *reinterpret_cast<uint32_t*>(&s.dh2[la_ * SH + c]) = dh2a[kk][2 * h];
    *reinterpret_cast<uint32_t*>(&s.dh2[lb_ * SH + c]) = dh2a[kk][2 * h + 1];
    const float e00 = lo_f(h1_a) > 0.f ? c3[j][0] : 0.f, e01 = hi_f(h1_a) > 0.f ? c3[j][1] : 0.f;
    const float e10 = lo_f(h1_b) > 0.f ? c3[j][2] : 0.f, e11 = hi_f(h1_b) > 0.f ? c3[j][3] : 0.f;
    *reinterpret_cast<uint32_t*>(&s.dh1[la_ * SH + c]) = pack_bf16(e00, e01);
    *reinterpret_cast<uint32_t*>(&s.dh1[lb_ * SH + c]) = pack_bf16(e10, e11);
  }
  // warp partials of dW3 (sum over the 8 row groups), db3 and loss
#pragma unroll
  for (int j = 0; j < 8; j++)
#pragma unroll
    for (int e = 0; e < 2; e++) {
      float v = dw3[j][e];
      v += __shfl_xor_sync(0xffffffffu, v, 4);
      v += __shfl_xor_sync(0xffffffffu, v, 8);
      v += __shfl_xor_sync(0xffffffffu, v, 16);
      if (g == 0) s.wpart[wid][8 * j + 2 * t + e] = v;
    }
  {
    float db = (t == 0) ? dza + dzb : 0.f, ls = la + lb;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      db += __shfl_xor_sync(0xffffffffu, db, o);
      ls += __shfl_xor_sync(0xffffffffu, ls, o);
    }
    if (lane == 0) {
      s.wpart[wid][64] = db;
      s.wpart[wid][65] = ls;
    }
  }
  __syncthreads();
  // dW2[i][j] = sum_r h1[r][i] dh2[r][j], dW1[i][j] = sum_r x[r][i] dh1[r][j]:
  // both operands lie with K (the rows r) along the stored rows
  float a2[8][4], a1[2][4];
#pragma unroll
  for (int j = 0; j < 8; j++) a2[j][0] = a2[j][1] = a2[j][2] = a2[j][3] = 0.f;
#pragma unroll
  for (int j = 0; j < 2; j++) a1[j][0] = a1[j][1] = a1[j][2] = a1[j][3] = 0.f;
  const int tr = lane & 7, tq = lane >> 3;
#pragma unroll
  for (int kk = 0; kk < 4; kk++) {
    // A tiles: (rows 0-7 | 8-15 of K) x (columns 0-7 | 8-15 of M), in the
    // order of the A registers: (m0, k0), (m8, k0), (m0, k8), (m8, k8)
    const int ar = 16 * kk + (tq >> 1) * 8 + tr, ac = (tq & 1) * 8;
    uint32_t a[4];
    ldsm_t(a, s.h1 + ar * SH + 16 * wid + ac);
#pragma unroll
    for (int jp = 0; jp < 4; jp++) {
      // B tiles: (k0, n0), (k8, n0), (k0, n8), (k8, n8)
      uint32_t b[4];
      ldsm_t(b, s.dh2 + (16 * kk + (tq & 1) * 8 + tr) * SH + 16 * jp + (tq >> 1) * 8);
      mma16816(a2[2 * jp], a, b[0], b[1]);
      mma16816(a2[2 * jp + 1], a, b[2], b[3]);
    }
    uint32_t ax[4], bx[4];
    ldsm_t(ax, s.x + ar * SX + ac);
    ldsm_t(bx, s.dh1 + (16 * kk + (tq & 1) * 8 + tr) * SH + 16 * wid + (tq >> 1) * 8);
    mma16816(a1[0], ax, bx[0], bx[1]);
    mma16816(a1[1], ax, bx[2], bx[3]);
  }
  const int i0 = 16 * wid + g;
#pragma unroll
  for (int j = 0; j < 8; j++) {
    const int c = 8 * j + 2 * t;
    __stcg(reinterpret_cast<float2*>(out + OFF_W2 + i0 * 64 + c), make_float2(a2[j][0], a2[j][1]));
    __stcg(reinterpret_cast<float2*>(out + OFF_W2 + (i0 + 8) * 64 + c), make_float2(a2[j][2], a2[j][3]));
  }
#pragma unroll
  for (int jj = 0; jj < 2; jj++) {
    const int c = 16 * wid + 8 * jj + 2 * t;
    __stcg(reinterpret_cast<float2*>(out + OFF_W1 + g * NH + c), make_float2(a1[jj][0], a1[jj][1]));
    if (g + 8 < NF)
      __stcg(reinterpret_cast<float2*>(out + OFF_W1 + (g + 8) * NH + c), make_float2(a1[jj][2], a1[jj][3]));
  }
  // biases, W3, loss (fixed-order sums)
  {
    const int j = threadIdx.x & 63;
    const __nv_bfloat16* m = threadIdx.x < 64 ? s.dh1 : s.dh2;
    float v = 0.f;
#pragma unroll 16
    for (int r = 0; r < kRowsPerCta; r++) v += __bfloat162float(m[r * SH + j]);
    if (threadIdx.x < 64) {
      __stcg(out + OFF_B1 + j, v);
      __stcg(out + OFF_W3 + j, s.wpart[0][j] + s.wpart[1][j] + s.wpart[2][j] + s.wpart[3][j]);
    } else {
      __stcg(out + OFF_B2 + j, v);
    }
  }
  if (threadIdx.x == 0) __stcg(out + OFF_B3, s.wpart[0][64] + s.wpart[1][64] + s.wpart[2][64] + s.wpart[3][64]);
  if (threadIdx.x == 1)
    __stcg(lout, (double)s.wpart[0][65] + s.wpart[1][65] + s.wpart[2][65] + s.wpart[3][65]);
}

constexpr int kPartStride = 5060;  // floats a partial vector takes (float4 loads stay aligned)

// Gradient partials of the tiles [t0, t1) of rows [0, n), dealt to the CTAs in
// turn; part[x] is tile t0 + x.
__global__ void __launch_bounds__(128) mlp_grad_cta(Weights W, const float* __restrict__ X,
                                                    const float* __restrict__ Y, int64_t n, float inv_n, int64_t t0,
                                                    int64_t t1, float* __restrict__ part, double* __restrict__ lpart) {
  extern __shared__ __align__(16) unsigned char smem[];
  GradSmem& s = *reinterpret_cast<GradSmem*>(smem);
  load_grad_weights(s, W);
  __syncthreads();
  for (int64_t x = blockIdx.x; x < t1 - t0; x += gridDim.x) {
    const int64_t r = (t0 + x) * kRowsPerCta;
    TileIn in;
    load_tile(X, Y, r, n, in);
    grad_tile(s, in, r, n, inv_n, part + x * kPartStride, lpart + x);
  }
}

// carry + part[0][k] + part[1][k] + ... for the kSumBlock parameters k of block
// b, in this order: thread j < 64 gets parameter 64 b + j.  128 threads, all
// calling.  The order makes the sum a chain of additions, so only the loads are
// spread: the partials of kSumTiles tiles come 16 bytes a thread, all in flight,
// into shared memory, from where 64 threads add them (4 cycles each; 128 tiles:
// 0.3 us), while the loads of the next kSumTiles run.
constexpr int kSumBlock = 64;
constexpr int kSumBlocks = (NP + kSumBlock - 1) / kSumBlock;
constexpr int kSumTiles = 160;
constexpr int kSumLoads = kSumTiles / 8;  // 16 threads a tile
using SumStage = float[kSumTiles][kSumBlock];
__device__ __forceinline__ float grad_sum(const float* __restrict__ part, int tiles, int b, float carry,
                                          SumStage& stage) {
  const int tid = threadIdx.x, row = tid >> 4, col = (tid & 15) * 4;
  const bool in = b * kSumBlock + col < kPartStride;  // the last block is short
  const float* src = part + b * kSumBlock + col;
  float4 x[kSumLoads];
  auto load = [&](int c0) {
#pragma unroll
    for (int i = 0; i < kSumLoads; i++) {
      const int c = c0 + i * 8 + row;
      x[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (in && c < tiles) x[i] = __ldcg(reinterpret_cast<const float4*>(src + (int64_t)c * kPartStride));
    }
  };
  float s = carry;
  load(0);
  for (int c0 = 0; c0 < tiles; c0 += kSumTiles) {
    const int m = tiles - c0 < kSumTiles ? tiles - c0 : kSumTiles;
#pragma unroll
    for (int i = 0; i < kSumLoads; i++)
      if (i * 8 + row < m) *reinterpret_cast<float4*>(&stage[i * 8 + row][col]) = x[i];
    __syncthreads();
    if (c0 + kSumTiles < tiles) load(c0 + kSumTiles);
    if (tid < kSumBlock) {
      int c = 0;
      for (; c + 16 <= m; c += 16) {
        float v[16];
#pragma unroll
        for (int i = 0; i < 16; i++) v[i] = stage[c + i][tid];
#pragma unroll
        for (int i = 0; i < 16; i++) s += v[i];
      }
      for (; c < m; c++) s += stage[c][tid];
    }
    __syncthreads();
  }
  return s;
}

// The losses of the tiles, in tile order.
__device__ __forceinline__ double loss_sum(const double* __restrict__ lpart, int tiles, double l) {
  for (int c = 0; c < tiles; c++) l += __ldcg(lpart + c);
  return l;
}

// first: the tiles are the first of the rows; else grad and loss hold the sums
// of those before.  inv_n (not zero on the last call): the loss becomes a mean.
__global__ void __launch_bounds__(128) grad_reduce(const float* __restrict__ part, int tiles, int first,
                                                   float* __restrict__ grad, const double* __restrict__ lpart,
                                                   double* __restrict__ loss, double inv_n) {
  __shared__ __align__(16) SumStage stage;
  const int k = blockIdx.x * kSumBlock + threadIdx.x;
  const bool mine = threadIdx.x < kSumBlock && k < NP;
  const float v = grad_sum(part, tiles, blockIdx.x, mine && !first ? grad[k] : 0.f, stage);
  if (mine) grad[k] = v;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const double l = loss_sum(lpart, tiles, first ? 0.0 : *loss);
    *loss = inv_n != 0 ? l * inv_n : l;
  }
}

// Adam on one parameter, and its BF16 copies.
struct Master {
  float *P, *m, *v;
  __nv_bfloat16 *w1t, *w2, *w2t, *w3;
};
struct Moments {
  float p, m, v;
};
__device__ __forceinline__ Moments load_moments(const Master& M, int k) {
  return k < NP ? Moments{M.P[k], M.m[k], M.v[k]} : Moments{0.f, 0.f, 0.f};
}
__device__ __forceinline__ void adam_one(const Master& M, int k, const Moments& o, float gk, float lr, float b1,
                                         float b2, float eps, float c1, float c2) {
  // the roundings are spelled out: which product of a sum is fused is otherwise
  // the compiler's choice, which may change with the code around it, and these
  // bits decide where a run ends
  const float mk = __fmaf_rn(1.f - b1, gk, __fmul_rn(b1, o.m));
  const float vk = __fmaf_rn(__fmul_rn(1.f - b2, gk), gk, __fmul_rn(b2, o.v));
  M.m[k] = mk;
  M.v[k] = vk;
  const float p = o.p - lr * (mk / c1) / (sqrtf(vk / c2) + eps);
  __stcg(M.P + k, p);
  const __nv_bfloat16 q = __float2bfloat16_rn(p);
  if (k < OFF_B1) {
    M.w1t[(k % NH) * 16 + k / NH] = q;  // w1t[o][i] = W1[i][o]
  } else if (k >= OFF_W2 && k < OFF_B2) {
    const int i = k - OFF_W2;
    M.w2[i] = q;
    M.w2t[(i % NH) * NH + i / NH] = q;
  } else if (k >= OFF_W3 && k < OFF_B3) {
    M.w3[k - OFF_W3] = q;
  }
}

// All CTAs of the (cooperative) grid; false when the wait ran out (they are
// co-resident and a step's work is evenly dealt, so only a wait made to, or a CTA
// that is seconds behind, does), after which every CTA leaves.
constexpr int64_t kWaitPolls = (int64_t)1 << 24;  // about ten seconds
__device__ __forceinline__ bool grid_wait(unsigned* bar, unsigned target, int64_t polls, int* err) {
  __shared__ int bad;
  __syncthreads();
  if (threadIdx.x == 0) {
    bad = 0;
    __threadfence();
    atomicAdd(bar, 1u);
    int64_t left = polls;
    unsigned x;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(bar) : "memory");
    } while (x < target && --left > 0);
    if (x < target) {
      bad = 1;
      *err = 1;
    }
  }
  __syncthreads();
  return bad == 0;
}

// Steps [s0, s1) of a training run: step s takes mini-batch s % per_epoch.  A
// step is: gradient partials of the tiles, dealt to the first `rows` CTAs | wait
// | the CTAs' shares of the parameters summed and updated | wait.  A batch of more
// tiles than there is room for partials takes them in chunks, the sums so far in
// grad.  corr: Adam's bias corrections (two floats a step).  Bound by the latency
// of its two waits and of the passes through L2 between them (weights in,
// partials out and in), so what does not depend on the other CTAs is loaded
// before each wait: the parameters and moments to update, the next step's rows.
// 32 steps of 8192 rows take 402 us (386 with sums split over four warps, which
// depend on the split); as four kernels a step (partials 18, sums 19, Adam 4, BF16
// copies 3 us) 1300.
struct TrainArgs {
  const float* X;
  const float* Y;
  int64_t n, batch, per_epoch;
  int64_t s0, s1;
  int64_t chunk;  // tiles there is room for
  int rows;       // CTAs that take tiles; the others only parameters
  float lr, b1, b2, eps;
  const float* corr;
  float* part;
  double* lpart;
  float* grad;
  double* loss;
  float* saved;   // not NULL: P, m and v as they are before the first step (kSavedStride floats each)
  unsigned* bar;  // zero
  unsigned more;  // CTAs waited for that do not exist
  int64_t polls;
  int* err;
};
constexpr int kSavedStride = (NP * 4 + 255) / 256 * 256 / 4;
constexpr size_t kTrainSmem = sizeof(GradSmem) + sizeof(SumStage);
__global__ void __launch_bounds__(128) mlp_train_steps(Weights W, Master M, TrainArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  GradSmem& s = *reinterpret_cast<GradSmem*>(smem);
  SumStage& stage = *reinterpret_cast<SumStage*>(smem + sizeof(GradSmem));
  const int G = gridDim.x, rows = a.rows;
  const bool works = (int)blockIdx.x < rows;
  const int j = threadIdx.x < kSumBlock ? (int)threadIdx.x : NP;  // (NP: no parameter)
  auto batch_of = [&](int64_t st, int64_t& r0, int64_t& nb) {
    r0 = (st % a.per_epoch) * a.batch;
    nb = r0 + a.batch <= a.n ? a.batch : a.n - r0;
  };
  if (a.saved)  // before the first wait: what a CTA that leaves there has not touched yet is saved too
    for (int b = blockIdx.x; b < kSumBlocks; b += G) {
      const int k = b * kSumBlock + j;
      const Moments o = load_moments(M, k);
      if (k >= NP) continue;
      a.saved[k] = o.p;
      a.saved[kSavedStride + k] = o.m;
      a.saved[2 * kSavedStride + k] = o.v;
    }
  unsigned target = a.more;
  int64_t r0, nb;
  batch_of(a.s0, r0, nb);
  TileIn in;
  const int64_t mine = (int64_t)blockIdx.x * kRowsPerCta;
  if (works) load_tile(a.X + r0 * NF, a.Y + r0, mine, nb, in);
  for (int64_t st = a.s0; st < a.s1; st++) {
    const float inv_n = 1.f / (float)nb;
    const int64_t tiles = (nb + kRowsPerCta - 1) / kRowsPerCta;
    const float c1 = a.corr[2 * (st - a.s0)], c2 = a.corr[2 * (st - a.s0) + 1];
    if (works) {
      load_grad_weights(s, W);
      __syncthreads();
    }
    double l = 0;  // CTA 0's first thread
    for (int64_t t0 = 0; t0 < tiles; t0 += a.chunk) {
      const int m = (int)(tiles - t0 < a.chunk ? tiles - t0 : a.chunk);
      const bool last = t0 + m == tiles;
      if (works)
        for (int x = blockIdx.x; x < m; x += rows) {
          const int64_t r = (t0 + x) * kRowsPerCta;
          if (r != mine) load_tile(a.X + r0 * NF, a.Y + r0, r, nb, in);
          grad_tile(s, in, r, nb, inv_n, a.part + (int64_t)x * kPartStride, a.lpart + x);
        }
      int k = (int)blockIdx.x * kSumBlock + j;
      Moments o = load_moments(M, k);
      if (!grid_wait(a.bar, target += G, a.polls, a.err)) return;
      for (int b = blockIdx.x; b < kSumBlocks; b += G) {
        if (b != (int)blockIdx.x) {
          k = b * kSumBlock + j;
          o = load_moments(M, k);
        }
        const float gk = grad_sum(a.part, m, b, t0 > 0 && k < NP ? a.grad[k] : 0.f, stage);
        if (k >= NP) continue;
        if (last) adam_one(M, k, o, gk, a.lr, a.b1, a.b2, a.eps, c1, c2);
        else a.grad[k] = gk;
      }
      if (st + 1 == a.s1 && blockIdx.x == 0 && threadIdx.x == 0) l = loss_sum(a.lpart, m, l);
      if (last) break;
      if (!grid_wait(a.bar, target += G, a.polls, a.err)) return;
    }
    if (st + 1 == a.s1) {
      if (blockIdx.x == 0 && threadIdx.x == 0) *a.loss = l * (1.0 / (double)nb);
      break;
    }
    batch_of(st + 1, r0, nb);
    if (works) load_tile(a.X + r0 * NF, a.Y + r0, mine, nb, in);
    if (!grid_wait(a.bar, target += G, a.polls, a.err)) return;
  }
}

}  // namespace
}  // namespace dcd

struct dcd_mlp {
  cudaStream_t stream = nullptr;
  int device = 0;
  unsigned char* block = nullptr;  // the allocation all of the following lie in
  float* P = nullptr;  // master params
  float* m = nullptr;
  float* v = nullptr;
  float* grad = nullptr;
  double* loss = nullptr;
  __nv_bfloat16* w1t = nullptr;
  __nv_bfloat16* w2 = nullptr;
  __nv_bfloat16* w2t = nullptr;
  __nv_bfloat16* w3 = nullptr;
  float* part = nullptr;     // partials of part_tiles tiles, in block or in more
  double* lpart = nullptr;
  int64_t part_tiles = 0;
  unsigned char* more = nullptr;  // allocation for batches of more tiles than block has room for
  unsigned* sync = nullptr;  // [0] the training kernel's barrier, [1] its error word
  float* corr = nullptr;     // Adam's bias corrections of kTrainSteps steps
  float* saved = nullptr;    // P, m, v before the training run (they lie behind each other in block, as here)
  int64_t adam_t = 0;
};

namespace {
using namespace dcd;

Weights weights_of(const dcd_mlp* m) { return Weights{m->w1t, m->w2, m->w2t, m->w3, m->P}; }

int refresh(dcd_mlp* m) {
  count_launch(), prepare<<<16, 256, 0, m->stream>>>(m->P, m->w1t, m->w2, m->w2t, m->w3);
  DCD_LAUNCH_CHECK();
  return DCD_OK;
}

// CTAs that take tiles: one an SM at most.
int64_t grad_ctas(int64_t tiles) { return tiles < num_sms() ? tiles : num_sms(); }

// Tiles whose partials (20 KB each) are held at once: what dcd_mlp_create has
// room for (kPartFew an SM; batches to 19,456 rows), for larger batches up to kPartMost
// an SM (25 MB, within L2); a batch of more takes them in chunks.  Growth that
// fails leaves smaller chunks.
constexpr int64_t kPartFew = 2, kPartMost = 8;
void part_room(dcd_mlp* m, int64_t tiles) {
  const int64_t want = tiles < kPartMost * num_sms() ? tiles : kPartMost * num_sms();
  if (want <= m->part_tiles) return;
  const int64_t room = kPartMost * num_sms();
  unsigned char* q = nullptr;
  if (fault_hit(kFaultAlloc) || cudaMalloc(&q, (size_t)room * (kPartStride * sizeof(float) + sizeof(double))) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  m->more = q;  // (growth happens once: block's own room is the only smaller one)
  m->lpart = reinterpret_cast<double*>(q);
  m->part = reinterpret_cast<float*>(q + (size_t)room * sizeof(double));
  m->part_tiles = room;
}

constexpr int64_t kTrainSteps = 4096;  // steps a launch of the training kernel takes at most

int grad_attrs() {
  DCD_TRY_CUDA(cudaFuncSetAttribute(mlp_grad_cta, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSmem)));
  DCD_TRY_CUDA(cudaFuncSetAttribute(mlp_train_steps, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTrainSmem));
  return DCD_OK;
}

// Mean BCE gradient of rows [0, n) into m->grad and m->loss.
int grad_pass(dcd_mlp* m, const float* X, const float* Y, int64_t n) {
  const int64_t tiles = cdiv(n, kRowsPerCta);
  part_room(m, tiles);
  DCD_TRY(grad_attrs());
  for (int64_t t0 = 0; t0 < tiles; t0 += m->part_tiles) {
    const int64_t t1 = t0 + m->part_tiles < tiles ? t0 + m->part_tiles : tiles;
    count_launch(), mlp_grad_cta<<<(unsigned)grad_ctas(t1 - t0), 128, sizeof(GradSmem), m->stream>>>(
        weights_of(m), X, Y, n, 1.f / (float)n, t0, t1, m->part, m->lpart);
    count_launch(), grad_reduce<<<kSumBlocks, 128, 0, m->stream>>>(m->part, (int)(t1 - t0), t0 == 0, m->grad, m->lpart,
                                                                   m->loss, t1 == tiles ? 1.0 / (double)n : 0.0);
    DCD_LAUNCH_CHECK();
  }
  return DCD_OK;
}

uint64_t splitmix(uint64_t& s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ULL);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

}  // namespace

namespace dcd {
int mlp_forward_on(dcd_mlp* m, const float* X, int64_t n, float* p, cudaStream_t s) {
  if (n <= 0) return DCD_OK;
  const int64_t tiles = cdiv(n, 16);
  const int64_t ctas = cdiv(tiles, 4) < 8 * (int64_t)num_sms() ? cdiv(tiles, 4) : 8 * (int64_t)num_sms();
  count_launch(), mlp_infer<<<(unsigned)ctas, 128, 0, s>>>(weights_of(m), X, n, p);
  DCD_LAUNCH_CHECK();
  return DCD_OK;
}
}  // namespace dcd

extern "C" {

int dcd_mlp_create(uint64_t seed, void* cuda_stream, dcd_mlp** out) {
  if (!out) return DCD_EINVAL;
  *out = nullptr;
  dcd_mlp* m = new (std::nothrow) dcd_mlp();
  if (!m) return DCD_ENOMEM;
  m->stream = static_cast<cudaStream_t>(cuda_stream);
  int rc = DCD_OK;
  do {
    if (cudaGetDevice(&m->device) != cudaSuccess) { rc = DCD_ECUDA; break; }
    // one allocation, cut into 256-byte aligned parts
    size_t at = 0;
    auto part = [&](size_t bytes) {
      const size_t o = at;
      at += (bytes + 255) & ~(size_t)255;
      return o;
    };
    const size_t oP = part(NP * sizeof(float)), om = part(NP * sizeof(float)), ov = part(NP * sizeof(float)),
                 og = part(NP * sizeof(float)), ol = part(sizeof(double)), o1 = part(64 * 16 * sizeof(__nv_bfloat16)),
                 o2 = part(64 * 64 * sizeof(__nv_bfloat16)), o2t = part(64 * 64 * sizeof(__nv_bfloat16)),
                 o3 = part(64 * sizeof(__nv_bfloat16)),
                 op = part((size_t)(kPartFew * num_sms()) * kPartStride * sizeof(float)),
                 olp = part((size_t)(kPartFew * num_sms()) * sizeof(double)), os = part(2 * sizeof(unsigned)),
                 oc = part(2 * kTrainSteps * sizeof(float)), ov0 = part(3 * kSavedStride * sizeof(float));
    if (cudaMalloc(&m->block, at) != cudaSuccess) {
      cudaGetLastError();
      rc = DCD_ENOMEM;
      break;
    }
    m->P = reinterpret_cast<float*>(m->block + oP);
    m->m = reinterpret_cast<float*>(m->block + om);
    m->v = reinterpret_cast<float*>(m->block + ov);
    m->grad = reinterpret_cast<float*>(m->block + og);
    m->loss = reinterpret_cast<double*>(m->block + ol);
    m->w1t = reinterpret_cast<__nv_bfloat16*>(m->block + o1);
    m->w2 = reinterpret_cast<__nv_bfloat16*>(m->block + o2);
    m->w2t = reinterpret_cast<__nv_bfloat16*>(m->block + o2t);
    m->w3 = reinterpret_cast<__nv_bfloat16*>(m->block + o3);
    m->part = reinterpret_cast<float*>(m->block + op);
    m->lpart = reinterpret_cast<double*>(m->block + olp);
    m->part_tiles = kPartFew * num_sms();
    m->sync = reinterpret_cast<unsigned*>(m->block + os);
    m->corr = reinterpret_cast<float*>(m->block + oc);
    m->saved = reinterpret_cast<float*>(m->block + ov0);
    // He-uniform initialisation from SplitMix64; biases zero
    std::vector<float> P(NP, 0.f);
    uint64_t s = seed;
    auto unif = [&](float lim) { return (float)(((splitmix(s) >> 11) * (1.0 / 9007199254740992.0)) * 2 - 1) * lim; };
    for (int i = 0; i < NF * NH; i++) P[OFF_W1 + i] = unif(std::sqrt(6.f / NF));
    for (int i = 0; i < NH * NH; i++) P[OFF_W2 + i] = unif(std::sqrt(6.f / NH));
    for (int i = 0; i < NH; i++) P[OFF_W3 + i] = unif(std::sqrt(6.f / NH));
    rc = dcd_mlp_set_params(m, P.data());
  } while (0);
  if (rc) {
    dcd_mlp_destroy(m);
    return rc;
  }
  *out = m;
  return DCD_OK;
}

int dcd_mlp_destroy(dcd_mlp* m) {
  if (!m) return DCD_OK;
  cudaStreamSynchronize(m->stream);
  if (m->more) cudaFree(m->more);
  if (m->block) cudaFree(m->block);
  delete m;
  return DCD_OK;
}

int dcd_mlp_set_params(dcd_mlp* m, const float* params) {
  if (!m || !params) return DCD_EINVAL;
  DCD_TRY_CUDA(cudaMemcpyAsync(m->P, params, NP * sizeof(float), cudaMemcpyHostToDevice, m->stream));
  DCD_TRY_CUDA(cudaMemsetAsync(m->m, 0, NP * sizeof(float), m->stream));
  DCD_TRY_CUDA(cudaMemsetAsync(m->v, 0, NP * sizeof(float), m->stream));
  m->adam_t = 0;
  DCD_TRY(refresh(m));
  DCD_TRY_CUDA(cudaStreamSynchronize(m->stream));
  return DCD_OK;
}

int dcd_mlp_get_params(dcd_mlp* m, float* params_out) {
  if (!m || !params_out) return DCD_EINVAL;
  DCD_TRY_CUDA(cudaMemcpyAsync(params_out, m->P, NP * sizeof(float), cudaMemcpyDeviceToHost, m->stream));
  DCD_TRY_CUDA(cudaStreamSynchronize(m->stream));
  return DCD_OK;
}

int dcd_mlp_forward(dcd_mlp* m, const float* d_X, int64_t n, float* d_p) {
  if (!m || n < 0 || (n && (!d_X || !d_p))) return DCD_EINVAL;
  if (n == 0) return DCD_OK;
  const int64_t tiles = cdiv(n, 16);
  const int64_t ctas = cdiv(tiles, 4) < 8 * (int64_t)num_sms() ? cdiv(tiles, 4) : 8 * (int64_t)num_sms();
  count_launch(), mlp_infer<<<(unsigned)ctas, 128, 0, m->stream>>>(weights_of(m), d_X, n, d_p);
  DCD_LAUNCH_CHECK();
  DCD_TRY_CUDA(cudaStreamSynchronize(m->stream));
  return DCD_OK;
}

int dcd_mlp_grad(dcd_mlp* m, const float* d_X, const float* d_y, int64_t n, float* grad_out, double* loss_out) {
  if (!m || n <= 0 || !d_X || !d_y) return DCD_EINVAL;
  DCD_TRY(grad_pass(m, d_X, d_y, n));
  if (grad_out)
    DCD_TRY_CUDA(cudaMemcpyAsync(grad_out, m->grad, NP * sizeof(float), cudaMemcpyDeviceToHost, m->stream));
  if (loss_out) DCD_TRY_CUDA(cudaMemcpyAsync(loss_out, m->loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
  DCD_TRY_CUDA(cudaStreamSynchronize(m->stream));
  return DCD_OK;
}

}  // extern "C"

namespace {
// The run of dcd_mlp_train.  *saved: m->saved holds the state from before it.
int train_run(dcd_mlp* m, const float* d_X, const float* d_y, int64_t n, int64_t batch, int32_t epochs, float lr,
              double* last, bool* saved) {
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  DCD_TRY(grad_attrs());
  const int64_t per_epoch = cdiv(n, batch), steps = per_epoch * epochs;
  TrainArgs a{};
  a.X = d_X;
  a.Y = d_y;
  a.n = n;
  a.batch = batch;
  a.per_epoch = per_epoch;
  a.lr = lr;
  a.b1 = b1;
  a.b2 = b2;
  a.eps = eps;
  a.corr = m->corr;
  const int64_t tiles = cdiv(batch < n ? batch : n, kRowsPerCta);
  part_room(m, tiles);
  a.chunk = m->part_tiles;
  a.part = m->part;
  a.lpart = m->lpart;
  a.grad = m->grad;
  a.loss = m->loss;
  a.bar = m->sync;
  a.err = reinterpret_cast<int*>(m->sync + 1);
  Weights W = weights_of(m);
  Master M{m->P, m->m, m->v, m->w1t, m->w2, m->w2t, m->w3};
  a.rows = (int)grad_ctas(tiles < a.chunk ? tiles : a.chunk);
  // every parameter block a CTA of its own, co-resident (one CTA an SM)
  unsigned ctas = (unsigned)(a.rows >= kSumBlocks ? a.rows : kSumBlocks < num_sms() ? kSumBlocks : num_sms());
  std::vector<float> corr;
  int err = 0;
  for (int64_t s0 = 0; s0 < steps; s0 += kTrainSteps) {
    a.s0 = s0;
    a.s1 = s0 + kTrainSteps < steps ? s0 + kTrainSteps : steps;
    corr.resize(2 * (a.s1 - a.s0));
    for (int64_t s = a.s0; s < a.s1; s++) {
      m->adam_t++;
      corr[2 * (s - a.s0)] = 1.f - std::pow(b1, (float)m->adam_t);
      corr[2 * (s - a.s0) + 1] = 1.f - std::pow(b2, (float)m->adam_t);
    }
    DCD_TRY_CUDA(cudaMemcpyAsync(m->corr, corr.data(), corr.size() * sizeof(float), cudaMemcpyHostToDevice, m->stream));
    DCD_TRY_CUDA(cudaMemsetAsync(m->sync, 0, 2 * sizeof(unsigned), m->stream));
    const bool stuck = fault_hit(kFaultWait);
    a.more = stuck ? 1 : 0;
    a.polls = stuck ? 4096 : kWaitPolls;
    a.saved = s0 == 0 ? m->saved : nullptr;
    // a stream that has fewer SMs than the device reports (a partition of it) refuses
    // the grid: any smaller one gives the same results
    auto launch = [&] {
      for (;;) {
        void* args[] = {&W, &M, &a};
        const int64_t most = g_fault_left[kFaultGrid].load(std::memory_order_relaxed);
        const cudaError_t e =
            most > 0 && (int64_t)ctas > most
                ? cudaErrorCooperativeLaunchTooLarge
                : cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(mlp_train_steps), dim3(ctas), dim3(128),
                                              args, kTrainSmem, m->stream);
        if (e != cudaErrorCooperativeLaunchTooLarge || ctas == 1) return e;
        cudaGetLastError();
        ctas /= 2;
        if (a.rows > (int)ctas) a.rows = (int)ctas;
      }
    };
    count_launch();
    DCD_TRY_CUDA(launch());
    *saved = true;
    DCD_TRY_CUDA(cudaMemcpyAsync(last, m->loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
    DCD_TRY_CUDA(cudaMemcpyAsync(&err, m->sync + 1, sizeof(int), cudaMemcpyDeviceToHost, m->stream));
    DCD_TRY_CUDA(cudaStreamSynchronize(m->stream));
    if (err) return DCD_ETIMEOUT;
  }
  return DCD_OK;
}

// The network as it was before a run that failed.
void train_undo(dcd_mlp* m, int64_t adam_t, bool saved) {
  m->adam_t = adam_t;
  if (saved) {
    cudaMemcpyAsync(m->P, m->saved, 3 * kSavedStride * sizeof(float), cudaMemcpyDeviceToDevice, m->stream);
    count_launch(), prepare<<<16, 256, 0, m->stream>>>(m->P, m->w1t, m->w2, m->w2t, m->w3);
  }
  cudaStreamSynchronize(m->stream);
}
}  // namespace

extern "C" {

int dcd_mlp_train(dcd_mlp* m, const float* d_X, const float* d_y, int64_t n, int64_t batch, int32_t epochs,
                  float lr, double* loss_out) {
  if (!m || n <= 0 || batch <= 0 || epochs <= 0 || !d_X || !d_y || !(lr > 0.f)) return DCD_EINVAL;
  const int64_t adam_t = m->adam_t;
  double last = 0;
  bool saved = false;
  const int rc = train_run(m, d_X, d_y, n, batch, epochs, lr, &last, &saved);
  if (rc != DCD_OK) {
    train_undo(m, adam_t, saved);
    return rc;
  }
  if (loss_out) *loss_out = last;
  return DCD_OK;
}

}  // extern "C"

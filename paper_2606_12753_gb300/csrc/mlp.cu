// Training and evaluation kernels of the learned face switch, and the face
// sampler that produces its training data from a state (see mlp.cuh).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include "../../include/mhd_gb300.h"
#include "mlp.cuh"
#include "stage.cuh"
#include "tc05.cuh"

namespace mhd {

__device__ __forceinline__ uint16_t to_bf16_bits(float x) {
  const __nv_bfloat16 b = __float2bfloat16_rn(x);
  return *reinterpret_cast<const uint16_t*>(&b);
}
__device__ __forceinline__ float from_bf16_bits(uint16_t u) {
  return __uint_as_float((uint32_t)u << 16);
}

// ---------------------------------------------------------------------------
// Training-size products on the fifth-generation tensor cores (tcgen05).
// A CTA of 128 threads takes 128 rows at a time (thread t owns row t): layer 1
// (128 x 32 x 16), layer 2 (128 x 32 x 32) and, in the backward pass, dh1 =
// delta2 W2 (128 x 32 x 32) and the weight gradients run as tcgen05.mma from
// shared memory into TMEM, issued by one thread and completed on an mbarrier;
// each warp then reads its 32 rows of the accumulator with tcgen05.ld.
// Operands are bf16 in the canonical layouts of tc05.cuh, side by side in two
// row blocks: XH = [h1 (32 columns) | x (16) | dz (16) | m1 (32)] and DD =
// [delta2 (32) | delta1 (32) | m2 (32) | h2 (32)], m = [a > 0] of a layer.  What
// contracts over the rows reads both blocks as MN-major operands in place:
// DD^T XH accumulates in TMEM over all tiles of the CTA and holds dW2 =
// delta2^T h1 and dW1 = delta1^T x; with the first three columns of dz -- dz
// cut into three bf16 terms, which hold its 24 bits exactly -- dW3 = h2^T dz
// and m2^T dz, of which db2 = w3 (m2^T dz); and C = delta2^T m1, of which db1_j =
// sum_o W2_oj C_oj: exact products summed in FP32.  (Its other blocks are not
// read.)
// ---------------------------------------------------------------------------

constexpr int TC_ROWS = 128;
constexpr uint32_t TC_LBO = 128;   // bytes between core matrices along K
// columns of the row blocks (the forward pass needs h1 and x only) and where x, dz, m1 start
template <bool BWD> constexpr int XH_COLS = BWD ? 96 : 48;
constexpr int XH_X = 32, XH_DZ = 48, XH_M1 = 64;
constexpr int DD_COLS = 128, DD_D1 = 32, DD_M2 = 64, DD_H2 = 96;
template <bool BWD> constexpr uint32_t XH_GROUP = XH_COLS<BWD> * 16;   // bytes of a group of 8 rows
constexpr uint32_t DD_GROUP = DD_COLS * 16;

// Shared memory of a CTA; BWD adds the backward pass's operands.
template <bool BWD>
struct TcShared {
  __align__(128) unsigned char DD[BWD ? TC_ROWS * DD_COLS * 2 : 128];
  __align__(128) unsigned char XH[TC_ROWS * XH_COLS<BWD> * 2];
  __align__(128) unsigned char B1[MLP_NH * MLP_NF * 2];                 // W1 [32 x 16]
  __align__(128) unsigned char B2[MLP_NH * MLP_NH * 2];                 // W2 [32 x 32]
  __align__(128) unsigned char B3[BWD ? MLP_NH * MLP_NH * 2 : 128];     // W2^T [32 x 32]
  __align__(16) float b1[MLP_NH];
  __align__(16) float b2[MLP_NH];
  __align__(16) float w3[MLP_NH];
  __align__(8) uint64_t mbar;
  uint32_t tmem;
};

// eight columns k0..k0+7 (bf16 pairs) of this thread's row of a block of K columns
__device__ __forceinline__ void tc_store8(unsigned char* A, int K, int k0, const uint32_t* p) {
  *reinterpret_cast<uint4*>(A + tc05::kmajor_offset(threadIdx.x, k0, K)) = make_uint4(p[0], p[1], p[2], p[3]);
}
__device__ __forceinline__ void tc_store32(unsigned char* A, int K, int k0, const uint32_t (&p)[16]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) tc_store8(A, K, k0 + 8 * c, p + 4 * c);
}

// relu and [a > 0] (all bits of each half) of an accumulator row plus its bias,
// rounded to bf16, by pairs: rounding keeps the sign, so both are packed
// operations on the rounded pair
__device__ __forceinline__ void tc_activate(const float (&v)[32], const float* bias, uint32_t (&h)[16],
                                            uint32_t (&m)[16]) {
  const __nv_bfloat162 zero = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
  for (int j = 0; j < 32; j += 4) {
    const float4 b = *reinterpret_cast<const float4*>(bias + j);
    const __nv_bfloat162 p = __floats2bfloat162_rn(v[j] + b.x, v[j + 1] + b.y);
    const __nv_bfloat162 q = __floats2bfloat162_rn(v[j + 2] + b.z, v[j + 3] + b.w);
    const __nv_bfloat162 rp = __hmax2(p, zero), rq = __hmax2(q, zero);
    h[j / 2] = *reinterpret_cast<const uint32_t*>(&rp);
    h[j / 2 + 1] = *reinterpret_cast<const uint32_t*>(&rq);
    m[j / 2] = __hgt2_mask(p, zero);
    m[j / 2 + 1] = __hgt2_mask(q, zero);
  }
}
// logit of a row from its second hidden layer
__device__ __forceinline__ float tc_logit(const uint32_t (&h)[16], const float* w3, float b3) {
  float z = b3;
#pragma unroll
  for (int j = 0; j < 32; j += 4) {
    const float4 w = *reinterpret_cast<const float4*>(w3 + j);
    z += __uint_as_float(h[j / 2] << 16) * w.x;
    z += __uint_as_float(h[j / 2] & 0xffff0000u) * w.y;
    z += __uint_as_float(h[j / 2 + 1] << 16) * w.z;
    z += __uint_as_float(h[j / 2 + 1] & 0xffff0000u) * w.w;
  }
  return z;
}

// weights into the operand layout, biases, TMEM and the mbarrier
template <bool BWD>
__device__ __forceinline__ void tc_setup(TcShared<BWD>& S, const unsigned char* block, uint32_t ncols) {
  const float* master = reinterpret_cast<const float*>(block);
  const uint16_t* wb = reinterpret_cast<const uint16_t*>(block + MLP_MASTER_BYTES);
  const int t = threadIdx.x;
  if (t < 32) tc05::alloc(&S.tmem, ncols);   // warp 0
  for (int e = t; e < MLP_NH * MLP_NF; e += blockDim.x) {
    const int n = e / MLP_NF, k = e % MLP_NF;
    *reinterpret_cast<uint16_t*>(S.B1 + tc05::kmajor_offset(n, k, MLP_NF)) = wb[MLP_WB_W1 + n * MLP_NF + k];
  }
  for (int e = t; e < MLP_NH * MLP_NH; e += blockDim.x) {
    const int n = e / MLP_NH, k = e % MLP_NH;
    const uint16_t w = wb[MLP_WB_W2 + e];
    *reinterpret_cast<uint16_t*>(S.B2 + tc05::kmajor_offset(n, k, MLP_NH)) = w;
    if (BWD) *reinterpret_cast<uint16_t*>(S.B3 + tc05::kmajor_offset(k, n, MLP_NH)) = w;   // B3[h][o] = W2[o][h]
  }
  if (t < MLP_NH) {
    S.b1[t] = master[MLP_OFF_B1 + t];
    S.b2[t] = master[MLP_OFF_B2 + t];
    S.w3[t] = from_bf16_bits(wb[MLP_WB_W3 + t]);
  }
  if (t == 0) tc05::mbar_init(&S.mbar);
  tc05::fence_smem_to_async();
  tc05::fence_before_sync();
  __syncthreads();
  tc05::fence_after_sync();
}

// D = A B^T over K columns of a row block (one thread): A starts at its first
// column in a block whose groups of 8 rows are `group` bytes, B is a weight.
__device__ __forceinline__ void tc_layer(uint32_t d, const unsigned char* A, uint32_t group, const unsigned char* B,
                                         int K) {
  const uint32_t id = tc05::idesc_bf16_f32(TC_ROWS, MLP_NH);
  for (int ks = 0; ks < K / 16; ++ks) {
    const uint64_t da = tc05::smem_desc(tc05::smem_addr(A) + ks * 2 * TC_LBO, TC_LBO, group);
    const uint64_t db = tc05::smem_desc(tc05::smem_addr(B) + ks * 2 * TC_LBO, TC_LBO, (uint32_t)K * 16);
    tc05::mma_bf16(d, da, db, id, ks > 0 ? 1u : 0u);
  }
}

// the weight gradients of a tile, DD^T XH over its 128 rows (one thread)
__device__ __forceinline__ void tc_weight_grads(uint32_t d, const unsigned char* DD, const unsigned char* XH,
                                                bool accumulate) {
  const uint32_t id = tc05::idesc_bf16_f32_mn(TC_ROWS, XH_COLS<true>);
#pragma unroll
  for (int ks = 0; ks < TC_ROWS / 16; ++ks) {
    const uint64_t da = tc05::smem_desc(tc05::smem_addr(DD) + ks * 2 * DD_GROUP, DD_GROUP, TC_LBO);
    const uint64_t db = tc05::smem_desc(tc05::smem_addr(XH) + ks * 2 * XH_GROUP<true>, XH_GROUP<true>, TC_LBO);
    tc05::mma_bf16(d, da, db, id, ks > 0 || accumulate ? 1u : 0u);
  }
}

// all threads: wait for the products committed last
template <bool BWD>
__device__ __forceinline__ bool tc_wait(TcShared<BWD>& S, uint32_t& phase) {
  const bool ok = tc05::mbar_wait(&S.mbar, phase);
  phase ^= 1u;
  tc05::fence_after_sync();
  return ok;
}
// this thread's row of 32 columns of an accumulator
__device__ __forceinline__ void tc_row(uint32_t tmem, uint32_t col, float (&v)[32]) {
  tc05::ld_32cols(tmem + ((uint32_t)(threadIdx.x & ~31) << 16) + col, v);
}

// threads' shared-memory writes visible to the next product, TMEM reads done
__device__ __forceinline__ void tc_sync() {
  tc05::fence_smem_to_async();
  tc05::fence_before_sync();
  __syncthreads();
}

template <bool BWD>
__device__ __forceinline__ void tc_teardown(TcShared<BWD>& S, uint32_t ncols) {
  tc05::fence_before_sync();
  __syncthreads();
  if (threadIdx.x < 32) {
    tc05::fence_after_sync();
    tc05::dealloc(S.tmem, ncols);
  }
}

// Features of a tile's rows (zero past n): the warp that owns rows 32w..32w+31
// reads their 2 KB front to back, 16 bytes a lane -- lane l takes features
// 4 (l & 3).. of row l / 4 of each group of eight -- and stores them as bf16
// where the operand wants them; no lane needs a row of its own.
__device__ __forceinline__ void tc_fetch_x(const float* X, long long tile_row, long long n, float4 (&x)[4]) {
  const int lane = threadIdx.x & 31;
  const long long r0 = tile_row + (threadIdx.x & ~31) + (lane >> 2);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const long long r = r0 + 8 * q;
    x[q] = r < n ? __ldg(reinterpret_cast<const float4*>(X + r * MLP_NF) + (lane & 3)) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
}
template <bool BWD>
__device__ __forceinline__ void tc_store_x(TcShared<BWD>& S, const float4 (&x)[4]) {
  const int lane = threadIdx.x & 31, r0 = (threadIdx.x & ~31) + (lane >> 2);
#pragma unroll
  for (int q = 0; q < 4; ++q)
    *reinterpret_cast<uint2*>(S.XH + tc05::kmajor_offset(r0 + 8 * q, XH_X + 4 * (lane & 3), XH_COLS<BWD>)) =
        make_uint2(pack_bf16x2(x[q].x, x[q].y), pack_bf16x2(x[q].z, x[q].w));
}

// Logits of n rows; a product that never completes gives NaN logits (no hang).
// Layer 2 of a tile and layer 1 of the next are issued together, so a tile
// costs one barrier and one wait for the tensor cores instead of two.
// Bound by instruction issue and the latency of the products, not by memory
// (68 bytes a row).  Measured (GB300), 1e6 / 4e6 rows: 25 / 77 us; 32 / 93 with two
// waits a tile, rows read by their own threads and scalar bf16 conversions.
__global__ void __launch_bounds__(TC_ROWS, 8) mlp_forward_tc_kernel(const unsigned char* block, const float* X,
                                                                  long long n, float* z) {
  __shared__ TcShared<false> S;
  const float b3 = reinterpret_cast<const float*>(block)[MLP_OFF_B3];
  const long long stride = (long long)gridDim.x * TC_ROWS;
  long long base = (long long)blockIdx.x * TC_ROWS;
  float4 x[4];
  tc_fetch_x(X, base, n, x);
  tc_setup(S, block, 64);
  uint32_t phase = 0;
  bool ok = true;
  tc_store_x(S, x);
  tc_sync();
  if (threadIdx.x == 0) {
    tc05::fence_after_sync();
    tc_layer(S.tmem, S.XH + XH_X / 8 * TC_LBO, XH_GROUP<false>, S.B1, MLP_NF);
    tc05::commit(&S.mbar);
  }
  tc_fetch_x(X, base + stride, n, x);
  ok &= tc_wait(S, phase);
  for (; base < n; base += stride) {
    float a[32];
    uint32_t h[16], m[16];
    tc_row(S.tmem, 0, a);
    tc_activate(a, S.b1, h, m);
    tc_store32(S.XH, XH_COLS<false>, 0, h);
    tc_store_x(S, x);
    tc_sync();
    if (threadIdx.x == 0) {
      tc05::fence_after_sync();
      tc_layer(S.tmem + 32, S.XH, XH_GROUP<false>, S.B2, MLP_NH);
      if (base + stride < n) tc_layer(S.tmem, S.XH + XH_X / 8 * TC_LBO, XH_GROUP<false>, S.B1, MLP_NF);
      tc05::commit(&S.mbar);
    }
    tc_fetch_x(X, base + 2 * stride, n, x);   // two tiles on, while the products run
    ok &= tc_wait(S, phase);
    tc_row(S.tmem, 32, a);
    tc_activate(a, S.b2, h, m);
    const float zz = tc_logit(h, S.w3, b3);
    const long long row = base + threadIdx.x;
    if (row < n) z[row] = ok ? zz : __int_as_float(0x7fc00000);
  }
  tc_teardown(S, 64);
}

// Sum of v[j] over the warp's lanes, in lane j: halves of the columns change
// places between lane pairs, 31 exchanges for 32 columns instead of 160.
__device__ __forceinline__ float column_sums(float (&v)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int w = 16; w > 0; w >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int j = 0; j < w; ++j) {
      const float give = up ? v[j] : v[j + w], keep = up ? v[j + w] : v[j];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, give, w);
    }
  }
  return v[0];
}

// Four consecutive values added to grad[p..p+3] (one reduction of 16 bytes where
// grad is aligned to it; p is a multiple of four).
__device__ __forceinline__ void add4(float* grad, int p, float a, float b, float c, float d) {
  if (((uintptr_t)grad & 15) == 0) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(grad + p), "f"(a), "f"(b), "f"(c), "f"(d)
                 : "memory");
  } else {
    atomicAdd(&grad[p], a);
    atomicAdd(&grad[p + 1], b);
    atomicAdd(&grad[p + 2], c);
    atomicAdd(&grad[p + 3], d);
  }
}

// Backward pass of the mean binary cross-entropy, added into grad[NPARAM]
// (deltas and activations rounded to bf16 where they enter a product, sums in
// FP32).  A product that never completes makes the gradient NaN (no hang).
// TMEM columns: 0-31 layer 1, layer 2 and dh1 in turn (each is in registers
// before the next is issued); 32-127 DD^T XH.  Three CTAs per SM (their shared
// memory): the four products of a tile follow one another, and the other CTAs
// fill the waits.  Measured (GB300), 16384 / 1e6 / 4e6 rows: 8.8 / 54 / 178 us.
// With the sums of db and dW3 by warp shuffles and the weight gradients by
// mma.sync on operands gathered element by element it took 21.8 / 354 / 1438.
__global__ void __launch_bounds__(TC_ROWS, 3) mlp_backward_tc_kernel(const unsigned char* block, const float* X,
                                                                     const float* y, long long n, float* grad) {
  extern __shared__ __align__(128) unsigned char tc_smem[];
  TcShared<true>& S = *reinterpret_cast<TcShared<true>*>(tc_smem);
  __shared__ float G3[4];   // db3
  const float b3 = reinterpret_cast<const float*>(block)[MLP_OFF_B3];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float inv_n = 1.0f / (float)n;
  const long long stride = (long long)gridDim.x * TC_ROWS;
  const long long first = (long long)blockIdx.x * TC_ROWS;
  constexpr int XC = XH_COLS<true>;
  float4 x[4];
  tc_fetch_x(X, first, n, x);
  float label = first + threadIdx.x < n ? __ldg(y + first + threadIdx.x) : 0.f;
  tc_setup(S, block, 128);
  uint32_t phase = 0;
  bool ok = true;
  float sb3 = 0.f;   // this thread's rows: sum of dz
  const uint32_t none[4] = {0u, 0u, 0u, 0u};
  tc_store8(S.XH, XC, XH_DZ + 8, none);   // the dz columns that stay zero
  for (long long base = first; base < n; base += stride) {
    const long long row = base + threadIdx.x;
    tc_store_x(S, x);
    tc_sync();
    if (threadIdx.x == 0) {
      tc05::fence_after_sync();
      tc_layer(S.tmem, S.XH + XH_X / 8 * TC_LBO, XH_GROUP<true>, S.B1, MLP_NF);
      tc05::commit(&S.mbar);
    }
    const float yr = label;
    tc_fetch_x(X, base + stride, n, x);   // the next tile's rows, while the products run
    label = row + stride < n ? __ldg(y + row + stride) : 0.f;
    ok &= tc_wait(S, phase);
    float v[32];
    uint32_t h[16], m1[16], m2[16], p[16];
    tc_row(S.tmem, 0, v);
    tc_activate(v, S.b1, h, m1);
    tc_store32(S.XH, XC, 0, h);
    tc_sync();
    if (threadIdx.x == 0) {
      tc05::fence_after_sync();
      tc_layer(S.tmem, S.XH, XH_GROUP<true>, S.B2, MLP_NH);
      tc05::commit(&S.mbar);
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) p[j] = m1[j] & 0x3f803f80u;   // 0 or 1 in bf16
    tc_store32(S.XH, XC, XH_M1, p);
    ok &= tc_wait(S, phase);
    tc_row(S.tmem, 0, v);
    tc_activate(v, S.b2, h, m2);
    // output layer, its gradient, delta2 = dz W3 [a2 > 0]
    const float zz = tc_logit(h, S.w3, b3);
    const float dz = row < n ? ((1.f / (1.f + __expf(-zz))) - yr) * inv_n : 0.f;
    sb3 += dz;
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
      const float4 w = *reinterpret_cast<const float4*>(S.w3 + j);
      p[j / 2] = pack_bf16x2(dz * w.x, dz * w.y) & m2[j / 2];
      p[j / 2 + 1] = pack_bf16x2(dz * w.z, dz * w.w) & m2[j / 2 + 1];
    }
    tc_store32(S.DD, DD_COLS, 0, p);
    tc_sync();
    // dh1 = delta2 W2; delta1 = dh1 [a1 > 0]
    if (threadIdx.x == 0) {
      tc05::fence_after_sync();
      tc_layer(S.tmem, S.DD, DD_GROUP, S.B3, MLP_NH);
      tc05::commit(&S.mbar);
    }
    tc_store32(S.DD, DD_COLS, DD_H2, h);
#pragma unroll
    for (int j = 0; j < 16; ++j) p[j] = m2[j] & 0x3f803f80u;
    tc_store32(S.DD, DD_COLS, DD_M2, p);
    {
      const float hi = from_bf16_bits(to_bf16_bits(dz)), r1 = dz - hi;
      const float mid = from_bf16_bits(to_bf16_bits(r1));
      const uint32_t terms[4] = {pack_bf16x2(hi, mid), pack_bf16x2(r1 - mid, 0.f), 0u, 0u};
      tc_store8(S.XH, XC, XH_DZ, terms);
    }
    ok &= tc_wait(S, phase);
    tc_row(S.tmem, 0, v);
#pragma unroll
    for (int j = 0; j < 16; ++j) p[j] = pack_bf16x2(v[2 * j], v[2 * j + 1]) & m1[j];
    tc_store32(S.DD, DD_COLS, DD_D1, p);
    tc_sync();
    if (threadIdx.x == 0) {
      tc05::fence_after_sync();
      tc_weight_grads(S.tmem + 32, S.DD, S.XH, base != first);
      tc05::commit(&S.mbar);
    }
    ok &= tc_wait(S, phase);   // before the operands are overwritten
  }
  // DD^T XH, 32 rows a warp: warp 0 (delta2) dW2 in columns 0-31 and C in
  // 64-95, warp 1 (delta1) dW1 in 32-47, warps 2 (m2) and 3 (h2) their sums
  // over dz in 48-50
  ok = __syncthreads_and(ok);
  const float nan = __int_as_float(0x7fc00000);
  float w[32];
  tc_row(S.tmem, warp == 0 ? 32 : 32 + 32, w);   // (columns 0-31 or 32-63 of the block)
  if (warp < 2) {
    const int cols = warp == 0 ? MLP_NH : MLP_NF;
    float* g = grad + (warp == 0 ? MLP_OFF_W2 + lane * MLP_NH : MLP_OFF_W1 + lane * MLP_NF);
#pragma unroll
    for (int c = 0; c < 32; c += 4)
      if (c < cols) add4(g, c, ok ? w[c] : nan, ok ? w[c + 1] : nan, ok ? w[c + 2] : nan, ok ? w[c + 3] : nan);
  } else {
    const float sum = w[16] + (w[17] + w[18]);
    atomicAdd(&grad[(warp == 2 ? MLP_OFF_B2 : MLP_OFF_W3) + lane], ok ? (warp == 2 ? S.w3[lane] * sum : sum) : nan);
  }
  if (warp == 0) {   // db1_j = sum over o (lanes) of W2[o][j] C[o][j]
    tc_row(S.tmem, 32 + XH_M1, w);
    const uint16_t* w2 = reinterpret_cast<const uint16_t*>(block + MLP_MASTER_BYTES) + MLP_WB_W2 + lane * MLP_NH;
#pragma unroll
    for (int j = 0; j < 32; ++j) w[j] *= from_bf16_bits(w2[j]);
    const float s = column_sums(w);
    atomicAdd(&grad[MLP_OFF_B1 + lane], ok ? s : nan);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sb3 += __shfl_xor_sync(0xffffffffu, sb3, o);
  if (lane == 0) G3[warp] = sb3;
  tc_teardown(S, 128);   // (with a barrier)
  if (threadIdx.x == 0) atomicAdd(&grad[MLP_OFF_B3], ok ? (G3[0] + G3[1]) + (G3[2] + G3[3]) : nan);
}

// Adam on the FP32 master weights; refreshes the bf16 copies.
__global__ void mlp_adam_kernel(unsigned char* block, float* m, float* v, const float* grad, int step, float lr,
                                float beta1, float beta2, float eps) {
  float* master = reinterpret_cast<float*>(block);
  uint16_t* wb = reinterpret_cast<uint16_t*>(block + MLP_MASTER_BYTES);
  const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < MLP_NPARAM; p += gridDim.x * blockDim.x) {
    const float gp = grad[p];
    const float mp = beta1 * m[p] + (1.f - beta1) * gp;
    const float vp = beta2 * v[p] + (1.f - beta2) * gp * gp;
    m[p] = mp;
    v[p] = vp;
    const float w = master[p] - lr * (mp / c1) / (sqrtf(vp / c2) + eps);
    master[p] = w;
    int q = -1;
    if (p < MLP_OFF_B1) q = MLP_WB_W1 + p;
    else if (p >= MLP_OFF_W2 && p < MLP_OFF_B2) q = MLP_WB_W2 + (p - MLP_OFF_W2);
    else if (p >= MLP_OFF_W3 && p < MLP_OFF_B3) q = MLP_WB_W3 + (p - MLP_OFF_W3);
    if (q >= 0) wb[q] = to_bf16_bits(w);
  }
}

__global__ void mlp_refresh_kernel(unsigned char* block) {
  const float* master = reinterpret_cast<const float*>(block);
  uint16_t* wb = reinterpret_cast<uint16_t*>(block + MLP_MASTER_BYTES);
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < MLP_NPARAM; p += gridDim.x * blockDim.x) {
    int q = -1;
    if (p < MLP_OFF_B1) q = MLP_WB_W1 + p;
    else if (p >= MLP_OFF_W2 && p < MLP_OFF_B2) q = MLP_WB_W2 + (p - MLP_OFF_W2);
    else if (p >= MLP_OFF_W3 && p < MLP_OFF_B3) q = MLP_WB_W3 + (p - MLP_OFF_W3);
    if (q >= 0) wb[q] = to_bf16_bits(master[p]);
  }
}

// Face sampler: features and HLL/HLLD label of the face below cell s along
// axis d (face id = d * ncell + s) of a periodic box, from the primitives W
// of the current state (reconstruction and solvers in the state's arithmetic).
template <typename R>
__global__ void dump_faces_kernel(Geo g, const R* W, const long long* ids, long long n, float* X, float* y,
                                  float* score) {
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
    const long long id = ids[q];
    const int d = (int)(id / g.ncell);
    const long long s = id - (long long)d * g.ncell;
    int c[3];
    c[0] = (int)(s % g.n[0]);
    c[1] = (int)((s / g.n[0]) % g.n[1]);
    c[2] = (int)(s / ((long long)g.n[0] * g.n[1]));
    const int t1 = (d + 1) % 3, t2 = (d + 2) % 3;
    R cells[4][7];
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      int cc[3] = {c[0], c[1], c[2]};
      cc[d] = wrapc(cc[d] + o - 2, g.n[d], 0);
      const long long si = cc[0] + (long long)g.n[0] * (cc[1] + (long long)g.n[1] * cc[2]);
      cells[o][0] = W[0 * g.ncell + si];
      cells[o][1] = W[(1 + d) * g.ncell + si];
      cells[o][2] = W[(1 + t1) * g.ncell + si];
      cells[o][3] = W[(1 + t2) * g.ncell + si];
      cells[o][4] = W[4 * g.ncell + si];
      cells[o][5] = W[(5 + t1) * g.ncell + si];
      cells[o][6] = W[(5 + t2) * g.ncell + si];
    }
    const R bn = W[(8 + d) * g.ncell + s];
    R wl[7], wr[7], fd[7], fl[7];
    plm_face(cells[0], cells[1], cells[2], cells[3], wl, wr, gpar<R>(g.rho_floor, g.frho_floor), gpar<R>(g.p_floor, g.fp_floor));
    const R gam = gpar<R>(g.gamma, g.fgamma);
    const R cl = fast_speed(wl, bn, gam), cr = fast_speed(wr, bn, gam);
    hlld_flux(wl, wr, bn, gam, fd);
    hll_flux(wl, wr, bn, gam, fl);
    float f[MLP_NF];
    face_features(wl, wr, bn, cl, cr, f);
#pragma unroll
    for (int k = 0; k < MLP_NF; ++k) X[q * MLP_NF + k] = f[k];
    const R rho = R(0.5) * (wl[0] + wr[0]);
    const R cm = rmax(cl, cr);
    const R b = rsqrt_(rho) * cm;
    const R sc[7] = {rho * cm, rho * cm * cm, rho * cm * cm, rho * cm * cm, rho * cm * cm * cm, b * cm, b * cm};
    R m = R(0);
#pragma unroll
    for (int k = 0; k < 7; ++k) m = rmax(m, rabs(fd[k] - fl[k]) / sc[k]);
    y[q] = m > R(1e-3) ? 1.f : 0.f;
    if (score) score[q] = (float)m;
  }
}

}  // namespace mhd

using namespace mhd;

extern "C" size_t mlp_param_bytes(void) { return MLP_BLOCK_BYTES; }

extern "C" int mlp_init(void* block, const float* master_host, void* stream) {
  if (!block || !master_host) return MHD_ERR_INVALID;
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemcpyAsync(block, master_host, MLP_NPARAM * sizeof(float), cudaMemcpyHostToDevice, st) != cudaSuccess)
    return MHD_ERR_CUDA;
  mlp_refresh_kernel<<<7, 256, 0, st>>>((unsigned char*)block);
  if (cudaGetLastError() != cudaSuccess) return MHD_ERR_CUDA;
  return cudaStreamSynchronize(st) == cudaSuccess ? MHD_OK : MHD_ERR_CUDA;
}

// 128-row tiles over a grid of at most `per_sm` CTAs per SM (the forward
// kernel's 64 TMEM columns allow 8 per SM; the backward kernel's shared memory 3)
static unsigned grid_for_tiles(long long n, int per_sm) {
  long long tiles = (n + TC_ROWS - 1) / TC_ROWS;
  if (tiles > 152LL * per_sm) tiles = 152LL * per_sm;
  return (unsigned)(tiles < 1 ? 1 : tiles);
}

extern "C" int mlp_forward(const void* block, const float* X, long long n, float* z, void* stream) {
  if (!block || !X || !z || n < 0 || ((uintptr_t)X & 15)) return MHD_ERR_INVALID;
  if (n == 0) return MHD_OK;
  mlp_forward_tc_kernel<<<grid_for_tiles(n, 8), TC_ROWS, 0, (cudaStream_t)stream>>>((const unsigned char*)block, X, n,
                                                                                  z);
  return cudaGetLastError() == cudaSuccess ? MHD_OK : MHD_ERR_CUDA;
}

extern "C" int mlp_backward(const void* block, const float* X, const float* y, long long n, float* grad,
                            void* stream) {
  if (!block || !X || !y || !grad || n < 1 || ((uintptr_t)X & 15)) return MHD_ERR_INVALID;
  constexpr int smem = (int)sizeof(TcShared<true>);   // beyond the 48 KB a kernel gets unasked
  if (cudaFuncSetAttribute(mlp_backward_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
    return MHD_ERR_CUDA;
  mlp_backward_tc_kernel<<<grid_for_tiles(n, 3), TC_ROWS, smem, (cudaStream_t)stream>>>((const unsigned char*)block, X,
                                                                                      y, n, grad);
  return cudaGetLastError() == cudaSuccess ? MHD_OK : MHD_ERR_CUDA;
}

extern "C" int mlp_adam(void* block, float* m, float* v, const float* grad, int step, double lr, double beta1,
                        double beta2, double eps, void* stream) {
  if (!block || !m || !v || !grad || step < 1) return MHD_ERR_INVALID;
  mlp_adam_kernel<<<7, 256, 0, (cudaStream_t)stream>>>((unsigned char*)block, m, v, grad, step, (float)lr,
                                                       (float)beta1, (float)beta2, (float)eps);
  return cudaGetLastError() == cudaSuccess ? MHD_OK : MHD_ERR_CUDA;
}

// The three launches of a training step from one call.  On the default minibatch
// (16384 rows) the device takes about 15 us a step (gradient 8.7, Adam 4.9) and
// the three calls from Python 30.7; from one call a step takes 18.2.
extern "C" int mlp_train_step(void* block, const float* X, const float* y, long long n, float* grad, float* m,
                              float* v, int step, double lr, double beta1, double beta2, double eps, void* stream) {
  if (!grad || !m || !v || step < 1) return MHD_ERR_INVALID;
  if (cudaMemsetAsync(grad, 0, MLP_NPARAM * sizeof(float), (cudaStream_t)stream) != cudaSuccess) return MHD_ERR_CUDA;
  const int rc = mlp_backward(block, X, y, n, grad, stream);
  return rc == MHD_OK ? mlp_adam(block, m, v, grad, step, lr, beta1, beta2, eps, stream) : rc;
}

// Face sampler entry (needs the handle's current primitives).
namespace mhd {
int dump_faces_launch(int prec, const Geo& g, const void* W, const long long* ids, long long n, float* X, float* y,
                      float* score, cudaStream_t st) {
  unsigned nb = (unsigned)((n + 255) / 256);
  if (nb > 152u * 16u) nb = 152u * 16u;
  if (nb < 1) nb = 1;
  if (prec == P_FP64) dump_faces_kernel<double><<<nb, 256, 0, st>>>(g, (const double*)W, ids, n, X, y, score);
  else dump_faces_kernel<float><<<nb, 256, 0, st>>>(g, (const float*)W, ids, n, X, y, score);
  return cudaGetLastError() == cudaSuccess ? MHD_OK : MHD_ERR_CUDA;
}
}  // namespace mhd

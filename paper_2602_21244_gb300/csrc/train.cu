// Training of the neural collision operator: forward, loss, hand-written
// backward with activation recomputation, Adam (Sec. 2.6: MSE against the
// harvested post-collision state; Sec. 2.3 shell projection and pair update
// and Sec. 2.5 moment matching in the graph; Adam as in Sec. 3.4.2).
//
// Per CTA (persistent, 512 threads, one 128-pair tile at a time):
//   forward   X -> z1..z3 (tcgen05, input and activations as bf16 hi + lo),
//             y, u = y/|y|, v_r' = |v_r| u, centre-of-mass update, moment
//             matching over pseudo-cells of 16 pairs (32 particles), loss
//   backward  dL/dv_new -> closed-form moment-matching and projection
//             backward -> dz4 = dL/dy; z_3 is still in the accumulator that
//             the forward left it in (the output layer has columns of its
//             own), z_2 and z_1 are recomputed by an MMA from exactly the
//             forward's operands (h1's low bf16 terms stay in tensor memory until
//             z_2 is there, so nothing else has to be regenerated), so every z_l equals the
//             forward's bit for bit (the stored variant reads back the copy
//             the forward wrote to global memory instead),
//             dz_l = dh_l * act'(z_l), dW_l += dz_l^T h_{l-1} (MN-major
//             operands, accumulated in TMEM across the CTA's tiles),
//             dh_{l-1} = dz_l W_l (W_l read MN-major from the forward tile)
//   flush     per-CTA partial gradients to global memory; a second kernel
//             sums them over CTAs in a fixed order (deterministic)
// TMEM columns: 0..127 scratch, 128..255 dW2, 256..383 dW3, 384..415 dW1
// (hi|lo input columns), 416..431 dW4^T, 432..447 output layer, 448..511 the
// low terms of h1 (A operand), in the backward 64 columns of z_1.
#include <cuda_bf16.h>

#include "internal.cuh"
#include "tc.cuh"

namespace dsmc {

namespace {
constexpr int kT = 128;          // pairs per tile
constexpr int kNT = 512;         // threads
constexpr int kH = 128;          // width
constexpr int kXin = 32;         // input columns (hi | lo)
constexpr int kGroup = 16;       // pairs per pseudo-cell
// shared memory layout
constexpr uint32_t S_WOUT = 0;                         // [16 x 128]
constexpr uint32_t S_WIN = S_WOUT + 16 * kH * 2;       // [128 x 32]
constexpr uint32_t S_W2 = S_WIN + kH * kXin * 2;       // [128 x 128]
constexpr uint32_t S_W3 = S_W2 + kH * kH * 2;          // [128 x 128]
constexpr uint32_t S_X = S_W3 + kH * kH * 2;           // [128 x 32] hi | lo
constexpr uint32_t S_H1 = S_X + kT * kXin * 2;         // [128 x 128] h1 (single bf16 copy)
constexpr uint32_t S_H2 = S_H1 + kT * kH * 2;          // [128 x 128] h2 (single)
constexpr uint32_t S_WK = S_H2 + kT * kH * 2;          // [128 x 128] x 2: working hi, lo; later dz
constexpr uint32_t S_WKLO = S_WK + kT * kH * 2;
constexpr uint32_t S_DZ4 = S_WKLO + kT * kH * 2;       // [128 x 16] dz of the output layer (bf16)
constexpr uint32_t S_DZ4F = S_DZ4 + kT * 16 * 2;       // [128 x 3] FP32
constexpr uint32_t S_BIAS = S_DZ4F + kT * 4 * 4;       // 3*128 + 16 floats
constexpr uint32_t S_WO32 = S_BIAS + (3 * kH + 16) * 4;  // output weights in FP32 [3 x 128]
constexpr uint32_t S_MISC = S_WO32 + 3 * kH * 4;       // mbarrier, tmem ptr, flag, drain mbarrier
constexpr uint32_t S_PRE = S_MISC + 64;                // [5 x 128] FP64: d, |v_r|, Theta_pre term of each row
constexpr uint32_t S_MEAN = S_PRE + 5 * kT * 8;        // [8 x 4] FP64: mean velocity of each group
constexpr uint32_t S_TOTAL = S_MEAN + (kT / kGroup) * 4 * 8;
static_assert(S_PRE % 8 == 0 && S_TOTAL <= 227 * 1024, "shared memory");
constexpr int kIssuer = 256;     // thread that issues the MMAs (of a warp without rows)
// per-CTA partial: dW1 (128 x 32), dW2, dW3 (128 x 128), dW4^T (128 x 16), then the bias
// gradients of each of the 4 TMEM lane groups [4 x 400], then the loss of each lane group.
// The matrices lie as the threads hold them, four consecutive columns per thread and
// the threads side by side (wpos), so that a warp's stores fill whole lines (2^14 pairs, one
// tile per CTA: 48 us; row-major, 32 lines per store of a warp, 51).
constexpr int kPDB = kH * kXin + 2 * kH * kH + kH * 16;
constexpr int kPLOSS = kPDB + 4 * 400;
constexpr int kPartial = kPLOSS + 16;
// position of (row, column) in a matrix of `rows` rows held 4 columns at a time; of
// dW2 and dW3 with 32 columns per group of 128 threads
__host__ __device__ constexpr int wpos(int row, int col, int rows) { return ((col >> 2) * rows + row) * 4 + (col & 3); }
__host__ __device__ constexpr int wpos32(int row, int col) { return wpos((col >> 5) * kH + row, col & 31, 4 * kH); }
constexpr int kNW = kH * 8 + 2 * kH * kH + 3 * kH;   // weights (d_in 8)
constexpr int kNB = 3 * kH + 3;                      // biases
constexpr uint32_t TM_DW2 = 128, TM_DW3 = 256, TM_DW1 = 384, TM_DW4 = 416, TM_OUT = 432, TM_H1LO = 448;
}  // namespace

struct TrainArgs {
  int mode;                  // 0 forward only, 1 backward from given dL/dv_new, 2 MSE loss vs targets
  int act;
  int64_t n;                 // pairs (multiple of 16)
  uint64_t seed, t;
  double sigma_v_inv, T_ref_inv, eps;
  double grad_scale, loss_scale;   // 1 / (n sigma_v^2), 1 / (2 n sigma_v^2)
  const float* theta;        // FP32 parameters: weights (row-major per layer), then biases
  const double *vi, *vj, *T, *ti, *tj;   // [n x 3], [n], targets [n x 3]
  const double *gi, *gj;     // mode 1: dL/dv_new [n x 3]
  double *oi, *oj;           // mode 0: v_new [n x 3]
  float* zst;                // stored variant: z_l (accumulator, without bias) per tile, else null
  float* partial;            // [gridDim x kPartial]
  int* status;
};

__device__ __forceinline__ float act_fn(int act, float z) {
  if (act == 1) return fmaxf(z, 0.f);
  return __fdividef(z, 1.f + __expf(-z));
}
// SiLU'(z) = s (1 + z (1 - s)), s = 1/(1 + e^-z), of two values on the paired FP32
// pipe, the same roundings as one value at a time (which took the 16 warps 3,700
// cycles a layer, now 2,000).
__device__ __forceinline__ float2 silu_slope2(float2 z) {
  const float2 one = make_float2(1.f, 1.f), m1 = make_float2(-1.f, -1.f);
  const float2 t = __fmul2_rn(z, make_float2(-1.44269504f, -1.44269504f));   // -z log2(e)
  const float2 d = __fadd2_rn(make_float2(tc::ex2_approx(t.x), tc::ex2_approx(t.y)), one);
  const float2 s = make_float2(tc::rcp_approx(d.x), tc::rcp_approx(d.y));
  return __fmul2_rn(s, __ffma2_rn(z, __ffma2_rn(s, m1, one), one));
}

// v[32] per lane -> lane l returns the sum over the warp's lanes of v[l]
__device__ __forceinline__ float warp_colsum32(float* v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int w = 16; w >= 1; w >>= 1) {
#pragma unroll
    for (int k = 0; k < w; ++k) {
      const bool hi = lane & w;
      const float send = hi ? v[k] : v[k + w];
      const float keep = hi ? v[k + w] : v[k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, w);
    }
  }
  return v[0];
}

__device__ __forceinline__ uint16_t to_bf16(float x) {
  return __bfloat16_as_ushort(__float2bfloat16_rn(x));
}

// FP64 -> FP32 as the hardware converts, on the integer pipe where the result is
// a normal number (f64_to_f32), by the conversion instruction otherwise.
__device__ __forceinline__ float to_f32(double v) {
  const uint32_t e = ((uint32_t)__double2hiint(v) >> 20) & 0x7FFu;
  return e - 897u < 254u ? f64_to_f32(v) : (float)v;
}

// Two normals from the 53-bit uniforms of (a0, a1) and (b0, b1): 1 - u1 is a
// 53-bit integer over 2^53 too, rounded to FP32 from that integer.
__device__ __forceinline__ void box_muller2(uint32_t a0, uint32_t a1, uint32_t b0, uint32_t b1, float* z0, float* z1) {
  const uint64_t k = (((uint64_t)a0 << 32) | a1) >> 11;
  const float v1 = __ull2float_rn((1ull << 53) - k) * 1.1102230246251565e-16f;   // 2^-53
  const float rho = sqrtf(-2.f * __logf(v1));
  float s, c;
  __sincosf(f64_to_f32(2.0 * DSMC_PI * u53_int(b0, b1)), &s, &c);
  *z0 = rho * c;
  *z1 = rho * s;
}

__device__ __forceinline__ uint64_t kdesc(uint32_t a, int K) { return tc::sdesc(a, 128, (uint32_t)(K / 8) * 128); }
// MN-major view of a [rows x F] tile: MN = F (features), K = rows
__device__ __forceinline__ uint64_t mdesc(uint32_t a, int F) { return tc::sdesc(a, (uint32_t)(F / 8) * 128, 128); }

// sums over the 16 lanes of this half-warp (groups are 16 consecutive rows)
// of K values at once, K a power of two up to 8: each step halves the values a lane still adds (the
// other half goes to its partner), so K values take K + log2(16/K) - 1 or so FP64
// additions instead of 4 K; the totals come back by shuffles alone.
template <int K>
__device__ __forceinline__ void half_sums(double* v) {
  const int lane = threadIdx.x & 31;
  int w = 8;
#pragma unroll
  for (int k = K / 2; k >= 1; k >>= 1, w >>= 1) {
    const bool up = lane & w;
#pragma unroll
    for (int q = 0; q < k; ++q) {
      const double send = up ? v[q] : v[q + k], keep = up ? v[q + k] : v[q];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, send, w);
    }
  }
  double t = v[0];
  for (; w >= 1; w >>= 1) t += __shfl_xor_sync(0xffffffffu, t, w);
  // value q sits in the lanes whose upper bits of the half-warp index spell q
#pragma unroll
  for (int q = 0; q < K; ++q) v[q] = __shfl_sync(0xffffffffu, t, (lane & 16) | (q * (16 / K)));
}

__global__ void __launch_bounds__(kNT, 1) k_train(TrainArgs a) {
  dep_wait_alone();
  extern __shared__ __align__(1024) char sm[];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int row = ((warp & 3) << 5) | lane, cg = warp >> 2, c0 = cg * 32;
  const uint32_t sb = tc::smem_u32(sm);
  uint64_t* mbar = (uint64_t*)(sm + S_MISC);
  uint32_t* tptr = (uint32_t*)(sm + S_MISC + 8);
  volatile int* flag = (volatile int*)(sm + S_MISC + 12);
  uint64_t* drain = (uint64_t*)(sm + S_MISC + 16);   // after a wait that ran out: the MMAs in flight are done
  float* bias = (float*)(sm + S_BIAS);
  const float* wo32 = (const float*)(sm + S_WO32);
  // bias gradients and loss accumulate in registers of fixed threads (no atomics,
  // so the result does not depend on warp scheduling)
  float dbacc[3] = {0.f, 0.f, 0.f};  // layer l, column c0 + lane
  float dbo[3] = {0.f, 0.f, 0.f};    // output bias (lane 0 of warps 0..3)
  double lossw = 0.0;                // sum of |v_new - v_target|^2 of this thread's rows (warps 0..3)
  float* dz4f = (float*)(sm + S_DZ4F);
  // ---- weights into K-major tiles (eight columns, one 16-byte store, at a
  // time: a mini-batch of one tile per CTA pays this once per step), biases
  {
    uint32_t* z = (uint32_t*)(sm + S_WOUT);
    for (int q = t; q < (16 * kH * 2) / 4; q += kNT) z[q] = 0u;
    const float* bsrc = a.theta + kNW;
    for (int q = t; q < 3 * kH + 16; q += kNT) bias[q] = q < 3 * kH + 3 ? bsrc[q] : 0.f;
    __syncthreads();
    // (every row of eight then starts at 16 bytes; word by word the prologue took 2 us more of 2^14 pairs' 53)
    const bool wide = ((uintptr_t)a.theta & 15u) == 0;
    auto put8 = [&](uint32_t dst, const float* w8) {
      uint32_t r[4];
      if (wide) {
        const float4 x = ((const float4*)w8)[0], y = ((const float4*)w8)[1];
        r[0] = tc::pack_bf16x2(x.x, x.y); r[1] = tc::pack_bf16x2(x.z, x.w);
        r[2] = tc::pack_bf16x2(y.x, y.y); r[3] = tc::pack_bf16x2(y.z, y.w);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) r[q] = tc::pack_bf16x2(w8[2 * q], w8[2 * q + 1]);
      }
      tc::st_shared_v4(sb + dst, r[0], r[1], r[2], r[3]);
    };
    if (t < kH) {   // W1's eight columns, in columns 0..7 (hi) and 16..23 (lo) of its tile
      put8(S_WIN + tc::kmajor_offset(t, 0, kXin), a.theta + 8 * t);
      put8(S_WIN + tc::kmajor_offset(t, 16, kXin), a.theta + 8 * t);
      tc::st_shared_v4(sb + S_WIN + tc::kmajor_offset(t, 8, kXin), 0u, 0u, 0u, 0u);
      tc::st_shared_v4(sb + S_WIN + tc::kmajor_offset(t, 24, kXin), 0u, 0u, 0u, 0u);
    }
    const float* w2 = a.theta + kH * 8;
    for (int e = t; e < kH * kH / 8; e += kNT) {
      const int n = e >> 4, k = (e & 15) * 8;
      put8(S_W2 + tc::kmajor_offset(n, k, kH), w2 + n * kH + k);
      put8(S_W3 + tc::kmajor_offset(n, k, kH), w2 + kH * kH + n * kH + k);
    }
    const float* w4 = w2 + 2 * kH * kH;
    for (int e = t; e < 3 * kH; e += kNT) {
      const uint16_t b = to_bf16(w4[e]);
      *(uint16_t*)(sm + S_WOUT + tc::kmajor_offset(e >> 7, e & 127, kH)) = b;
      ((float*)(sm + S_WO32))[e] = __uint_as_float((uint32_t)b << 16);
    }
  }
  if (warp == 0) { tc::tmem_alloc(tptr, 512); tc::tmem_relinquish(); }
  if (t == 0) { tc::mbar_init(mbar, 1); tc::mbar_init(drain, 1); tc::mbar_fence_init(); *flag = 1; }
  tc::fence_async_smem();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tm = *(volatile uint32_t*)tptr;
  const uint32_t lane_tm = tm + ((uint32_t)((warp & 3) * 32) << 16);
  uint32_t phase = 0;
  int tiles_done = 0;

  // Every thread waits for the committed MMAs itself (each then reads TMEM
  // and reuses the operands' shared memory without a barrier); a timeout
  // clears the flag, read after the next barrier so that all threads leave together.
  auto wait_mma = [&]() {
    if (!tc::mbar_wait(mbar, phase, a.status, kBarrierLimitNs)) *flag = 0;
    phase ^= 1u;
    tc::fence_after();
  };
  // make shared-memory writes and TMEM accesses visible before an MMA; false after a timeout
  auto to_mma = [&]() -> bool {
    tc::fence_async_smem();
    tc::fence_before();
    __syncthreads();
    return *flag != 0;
  };

  // z1 from x (hi + lo): two K steps (thread kIssuer)
  auto input_mma = [&]() {
    const uint32_t id = tc::idesc_bf16(kT, kH);
    for (int s = 0; s < 2; ++s)
      tc::mma_bf16(tm, kdesc(sb + S_X + 256u * s, kXin), kdesc(sb + S_WIN + 256u * s, kXin), id, s > 0);
  };
  // columns 64 h .. 64 h + 63 of z1, for the backward (thread kIssuer)
  auto half_input_mma = [&](int h) {
    const uint32_t id = tc::idesc_bf16(kT, 64), w = sb + S_WIN + tc::kmajor_offset(64 * h, 0, kXin);
    for (int s = 0; s < 2; ++s) tc::mma_bf16(tm + TM_H1LO, kdesc(sb + S_X + 256u * s, kXin), kdesc(w + 256u * s, kXin), id, s > 0);
  };
  // The MMA of hidden layer l + 1 (l = 1, 2) on its input as hi + lo terms:
  // h1 = S_H1 + TM_H1LO (tensor memory), h2 = S_H2 + S_WK (thread kIssuer)
  auto hidden_mma = [&](int l) {
    const uint32_t id = tc::idesc_bf16(kT, kH);
    const uint32_t wl = l == 1 ? S_W2 : S_W3, hhi = l == 1 ? S_H1 : S_H2;
    for (int s = 0; s < 8; ++s)
      tc::mma_bf16(tm, kdesc(sb + hhi + 256u * s, kH), kdesc(sb + wl + 256u * s, kH), id, s > 0);
    for (int s = 0; s < 8; ++s) {
      if (l == 1) tc::mma_bf16_ta(tm, tm + TM_H1LO + 8u * s, kdesc(sb + wl + 256u * s, kH), id, 1);
      else tc::mma_bf16(tm, kdesc(sb + S_WK + 256u * s, kH), kdesc(sb + wl + 256u * s, kH), id, 1);
    }
  };
  // Epilogue of hidden layer l from this thread's 32 accumulator values v:
  // bias, activation (SiLU four values at a time on the paired FP32 pipe, as
  // in the collide kernel's epilogue), the hi + lo split; stored as the next
  // layer's input (l = 0: S_H1 and, the low terms, tensor memory; l = 1:
  // S_H2, S_WK; l = 2, the output layer's: S_WK, S_WKLO).
  auto hidden_epilogue = [&](int l, const float* v) {
    uint32_t pk[16], lo[16];
    const float2* b2 = (const float2*)(bias + l * kH + c0);
#pragma unroll
    for (int q = 0; q < 16; q += 2) {
      float2 va = __fadd2_rn(make_float2(v[2 * q], v[2 * q + 1]), b2[q]);
      float2 vb = __fadd2_rn(make_float2(v[2 * q + 2], v[2 * q + 3]), b2[q + 1]);
      if (a.act == 0) {
        tc::silu4x2(va, vb);
      } else {
        va = make_float2(act_fn(a.act, va.x), act_fn(a.act, va.y));
        vb = make_float2(act_fn(a.act, vb.x), act_fn(a.act, vb.y));
      }
      const float2 m1 = make_float2(-1.f, -1.f);
      pk[q] = tc::pack_bf16x2(va.x, va.y);
      pk[q + 1] = tc::pack_bf16x2(vb.x, vb.y);
      const float2 ra = __ffma2_rn(make_float2(__uint_as_float(pk[q] << 16), __uint_as_float(pk[q] & 0xFFFF0000u)), m1, va);
      const float2 rb = __ffma2_rn(make_float2(__uint_as_float(pk[q + 1] << 16), __uint_as_float(pk[q + 1] & 0xFFFF0000u)),
                                   m1, vb);
      lo[q] = tc::pack_bf16x2(ra.x, ra.y);
      lo[q + 1] = tc::pack_bf16x2(rb.x, rb.y);
    }
    const uint32_t dhi = l == 0 ? S_H1 : l == 1 ? S_H2 : S_WK, dlo = l == 1 ? S_WK : S_WKLO;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t off = tc::kmajor_offset(row, c0 + 8 * j, kH);
      tc::st_shared_v4(sb + dhi + off, pk[4 * j], pk[4 * j + 1], pk[4 * j + 2], pk[4 * j + 3]);
      if (l > 0) tc::st_shared_v4(sb + dlo + off, lo[4 * j], lo[4 * j + 1], lo[4 * j + 2], lo[4 * j + 3]);
    }
    if (l == 0) {   // row m in lane m, two bf16 per column
      tc::st16_async(lane_tm + TM_H1LO + (uint32_t)(c0 >> 1), lo);
      tc::wait_st();
    }
  };
  // The input row of pair p as its nonzero packed words: columns 0..7 of the
  // hi term in x[0..3], of the lo term in x[4..7].  Warps 4..7 form the next
  // tile's rows while warps 0..3 run the row stage.
  auto features = [&](int64_t p, uint32_t* x) {
    float f[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) f[q] = 0.f;
    if (p < a.n) {
#pragma unroll
      for (int c = 0; c < 3; ++c) f[c] = to_f32((a.vi[3 * p + c] - a.vj[3 * p + c]) * a.sigma_v_inv);
      f[3] = to_f32(a.T[p] * a.T_ref_inv);
      const u32x4 wa = draw(a.seed, (uint32_t)p, 0u, a.t, TAG_NOISE, 0);
      const u32x4 wb = draw(a.seed, (uint32_t)p, 0u, a.t, TAG_NOISE, 1);
      box_muller2(wa.x, wa.y, wa.z, wa.w, &f[4], &f[5]);
      box_muller2(wb.x, wb.y, wb.z, wb.w, &f[6], &f[7]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      x[q] = tc::pack_bf16x2(f[2 * q], f[2 * q + 1]);
      x[4 + q] = tc::pack_bf16x2(f[2 * q] - __uint_as_float(x[q] << 16), f[2 * q + 1] - __uint_as_float(x[q] & 0xFFFF0000u));
    }
  };
  // The row stage's part that needs no network, one row per thread of warps 0..3
  // in two halves of about an MMA wait each, handed to the row stage in shared
  // memory: the group moments over the 32 particles of the pseudo-cell, from the pairs'
  // sums and differences: the pair update keeps vi + vj, so the mean velocity
  // is the same before and after, and with d = (vi + vj)/2 - mean
  //   |vi - mean|^2 + |vj - mean|^2 = 2 |d|^2 + |v_r|^2 / 2
  // before it; after it the particles are at d +- v_r'/2.  (At the head of the
  // row stage 1M pairs take 1072 us, here 1010.)
  double* pre = (double*)(sm + S_PRE);
  double* mean = (double*)(sm + S_MEAN);
  auto row_pairs = [&](int64_t p, bool valid) {
    double g2 = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double vi = valid ? a.vi[3 * p + c] : 0.0, vj = valid ? a.vj[3 * p + c] : 0.0, ur = vi - vj;
      g2 = fma(ur, ur, g2);
      pre[c * kT + row] = vi + vj;
    }
    pre[3 * kT + row] = g2;
  };
  auto row_groups = [&]() {
    double d[4], sum[3], th = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) d[c] = sum[c] = pre[c * kT + row];
    d[3] = 0.0;
    half_sums<4>(d);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double u = d[c] * (1.0 / (2 * kGroup));
      if ((lane & (kGroup - 1)) == c) mean[4 * (row / kGroup) + c] = u;
      d[c] = fma(0.5, sum[c], -u);
      th = fma(d[c], d[c], th);
      pre[c * kT + row] = d[c];
    }
    const double g2 = pre[3 * kT + row];
    pre[3 * kT + row] = root64(g2);
    pre[4 * kT + row] = fma(0.5, g2, th + th);
  };
  // act'(z + bias) of this thread's 32 values of layer l
  auto act_slopes = [&](int l, const float* z, float* g) {
    const float2* b2 = (const float2*)(bias + l * kH + c0);
    if (a.act == 0) {
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const float2 v = silu_slope2(__fadd2_rn(make_float2(z[2 * q], z[2 * q + 1]), b2[q]));
        g[2 * q] = v.x; g[2 * q + 1] = v.y;
      }
    } else {
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const float2 v = __fadd2_rn(make_float2(z[2 * q], z[2 * q + 1]), b2[q]);
        g[2 * q] = v.x > 0.f ? 1.f : 0.f; g[2 * q + 1] = v.y > 0.f ? 1.f : 0.f;
      }
    }
  };
  // this tile's z_l of the stored variant, row-major [128 x 128]
  auto stored_z = [&](int64_t tile, int l) { return (float4*)(a.zst + (((size_t)tile * 3 + l) * kT + row) * kH + c0); };
  auto load_z = [&](int64_t tile, int l, float* z) {
    if (a.zst) {
      const float4* src = stored_z(tile, l);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float4 f = src[q];
        z[4 * q] = f.x; z[4 * q + 1] = f.y; z[4 * q + 2] = f.z; z[4 * q + 3] = f.w;
      }
    } else {
      // (z_1: its first 64 columns, later the others, in TM_H1LO)
      tc::ld32(lane_tm + (l == 0 ? TM_H1LO + (uint32_t)(c0 & 63) : (uint32_t)c0), z);
    }
  };

  const int64_t ntiles = (a.n + kT - 1) / kT;
  const bool rowthr = t < kT, xthr = cg == 1;
  uint32_t xw[8];   // warps 4..7: the coming tile's input row
  if (xthr) features((int64_t)blockIdx.x * kT + row, xw);
  bool alive = true, busy = false;   // busy: the last tile's final MMAs are not waited for yet
  for (int64_t tile = blockIdx.x; tile < ntiles && alive; tile += gridDim.x) {
    const int64_t p = tile * kT + row;
    const bool valid = rowthr && p < a.n;
    if (busy) wait_mma();   // dW1 of the last tile reads the input tile
    if (xthr) {
      tc::st_shared_v4(sb + S_X + tc::kmajor_offset(row, 0, kXin), xw[0], xw[1], xw[2], xw[3]);
      tc::st_shared_v4(sb + S_X + tc::kmajor_offset(row, 8, kXin), 0u, 0u, 0u, 0u);
      tc::st_shared_v4(sb + S_X + tc::kmajor_offset(row, 16, kXin), xw[4], xw[5], xw[6], xw[7]);
      tc::st_shared_v4(sb + S_X + tc::kmajor_offset(row, 24, kXin), 0u, 0u, 0u, 0u);
    }
    if (!(alive = to_mma())) break;
    // ---------------- forward, layers 1..3 (scratch accumulator at TMEM column 0)
    for (int l = 0; l < 3; ++l) {
      if (t == kIssuer) {
        tc::fence_after();
        if (l == 0) input_mma();
        else hidden_mma(l);
        tc::commit(mbar);
      }
      // beside the MMAs of layers 2 and 3, what the row stage needs of the pairs alone
      if (rowthr && l == 1) row_pairs(p, valid);
      if (rowthr && l == 2) row_groups();
      wait_mma();
      float v[32];
      tc::ld32(lane_tm + (uint32_t)c0, v);
      if (a.zst && a.mode != 0) {
        float4* dst = stored_z(tile, l);
#pragma unroll
        for (int q = 0; q < 8; ++q) dst[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
      }
      hidden_epilogue(l, v);
      if (!(alive = to_mma())) break;
    }
    if (!alive) break;
    // ---------------- output layer, into columns of its own: z3 stays in the
    // scratch accumulator for the backward
    if (t == kIssuer) {
      tc::fence_after();
      const uint32_t id = tc::idesc_bf16(kT, 16);
      for (int s = 0; s < 8; ++s)
        tc::mma_bf16(tm + TM_OUT, kdesc(sb + S_WK + 256u * s, kH), kdesc(sb + S_WOUT + 256u * s, kH), id, s > 0);
      for (int s = 0; s < 8; ++s)
        tc::mma_bf16(tm + TM_OUT, kdesc(sb + S_WKLO + 256u * s, kH), kdesc(sb + S_WOUT + 256u * s, kH), id, 1);
      tc::commit(mbar);
    }
    // ---------------- shell projection, pair update, moment matching, loss (rows)
    if (rowthr) {
      double u[3], d[3], upre[3], th[2] = {0.0, 0.0};
      for (int c = 0; c < 3; ++c) { d[c] = pre[c * kT + row]; upre[c] = mean[4 * (row / kGroup) + c]; }
      const double g = pre[3 * kT + row];
      th[0] = pre[4 * kT + row];
      double gi[3] = {0, 0, 0}, gj[3] = {0, 0, 0};   // targets (mode 2) or dL/dv_new (mode 1)
      if (valid && a.mode != 0) {
        const double* si = a.mode == 2 ? a.ti : a.gi;
        const double* sj = a.mode == 2 ? a.tj : a.gj;
        for (int c = 0; c < 3; ++c) { gi[c] = si[3 * p + c]; gj[c] = sj[3 * p + c]; }
      }
      wait_mma();
      float v[16];
      tc::ld16(lane_tm + TM_OUT, v);
      const double yd[3] = {f32_to_f64(v[0] + bias[3 * kH]), f32_to_f64(v[1] + bias[3 * kH + 1]),
                            f32_to_f64(v[2] + bias[3 * kH + 2])};
      const double ny2 = yd[0] * yd[0] + yd[1] * yd[1] + yd[2] * yd[2];
      // 1/|y| (0 for y = 0)
      const double iny = !valid ? 0.0 : plain64(ny2) ? rsqrt64(ny2) : ny2 > 0.0 ? 1.0 / sqrt(ny2) : 0.0;
      const double hg = 0.5 * g;
      double dpi[3], dpj[3];
      for (int c = 0; c < 3; ++c) {
        u[c] = yd[c] * iny;
        dpi[c] = fma(hg, u[c], d[c]);
        dpj[c] = fma(-hg, u[c], d[c]);
        th[1] = fma(dpi[c], dpi[c], fma(dpj[c], dpj[c], th[1]));
      }
      half_sums<2>(th);
      // alpha = sqrt(Theta_pre / Theta_post)
      const double thp = th[0] * th[1];
      const double alpha = plain64(thp) ? th[0] * rsqrt64(thp) : th[1] > 0.0 ? sqrt(th[0] / th[1]) : 1.0;
      double ni[3], nj[3];
      for (int c = 0; c < 3; ++c) { ni[c] = fma(alpha, dpi[c], upre[c]); nj[c] = fma(alpha, dpj[c], upre[c]); }
      if (a.mode == 0) {
        if (valid) for (int c = 0; c < 3; ++c) { a.oi[3 * p + c] = ni[c]; a.oj[3 * p + c] = nj[c]; }
      } else {
        double Gd[3] = {0, 0, 0};   // G_i - G_j
        double l2 = 0.0;
        if (valid) {
          if (a.mode == 2) {
            for (int c = 0; c < 3; ++c) {
              const double ri = ni[c] - gi[c], rj = nj[c] - gj[c];
              l2 = fma(ri, ri, fma(rj, rj, l2));
              Gd[c] = (ri - rj) * a.grad_scale;
            }
          } else {
            for (int c = 0; c < 3; ++c) Gd[c] = gi[c] - gj[c];
          }
        }
        lossw += l2;   // (summed over the lanes and scaled at the end)
        // Backward of moment matching, dL/dv = alpha (G - Gbar) - (alpha S /
        // Theta_post) (v - u_post), then of the centre-of-mass update (v_r'
        // enters as +1/2 for i, -1/2 for j) and of the projection, dy =
        // (g/|y|)(I - u u^T) dv_r'.  In dv_r' = (dL/dv_i - dL/dv_j)/2 the mean
        // Gbar cancels, and the last term, (v_i - v_j)/2 = g u / 2 along u,
        // is what (I - u u^T) removes: dv_r' = alpha (G_i - G_j)/2 gives the same dy.
        double dvr[3], ud = 0.0;
        for (int c = 0; c < 3; ++c) {
          dvr[c] = 0.5 * alpha * Gd[c];
          ud = fma(u[c], dvr[c], ud);
        }
        const double s = valid ? g * iny : 0.0;
        for (int c = 0; c < 3; ++c) {
          const float dy = valid ? to_f32(s * fma(-u[c], ud, dvr[c])) : 0.f;
          dz4f[4 * row + c] = dy;
        }
        uint32_t d0 = tc::pack_bf16x2(dz4f[4 * row], dz4f[4 * row + 1]);
        uint32_t d1 = tc::pack_bf16x2(dz4f[4 * row + 2], 0.f);
        tc::st_shared_v4(sb + S_DZ4 + tc::kmajor_offset(row, 0, 16), d0, d1, 0u, 0u);
        tc::st_shared_v4(sb + S_DZ4 + tc::kmajor_offset(row, 8, 16), 0u, 0u, 0u, 0u);
      }
    } else {
      phase ^= 1u;   // the output layer's MMAs, which only the row threads wait for
      if (xthr && tile + gridDim.x < ntiles) features((tile + gridDim.x) * kT + row, xw);
      // the coming tile's rows of the arrays that the row stage reads, into L2 (3 KB of each: 24 lines)
      if (cg == 2 && a.mode != 0 && lane < 24 && tile + gridDim.x < ntiles) {
        const double* arr[4] = {a.vi, a.vj, a.mode == 2 ? a.ti : a.gi, a.mode == 2 ? a.tj : a.gj};
        const double* q = arr[warp & 3] + 3 * (tile + gridDim.x) * kT + 16 * lane;
        if (q < arr[warp & 3] + 3 * a.n) asm volatile("prefetch.global.L2 [%0];" ::"l"(q));
      }
    }
    if (a.mode == 0) {
      tc::fence_before();
      __syncthreads();
      tc::fence_after();
      alive = *flag != 0;
      continue;
    }
    // ---------------- layers 3, 2, 1: z3 is still in the scratch accumulator
    // Every MMA that a layer needs is issued with the one before: z_2 beside
    // dW4, z_1 beside dh_2 and dh_1 (64 columns at a time, where h1's low terms
    // were), so a layer costs one barrier and one wait, and act' is formed while
    // the next MMAs run (z_2 and z_1 each behind a barrier and a wait of their own:
    // 1M pairs 1112 us, now 1072).
    float dh[32], g[32];
    load_z(tile, 2, g);
    act_slopes(2, g, dh);
    if (!(alive = to_mma())) break;
    // dW4^T += h3^T dz4 (hi and lo); z_2 from h1 (hi + lo)
    const uint32_t acc0 = tiles_done > 0 ? 1u : 0u;
    if (t == kIssuer) {
      tc::fence_after();
      const uint32_t id4 = tc::idesc_bf16(kT, 16) | (1u << 15) | (1u << 16);
      for (int s = 0; s < 8; ++s)
        tc::mma_bf16(tm + TM_DW4, mdesc(sb + S_WK + 2u * 2048u * s, kH), mdesc(sb + S_DZ4 + 2u * 256u * s, 16), id4,
                     (acc0 | (s > 0)) ? 1u : 0u);
      for (int s = 0; s < 8; ++s)
        tc::mma_bf16(tm + TM_DW4, mdesc(sb + S_WKLO + 2u * 2048u * s, kH), mdesc(sb + S_DZ4 + 2u * 256u * s, 16), id4, 1);
      if (!a.zst) hidden_mma(1);
      tc::commit(mbar);
    }
    // dz3 = dh3 act'(z3) with dh3 = dz4 W4 on CUDA cores (K = 3)
    {
      const float d0 = dz4f[4 * row], d1 = dz4f[4 * row + 1], d2 = dz4f[4 * row + 2];
#pragma unroll
      for (int q = 0; q < 32; ++q)
        dh[q] = (d0 * wo32[c0 + q] + d1 * wo32[kH + c0 + q] + d2 * wo32[2 * kH + c0 + q]) * dh[q];
      if (rowthr) {   // bias gradient of the output layer
        float s3[3] = {d0, d1, d2};
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
          for (int c = 0; c < 3; ++c) s3[c] += __shfl_xor_sync(0xffffffffu, s3[c], o);
        for (int c = 0; c < 3; ++c) dbo[c] += s3[c];
      }
    }
    for (int l = 2;; --l) {
      // dh holds dz_l: packed as the operand of dW_l and dh_{l-1}.  dz_3 and dz_1
      // go to S_WK, dz_2 to S_WKLO, whose last readers are done: h3's dW4 by
      // the first wait, dW_3 by the wait for dh_1, which was committed after it.
      const uint32_t dzb = l == 1 ? S_WKLO : S_WK;
      uint32_t pk[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) pk[q] = tc::pack_bf16x2(dh[2 * q], dh[2 * q + 1]);
      if (l == 2) {
        wait_mma();
        load_z(tile, 1, g);   // z_2, before dh_2 takes the accumulator
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
        tc::st_shared_v4(sb + dzb + tc::kmajor_offset(row, c0 + 8 * j, kH), pk[4 * j], pk[4 * j + 1], pk[4 * j + 2],
                         pk[4 * j + 3]);
      if (!(alive = to_mma())) break;
      // dh_{l-1} = dz W_l and a half of z_1 (not for l = 0), then dW_l += dz^T
      // h_{l-1}, which runs on while dh_{l-1} is read back
      if (t == kIssuer) {
        tc::fence_after();
        if (l > 0) {
          const uint32_t hprev = l == 2 ? S_H2 : S_H1;
          const uint32_t wl = l == 2 ? S_W3 : S_W2;
          const uint32_t dw = l == 2 ? TM_DW3 : TM_DW2;
          const uint32_t idh = tc::idesc_bf16(kT, kH) | (1u << 16);
          if (!a.zst) half_input_mma(2 - l);
          for (int s = 0; s < 8; ++s)
            tc::mma_bf16(tm, kdesc(sb + dzb + 256u * s, kH), mdesc(sb + wl + 2u * 2048u * s, kH), idh, s > 0);
          tc::commit(mbar);
          const uint32_t idw = tc::idesc_bf16(kH, kH) | (1u << 15) | (1u << 16);
          for (int s = 0; s < 8; ++s)
            tc::mma_bf16(tm + dw, mdesc(sb + dzb + 2u * 2048u * s, kH), mdesc(sb + hprev + 2u * 2048u * s, kH), idw,
                         (acc0 | (s > 0)) ? 1u : 0u);
        } else {
          const uint32_t idw = tc::idesc_bf16(kH, kXin) | (1u << 15) | (1u << 16);
          for (int s = 0; s < 8; ++s)
            tc::mma_bf16(tm + TM_DW1, mdesc(sb + dzb + 2u * 2048u * s, kH), mdesc(sb + S_X + 2u * 512u * s, kXin), idw,
                         (acc0 | (s > 0)) ? 1u : 0u);
          tc::commit(mbar);
        }
      }
      dbacc[l] += warp_colsum32(dh);   // (the column sums; dh is not used after)
      if (l == 0) break;
      // act'(z_{l-1}): formed here, beside the MMAs, but for the columns of z_1
      // that come with dh_1
      if (l == 2 || cg < 2) act_slopes(l - 1, g, g);
      wait_mma();
      tc::ld32(lane_tm + (uint32_t)c0, dh);
      if (l == 1 && cg >= 2) {
        load_z(tile, 0, g);
        act_slopes(0, g, g);
      }
#pragma unroll
      for (int q = 0; q < 32; ++q) dh[q] *= g[q];
      if (l == 2 && cg < 2) load_z(tile, 0, g);
    }
    if (!alive) break;
    busy = true;
    ++tiles_done;
  }
  if (busy && alive) wait_mma();
  // the tiles' loop was left early: MMAs that not every thread has waited for (a
  // layer's dW runs on beside the next one) end (bounded) before TMEM is released
  if (!alive && t == kIssuer) {
    tc::commit(drain);
    tc::mbar_wait(drain, 0, a.status, kBarrierLimitNs);
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  alive = alive && *flag != 0;
  // ---------------- flush this CTA's partial gradients
  if (alive && a.mode != 0) {
    float* P = a.partial + (size_t)blockIdx.x * kPartial;
    if (tiles_done == 0) {
      for (int q = t; q < kPartial; q += kNT) P[q] = 0.f;
    } else {
      float v[32];
      // k values of this thread, its 4 q-th to (4 q + 3)-th `stride` floats after the ones
      // before (16 bytes at a time where the workspace allows it)
      const bool wide = ((uintptr_t)a.partial & 15u) == 0;
      auto put = [&](float* dst, int k, int stride) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (4 * q >= k) break;
          float* d = dst + q * stride;
          if (wide) {
            *(float4*)d = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) d[e] = v[4 * q + e];
          }
        }
      };
      // dW2, dW3: [128 out x 128 in]
      tc::ld32(lane_tm + TM_DW2 + (uint32_t)c0, v);
      put(P + kH * kXin + wpos32(row, c0), 32, 4 * kNT);
      tc::ld32(lane_tm + TM_DW3 + (uint32_t)c0, v);
      put(P + kH * kXin + kH * kH + wpos32(row, c0), 32, 4 * kNT);
      if (cg == 0) {
        tc::ld32(lane_tm + TM_DW1, v);  // [128 out x 32 (hi | lo)]
        put(P + wpos(row, 0, kH), 32, 4 * kH);
      } else if (cg == 1) {
        tc::ld16(lane_tm + TM_DW4, v);  // [128 in x 16 out]
        put(P + kH * kXin + 2 * kH * kH + wpos(row, 0, kH), 16, 4 * kH);
      }
      const int g = warp & 3;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) lossw += __shfl_xor_sync(0xffffffffu, lossw, o);
      for (int l = 0; l < 3; ++l) P[kPDB + g * 400 + l * kH + c0 + lane] = dbacc[l];
      if (cg == 0 && lane == 0) {
        for (int c = 0; c < 3; ++c) P[kPDB + g * 400 + 3 * kH + c] = dbo[c];
        P[kPLOSS + g] = (float)(lossw * a.loss_scale);
      }
    }
  } else if (a.mode != 0 && t == 0 && !alive) {
    set_status(a.status, DSMC_ERR_TIMEOUT);
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tm, 512);
}

// Adam (Kingma & Ba 2015, Algorithm 1) on FP32 parameters [weights, biases];
// optionally writes the bf16 weights and FP32 biases the collide kernel takes.
struct AdamArgs {
  float *master, *m, *v;    // master null: no update
  uint16_t* w_bf16;
  float* bias;
  int n_w;
  float lr, b1, b2, eps, c1, c2;
};
__device__ __forceinline__ void adam_one(const AdamArgs& A, int q, float g) {
  const float mq = A.b1 * A.m[q] + (1.f - A.b1) * g;
  const float vq = A.b2 * A.v[q] + (1.f - A.b2) * g * g;
  A.m[q] = mq;
  A.v[q] = vq;
  const float th = A.master[q] - A.lr * (mq * A.c1) / (sqrtf(vq * A.c2) + A.eps);
  A.master[q] = th;
  if (q < A.n_w) {
    if (A.w_bf16) A.w_bf16[q] = to_bf16(th);
  } else if (A.bias) {
    A.bias[q - A.n_w] = th;
  }
}

// s plus n values `stride` floats apart, added in order; sixteen loads are
// in flight at a time (the sum is a chain of FP32 additions, the loads are not:
// one at a time, the 152 partials cost as many round trips to L2).
__device__ __forceinline__ float ordered_sum(float s, const float* __restrict__ p, int n, size_t stride) {
  constexpr int kFly = 16;
  float v[kFly];
  for (int b = 0; b < n; b += kFly) {
#pragma unroll
    for (int q = 0; q < kFly; ++q) v[q] = b + q < n ? p[(size_t)(b + q) * stride] : 0.f;
#pragma unroll
    for (int q = 0; q < kFly; ++q)
      if (b + q < n) s += v[q];
  }
  return s;
}

// Sum the per-CTA partials in CTA order; write gradients in the weight layout
// (row-major per layer, then biases) and the loss.  One output per thread, a
// warp for the loss; 16,384 threads with one load in flight each took 81 us
// for 34,563 outputs of 128 CTAs.
constexpr int kReduceThreads = 128;
__global__ void __launch_bounds__(kReduceThreads) k_train_reduce(const float* __restrict__ partial, int nblk,
                                                                 float* __restrict__ grad, double* loss, AdamArgs A) {
  dep_wait();
  const int nw = kNW;
  const int nb = kNB;
  if (blockIdx.x == 0) {   // the loss: lane l the values l, l + 32, ... of [CTA][lane group], then a tree
    if (threadIdx.x < 32) {
      double l = 0.0;
      for (int q = threadIdx.x; q < 4 * nblk; q += 32) l += partial[(size_t)(q >> 2) * kPartial + kPLOSS + (q & 3)];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
      if (threadIdx.x == 0 && loss) *loss = l;
    }
    return;
  }
  // thread q: the q-th value of the partials (neighbouring threads read
  // neighbouring words), out: where its sum goes in the weight layout
  const int q = (blockIdx.x - 1) * kReduceThreads + threadIdx.x;
  if (q >= nw + nb) return;
  int out = q;
  float s = 0.f;
  if (q < kH * 8) {                          // W1[o][k] = hi column k + lo column 16 + k
    const int o = (q >> 2) & (kH - 1), k = (q >> 9) * 4 + (q & 3);
    out = o * 8 + k;
    const float* p = partial + wpos(o, k, kH);
    constexpr int lo = wpos(0, 16, kH);
    for (int b = 0; b < nblk; b += 8) {
      float v[16];
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        v[2 * r] = b + r < nblk ? p[(size_t)(b + r) * kPartial] : 0.f;
        v[2 * r + 1] = b + r < nblk ? p[(size_t)(b + r) * kPartial + lo] : 0.f;
      }
#pragma unroll
      for (int r = 0; r < 8; ++r)
        if (b + r < nblk) s += v[2 * r] + v[2 * r + 1];
    }
  } else if (q < kH * 8 + 2 * kH * kH) {     // W2, W3
    const int j = q - kH * 8, m = j / (kH * kH), w = j % (kH * kH);
    const int t = (w >> 2) & (kNT - 1), o = t & (kH - 1), k = (t / kH) * 32 + (w / (4 * kNT)) * 4 + (w & 3);
    out = kH * 8 + m * kH * kH + o * kH + k;
    s = ordered_sum(s, partial + kH * kXin + j, nblk, kPartial);
  } else if (q < nw) {                       // W4[o][k] = dW4^T[k][o]
    const int r = q - kH * 8 - 2 * kH * kH, o = r / kH, k = r % kH;
    s = ordered_sum(s, partial + kH * kXin + 2 * kH * kH + wpos(k, o, kH), nblk, kPartial);
  } else {                                   // biases: lane groups 0..3 of every CTA, in order
    const float* p = partial + kPDB + (q - nw);
    for (int b = 0; b < nblk; b += 4) {
      float v[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) v[r] = b + r / 4 < nblk ? p[(size_t)(b + r / 4) * kPartial + (r & 3) * 400] : 0.f;
#pragma unroll
      for (int r = 0; r < 16; ++r)
        if (b + r / 4 < nblk) s += v[r];
    }
  }
  grad[out] = s;
  if (A.master) adam_one(A, out, s);   // (a training step: a launch less than Adam by itself, 2^14 pairs 48 us, now 45)
}

__global__ void k_adam(int n, const float* __restrict__ grad, AdamArgs A) {
  dep_wait();
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) adam_one(A, q, grad[q]);
}

size_t train_act_bytes(int64_t n) { return sizeof(float) * 3 * (size_t)kT * kH * (size_t)((n + kT - 1) / kT); }

size_t train_ws(int sms) { return align256(sizeof(float) * (size_t)kPartial * (size_t)(sms > 0 ? sms : 1)); }

static AdamArgs adam_args(const AdamStep& a) {
  AdamArgs A;
  A.master = a.master; A.m = a.m; A.v = a.v; A.w_bf16 = a.w_bf16; A.bias = a.bias; A.n_w = a.n_w;
  A.lr = a.lr; A.b1 = (float)a.b1; A.b2 = (float)a.b2; A.eps = a.eps;
  A.c1 = (float)(1.0 / (1.0 - pow(a.b1, (double)a.step)));
  A.c2 = (float)(1.0 / (1.0 - pow(a.b2, (double)a.step)));
  return A;
}

int launch_train(Ctx* c, const dsmc_mlp_t& mlp, int mode, uint64_t seed, uint64_t t, int64_t n,
                 const float* theta, const double* vi, const double* vj, const double* T,
                 const double* ti, const double* tj, const double* gi, const double* gj, double* oi, double* oj,
                 float* grad, double* loss, void* ws, size_t ws_bytes, cudaStream_t s, float* act, const AdamStep* adam) {
  const int sms = sm_count(c);
  if (mode != 0 && ws_bytes < train_ws(sms)) return record(c, DSMC_ERR_ARG, "train: workspace too small");
  if (cudaFuncSetAttribute((const void*)k_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S_TOTAL) !=
      cudaSuccess)
    return record(c, DSMC_ERR_CUDA, "train: shared-memory attribute");
  TrainArgs a;
  a.mode = mode; a.act = mlp.act; a.n = n; a.seed = seed; a.t = t;
  a.sigma_v_inv = 1.0 / mlp.sigma_v; a.T_ref_inv = 1.0 / mlp.T_ref; a.eps = mlp.eps;
  a.grad_scale = n > 0 ? a.sigma_v_inv * a.sigma_v_inv / (double)n : 0.0;
  a.loss_scale = 0.5 * a.grad_scale;
  a.theta = theta; a.vi = vi; a.vj = vj; a.T = T; a.ti = ti; a.tj = tj; a.gi = gi; a.gj = gj;
  a.oi = oi; a.oj = oj; a.zst = act; a.partial = (float*)ws; a.status = status_ptr(c);
  const int64_t tiles = (n + kT - 1) / kT;
  const int blocks = (int)(tiles < sms ? (tiles > 0 ? tiles : 1) : sms);
  launch_dep(k_train, blocks, kNT, S_TOTAL, s, a);
  count_launches(c, 1);
  if (mode != 0) {
    const int outs = kNW + kNB;
    launch_dep(k_train_reduce, 1 + (outs + kReduceThreads - 1) / kReduceThreads, kReduceThreads, 0, s, 
        (const float*)ws, blocks, grad, loss, adam ? adam_args(*adam) : AdamArgs{});
    count_launches(c, 1);
  }
  return cudaGetLastError() == cudaSuccess ? 0 : DSMC_ERR_CUDA;
}

int launch_adam(Ctx* c, int n, const float* grad, const AdamStep& adam, cudaStream_t s) {
  launch_dep(k_adam, 64, 256, 0, s, n, grad, adam_args(adam));
  count_launches(c, 1);
  return cudaGetLastError() == cudaSuccess ? 0 : DSMC_ERR_CUDA;
}

}  // namespace dsmc

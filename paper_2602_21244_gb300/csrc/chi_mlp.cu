// chi-MLP surrogate (Sec. 3.4, Fig. nn_architecture; reading R9) on the
// tcgen05 tensor cores: inputs [ln(E_r)*, b/b_max] -> 512, 512, 512, 256, 128
// (SiLU) -> 1 (Softplus); the Softplus output y approximates ln(1 + chi),
// so chi = e^y - 1.  It synthesises the look-up table of Sec. 3.4.4.
//
// One persistent CTA per SM works on 128-row tiles, a layer in passes of 128
// output columns: the MMAs of a pass (M = N = 128, FP32 accumulator in one of
// two 128-column halves of TMEM) run while the epilogue of the pass before
// reads the other half back, adds the bias and applies SiLU.  A layer's input
// is its A operand in the other 256 TMEM columns (two bf16 per column); the
// layer reads it until its last pass, so the earlier passes' outputs wait in the
// epilogue's registers and are stored once the last pass's MMAs are done, and
// the next layer starts on those while the last pass is still in the epilogue.
// (With every second layer's input in shared memory the MMAs read 8 KB of
// operands each from there and took twice as long: 652 against 452 us for the
// MMAs of the 512 x 512 table.)  The weights (1.39 MB, the same for every tile)
// stream from L2 all the time, 32 KB bulk copies (128 rows x 128 K columns,
// packed once in the operand layout and in the order of use by
// dsmc_chi_mlp_pack) through a ring of six buffers.  Roles: 16 epilogue warps
// (warp w: TMEM lanes 32 (w % 4), a quarter of the pass's columns), one lane
// issuing the MMAs, one the copies; the hand-offs are mbarriers.
//
// Measured on the 512 x 512 table (361 GFLOP): 1136 us when a layer's epilogue
// ran after all of its MMAs (tensor pipe and copies stood still meanwhile), 721
// us with the passes overlapped and operands alternating between tensor and
// shared memory, 522 us with all of them in tensor memory, 361 us (1.0
// PFLOP/s, 53 % of the measured bf16 peak) with 32 KB chunks and a shorter issue
// loop.  What bounds it now: the MMA lane's waits and issue (about 100 us over
// the pipe's 190 us), then the SiLU (320 us without it); the copies do not (the
// same time with three buffers).
//
// Precision: the input enters as two bf16 terms (about 16 bits); hidden
// activations 1-4 are stored as single bf16 terms (a second term would not
// fit 128 rows x 512 columns twice in shared memory); accumulation in FP32.
#include <vector>

#include "internal.cuh"
#include "tc.cuh"

namespace dsmc {

namespace {

constexpr int kRows = 128;
constexpr int kEpiWarps = 16;                  // epilogue warps: 4 TMEM lane quadrants x 4 column groups
constexpr int kMmaWarp = kEpiWarps, kCopyWarp = kEpiWarps + 1;
constexpr int kThr = (kEpiWarps + 2) * 32;
constexpr int kNbuf = 6;
constexpr int kMmaLayers = 5;                       // hidden layers 1..5 on the tensor cores
constexpr int kPassN = 128;                         // output columns of a pass
constexpr int kChunkK = 128;                        // K columns of a weight chunk (layer 1: all 16, every pass)
// widths 2, 512, 512, 512, 256, 128, 1; K and N of the MMA layers (input padded to K = 16)
__host__ __device__ constexpr int dims_of(int i) {
  return i == 0 ? 2 : i <= 3 ? 512 : i == 4 ? 256 : i == 5 ? 128 : 1;
}
__host__ __device__ constexpr int k_of(int l) { return l == 0 ? 16 : l <= 3 ? 512 : 256; }
__host__ __device__ constexpr int n_of(int l) { return l <= 2 ? 512 : l == 3 ? 256 : 128; }
__host__ __device__ constexpr int passes_of(int l) { return n_of(l) / kPassN; }
constexpr int kBiasTotal = 512 + 512 + 512 + 256 + 128 + 1;

// byte offset of layer l's first chunk in the packed weights
__host__ __device__ constexpr uint32_t layer_off(int l) {
  uint32_t o = 0;
  for (int q = 0; q < l; ++q) o += (uint32_t)(k_of(q) * n_of(q) * 2);
  return o;
}
constexpr uint32_t kChunkBytes = kPassN * kChunkK * 2;
constexpr uint32_t kFirstBytes = layer_off(1);                // layer 1 is one shorter chunk
static_assert(kFirstBytes <= kChunkBytes, "layer 1 fits a buffer");
constexpr uint32_t kWoutOff = layer_off(kMmaLayers);          // FP32 output weights [128]
constexpr uint32_t kPackedBytes = kWoutOff + 128 * 4;
constexpr int kPerTile = 1 + (int)((kWoutOff - kFirstBytes) / kChunkBytes);   // 43 chunks

// shared memory layout (bytes)
constexpr uint32_t kBufOff = 0;                                  // kNbuf x 32 KB
constexpr uint32_t kXOff = kBufOff + kNbuf * kChunkBytes;        // input tile [128 x 16]
constexpr uint32_t kBiasOff = kXOff + kRows * 16 * 2;
constexpr uint32_t kWoOff = kBiasOff + ((kBiasTotal * 4 + 15) / 16) * 16;
constexpr uint32_t kYpOff = kWoOff + 128 * 4;                    // 4 column groups x 128 rows
constexpr uint32_t kBarOff = kYpOff + 4 * kRows * 4;             // the mbarriers
constexpr uint32_t kTptrOff = kBarOff + (2 * kNbuf + 9) * 8;
constexpr uint32_t kFlagOff = kTptrOff + 8;
constexpr uint32_t kSmemBytes = kFlagOff + 16;
// TMEM: accumulators of even and odd passes in columns 0..127 and 128..255, the A operand in 256..511
constexpr uint32_t kTmemA = 256;

struct ChiArgs {
  const char* packed;
  const float* bias;
  int64_t n;
  const float* x;      // [n][2], or null (table mode)
  float* y;            // Softplus outputs, or null
  float* chi;          // e^y - 1, or null
  int32_t nb, nE;      // table mode: row g is node (g / nb, g % nb)
  int* status;
};

__device__ __forceinline__ float softplus_f(float z) { return fmaxf(z, 0.f) + log1pf(__expf(-fabsf(z))); }

}  // namespace

// ------------------------------------------------------------------ packing
// Chunks in the order of use, operands in the K-major core-matrix layout.
// Layer 1 (K = 2 in the network): one 16 KB chunk of four 128-row passes of
// 16 K columns, holding W1[n][0], W1[n][1] in columns 0, 1 (the inputs' bf16
// terms) and again in 2, 3 (their remainders), zeros elsewhere.  The other
// layers: per pass of 128 rows, 32 KB chunks of 128 K columns.
__global__ void k_chi_mlp_pack(const uint16_t* __restrict__ w, char* __restrict__ packed) {
  const int64_t total = (int64_t)layer_off(kMmaLayers) / 2;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total + 128;
       e += (int64_t)gridDim.x * blockDim.x) {
    if (e >= total) {   // output weights W6[0][k] as FP32
      const int k = (int)(e - total);
      uint32_t src_off = 0;
      for (int q = 0; q < 5; ++q) src_off += (uint32_t)(dims_of(q) * dims_of(q + 1));
      ((float*)(packed + kWoutOff))[k] = __uint_as_float((uint32_t)w[src_off + k] << 16);
      continue;
    }
    int l = 0;
    int64_t r = e;
    while (r >= (int64_t)k_of(l) * n_of(l)) { r -= (int64_t)k_of(l) * n_of(l); ++l; }
    // element e is the e-th of the packed array: its pass, chunk and place in the operand tile
    const int kc = l == 0 ? 16 : kChunkK;                      // K columns of the tile
    const int tile = (int)(r / (kPassN * kc)), rem = (int)(r % (kPassN * kc));
    const int per_pass = k_of(l) / kc, pass = tile / per_pass, k0 = (tile % per_pass) * kc;
    // invert kmajor_offset(n, k, kc) / 2: 8 rows x 8 columns are 64 elements, kc / 8 of them side by side
    const int grp = rem / (8 * kc), in_grp = rem % (8 * kc), within = in_grp % 64;
    const int n = pass * kPassN + grp * 8 + within / 8, k = k0 + (in_grp / 64) * 8 + within % 8;
    uint32_t src_off = 0;
    for (int q = 0; q < l; ++q) src_off += (uint32_t)(dims_of(q) * dims_of(q + 1));
    const int din = dims_of(l);
    uint16_t v = 0;
    if (l == 0) {
      if (k < 4) v = w[src_off + n * din + (k & 1)];
    } else {
      v = w[src_off + n * din + k];
    }
    ((uint16_t*)packed)[e] = v;
  }
}

// ------------------------------------------------------------------ forward
// Bounded wait of one role on a barrier: false after the limit (recorded), or
// once another role has failed.
__device__ __forceinline__ bool role_wait(uint64_t* bar, uint32_t parity, volatile int* fail, int* status) {
  if (tc::mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  while (!tc::mbar_try_wait_hint(bar, parity, 20000u)) {
    if (*fail) return false;
    if (globaltimer_ns() - t0 > kBarrierLimitNs) {
      set_status(status, DSMC_ERR_TIMEOUT);
      *fail = 1;
      return false;
    }
  }
  return true;
}
__device__ __forceinline__ void bar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}

__global__ void __launch_bounds__(kThr, 1) k_chi_mlp(ChiArgs a) {
  extern __shared__ __align__(1024) char smem[];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  uint64_t* full = (uint64_t*)(smem + kBarOff);   // chunk landed: the copy's arrival and bytes
  uint64_t* empty = full + kNbuf;                 // the MMAs that read the buffer are done
  uint64_t* dfull = empty + kNbuf;                // a pass's accumulators are complete (even, odd passes)
  uint64_t* dfree = dfull + 2;                    // its epilogue has read them
  uint64_t* aearly = dfree + 2;                   // a layer's outputs are stored, but for the last pass's
  uint64_t* alast = aearly + 1;                   // all of them
  uint64_t* xfull = alast + 1;                    // the tile's input rows are in shared memory
  uint64_t* yfull = xfull + 1;                    // the column groups' partial outputs are
  uint64_t* drain = yfull + 1;                    // at the end: the MMAs in flight are done
  volatile int* fail = (volatile int*)(smem + kFlagOff);
  const uint32_t sbase = tc::smem_u32(smem);
  float* bias = (float*)(smem + kBiasOff);
  float* wo = (float*)(smem + kWoOff);
  float* yp = (float*)(smem + kYpOff);
  for (int i = t; i < kBiasTotal; i += kThr) bias[i] = a.bias[i];
  for (int i = t; i < 128; i += kThr) wo[i] = ((const float*)(a.packed + kWoutOff))[i];
  if (w == 0) {
    tc::tmem_alloc((uint32_t*)(smem + kTptrOff), 512);
    tc::tmem_relinquish();
  }
  if (t == 0) {
    for (int b = 0; b < kNbuf; ++b) { tc::mbar_init(full + b, 1); tc::mbar_init(empty + b, 1); }
    for (int b = 0; b < 2; ++b) { tc::mbar_init(dfull + b, 1); tc::mbar_init(dfree + b, kEpiWarps); }
    tc::mbar_init(aearly, kEpiWarps);
    tc::mbar_init(alast, kEpiWarps);
    tc::mbar_init(xfull, kRows);
    tc::mbar_init(yfull, kEpiWarps);
    tc::mbar_init(drain, 1);
    tc::mbar_fence_init();
    *fail = 0;
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = *(volatile uint32_t*)(smem + kTptrOff);

  // Tiles blockIdx.x, blockIdx.x + gridDim.x, ...: every CTA streams the
  // whole weight sequence once per tile into its own buffers.
  const int64_t n_tiles = (a.n + kRows - 1) / kRows;
  const int my_its = (int64_t)blockIdx.x < n_tiles ? (int)((n_tiles - 1 - blockIdx.x) / gridDim.x + 1) : 0;

  if (w == kCopyWarp) {
    // ------------------------------------------------ weight copies
    if (lane == 0) {
      const int total = my_its * kPerTile;   // (below 2^31: n < 2^32 rows over at least 100 CTAs)
      int m = 0, b = 0, at = 0;              // chunk, its buffer, its place in the sequence
      uint32_t ph = 1;                       // parity of the buffer's last release
      for (; m < total; ++m) {
        if (m >= kNbuf && !role_wait(empty + b, ph, fail, a.status)) break;
        const uint32_t bytes = at ? kChunkBytes : kFirstBytes;
        tc::mbar_arrive_expect_tx(full + b, bytes);
        tc::bulk_g2s(sbase + kBufOff + (uint32_t)b * kChunkBytes,
                     a.packed + (at ? kFirstBytes + (size_t)(at - 1) * kChunkBytes : 0), bytes, full + b);
        if (++at == kPerTile) at = 0;
        if (++b == kNbuf) { b = 0; ph ^= 1u; }
      }
      // the copies in flight land (bounded) before the shared memory is released,
      // those of the last chunks too: another role may fail after they are issued
      for (int q = m > kNbuf ? m - kNbuf : 0; q < m; ++q)
        tc::mbar_wait(full + q % kNbuf, (uint32_t)(q / kNbuf) & 1u, a.status, kBarrierLimitNs);
    }
    __syncwarp();
  } else if (w == kMmaWarp) {
    // ------------------------------------------------ MMAs
    if (lane == 0) {
      const uint32_t idesc = tc::idesc_bf16(kRows, kPassN);
      // counters by increments and descriptors by additions: this one
      // thread's instructions paced the MMAs (64-bit divisions by the ring's
      // length and descriptors built from scratch cost 270 ns per 16 KB chunk)
      int b = 0;                 // ring buffer of the next chunk
      uint32_t bph = 0;          // its parity
      uint32_t g = 0;            // passes issued
      const uint64_t dx = tc::sdesc(sbase + kXOff, 128, 256);
      const uint64_t d16 = tc::sdesc(sbase + kBufOff, 128, 256), dk = tc::sdesc(sbase + kBufOff, 128, kChunkK * 16);
      constexpr uint32_t kBufStep = kChunkBytes >> 4;   // descriptor units
      bool ok = true;
      auto wait_chunk = [&]() { return role_wait(full + b, bph, fail, a.status); };
      auto next_chunk = [&]() {
        tc::commit(empty + b);
        if (++b == kNbuf) { b = 0; bph ^= 1u; }
      };
      for (int it = 0; it < my_its && ok; ++it) {
        for (int l = 0; l < kMmaLayers && ok; ++l) {
          const int nk = k_of(l) / kChunkK, np = passes_of(l);
          const uint32_t stored = (uint32_t)(it * (kMmaLayers - 1) + l - 1) & 1u;   // layers' outputs so far
          for (int p = 0; p < np && ok; ++p, ++g) {
            // the accumulator half was last read by the epilogue two passes ago
            if (g >= 2) ok = role_wait(dfree + (g & 1), ((g - 2) >> 1) & 1u, fail, a.status);
            const uint32_t d = tmem + (g & 1) * kPassN;
            if (l == 0) {
              if (ok && p == 0) ok = role_wait(xfull, (uint32_t)it & 1u, fail, a.status) && wait_chunk();
              if (!ok) break;
              tc::fence_after();
              tc::mma_bf16(d, dx, d16 + (uint32_t)b * kBufStep + (uint32_t)p * (kPassN * 16 * 2 >> 4), idesc, 0);
              if (p == np - 1) next_chunk();
            } else {
              for (int c = 0; c < nk; ++c) {
                if (p == 0) {
                  // the layer's last 128 input columns come from the last pass
                  if (c == 0) ok = role_wait(aearly, stored, fail, a.status);
                  if (ok && c == nk - 1) ok = role_wait(alast, stored, fail, a.status);
                }
                if (!ok || !(ok = wait_chunk())) break;
                tc::fence_after();
                const uint64_t db = dk + (uint32_t)b * kBufStep;
                const uint32_t ta = tmem + kTmemA + (uint32_t)c * (kChunkK / 2);
#pragma unroll
                for (int s = 0; s < kChunkK / 16; ++s)
                  tc::mma_bf16_ta(d, ta + 8u * s, db + 16u * s, idesc, c > 0 || s > 0);
                next_chunk();
              }
            }
            if (ok) tc::commit(dfull + (g & 1));
          }
        }
      }
      // MMAs in flight end (bounded) before TMEM and shared memory are released,
      // those of the last pass too: its epilogue may fail after they are issued
      tc::commit(drain);
      tc::mbar_wait(drain, 0, a.status, kBarrierLimitNs);
    }
    __syncwarp();
  } else {
    // ------------------------------------------------ input rows and epilogues
    const int q = w & 3, cg = w >> 2;           // TMEM lane quadrant, column group
    const int row = q * 32 + lane;
    const uint32_t lane_tm = tmem + ((uint32_t)(q * 32) << 16);
    // input row of a tile (warps 0..3): [x0 hi, x1 hi, x0 lo, x1 lo, 0 ...] as a K = 16 tile
    auto input_row = [&](int64_t tile) {
      const int64_t gr = tile * kRows + row;
      float x0 = 0.f, x1 = 0.f;
      if (gr < a.n) {
        if (a.x) { x0 = a.x[2 * gr]; x1 = a.x[2 * gr + 1]; }
        else {
          x0 = (float)(gr / a.nb) / (float)(a.nE - 1);
          x1 = (float)(gr % a.nb) / (float)(a.nb - 1);
        }
      }
      const uint32_t hi = tc::pack_bf16x2(x0, x1);
      const float h0 = __uint_as_float(hi << 16), h1 = __uint_as_float(hi & 0xFFFF0000u);
      const uint32_t lo = tc::pack_bf16x2(x0 - h0, x1 - h1);
      tc::st_shared_v4(sbase + kXOff + tc::kmajor_offset(row, 0, 16), hi, lo, 0u, 0u);
      tc::st_shared_v4(sbase + kXOff + tc::kmajor_offset(row, 8, 16), 0u, 0u, 0u, 0u);
      tc::fence_async_smem();
      bar_arrive(xfull);
    };
    if (cg == 0 && my_its > 0) input_row(blockIdx.x);
    uint32_t g = 0;
    auto arrive = [&](uint64_t* bar) {
      tc::fence_before();
      __syncwarp();
      if (lane == 0) bar_arrive(bar);
    };
    // wait for pass g's accumulators
    auto wait_pass = [&]() {
      const bool ok = __all_sync(0xffffffffu, role_wait(dfull + (g & 1), (g >> 1) & 1u, fail, a.status));
      tc::fence_after();
      return ok;
    };
    // this warp's 32 columns of pass g (layer columns n0 ..), 16 at a time:
    // bias, SiLU, then put(h, z) for each half; the accumulators are free after the
    // second read
    auto activate = [&](const float* b, auto&& put) {
      const uint32_t at = lane_tm + (g & 1) * kPassN + 32u * (uint32_t)cg;
      uint32_t ra[16], rb[16];
      tc::ld16_async(at, ra);
      tc::wait_ld16(ra);
      tc::ld16_async(at + 16, rb);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t* r = h ? rb : ra;
        const float2* b2 = (const float2*)(b + 16 * h);
        float2 z[8];
        if (h) {
          tc::wait_ld16(rb);
          arrive(dfree + (g & 1));
        }
#pragma unroll
        for (int k = 0; k < 8; ++k)
          z[k] = __fadd2_rn(make_float2(__uint_as_float(r[2 * k]), __uint_as_float(r[2 * k + 1])), b2[k]);
#pragma unroll
        for (int k = 0; k < 8; k += 2) tc::silu4x2(z[k], z[k + 1]);
        put(h, z);
      }
    };
    // columns n0 .. n0 + 31 of a layer's output into the A operand
    auto store = [&](int n0, const uint32_t* pk) { tc::st16_async(lane_tm + kTmemA + (uint32_t)(n0 >> 1), pk); };
    bool ok = true;
    for (int it = 0; it < my_its && ok; ++it) {
      const int64_t tile = (int64_t)blockIdx.x + (int64_t)it * gridDim.x;
      float2 yq = make_float2(0.f, 0.f);
      uint32_t boff = 0;
      for (int l = 0; l < kMmaLayers - 1 && ok; ++l) {
        const int np = passes_of(l);
        // the layer's own MMAs read the A operand until its last pass: the
        // earlier passes' outputs are held in registers till then (the first
        // layer reads the input tile instead, and stores as it goes)
        uint32_t held[4][16];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          if (p >= np || !ok) continue;
          ok = wait_pass();
          if (!ok) continue;
          const bool last = p == np - 1;
          if (l > 0 && last) {
#pragma unroll
            for (int q2 = 0; q2 < 3; ++q2)
              if (q2 < np - 1) store(q2 * kPassN + 32 * cg, held[q2]);
            tc::wait_st();
            arrive(aearly);
          }
          // the first layer's MMAs are done with the input tile: the next one's rows
          if (l == 0 && last && cg == 0 && it + 1 < my_its) input_row(tile + gridDim.x);
          const int n0 = p * kPassN + 32 * cg;
          activate(bias + boff + n0, [&](int h, const float2* z) {
#pragma unroll
            for (int k = 0; k < 8; ++k) held[p][8 * h + k] = tc::pack_bf16x2(z[k].x, z[k].y);
          });
          ++g;
          if (l == 0 || last) {
            store(n0, held[p]);
            tc::wait_st();
            if (last) arrive(alast);
            else if (p == np - 2) arrive(aearly);   // (first layer)
          }
        }
        boff += (uint32_t)n_of(l);
      }
      if (ok && (ok = wait_pass())) {   // the last hidden layer, into the output's dot products
        const int n0 = 32 * cg;
        activate(bias + boff + n0, [&](int h, const float2* z) {
          const float2* w2 = (const float2*)(wo + n0 + 16 * h);
#pragma unroll
          for (int k = 0; k < 8; ++k) yq = __ffma2_rn(z[k], w2[k], yq);
        });
        ++g;
        boff += (uint32_t)n_of(kMmaLayers - 1);
      }
      if (!ok) break;
      // output layer: the four column groups' partial dot products, bias, Softplus
      yp[cg * kRows + row] = yq.x + yq.y;
      __syncwarp();
      if (lane == 0) bar_arrive(yfull);
      if (cg == 0) {
        if (!__all_sync(0xffffffffu, role_wait(yfull, (uint32_t)it & 1u, fail, a.status))) break;
        const int64_t gr = tile * kRows + row;
        if (gr < a.n) {
          const float z = yp[row] + yp[kRows + row] + yp[2 * kRows + row] + yp[3 * kRows + row] + bias[boff];
          const float y = softplus_f(z);
          if (a.y) a.y[gr] = y;
          if (a.chi) a.chi[gr] = expm1f(y);
        }
      }
      // (yp is written again only after every warp has been through the next
      // tile's earlier passes)
    }
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (w == 0) tc::tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------ host side
size_t chi_mlp_packed_size() { return kPackedBytes; }

int launch_chi_mlp_pack(Ctx* c, const uint16_t* w_bits, void* packed, cudaStream_t s) {
  k_chi_mlp_pack<<<sm_count(c) * 4, 256, 0, s>>>(w_bits, (char*)packed);
  count_launches(c, 1);
  return cudaGetLastError() == cudaSuccess ? 0 : DSMC_ERR_CUDA;
}

static int launch_chi_mlp(Ctx* c, const ChiArgs& a, cudaStream_t s) {
  if (a.n == 0) return 0;
  if (cudaFuncSetAttribute((const void*)k_chi_mlp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes) !=
      cudaSuccess)
    return record(c, DSMC_ERR_CUDA, "chi_mlp: shared memory attribute");
  // one wave of persistent CTAs, one per SM (206 KB of shared memory each)
  const int64_t tiles = (a.n + kRows - 1) / kRows;
  const int64_t grid = tiles < sm_count(c) ? tiles : sm_count(c);
  k_chi_mlp<<<(unsigned)grid, kThr, kSmemBytes, s>>>(a);
  count_launches(c, 1);
  return cudaGetLastError() == cudaSuccess ? 0 : DSMC_ERR_CUDA;
}

int launch_chi_mlp_forward(Ctx* c, const void* packed, const float* bias, int64_t n, const float* x, float* y,
                           float* chi, cudaStream_t s) {
  ChiArgs a = {};
  a.packed = (const char*)packed; a.bias = bias; a.n = n; a.x = x; a.y = y; a.chi = chi;
  a.status = status_ptr(c);
  return launch_chi_mlp(c, a, s);
}

int launch_chi_mlp_table(Ctx* c, const void* packed, const float* bias, int32_t nb, int32_t nE, float* table,
                         cudaStream_t s) {
  ChiArgs a = {};
  a.packed = (const char*)packed; a.bias = bias; a.n = (int64_t)nb * nE; a.chi = table;
  a.nb = nb; a.nE = nE;
  a.status = status_ptr(c);
  return launch_chi_mlp(c, a, s);
}

}  // namespace dsmc

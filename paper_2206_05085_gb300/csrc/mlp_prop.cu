// Learned-proposal network (not part of the paper): position encoding
// [x, sin(2^f x_a), cos(2^f x_a)], f < 6 (39 values) -> ReLU 64 -> ReLU 64 ->
// 1 logit, on the 5th-generation tensor cores (tcgen05, FP32 accumulation in
// tensor memory).  128-sample tiles, persistent CTAs (forward: thread = tile
// row = TMEM lane; the backward has two threads per row and two tiles in
// flight).
//
// BF16 form.  The parameters are the stored BF16 values (W1, b1, W2 are one
// BF16 term each; W3, b2, b3 are BF16-rounded and used in FP32 on the CUDA
// cores).  Every other MMA operand -- the encoded inputs X, the hidden
// activations H1, the gradient rows G -- is kept as two BF16 terms, hi =
// bf16(v) and lo = bf16(v - hi) (16 significant bits between them), so no
// value is rounded to BF16 between layers: a product with a weight matrix is
// hi W + lo W (two MMAs), a weight gradient G^T A is Gh^T Ah + Gh^T Al +
// Gl^T Ah (three; the dropped lo*lo term is 2^-16 of the product).
//
// Forward, per tile:  X [128 x 48] (39 inputs, a 1 carrying b1, zero pad) ->
//   D1 = X W1^T -> H1 = relu(D1), split in tensor memory in place -> D2 = H1
//   W2^T -> z = b3 + W3 relu(D2 + b2) (output layer on the CUDA cores).
// Backward, per tile (the forward is recomputed): g_z -> G2 = (W3^T g_z) *
//   (z2 > 0) -> dW2 += G2^T H1, db2 += G2^T 1, g_h1 = G2 W2 -> G1 = g_h1 *
//   (H1 > 0) -> dW1|db1 += G1^T X (X's ones column yields db1).  The
//   weight-gradient accumulators stay in tensor memory for the whole kernel.
//   One warp issues the MMAs, two groups of eight warps run the epilogues of
//   two tiles.
// Every wait on an mbarrier is bounded (DVGO_ERR_TIMEOUT).
#include "common.cuh"
#include "mlp_common.cuh"
#include "tcgen05.cuh"

namespace dvgo {

__device__ int g_mlp_status;  // DVGO_ERR_TIMEOUT if a bounded wait gave up

namespace prop {

constexpr int kH = 64;                        // hidden width
constexpr int kPropFreq = 6;
constexpr int oW1 = 0, oB1 = kH * kIn, oW2 = oB1 + kH, oB2 = oW2 + kH * kH, oW3 = oB2 + kH, oB3 = oW3 + kH;
constexpr int kK1 = 48;                       // padded input width
constexpr uint32_t kSboX = (kK1 / 8) * 128;   // 768: forward X rows
constexpr uint32_t kSboW2 = (kH / 8) * 128;   // 1024
constexpr uint32_t kSboH = (kH / 8) * 128;    // 1024: backward H1 and G rows
constexpr uint32_t kXBytes = kTile * kK1 * 2;
constexpr uint32_t kHBytes = kTile * kH * 2;
constexpr uint32_t kSpin = 1u << 24;

// forward shared memory
constexpr uint32_t fW1 = 0, fW2 = fW1 + kH * kK1 * 2, fXh = fW2 + kH * kH * 2, fXl = fXh + kXBytes,
                   fEnd = fXl + kXBytes;
// backward shared memory: the weights, then one tile's operands per group of epilogue warps
constexpr uint32_t bW1 = 0, bW2 = bW1 + kH * kK1 * 2, bGroup = bW2 + kH * kH * 2;
constexpr uint32_t oXh = 0, oXl = oXh + kXBytes, oHh = oXl + kXBytes, oHl = oHh + kHBytes, oGh = oHl + kHBytes,
                   oGl = oGh + kHBytes, kGroupBytes = oGl + kHBytes, bEnd = bGroup + 2 * kGroupBytes;
// backward tensor-memory columns: D of each group (D1, D2, g_h1 in turn), then
// dW2, dW1 and db2 (M = 64 products: output unit 16 w + i in lane 32 w + i)
constexpr uint32_t cD = 0, cDW2 = 128, cDW1 = 192, cDB2 = 240;

struct Side {
  alignas(16) float2 ob[kH];    // per hidden unit: (b2, W3)
  float b3;
  uint64_t ready[2];   // backward, per group: its operands of the next stage are written (8 warps)
  uint64_t gdone[2];   // backward, per group: MMAs of the stage finished
  uint64_t done;       // forward: MMAs of the layer finished
  uint64_t fin;     // backward: every MMA of the kernel finished
  uint32_t tmem_slot;
  int error;
};
constexpr int kFwdPerSM = 4;   // resident forward CTAs (128 TMEM columns each)
constexpr int kBwdThreads = 544;   // two groups of 8 epilogue warps and the MMA warp
static_assert(kFwdPerSM * (fEnd + sizeof(Side) + 1024) <= 227 * 1024, "forward shared memory");
static_assert(bEnd + sizeof(Side) <= 227 * 1024, "backward shared memory");

__device__ __forceinline__ float bfr(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__device__ __forceinline__ uint32_t u32_of(__nv_bfloat162 v) { return *reinterpret_cast<const uint32_t*>(&v); }

// Eight values of row `row` from column k8 as hi / lo BF16 core-matrix rows.
__device__ __forceinline__ void st_split8(uint8_t* hi, uint8_t* lo, int row, int k8, uint32_t sbo,
                                          const float* v) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __nv_bfloat162 h2 = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    const float2 hf = __bfloat1622float2(h2);
    h[i] = u32_of(h2);
    l[i] = u32_of(__floats2bfloat162_rn(v[2 * i] - hf.x, v[2 * i + 1] - hf.y));
  }
  const uint32_t off = tc::cm_off(row, k8, sbo);
  *reinterpret_cast<uint4*>(hi + off) = make_uint4(h[0], h[1], h[2], h[3]);
  *reinterpret_cast<uint4*>(lo + off) = make_uint4(l[0], l[1], l[2], l[3]);
}

// One stored BF16 parameter.
__device__ __forceinline__ void st_w(uint8_t* base, uint32_t off, float x) {
  *reinterpret_cast<__nv_bfloat16*>(base + off) = __float2bfloat16_rn(x);
}

// Column k of the padded input in the parameters' order: W1's column, the
// bias (kIn) or none (-1).  Forward: the order of the encoding.  Backward (kBwd): each
// thread of a row encodes whole sine-cosine pairs, so columns 0-23 hold x and
// the pairs p = 0..8, columns 24-47 the pairs 9..17 and the constant 1.
constexpr int kOneColBwd = 42;
template <bool kBwd>
__device__ __forceinline__ int param_col(int k) {
  if constexpr (!kBwd) return k <= kIn ? k : -1;
  if (k < 3) return k;
  const int q = k < 24 ? k - 3 : k - 24;
  if (q < 18) {
    const int p = (q >> 1) + (k < 24 ? 0 : 9);
    return 3 + p + ((q & 1) ? 3 * kPropFreq : 0);
  }
  return k == kOneColBwd ? kIn : -1;
}

// W1 | b1 | 0 and W2 as BF16 core matrices; W3, b2, b3 BF16-rounded.
template <bool kBwd>
__device__ __forceinline__ void load_weights(const float* __restrict__ params, uint8_t* w1, uint8_t* w2, Side* fs) {
#pragma unroll 8
  for (int e = threadIdx.x; e < kH * kK1; e += blockDim.x) {
    const int o = e / kK1, k = e % kK1, c = param_col<kBwd>(k);
    const float v = c < 0 ? 0.0f : __ldg(params + (c < kIn ? oW1 + o * kIn + c : oB1 + o));
    st_w(w1, tc::cm_off(o, k, kSboX), v);
  }
#pragma unroll 8
  for (int e = threadIdx.x; e < kH * kH; e += blockDim.x)
    st_w(w2, tc::cm_off(e / kH, e % kH, kSboW2), __ldg(params + oW2 + e));
  for (int e = threadIdx.x; e < kH; e += blockDim.x)
    fs->ob[e] = make_float2(bfr(__ldg(params + oB2 + e)), bfr(__ldg(params + oW3 + e)));
  if (threadIdx.x == 0) fs->b3 = bfr(__ldg(params + oB3));
}

// Position of list position j (valid: j < n).
__device__ __forceinline__ void load_pos(const float* __restrict__ xyz, const int32_t* __restrict__ idx, int64_t j,
                                         int64_t n, float (&x)[3]) {
  if (j >= n) return;
  const int64_t s = idx ? (int64_t)__ldg(idx + j) : j;
#pragma unroll
  for (int a = 0; a < 3; ++a) x[a] = __ldg(xyz + 3 * s + a);
}

// Input row [x (3), sin(2^f x_a) (a major, f inner), cos(2^f x_a), 1, 0 ...];
// rows past the list end are zero.
__device__ __forceinline__ void encode(const float (&x)[3], bool valid, float row[kK1]) {
#pragma unroll
  for (int k = 0; k < kK1; ++k) row[k] = 0.0f;
  if (!valid) return;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    row[a] = x[a];
#pragma unroll
    for (int f = 0; f < kPropFreq; ++f) {
      float sn, cs;
      sincosf(x[a] * (float)(1 << f), &sn, &cs);
      row[3 + a * kPropFreq + f] = sn;
      row[3 + 3 * kPropFreq + a * kPropFreq + f] = cs;
    }
  }
  row[kIn] = 1.0f;
}

// The backward's 24 columns of half `half` of the row, split: hi terms of
// column pairs in words 0-11, lo terms in 12-23.
__device__ __forceinline__ void encode_half(const float (&x)[3], bool valid, int half, uint32_t (&w)[24]) {
  float v[24];
#pragma unroll
  for (int k = 0; k < 24; ++k) v[k] = 0.0f;
  if (valid) {
    const int base = half ? 0 : 3;
    if (!half) {
#pragma unroll
      for (int a = 0; a < 3; ++a) v[a] = x[a];
    }
    float sc[18];
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      // pair p = 9 half + q: axis p / 6, frequency p % 6
      const float xa = half ? (q < 3 ? x[1] : x[2]) : (q < 6 ? x[0] : x[1]);
      const int f0 = q % 6, f1 = (q + 3) % 6;
      sincosf(xa * (half ? (float)(1 << f1) : (float)(1 << f0)), &sc[2 * q], &sc[2 * q + 1]);
    }
    if (base == 3) {
#pragma unroll
      for (int i = 0; i < 18; ++i) v[3 + i] = sc[i];
    } else {
#pragma unroll
      for (int i = 0; i < 18; ++i) v[i] = sc[i];
      v[kOneColBwd - 24] = 1.0f;
    }
  }
#pragma unroll
  for (int i = 0; i < 12; ++i) {
    const __nv_bfloat162 h2 = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    const float2 hf = __bfloat1622float2(h2);
    w[i] = u32_of(h2);
    w[12 + i] = u32_of(__floats2bfloat162_rn(v[2 * i] - hf.x, v[2 * i + 1] - hf.y));
  }
}

__device__ __forceinline__ void write_x(uint8_t* xh, uint8_t* xl, int row, const float (&x)[kK1]) {
#pragma unroll
  for (int kb = 0; kb < kK1 / 8; ++kb) st_split8(xh, xl, row, kb * 8, kSboX, x + 8 * kb);
}

// D = A W^T with A split (hi, lo) and W one term: two MMAs per K step of 16.
// (One elected thread; unrolled: see the colour MLP's issue loops.)
// Descriptors are formed once and advanced by addition: forming them per
// instruction made the issue, not the product, the cost (125 cycles each).
template <int kSteps>
__device__ __forceinline__ void mma_split_w(uint32_t d, uint32_t ah, uint32_t al, uint32_t a_sbo, uint32_t w,
                                            uint32_t w_sbo, uint32_t idesc) {
  uint64_t dah = tc::smem_desc(ah, 128, a_sbo), dal = tc::smem_desc(al, 128, a_sbo), dw = tc::smem_desc(w, 128, w_sbo);
#pragma unroll
  for (int j = 0; j < kSteps; ++j) {
    tc::mma_bf16(d, dah, dw, idesc, j > 0 ? 1u : 0u);
    tc::mma_bf16(d, dal, dw, idesc, 1u);
    dah += 256 >> 4;
    dal += 256 >> 4;
    dw += 256 >> 4;
  }
}

// D += A^T B over the tile's 128 rows, A (G) and B (H1 or X) split, both
// MN-major: Gh Bh + Gh Bl + Gl Bh per K step of 16 rows.
__device__ __forceinline__ void mma_grad(uint32_t d, uint32_t gh, uint32_t gl, uint32_t bh, uint32_t bl,
                                         uint32_t b_sbo, uint32_t idesc, bool accumulate) {
  uint64_t dgh = tc::smem_desc_mn(gh, kSboH, 128), dgl = tc::smem_desc_mn(gl, kSboH, 128);
  uint64_t dbh = tc::smem_desc_mn(bh, b_sbo, 128), dbl = tc::smem_desc_mn(bl, b_sbo, 128);
  const uint64_t ib = (2 * b_sbo) >> 4;
#pragma unroll
  for (int q = 0; q < kTile / 16; ++q) {
    tc::mma_bf16(d, dgh, dbh, idesc, (accumulate || q > 0) ? 1u : 0u);
    tc::mma_bf16(d, dgh, dbl, idesc, 1u);
    tc::mma_bf16(d, dgl, dbh, idesc, 1u);
    dgh += (2 * kSboH) >> 4;
    dgl += (2 * kSboH) >> 4;
    dbh += ib;
    dbl += ib;
  }
}

}  // namespace prop

using namespace prop;

// 128 threads.  Per tile: X -> layer 1 -> H1 -> layer 2 -> output layer.  The
// phases of a tile follow one another; four resident CTAs per SM (H1 stays in
// tensor memory, so a CTA needs 39 KB of shared memory and 128 TMEM columns)
// fill each other's waits.  What bounds it: the encoding and the epilogues on
// the CUDA cores (about 1.5k instructions a row).  Measured, 5.3e6
// candidates: 615 us with H1 in shared memory and two CTAs per SM, 324 us now;
// a tile's rows on twice the warps (half the encoding and the columns each)
// took 328 us, so it is the instructions and not their latency.
__global__ void __launch_bounds__(128, kFwdPerSM) prop_fwd_kernel(const float* __restrict__ xyz,
                                                                  const int32_t* __restrict__ idx, int64_t n_cap,
                                                                  const int64_t* __restrict__ n_dev,
                                                                  const float* __restrict__ params,
                                                                  float* __restrict__ out) {
  extern __shared__ __align__(1024) uint8_t sm[];
  Side* fs = reinterpret_cast<Side*>(sm + fEnd);
  const int tid = threadIdx.x, warp = tid >> 5;
  const int64_t n = mlp_count(n_cap, n_dev);
  const int64_t ntiles = (n + kTile - 1) / kTile;
  if ((int64_t)blockIdx.x >= ntiles) return;
  float x[3] = {0.0f, 0.0f, 0.0f};
  load_pos(xyz, idx, (int64_t)blockIdx.x * kTile + tid, n, x);
  if (warp == 0) tc::tmem_alloc(&fs->tmem_slot, 128);
  if (tid == 0) tc::mbar_init(&fs->done, 1);
  load_weights<false>(params, sm + fW1, sm + fW2, fs);
  tc::fence_proxy_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = fs->tmem_slot;
  const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
  const uint32_t sW1 = tc::smem_u32(sm + fW1), sW2 = tc::smem_u32(sm + fW2);
  const uint32_t sXh = tc::smem_u32(sm + fXh), sXl = tc::smem_u32(sm + fXl);
  const uint32_t id = tc::idesc_bf16(128, kH, 0, 0);
  uint32_t phase = 0;
  bool ok = true;
  for (int64_t t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
    const int64_t j = t * kTile + tid;
    {
      float v[kK1];
      encode(x, j < n, v);
      write_x(sm + fXh, sm + fXl, tid, v);
    }
    tc::fence_proxy_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) {
      tc::fence_after_sync();
      if (tc::elect_one()) {
        mma_split_w<kK1 / 16>(tmem, sXh, sXl, kSboX, sW1, kSboX, id);
        tc::mma_commit(&fs->done);
      }
      __syncwarp();
    }
    load_pos(xyz, idx, j + (int64_t)gridDim.x * kTile, n, x);   // the next tile's position
    ok = __syncthreads_and(tc::mbar_wait(&fs->done, phase, kSpin));
    phase ^= 1;
    if (!ok) break;
    tc::fence_after_sync();
#pragma unroll 1
    for (int ch = 0; ch < kH / 32; ++ch) {          // H1 = relu(D1), split: per 16 units 8 hi, 8 lo columns
      float v[32];
      tc::tmem_ld32(lane_base + ch * 32, v);
      uint32_t w[32];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float a = fmaxf(v[2 * i], 0.0f), b = fmaxf(v[2 * i + 1], 0.0f);
        const __nv_bfloat162 h2 = __floats2bfloat162_rn(a, b);
        const float2 hf = __bfloat1622float2(h2);
        w[(i >> 3) * 16 + (i & 7)] = u32_of(h2);
        w[(i >> 3) * 16 + 8 + (i & 7)] = u32_of(__floats2bfloat162_rn(a - hf.x, b - hf.y));
      }
      tc::tmem_st32(lane_base + ch * 32, w);
    }
    tc::tmem_wait_st();
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) {
      tc::fence_after_sync();
      if (tc::elect_one()) {
        uint64_t dw = tc::smem_desc(sW2, 128, kSboW2);
#pragma unroll
        for (uint32_t k = 0; k < kH / 16; ++k) {
          tc::mma_ts(tmem + kH, tmem + 16 * k, dw, id, k > 0 ? 1u : 0u);
          tc::mma_ts(tmem + kH, tmem + 16 * k + 8, dw, id, 1u);
          dw += 256 >> 4;
        }
        tc::mma_commit(&fs->done);
      }
      __syncwarp();
    }
    ok = __syncthreads_and(tc::mbar_wait(&fs->done, phase, kSpin));
    phase ^= 1;
    if (!ok) break;
    tc::fence_after_sync();
    float z = fs->b3;
#pragma unroll 1
    for (int ch = 0; ch < kH / 32; ++ch) {
      float v[32];
      tc::tmem_ld32(lane_base + kH + ch * 32, v);
#pragma unroll
      for (int i = 0; i < 32; i += 2) {
        const float4 q = *reinterpret_cast<const float4*>(&fs->ob[ch * 32 + i]);
        z = fmaf(q.y, fmaxf(v[i] + q.x, 0.0f), z);
        z = fmaf(q.w, fmaxf(v[i + 1] + q.z, 0.0f), z);
      }
    }
    if (j < n) out[idx ? (int64_t)__ldg(idx + j) : j] = z;
    tc::fence_before_sync();
  }
  if (!ok && tid == 0) atomicExch(&g_mlp_status, (int)DVGO_ERR_TIMEOUT);
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(tmem, 128);
}

// Backward, 544 threads: two groups of 8 epilogue warps, each on its own tile
// (the CTA's tiles alternate between them), and warp 16 that issues the MMAs
// of each stage once the group's warps signal that its operands are in shared
// memory, and commits them to the group's `gdone`.  Warp w: group w / 8, tile
// rows 32 (w & 3) .., hidden columns 32 ((w >> 2) & 1) .. and that half of the
// input columns.
//   stage 0: D = X W1^T
//   stage 1: D = H1 W2^T
//   stage 2: dW2 += G2^T H1;  db2 += G2^T 1 (X's ones column);  D = G2 W2
//   stage 3: dW1|db1 += G1^T X
// The groups run two stages apart, so that one's epilogues go beside the
// other's MMAs; the weight gradients of both sum in one set of accumulators,
// tile after tile.  g_params += the CTA's sums (atomics at the end).
// What bounds it: the epilogues (about 650 instructions a thread and tile);
// the MMAs are 2.8k cycles a tile.  The weight gradients are M = 64 products
// (32 cycles each for N = 64; the 128-row form with the gradient padded to
// 128 took 48); dW3 is summed per thread over all tiles and reduced over the
// rows once.  Measured, 5.3e6 candidates: 2605 us with one group, 128-row
// gradients and rolled issue loops; 840 us in this form with waits that read
// the error word before the barrier (a shared-memory round trip on every
// stage's chain), 813 us with the barrier polled first, 804 us with the output
// layer's constants read for two units at a time.  An MMA warp that polls
// both groups and takes whichever is ready is slower (914 us): its polling
// competes for shared memory.
__global__ void __launch_bounds__(kBwdThreads, 1) prop_bwd_kernel(const float* __restrict__ g_out,
                                                                  const float* __restrict__ xyz,
                                                                  const int32_t* __restrict__ idx, int64_t n_cap,
                                                                  const int64_t* __restrict__ n_dev,
                                                                  const float* __restrict__ params,
                                                                  float* __restrict__ g_params) {
  extern __shared__ __align__(1024) uint8_t sm[];
  Side* fs = reinterpret_cast<Side*>(sm + bEnd);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t n = mlp_count(n_cap, n_dev);
  const int64_t ntiles = (n + kTile - 1) / kTile;
  if ((int64_t)blockIdx.x >= ntiles) return;
  const int64_t tiles = (ntiles - 1 - blockIdx.x) / gridDim.x + 1;
  if (warp == 16) tc::tmem_alloc(&fs->tmem_slot, 256);
  if (tid == 0) {
    for (int g = 0; g < 2; ++g) {
      tc::mbar_init(&fs->ready[g], 8);
      tc::mbar_init(&fs->gdone[g], 1);
    }
    tc::mbar_init(&fs->fin, 1);
    fs->error = 0;
  }
  load_weights<true>(params, sm + bW1, sm + bW2, fs);
  tc::fence_proxy_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = fs->tmem_slot;
  const int group = (warp >> 3) & 1, quarter = warp & 3, half = (warp >> 2) & 1, row = quarter * 32 + lane;
  const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
  float dW3acc[32], db3acc = 0.0f;
#pragma unroll
  for (int i = 0; i < 32; ++i) dW3acc[i] = 0.0f;
  if (warp == 16) {
    // ------------------------------------------------------- MMA issuer
    const uint32_t sW1 = tc::smem_u32(sm + bW1), sW2 = tc::smem_u32(sm + bW2);
    uint32_t ph[2] = {0u, 0u};
    bool ok = true;
    // stage `st` of tile k (group k & 1) once its operands are in (lane 0 polls)
    auto stage = [&](int64_t k, int st) {
      if (!ok || k < 0 || k >= tiles) return;
      const int g = (int)(k & 1);
      int r = 0;
      if (lane == 0) {
        r = tc::mbar_try_wait(&fs->ready[g], ph[g]) ||
                    (!*(volatile int*)&fs->error && tc::mbar_wait(&fs->ready[g], ph[g], kSpin))
                ? 1
                : 0;
        if (!r) atomicExch(&fs->error, 1);
      }
      ph[g] ^= 1;
      ok = __shfl_sync(0xffffffffu, r, 0) != 0;
      if (!ok) return;
      tc::fence_after_sync();
      if (tc::elect_one()) {
        const uint32_t base = tc::smem_u32(sm + bGroup) + (uint32_t)g * kGroupBytes, D = tmem + cD + kH * (uint32_t)g;
        if (st == 0) {
          mma_split_w<kK1 / 16>(D, base + oXh, base + oXl, kSboX, sW1, kSboX, tc::idesc_bf16(128, kH, 0, 0));
        } else if (st == 1) {
          mma_split_w<kH / 16>(D, base + oHh, base + oHl, kSboH, sW2, kSboW2, tc::idesc_bf16(128, kH, 0, 0));
        } else if (st == 2) {
          // D = G2 W2: Gh W2 + Gl W2 (G K-major, W2 MN-major)
          uint64_t dgh = tc::smem_desc(base + oGh, 128, kSboH), dgl = tc::smem_desc(base + oGl, 128, kSboH);
          uint64_t dw = tc::smem_desc_mn(sW2, kSboW2, 128);
          const uint32_t id_gh = tc::idesc_bf16(128, kH, 0, 1);
#pragma unroll
          for (int q = 0; q < kH / 16; ++q) {
            tc::mma_bf16(D, dgh, dw, id_gh, q > 0 ? 1u : 0u);
            tc::mma_bf16(D, dgl, dw, id_gh, 1u);
            dgh += 256 >> 4;
            dgl += 256 >> 4;
            dw += (2 * kSboW2) >> 4;
          }
          mma_grad(tmem + cDW2, base + oGh, base + oGl, base + oHh, base + oHl, kSboH, tc::idesc_bf16(64, kH, 1, 1),
                   k > 0);
          // db2: X's columns 32-47 hold the exact ones column
          uint64_t gh = tc::smem_desc_mn(base + oGh, kSboH, 128), gl = tc::smem_desc_mn(base + oGl, kSboH, 128);
          uint64_t dx = tc::smem_desc_mn(base + oXh + 4 * 128, kSboX, 128);
          const uint32_t id16 = tc::idesc_bf16(64, 16, 1, 1);
#pragma unroll
          for (int q = 0; q < kTile / 16; ++q) {
            tc::mma_bf16(tmem + cDB2, gh, dx, id16, (k > 0 || q > 0) ? 1u : 0u);
            tc::mma_bf16(tmem + cDB2, gl, dx, id16, 1u);
            gh += (2 * kSboH) >> 4;
            gl += (2 * kSboH) >> 4;
            dx += (2 * kSboX) >> 4;
          }
        } else {
          mma_grad(tmem + cDW1, base + oGh, base + oGl, base + oXh, base + oXl, kSboX, tc::idesc_bf16(64, kK1, 1, 1),
                   k > 0);
        }
        tc::mma_commit(&fs->gdone[g]);
      }
      __syncwarp();
    };
    // group 0 on tile k (even), group 1 two stages behind it on tile k + 1
    stage(0, 0);
    stage(0, 1);
    for (int64_t k = 0; k < tiles; k += 2) {
      stage(k, 2);
      stage(k + 1, 0);
      stage(k, 3);
      stage(k + 1, 1);
      stage(k + 2, 0);
      stage(k + 1, 2);
      stage(k + 2, 1);
      stage(k + 1, 3);
    }
    // every MMA issued has finished before tensor memory is read or released
    if (tc::elect_one()) {
      tc::mma_commit(&fs->fin);
      if (!tc::mbar_wait(&fs->fin, 0, kSpin)) atomicExch(&fs->error, 1);
    }
    __syncwarp();
  } else {
    // --------------------------------------------------- epilogue warps
    uint32_t ph = 0;
    uint8_t* const gb = sm + bGroup + (uint32_t)group * kGroupBytes;
    const uint32_t Dt = lane_base + cD + kH * (uint32_t)group + 32u * (uint32_t)half;
    auto signal = [&]() {
      tc::fence_proxy_async_smem();
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&fs->ready[group]);
    };
    auto await = [&]() -> bool {   // the outcome is the warp's
      const bool ok = tc::mbar_try_wait(&fs->gdone[group], ph) ||
                      (!*(volatile int*)&fs->error && tc::mbar_wait(&fs->gdone[group], ph, kSpin));
      ph ^= 1;
      if (!ok) atomicExch(&fs->error, 1);
      const bool all = __all_sync(0xffffffffu, ok);
      tc::fence_after_sync();
      return all;
    };
    auto row_of = [&](int64_t k) { return ((int64_t)blockIdx.x + k * gridDim.x) * kTile + row; };
    auto upstream = [&](int64_t j) { return j < n ? __ldg(g_out + (idx ? (int64_t)__ldg(idx + j) : j)) : 0.0f; };
    float pos[3] = {0.0f, 0.0f, 0.0f};
    load_pos(xyz, idx, row_of(group), n, pos);
    float gup = upstream(row_of(group)), gup_next = 0.0f;
    uint32_t xw[24];
    encode_half(pos, row_of(group) < n, half, xw);
    for (int64_t k = group; k < tiles; k += 2) {
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const uint32_t off = tc::cm_off(row, 24 * half + 8 * q, kSboX);
        *reinterpret_cast<uint4*>(gb + oXh + off) = make_uint4(xw[4 * q], xw[4 * q + 1], xw[4 * q + 2], xw[4 * q + 3]);
        *reinterpret_cast<uint4*>(gb + oXl + off) =
            make_uint4(xw[12 + 4 * q], xw[13 + 4 * q], xw[14 + 4 * q], xw[15 + 4 * q]);
      }
      signal();                                     // stage 0
      load_pos(xyz, idx, row_of(k + 2), n, pos);    // the group's next position and upstream gradient
      gup_next = upstream(row_of(k + 2));
      if (!await()) break;
      uint32_t mask = 0u;                           // H1 > 0 on this thread's columns
#pragma unroll 1
      for (int c = 0; c < 2; ++c) {                 // H1 = relu(D1), split
        float v[16];
        tc::tmem_ld16(Dt + 16 * c, v);
        uint32_t m = 0u;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          v[i] = fmaxf(v[i], 0.0f);
          if (v[i] > 0.0f) m |= 1u << i;
        }
        mask |= m << (16 * c);
#pragma unroll
        for (int q = 0; q < 2; ++q) st_split8(gb + oHh, gb + oHl, row, 32 * half + 16 * c + 8 * q, kSboH, v + 8 * q);
      }
      signal();                                     // stage 1
      if (!await()) break;
      // output layer: g_z = the upstream logit gradient; G2 = (W3^T g_z) * (z2 > 0);
      // dW3 += g_z h2
      if (half == 0) db3acc += gup;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        float v[16];
        tc::tmem_ld16(Dt + 16 * c, v);
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
          const float4 q = *reinterpret_cast<const float4*>(&fs->ob[32 * half + 16 * c + i]);
          const float z0 = v[i] + q.x, z1 = v[i + 1] + q.z;
          dW3acc[16 * c + i] = fmaf(gup, fmaxf(z0, 0.0f), dW3acc[16 * c + i]);
          dW3acc[16 * c + i + 1] = fmaf(gup, fmaxf(z1, 0.0f), dW3acc[16 * c + i + 1]);
          v[i] = z0 > 0.0f ? gup * q.y : 0.0f;
          v[i + 1] = z1 > 0.0f ? gup * q.w : 0.0f;
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) st_split8(gb + oGh, gb + oGl, row, 32 * half + 16 * c + 8 * q, kSboH, v + 8 * q);
      }
      signal();                                     // stage 2
      if (!await()) break;
#pragma unroll 1
      for (int c = 0; c < 2; ++c) {                 // G1 = g_h1 * (H1 > 0), split
        float v[16];
        tc::tmem_ld16(Dt + 16 * c, v);
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = (mask >> i) & 1u ? v[i] : 0.0f;
        mask >>= 16;
#pragma unroll
        for (int q = 0; q < 2; ++q) st_split8(gb + oGh, gb + oGl, row, 32 * half + 16 * c + 8 * q, kSboH, v + 8 * q);
      }
      signal();                                     // stage 3
      encode_half(pos, row_of(k + 2) < n, half, xw);
      gup = gup_next;
      if (!await()) break;
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const bool ok = fs->error == 0;
  if (ok && warp < 16) {
    // output layer: this warp's row sums (lane = hidden unit 32 half + lane)
    atomicAdd(g_params + oW3 + 32 * half + lane, reduce_scatter32(dW3acc, lane));
    if (half == 0) {
      float v = db3acc;
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) atomicAdd(g_params + oB3, v);
    }
    // dW2, db2 and dW1|db1: output unit o in lanes 0-15 of each quarter; one
    // 16-column block per warp of a quarter (dW2: warps / 4 = 0..3, then dW1 and db2)
    const int o = 16 * quarter + lane, blk = warp >> 2;
    float d[16];
    tc::tmem_ld16(lane_base + cDW2 + 16 * blk, d);
    if (lane < 16) {
#pragma unroll
      for (int i = 0; i < 16; ++i) atomicAdd(g_params + oW2 + o * kH + 16 * blk + i, d[i]);
    }
    __syncwarp();
    if (blk < 3) {
      tc::tmem_ld16(lane_base + cDW1 + 16 * blk, d);
      if (lane < 16) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int c = param_col<true>(16 * blk + i);
          if (c >= 0) atomicAdd(g_params + (c < kIn ? oW1 + o * kIn + c : oB1 + o), d[i]);
        }
      }
    } else {
      tc::tmem_ld16(lane_base + cDB2, d);
      if (lane < 16) atomicAdd(g_params + oB2 + o, d[kOneColBwd - 32]);
    }
  }
  if (!ok && tid == 0) atomicExch(&g_mlp_status, (int)DVGO_ERR_TIMEOUT);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 16) tc::tmem_dealloc(tmem, 256);
}

}  // namespace dvgo

using namespace dvgo;

int dvgo_proposal_fwd_bf16(const float* xyz, const int32_t* idx, int64_t n_cap, const int64_t* n_dev,
                           const float* params, float* logits, cudaStream_t st) {
  const size_t smem = fEnd + sizeof(Side);
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(prop_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    attr = true;
  }
  const int grid = (int)std::min<int64_t>((n_cap + kTile - 1) / kTile, kFwdPerSM * kNumSMs);
  if (grid < 1) return DVGO_OK;
  prop_fwd_kernel<<<grid, 128, smem, st>>>(xyz, idx, n_cap, n_dev, params, logits);
  return launch_status();
}

int dvgo_proposal_bwd_bf16(const float* g_logits, const float* xyz, const int32_t* idx, int64_t n_cap,
                           const int64_t* n_dev, const float* params, float* g_params, cudaStream_t st) {
  const size_t smem = bEnd + sizeof(Side);
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(prop_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    attr = true;
  }
  const int grid = (int)std::min<int64_t>((n_cap + kTile - 1) / kTile, kNumSMs);
  if (grid < 1) return DVGO_OK;
  prop_bwd_kernel<<<grid, kBwdThreads, smem, st>>>(g_logits, xyz, idx, n_cap, n_dev, params, g_params);
  return launch_status();
}

int dvgo_mlp_status_read_and_clear(cudaStream_t st) {
  int v = 0, zero = 0;
  cudaMemcpyFromSymbolAsync(&v, g_mlp_status, sizeof(int), 0, cudaMemcpyDeviceToHost, st);
  cudaMemcpyToSymbolAsync(g_mlp_status, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, st);
  cudaStreamSynchronize(st);
  return v;
}

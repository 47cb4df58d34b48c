// Colour MLP (rgbnet, the shallow decoder of the hybrid representation of
// Tab. 1) in exact FP32 on the CUDA cores: 39 -> ReLU 128 -> ReLU 128 ->
// sigmoid 3.  Fused per tile of 128 samples.  The forward can store both
// hidden activations (list position j: act[j][0:128] = h1, act[j][128:256]
// = h2); the backward then reads them instead of recomputing the forward.
// Persistent CTAs keep their share of the weight gradients in registers
// across tiles and flush them once with atomics.
//
// 512 threads.  Shared-memory rows have pitches 44 (40-wide) and 132
// (128-wide).  The large products run on packed pairs of neighbouring columns
// (one instruction, two FMAs, each element still summed in k order) in 8 x 4
// register blocks: warp w rows 8w .. 8w+7, lane columns 4 lane .. + 3, so that
// one operand is a uniform load (one wavefront) and the other 512 contiguous
// bytes: 6 shared-memory wavefronts per 16 packed FMAs and warp.
//   NN products (reduction along the rows of B): A by row, B by k.
//   TN products (reduction over the tile's samples): both by sample.
//   NT products (the backward's recomputed forward; ty = tid / 16, tx = tid %
//     16): thread rows ty + 32a, columns tx + 16b, 128-bit loads along k.
// What bounds them: FMA issue and shared-memory bandwidth together.  Measured,
// 130,000 samples: forward 170 us with scalar FMAs in 8 x 8 blocks on 8 warps
// (half the FMA pipe idle on dependences), 141 us packed in 4 x 8 blocks of
// 32 x 16 threads (12 wavefronts per 16 packed FMAs: bandwidth), 137 us in this
// form with the X tile built by four warps between two barriers, 127 us with
// each warp building its own rows (250,000 samples: 248 and 225 us); backward
// 362, 317 and 300 us (292 with g_k0 on the threads that do not build the
// input tile; dW1 in 2 x 5 blocks, with fewer wavefronts, was not faster).  The
// backward's 128 registers leave 80 bytes of it in local memory.
#include "common.cuh"
#include "mlp_common.cuh"

namespace dvgo {

constexpr int kP40 = 44;   // pitch of 40-wide rows
constexpr int kP128 = 132; // pitch of 128-wide rows
constexpr int kAct = 2 * kHid;
constexpr int kF32Threads = 512;
constexpr int kRowsT = 8;   // tile rows (or output units) per thread in the NN and TN products

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ float dot4(float4 a, float4 b, float acc) {
  acc = fmaf(a.x, b.x, acc);
  acc = fmaf(a.y, b.y, acc);
  acc = fmaf(a.z, b.z, acc);
  return fmaf(a.w, b.w, acc);
}
__device__ __forceinline__ float comp(float4 v, int q) {
  return q == 0 ? v.x : (q == 1 ? v.y : (q == 2 ? v.z : v.w));
}

// W1 (+ b1 as column 39) into [128][44]; W2 into [128][132].
__device__ __forceinline__ void load_w1(const float* __restrict__ params, float* W1S) {
  for (int e = threadIdx.x; e < kHid * kP40; e += blockDim.x) {
    const int o = e / kP40, k = e % kP40;
    W1S[e] = k < kIn ? params[kOffW1 + o * kIn + k] : (k == kIn ? params[kOffB1 + o] : 0.0f);
  }
}
__device__ __forceinline__ void load_w2(const float* __restrict__ params, float* W2S) {
  for (int e = threadIdx.x; e < kHid * kHid; e += blockDim.x) {
    const int o = e / kHid, i = e % kHid;
    W2S[o * kP128 + i] = params[kOffW2 + e];
  }
}

// W1 | b1 transposed, [40][132] (row k, column o), and W2 transposed, [128][132].
__device__ __forceinline__ void load_w1t(const float* __restrict__ params, float* W1T) {
  for (int e = threadIdx.x; e < kHid * kInP; e += blockDim.x) {
    const int o = e / kInP, k = e % kInP;
    W1T[k * kP128 + o] = __ldg(params + (k < kIn ? kOffW1 + o * kIn + k : kOffB1 + o));
  }
}
__device__ __forceinline__ void load_w2t(const float* __restrict__ params, float* W2T) {
#pragma unroll 8
  for (int e = threadIdx.x; e < kHid * kHid; e += blockDim.x)
    W2T[(e % kHid) * kP128 + e / kHid] = __ldg(params + kOffW2 + e);
}

// acc[a][p] = sum_k A[(8 warp + a)*lda + k] * B[k*ldb + 4 lane + 2p, + 1], K % 4 == 0
template <int K>
__device__ __forceinline__ void gemm_nn(const float* A, int lda, const float* B, int ldb, f32x2 acc[kRowsT][2]) {
  const float* a0 = A + kRowsT * (threadIdx.x >> 5) * lda;
  const float* b0 = B + 4 * (threadIdx.x & 31);
#pragma unroll
  for (int a = 0; a < kRowsT; ++a) acc[a][0] = acc[a][1] = 0ull;
#pragma unroll 2
  for (int k = 0; k < K; k += 4) {
    float4 av[kRowsT];
#pragma unroll
    for (int a = 0; a < kRowsT; ++a) av[a] = ld4(a0 + a * lda + k);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 b = ld4(b0 + (k + q) * ldb);
      const f32x2 bl = pack2(b.x, b.y), bh = pack2(b.z, b.w);
#pragma unroll
      for (int a = 0; a < kRowsT; ++a) {
        const float x = comp(av[a], q);
        const f32x2 d = pack2(x, x);
        acc[a][0] = fma2(d, bl, acc[a][0]);
        acc[a][1] = fma2(d, bh, acc[a][1]);
      }
    }
  }
}

// max(v + bias, 0) of a row's four columns
__device__ __forceinline__ float4 relu4(const f32x2 acc[2], const float4& bias) {
  const float2 l = unpack2(acc[0]), h = unpack2(acc[1]);
  return make_float4(fmaxf(l.x + bias.x, 0.0f), fmaxf(l.y + bias.y, 0.0f), fmaxf(h.x + bias.z, 0.0f),
                     fmaxf(h.y + bias.w, 0.0f));
}

// acc[a][b] = sum_k A[(ty+32a)*lda + k] * B[(tx+16b)*ldb + k], K % 4 == 0
template <int K>
__device__ __forceinline__ void gemm_nt(const float* A, int lda, const float* B, int ldb, int ty,
                                        int tx, float acc[4][8]) {
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 8; ++b) acc[a][b] = 0.0f;
#pragma unroll 2
  for (int k = 0; k < K; k += 4) {
    float4 av[4], bv[8];
#pragma unroll
    for (int a = 0; a < 4; ++a) av[a] = ld4(A + (ty + 32 * a) * lda + k);
#pragma unroll
    for (int b = 0; b < 8; ++b) bv[b] = ld4(B + (tx + 16 * b) * ldb + k);
    // outer-product order: 32 independent FMAs per k
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) acc[a][b] = fmaf(comp(av[a], q), comp(bv[b], q), acc[a][b]);
  }
}

// Write the thread's 4x8 block (rows ty + 32a, columns tx + 16b) of a tile.
__device__ __forceinline__ void store_block(float* S, int ld, int ty, int tx, const float v[4][8]) {
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 8; ++b) S[(ty + 32 * a) * ld + tx + 16 * b] = v[a][b];
}

// Rows j0.. of a global [.][256] activation buffer, column offset col, into a
// [128][128] shared-memory tile (pitch 132; rows past n zero), by asynchronous
// 16-byte copies (all of a thread's in flight); ends with copies_done().
__device__ __forceinline__ void tile_from_global(float* S, const float* __restrict__ act, int64_t j0,
                                                 int64_t n, int col) {
  for (int e = threadIdx.x; e < kTile * (kHid / 4); e += blockDim.x) {
    const int r = e >> 5, c4 = (e & 31) * 4;
    if (j0 + r < n) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                       (uint32_t)__cvta_generic_to_shared(S + r * kP128 + c4)),
                   "l"(act + (j0 + r) * kAct + col + c4)
                   : "memory");
    } else {
      st4(S + r * kP128 + c4, make_float4(0.f, 0.f, 0.f, 0.f));
    }
  }
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ void build_x_tile(float* XS, const float* __restrict__ k0,
                                             const float* __restrict__ rays_d,
                                             const int32_t* __restrict__ ray_id,
                                             const int32_t* __restrict__ idx, int64_t j0, int64_t n) {
  if (threadIdx.x < kTile) {
    float row[kInP];
    encode_row(k0, rays_d, ray_id, idx, j0 + threadIdx.x, n, row);
    float* dst = XS + threadIdx.x * kP40;
#pragma unroll
    for (int k = 0; k < kInP; k += 4) st4(dst + k, make_float4(row[k], row[k + 1], row[k + 2], row[k + 3]));
  }
}

// What a lane of the forward loads for its tile row (row lane / 4 of the warp's
// eight, q = lane % 4): features 4 q .. + 3 (q < 3) and the ray's direction.
// The loads depend on each other (list index; feature row and ray id;
// direction), so they are issued in three steps, spread over the tile before.
struct XRow {
  int64_t s;   // sample index (-1 past the list end)
  int32_t r;
  float4 f;
  float d[3];
  __device__ __forceinline__ void l1(const int32_t* __restrict__ idx, int64_t j, int64_t n) {
    s = j < n ? (idx ? (int64_t)__ldg(idx + j) : j) : -1;
  }
  __device__ __forceinline__ void l2(const float* __restrict__ k0, const int32_t* __restrict__ ray_id, int q) {
    f = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    r = -1;
    if (s < 0) return;
    if (q < 3) f = __ldg(reinterpret_cast<const float4*>(k0 + s * kFeat) + q);
    r = __ldg(ray_id + s);
  }
  __device__ __forceinline__ void l3(const float* __restrict__ rays_d) {
#pragma unroll
    for (int a = 0; a < 3; ++a) d[a] = r >= 0 ? __ldg(rays_d + 3 * (int64_t)r + a) : 0.0f;
  }
  // This lane's part of the input row (the row of encode_row): its features
  // (q = 3: the direction and the constant) and the pairs p = 3 q .. + 2.
  __device__ __forceinline__ void store(float* x, int q) const {
    const bool valid = s >= 0;
    if (q < 3) {
      st4(x + 4 * q, f);
    } else {
#pragma unroll
      for (int a = 0; a < 3; ++a) x[kFeat + a] = d[a];
      x[kIn] = valid ? 1.0f : 0.0f;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int p = 3 * q + i, a = p >> 2;
      float sn, cs;
      sincosf((a == 0 ? d[0] : (a == 1 ? d[1] : d[2])) * (float)(1 << (p & 3)), &sn, &cs);
      x[kFeat + 3 + p] = valid ? sn : 0.0f;
      x[kFeat + 3 + 3 * kNumFreq + p] = valid ? cs : 0.0f;
    }
  }
};

__global__ void __launch_bounds__(kF32Threads, 1) rgbnet_fwd_f32_kernel(
    const float* __restrict__ k0, const float* __restrict__ rays_d,
    const int32_t* __restrict__ ray_id, const int32_t* __restrict__ idx, int64_t n_cap,
    const int64_t* __restrict__ n_dev, const float* __restrict__ params, float* __restrict__ rgb,
    float* __restrict__ act) {
  extern __shared__ float4 smem4[];
  float* smem = reinterpret_cast<float*>(smem4);
  float* W1T = smem;                   // [40][132]
  float* W2T = W1T + kInP * kP128;     // [128][132]
  float* XS = W2T + kHid * kP128;      // [128][44]
  float* HS = XS + kTile * kP40;       // [128][132]  h1
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n = mlp_count(n_cap, n_dev);
  const int64_t ntiles = (n + kTile - 1) / kTile;
  load_w1t(params, W1T);
  load_w2t(params, W2T);
  // this thread's columns 4 lane ..
  float w3[3][4], b2a[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    b2a[b] = __ldg(params + kOffB2 + 4 * lane + b);
#pragma unroll
    for (int c = 0; c < 3; ++c) w3[c][b] = __ldg(params + kOffW3 + c * kHid + 4 * lane + b);
  }
  const float4 b2v = make_float4(b2a[0], b2a[1], b2a[2], b2a[3]), zero = make_float4(0.f, 0.f, 0.f, 0.f);
  const int xq = lane & 3, xrow = kRowsT * warp + (lane >> 2);
  XRow xr;
  xr.l1(idx, (int64_t)blockIdx.x * kTile + xrow, n);
  xr.l2(k0, ray_id, xq);
  xr.l3(rays_d);
  __syncthreads();   // the weights are in; from here on a warp touches its own eight rows only
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int64_t j0 = t * kTile;
    xr.store(XS + xrow * kP40, xq);
    xr.l1(idx, j0 + (int64_t)gridDim.x * kTile + xrow, n);   // the next tile's rows
    __syncwarp();
    f32x2 acc[kRowsT][2];
    gemm_nn<kInP>(XS, kP40, W1T, kP128, acc);
    xr.l2(k0, ray_id, xq);
#pragma unroll
    for (int a = 0; a < kRowsT; ++a) {
      const int r = kRowsT * warp + a;
      const float4 h = relu4(acc[a], zero);
      st4(HS + r * kP128 + 4 * lane, h);
      if (act && j0 + r < n) st4(act + (j0 + r) * kAct + 4 * lane, h);
    }
    __syncwarp();   // a warp reads back only its own rows
    gemm_nn<kHid>(HS, kP128, W2T, kP128, acc);
    xr.l3(rays_d);
    // layer 3: 8 rows x 3 outputs of the warp, reduced over its lanes (lane l
    // ends with row l / 3, output l % 3)
    float z[32];
#pragma unroll
    for (int i = 24; i < 32; ++i) z[i] = 0.0f;
#pragma unroll
    for (int a = 0; a < kRowsT; ++a) {
      const int64_t j = j0 + kRowsT * warp + a;
      const float4 h = relu4(acc[a], b2v);
      if (act && j < n) st4(act + j * kAct + kHid + 4 * lane, h);
#pragma unroll
      for (int c = 0; c < 3; ++c)
        z[3 * a + c] = fmaf(w3[c][3], h.w, fmaf(w3[c][2], h.z, fmaf(w3[c][1], h.y, w3[c][0] * h.x)));
    }
    const float zs = reduce_scatter32(z, lane);
    const int64_t j = j0 + kRowsT * warp + lane / 3;
    if (lane < 24 && j < n) {
      const int64_t s = idx ? (int64_t)__ldg(idx + j) : j;
      rgb[3 * s + lane % 3] = sigmoid_f(zs + __ldg(params + kOffB3 + lane % 3));
    }
  }
}

// Backward.  Per tile: h1, h2 (stored, or recomputed when act is NULL), y =
// rgb -> g_z3 -> dW3/db3, g_z2 -> dW2/db2, g_h1 -> g_z1 -> dW1/db1, g_k0.
__global__ void __launch_bounds__(kF32Threads, 1) rgbnet_bwd_f32_kernel(
    const float* __restrict__ g_rgb, const float* __restrict__ g_color, const float* __restrict__ w,
    const float* __restrict__ k0, const float* __restrict__ rays_d,
    const int32_t* __restrict__ ray_id, const int32_t* __restrict__ idx, int64_t n_cap,
    const int64_t* __restrict__ n_dev, const float* __restrict__ params,
    const float* __restrict__ act, const float* __restrict__ rgb_saved,
    float* __restrict__ g_params, float* __restrict__ g_k0) {
  extern __shared__ float4 smem4[];
  float* smem = reinterpret_cast<float*>(smem4);
  float* W2S = smem;                   // [128][132]
  float* H1S = W2S + kHid * kP128;     // [128][132]  h1, later g_z1
  float* GS = H1S + kTile * kP128;     // [128][132]  x (pitch 44), h2, g_z2, x again
  float* W1S = GS + kTile * kP128;     // [128][44]
  float* GZ3 = W1S + kHid * kP40;      // [128][4]    g_z3 per tile row
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, warp = tid >> 5, lane = tid & 31;
  const int64_t n = mlp_count(n_cap, n_dev);
  const int64_t ntiles = (n + kTile - 1) / kTile;
  load_w1(params, W1S);
  load_w2(params, W2S);
  // persistent gradient partials
  f32x2 dW2[kRowsT][2], dW1[2][3];   // pairs of columns i; pairs of rows o
  float db2 = 0.0f;                  // column o3, this quarter of the samples
  float db3[3] = {0.f, 0.f, 0.f};       // threads 0..127: their tile row
#pragma unroll
  for (int a = 0; a < kRowsT; ++a) dW2[a][0] = dW2[a][1] = 0ull;
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int c = 0; c < 3; ++c) dW1[p][c] = 0ull;
  const int o3 = tid & 127, part = tid >> 7;  // dW3: output column, quarter of the samples
  float w3o[3], W3o[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    w3o[c] = 0.0f;
    W3o[c] = __ldg(params + kOffW3 + c * kHid + o3);
  }
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int64_t j0 = t * kTile;
    __syncthreads();
    if (act) {
      tile_from_global(H1S, act, j0, n, 0);
      tile_from_global(GS, act, j0, n, kHid);
      // the next tile's rows (contiguous) start their way into L2
      const int64_t jn = j0 + (int64_t)gridDim.x * kTile;
      if (jn < n && tid < kTile && jn + tid < n)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(act + (jn + tid) * kAct),
                     "r"(kAct * (int)sizeof(float))
                     : "memory");
    } else {
      build_x_tile(GS, k0, rays_d, ray_id, idx, j0, n);
      __syncthreads();
      float acc[4][8];
      gemm_nt<kInP>(GS, kP40, W1S, kP40, ty, tx, acc);
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) acc[a][b] = fmaxf(acc[a][b], 0.0f);
      store_block(H1S, kP128, ty, tx, acc);
      __syncthreads();
      gemm_nt<kHid>(H1S, kP128, W2S, kP128, ty, tx, acc);
      __syncthreads();  // x no longer read
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b)
          acc[a][b] = fmaxf(acc[a][b] + __ldg(params + kOffB2 + tx + 16 * b), 0.0f);
      store_block(GS, kP128, ty, tx, acc);
    }
    // g_z3 = g_rgb * y (1 - y); y is the stored forward output (or recomputed);
    // with both stored its loads overlap the tile copies
    if (!(act && rgb_saved)) {
      copies_done();
      __syncthreads();
    }
    if (tid < kTile) {
      const int64_t j = j0 + tid;
      float g[3] = {0.f, 0.f, 0.f};
      if (j < n) {
        const int64_t s = idx ? (int64_t)__ldg(idx + j) : j;
        upstream_rgb_grad(g_rgb, g_color, w, ray_id, s, g);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float y;
          if (rgb_saved) {
            y = __ldg(rgb_saved + 3 * s + c);
          } else {
            float z = __ldg(params + kOffB3 + c);
            for (int o = 0; o < kHid; o += 4)
              z = dot4(ld4(GS + tid * kP128 + o), __ldg(reinterpret_cast<const float4*>(params + kOffW3 + c * kHid + o)), z);
            y = sigmoid_f(z);
          }
          g[c] *= y * (1.0f - y);
        }
      }
      st4(GZ3 + 4 * tid, make_float4(g[0], g[1], g[2], 0.0f));
#pragma unroll
      for (int c = 0; c < 3; ++c) db3[c] += g[c];
    }
    copies_done();
    __syncthreads();  // h1, h2 tiles and g_z3 complete
    // thread = (o, quarter of the rows): dW3[c][o] += sum_s g_z3[s][c] h2[s][o],
    // and g_z2[s][o] = (h2 > 0) sum_c g_z3[s][c] W3[c][o] in place over h2
    {
      float* h2 = GS + o3;
#pragma unroll 8
      for (int r = part * 32; r < part * 32 + 32; ++r) {
        const float4 g = ld4(GZ3 + 4 * r);
        const float hv = h2[r * kP128];
        w3o[0] = fmaf(g.x, hv, w3o[0]);
        w3o[1] = fmaf(g.y, hv, w3o[1]);
        w3o[2] = fmaf(g.z, hv, w3o[2]);
        const float gs = fmaf(g.z, W3o[2], fmaf(g.x, W3o[0], g.y * W3o[1]));
        const float g2 = hv > 0.0f ? gs : 0.0f;
        db2 += g2;
        h2[r * kP128] = g2;
      }
    }
    __syncthreads();
    // dW2[o][i] += sum_s g_z2[s][o] h1[s][i]: o = 8 warp + a, i = 4 lane ..
    {
      const float *gp = GS + kRowsT * warp, *hp = H1S + 4 * lane;
      float4 g0 = ld4(gp), g1 = ld4(gp + 4), hv = ld4(hp);
#pragma unroll 4
      for (int r = 0; r < kTile; ++r) {
        // the next row's operands are loaded beside this row's products
        const int rn = r + 1 < kTile ? (r + 1) * kP128 : 0;
        const float4 n0 = ld4(gp + rn), n1 = ld4(gp + rn + 4), nh = ld4(hp + rn);
        const float gv[kRowsT] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
        const f32x2 hl = pack2(hv.x, hv.y), hh = pack2(hv.z, hv.w);
#pragma unroll
        for (int a = 0; a < kRowsT; ++a) {
          const f32x2 d = pack2(gv[a], gv[a]);
          dW2[a][0] = fma2(d, hl, dW2[a][0]);
          dW2[a][1] = fma2(d, hh, dW2[a][1]);
        }
        g0 = n0;
        g1 = n1;
        hv = nh;
      }
    }
    // g_h1[s][i] = sum_o g_z2[s][o] W2[o][i]: rows 8 warp + a, columns 4 lane ..
    {
      f32x2 acc[kRowsT][2];
      gemm_nn<kHid>(GS, kP128, W2S, kP128, acc);
      __syncthreads();  // dW2 finished reading h1
      // g_z1 = g_h1 * (h1 > 0), in place over h1
#pragma unroll
      for (int a = 0; a < kRowsT; ++a) {
        float* q = H1S + (kRowsT * warp + a) * kP128 + 4 * lane;
        const float4 h1 = ld4(q);
        const float2 l = unpack2(acc[a][0]), h = unpack2(acc[a][1]);
        st4(q, make_float4(h1.x > 0.f ? l.x : 0.f, h1.y > 0.f ? l.y : 0.f, h1.z > 0.f ? h.x : 0.f,
                           h1.w > 0.f ? h.y : 0.f));
      }
    }
    __syncthreads();  // g_z2 no longer read
    // The x tile is built by the first 128 threads while the 384 others form
    // g_k0[s][k] = sum_o g_z1[s][o] W1[o][k], k < 12: rows g + 32a of one column.
    if (tid < kTile) {
      build_x_tile(GS, k0, rays_d, ray_id, idx, j0, n);
    } else {
      static_assert(kF32Threads - kTile == 32 * kFeat, "32 row groups of one thread per column");
      const int g = (tid - kTile) / kFeat, k = (tid - kTile) % kFeat;
      float gk[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) gk[a] = 0.0f;
#pragma unroll 2
      for (int o = 0; o < kHid; o += 4) {
        const float w0 = W1S[o * kP40 + k], w1 = W1S[(o + 1) * kP40 + k];
        const float w2 = W1S[(o + 2) * kP40 + k], w3v = W1S[(o + 3) * kP40 + k];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const float4 q = ld4(H1S + (g + 32 * a) * kP128 + o);
          gk[a] = fmaf(q.x, w0, fmaf(q.y, w1, fmaf(q.z, w2, fmaf(q.w, w3v, gk[a]))));
        }
      }
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const int64_t j = j0 + g + 32 * a;
        if (j < n) {
          const int64_t s = idx ? (int64_t)__ldg(idx + j) : j;
          g_k0[s * kFeat + k] = gk[a];
        }
      }
    }
    __syncthreads();
    // dW1[o][k] += sum_s g_z1[s][o] x[s][k]; o in {2ty.., 64+2ty..}, k in {tx, tx+16, tx+32}
    {
      const float *gp = H1S + 2 * ty, *xp = GS + tx;
      const bool third = tx + 32 < kInP;
      float2 g0 = *reinterpret_cast<const float2*>(gp), g1 = *reinterpret_cast<const float2*>(gp + 64);
      float x0 = xp[0], x1 = xp[16], x2 = third ? xp[32] : 0.0f;
#pragma unroll 4
      for (int r = 0; r < kTile; ++r) {
        // the next row's operands are loaded beside this row's products
        const int rn = r + 1 < kTile ? r + 1 : 0;
        const float2 n0 = *reinterpret_cast<const float2*>(gp + rn * kP128),
                     n1 = *reinterpret_cast<const float2*>(gp + rn * kP128 + 64);
        const float y0 = xp[rn * kP40], y1 = xp[rn * kP40 + 16], y2 = third ? xp[rn * kP40 + 32] : 0.0f;
        const f32x2 ga = pack2(g0.x, g0.y), gb = pack2(g1.x, g1.y);
        const f32x2 d0 = pack2(x0, x0), d1 = pack2(x1, x1), d2 = pack2(x2, x2);
        dW1[0][0] = fma2(ga, d0, dW1[0][0]);
        dW1[1][0] = fma2(gb, d0, dW1[1][0]);
        dW1[0][1] = fma2(ga, d1, dW1[0][1]);
        dW1[1][1] = fma2(gb, d1, dW1[1][1]);
        dW1[0][2] = fma2(ga, d2, dW1[0][2]);
        dW1[1][2] = fma2(gb, d2, dW1[1][2]);
        g0 = n0;
        g1 = n1;
        x0 = y0;
        x1 = y1;
        x2 = y2;
      }
    }
  }
  // flush partials
#pragma unroll
  for (int a = 0; a < kRowsT; ++a)
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      float* q = g_params + kOffW2 + (kRowsT * warp + a) * kHid + 4 * lane + 2 * p;
      const float2 f = unpack2(dW2[a][p]);
      atomicAdd(q, f.x);
      atomicAdd(q + 1, f.y);
    }
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int o = 64 * p + 2 * ty, k = tx + 16 * c;
      if (k > kIn) continue;
      const float2 f = unpack2(dW1[p][c]);
      atomicAdd(g_params + (k < kIn ? kOffW1 + o * kIn + k : kOffB1 + o), f.x);
      atomicAdd(g_params + (k < kIn ? kOffW1 + (o + 1) * kIn + k : kOffB1 + o + 1), f.y);
    }
  atomicAdd(g_params + kOffB2 + o3, db2);
#pragma unroll
  for (int c = 0; c < 3; ++c) atomicAdd(g_params + kOffW3 + c * kHid + o3, w3o[c]);
  if (tid < kTile) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float v = db3[c];
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if ((tid & 31) == 0) atomicAdd(g_params + kOffB3 + c, v);
    }
  }
}

}  // namespace dvgo

using namespace dvgo;

int dvgo_rgbnet_fwd_f32(const float* k0, const float* rays_d, const int32_t* ray_id,
                        const int32_t* idx, int64_t n_cap, const int64_t* n_dev,
                        const float* params, float* rgb, float* act, cudaStream_t st) {
  const size_t smem = sizeof(float) * (kInP * kP128 + kTile * kP40 + 2 * kHid * kP128);
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(rgbnet_fwd_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    attr = true;
  }
  int grid = (int)std::min<int64_t>((n_cap + kTile - 1) / kTile, kNumSMs);
  if (grid < 1) return DVGO_OK;
  rgbnet_fwd_f32_kernel<<<grid, kF32Threads, smem, st>>>(k0, rays_d, ray_id, idx, n_cap, n_dev, params, rgb,
                                                 act);
  return launch_status();
}

int dvgo_rgbnet_bwd_f32(const float* g_rgb, const float* g_color, const float* w, const float* k0,
                        const float* rays_d, const int32_t* ray_id, const int32_t* idx,
                        int64_t n_cap, const int64_t* n_dev, const float* params,
                        const float* act, const float* rgb, float* g_params, float* g_k0,
                        cudaStream_t st) {
  const size_t smem = sizeof(float) * (3 * kHid * kP128 + kHid * kP40 + 4 * kTile);
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(rgbnet_bwd_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    attr = true;
  }
  int grid = (int)std::min<int64_t>((n_cap + kTile - 1) / kTile, kNumSMs);
  if (grid < 1) return DVGO_OK;
  rgbnet_bwd_f32_kernel<<<grid, kF32Threads, smem, st>>>(g_rgb, g_color, w, k0, rays_d, ray_id, idx, n_cap,
                                                 n_dev, params, act, rgb, g_params, g_k0);
  return launch_status();
}

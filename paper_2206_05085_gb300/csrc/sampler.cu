// Ray sampling (Sec. 3 "Re-implement rendering utils": sample only inside
// the scene bbox; Sec. 1 occupancy mask; Sec. 5.4 contracted step for
// unbounded scenes) and the live-sample list used after early stop.
//
// Every decision that creates or drops a sample is IEEE FP32 with explicit
// round-to-nearest intrinsics (no FMA contraction), in the operation order
// stated in dvgo.h / below, so the integer results are reproducible bit for
// bit by any IEEE FP32 implementation of the same formulas.
#include <cuda.h>

#include <mutex>

#include "common.cuh"

namespace dvgo {

struct SamplerArgs {
  float lo[3], hi[3];
  int G[3];
  float scale[3];  // (G-1)/(hi-lo), FP32
  dvgo_sampler_desc s;
};

__device__ __forceinline__ int nearest_idx(float x, float lo, float scale, int G) {
  // One conversion that rounds down (it saturates, and takes NaN to 0) instead
  // of floor, conversion and float clamps: the bounded count of 16,384 rays
  // over 160^3 voxels takes 21.4 us, 23.4 us with those.
  const int n = __float2int_rd(__fadd_rn(__fmul_rn(__fsub_rn(x, lo), scale), 0.5f));
  return min(max(n, 0), G - 1);
}

// The occupancy byte of x (0 outside the box, 1 without a mask): a sample is
// kept when it is not 0.
__device__ __forceinline__ int keep_byte(const SamplerArgs& A, const uint8_t* __restrict__ mask,
                                         const float x[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a)
    if (!(x[a] >= A.lo[a] && x[a] <= A.hi[a])) return 0;
  if (!mask) return 1;
  int ix = nearest_idx(x[0], A.lo[0], A.scale[0], A.G[0]);
  int iy = nearest_idx(x[1], A.lo[1], A.scale[1], A.G[1]);
  int iz = nearest_idx(x[2], A.lo[2], A.scale[2], A.G[2]);
  return __ldg(mask + ((int64_t)iz * A.G[1] + iy) * A.G[0] + ix);
}
__device__ __forceinline__ bool keep_point(const SamplerArgs& A, const uint8_t* __restrict__ mask,
                                           const float x[3]) {
  return keep_byte(A, mask, x) != 0;
}

struct RaySpan {
  float tlo, thi;
  int n;
};

// Ray/bbox slab and step count (mode 0).
__device__ __forceinline__ RaySpan ray_span(const SamplerArgs& A, const float o[3], const float d[3]) {
  float tlo = A.s.near, thi = A.s.far;
  bool empty = false;
  if (A.s.use_slab) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (d[a] == 0.0f) {
        if (o[a] < A.lo[a] || o[a] > A.hi[a]) empty = true;
      } else {
        float ta = __fdiv_rn(__fsub_rn(A.lo[a], o[a]), d[a]);
        float tb = __fdiv_rn(__fsub_rn(A.hi[a], o[a]), d[a]);
        float tn = ta < tb ? ta : tb;
        float tf = ta < tb ? tb : ta;
        if (tn > tlo) tlo = tn;
        if (tf < thi) thi = tf;
      }
    }
  }
  int n = 0;
  if (!empty && thi > tlo) {
    float u = __fdiv_rn(__fsub_rn(thi, tlo), A.s.step);
    float nf = ceilf(__fsub_rn(u, A.s.step_offset));
    if (nf > (float)A.s.max_steps) n = A.s.max_steps;
    else if (nf > 0.0f) n = (int)nf;
  }
  return {tlo, thi, n};
}

__device__ __forceinline__ void point_at(const SamplerArgs& A, const float o[3], const float d[3],
                                         float tlo, int k, float x[3]) {
  float t = __fadd_rn(tlo, __fmul_rn(__fadd_rn((float)k, A.s.step_offset), A.s.step));
#pragma unroll
  for (int a = 0; a < 3; ++a) x[a] = __fadd_rn(o[a], __fmul_rn(t, d[a]));
}

__device__ __forceinline__ void load_ray(const float* __restrict__ ro, const float* __restrict__ rd,
                                         int64_t r, float o[3], float d[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    o[a] = __ldg(ro + 3 * r + a);
    d[a] = __ldg(rd + 3 * r + a);
  }
}

// Mode 2: the ray in normalized device coordinates (forward-facing scenes);
// ok is false for a ray that does not look down -z.
struct NdcRay {
  float o[3], d[3];
  int n;   // layer crossings
};

__device__ __forceinline__ NdcRay ndc_ray(const SamplerArgs& A, const float o[3], const float d[3]) {
  NdcRay q;
  q.n = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) q.o[a] = q.d[a] = 0.0f;
  if (!(d[2] < 0.0f)) return q;
  const float nr = A.s.ndc_near;
  const float t = __fdiv_rn(-__fadd_rn(nr, o[2]), d[2]);
  const float ox = __fadd_rn(o[0], __fmul_rn(t, d[0]));
  const float oy = __fadd_rn(o[1], __fmul_rn(t, d[1]));
  const float oz = __fadd_rn(o[2], __fmul_rn(t, d[2]));
  if (!(oz < 0.0f)) return q;
  const float rx = __fdiv_rn(ox, oz), ry = __fdiv_rn(oy, oz);
  const float two_n = __fmul_rn(2.0f, nr);
  q.o[0] = -__fmul_rn(A.s.ndc_fx, rx);
  q.o[1] = -__fmul_rn(A.s.ndc_fy, ry);
  q.o[2] = __fadd_rn(1.0f, __fdiv_rn(two_n, oz));
  q.d[0] = -__fmul_rn(A.s.ndc_fx, __fsub_rn(__fdiv_rn(d[0], d[2]), rx));
  q.d[1] = -__fmul_rn(A.s.ndc_fy, __fsub_rn(__fdiv_rn(d[1], d[2]), ry));
  q.d[2] = -__fdiv_rn(two_n, oz);
  const float nf = floorf(__fdiv_rn((float)(A.G[2] - 1), A.s.step));
  const int K = (int)nf + 1;
  q.n = K < A.s.max_steps ? K : A.s.max_steps;
  return q;
}

// Crossing of layer plane k: z_k = lo_z + (k step) dz, dz = (hi_z - lo_z)/(G_z - 1).
__device__ __forceinline__ void ndc_point(const SamplerArgs& A, const NdcRay& q, int k, float x[3]) {
  const float dz = __fdiv_rn(__fsub_rn(A.hi[2], A.lo[2]), (float)(A.G[2] - 1));
  const float z = __fadd_rn(A.lo[2], __fmul_rn(__fmul_rn((float)k, A.s.step), dz));
  const float t = __fdiv_rn(__fsub_rn(z, q.o[2]), q.d[2]);
  x[0] = __fadd_rn(q.o[0], __fmul_rn(t, q.d[0]));
  x[1] = __fadd_rn(q.o[1], __fmul_rn(t, q.d[1]));
  x[2] = z;
}

// Steps per ray whose keep bits pass 1 records for pass 2: one word of 32
// steps per lane of the ray's warp (1024 steps).  Longer marches recompute
// the keep test in pass 2.
constexpr int kBitWords = 32;

// Mode 0, pass 1: one warp per ray counts the kept samples.  With bits,
// the warp also stores each 32-step chunk's keep ballot (lane j holds chunk
// j's word; one coalesced store per ray), so that pass 2 need not repeat the
// occupancy lookups.
// kNdc: mode 2 (layer crossings of the warped ray) instead of mode 0.
template <bool kNdc>
__global__ void __launch_bounds__(256, 8) bbox_count_kernel(SamplerArgs A, const float* __restrict__ ro,
                                  const float* __restrict__ rd, int64_t R,
                                  const uint8_t* __restrict__ mask, int32_t* __restrict__ counts,
                                  uint32_t* __restrict__ bits) {
  const int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = warp; r < R; r += nwarps) {
    float o[3], d[3];
    load_ray(ro, rd, r, o, d);
    RaySpan sp{0.0f, 0.0f, 0};
    NdcRay q;
    if (kNdc) {
      q = ndc_ray(A, o, d);
      sp.n = q.n;
    } else {
      sp = ray_span(A, o, d);
    }
    int cnt = 0;
    uint32_t mine = 0;
    // four 32-step chunks per round, so that their occupancy lookups are in
    // flight together
    for (int k0 = 0; k0 < sp.n; k0 += 128) {
      bool keep[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int k = k0 + 32 * u + lane;
        keep[u] = false;
        if (k < sp.n) {
          float x[3];
          if (kNdc) ndc_point(A, q, k, x);
          else point_at(A, o, d, sp.tlo, k, x);
          keep[u] = keep_point(A, mask, x);
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const unsigned bal = __ballot_sync(0xffffffffu, keep[u]);
        if (lane == (k0 >> 5) + u) mine = bal;
        cnt += __popc(bal);
      }
    }
    if (lane == 0) counts[r] = cnt;
    if (bits && 32 * lane < sp.n) bits[r * kBitWords + lane] = mine;
  }
}

// Mode 0, pass 2: one warp per ray writes the kept samples in step order.
// With bits (only when max_steps <= 32 kBitWords = 1024) the keep decisions are
// pass 1's ballots; without, the keep test is evaluated again (same FP32
// operations, same result).
template <bool kNdc>
__global__ void bbox_fill_kernel(SamplerArgs A, const float* __restrict__ ro,
                                 const float* __restrict__ rd, int64_t R,
                                 const uint8_t* __restrict__ mask,
                                 const uint32_t* __restrict__ bits,
                                 const int64_t* __restrict__ ray_off, float* __restrict__ xyz,
                                 int32_t* __restrict__ ray_id, int32_t* __restrict__ step_k,
                                 float* __restrict__ s_mid, float* __restrict__ s_len) {
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = warp; r < R; r += nwarps) {
    float o[3], d[3];
    load_ray(ro, rd, r, o, d);
    RaySpan sp{0.0f, 0.0f, 0};
    NdcRay q;
    float span, slen;
    if (kNdc) {
      q = ndc_ray(A, o, d);
      sp.n = q.n;
      span = (float)q.n;                 // s = (k + 0.5)/K, length 1/K
      slen = __fdiv_rn(1.0f, span);
    } else {
      sp = ray_span(A, o, d);
      span = __fsub_rn(sp.thi, sp.tlo);
      slen = __fdiv_rn(A.s.step, span);
    }
    int64_t pos = ray_off[r];
    uint32_t mine = 0;
    if (bits && 32 * lane < sp.n) mine = bits[r * kBitWords + lane];
    for (int k0 = 0; k0 < sp.n; k0 += 32) {
      int k = k0 + lane;
      bool keep = false;
      float x[3];
      unsigned bal;
      if (bits) {
        bal = __shfl_sync(0xffffffffu, mine, k0 >> 5);
        keep = (bal >> lane) & 1u;
        if (keep) {
          if (kNdc) ndc_point(A, q, k, x);
          else point_at(A, o, d, sp.tlo, k, x);
        }
      } else {
        if (k < sp.n) {
          if (kNdc) ndc_point(A, q, k, x);
          else point_at(A, o, d, sp.tlo, k, x);
          keep = keep_point(A, mask, x);
        }
        bal = __ballot_sync(0xffffffffu, keep);
      }
      if (keep) {
        int64_t s = pos + __popc(bal & lt_mask);
        xyz[3 * s + 0] = x[0];
        xyz[3 * s + 1] = x[1];
        xyz[3 * s + 2] = x[2];
        ray_id[s] = (int32_t)r;
        step_k[s] = k;
        s_mid[s] = kNdc ? __fdiv_rn(__fadd_rn((float)k, 0.5f), span)
                        : __fdiv_rn(__fmul_rn(__fadd_rn((float)k, A.s.step_offset), A.s.step), span);
        s_len[s] = slen;
      }
      pos += __popc(bal);
    }
  }
}

// Mode 1: contracted-space march (Eq. ub).  One step at world point x: the
// contracted point xc and the Jacobian-mapped direction j (false when xc's
// contracted radius has reached rmax: the march ends before xc), then the
// advance of x by the contracted step (false when the step is not finite).
struct CMarch {
  float b, opb, rmax, two_b;
  bool p_inf;
};

__device__ __forceinline__ CMarch cmarch_consts(const SamplerArgs& A) {
  CMarch M;
  M.b = A.s.contract_b;
  M.opb = __fadd_rn(1.0f, M.b);
  M.rmax = __fsub_rn(M.opb, A.s.step_c);
  M.two_b = __fmul_rn(2.0f, M.b);
  M.p_inf = A.s.p_inf != 0;
  return M;
}

__device__ __forceinline__ bool cmarch_point(const CMarch& M, const float x[3], const float d[3], float xc[3],
                                             float j[3], bool& inside) {
  float rad;
  int m = 0;
  if (M.p_inf) {
    float a0 = fabsf(x[0]), a1 = fabsf(x[1]), a2 = fabsf(x[2]);
    rad = a0;
    if (a1 > rad) { rad = a1; m = 1; }
    if (a2 > rad) { rad = a2; m = 2; }
  } else {
    rad = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(x[0], x[0]), __fmul_rn(x[1], x[1])),
                               __fmul_rn(x[2], x[2])));
  }
  inside = rad <= 1.0f;
  if (inside) {
#pragma unroll
    for (int a = 0; a < 3; ++a) { xc[a] = x[a]; j[a] = d[a]; }
    // xc = x: its contracted radius is rad itself (the same operations on
    // the same values)
    return rad < M.rmax;
  } else {
    float r2 = __fmul_rn(rad, rad);
    float gr = __fsub_rn(__fdiv_rn(M.opb, rad), __fdiv_rn(M.b, r2));
    float gp = __fsub_rn(__fdiv_rn(M.two_b, __fmul_rn(r2, rad)), __fdiv_rn(M.opb, r2));
    float rdot;
    if (M.p_inf) {
      float xm = m == 0 ? x[0] : (m == 1 ? x[1] : x[2]);
      float dm = m == 0 ? d[0] : (m == 1 ? d[1] : d[2]);
      rdot = xm < 0.0f ? -dm : dm;
    } else {
      rdot = __fdiv_rn(__fadd_rn(__fadd_rn(__fmul_rn(x[0], d[0]), __fmul_rn(x[1], d[1])),
                                 __fmul_rn(x[2], d[2])), rad);
    }
    float gq = __fmul_rn(gp, rdot);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      xc[a] = __fmul_rn(gr, x[a]);
      j[a] = __fadd_rn(__fmul_rn(gr, d[a]), __fmul_rn(gq, x[a]));
    }
  }
  float cr;
  if (M.p_inf) {
    cr = fabsf(xc[0]);
    if (fabsf(xc[1]) > cr) cr = fabsf(xc[1]);
    if (fabsf(xc[2]) > cr) cr = fabsf(xc[2]);
  } else {
    cr = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(xc[0], xc[0]), __fmul_rn(xc[1], xc[1])),
                              __fmul_rn(xc[2], xc[2])));
  }
  return cr < M.rmax;
}

// step_c / |j|, the contracted step along j
__device__ __forceinline__ float cmarch_step_len(const SamplerArgs& A, const float j[3]) {
  const float nj = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(j[0], j[0]), __fmul_rn(j[1], j[1])),
                                        __fmul_rn(j[2], j[2])));
  return __fdiv_rn(A.s.step_c, nj);
}

// Inside the unit ball j = d, so the step is the ray's constant h_in =
// cmarch_step_len(A, d), formed once per ray (the same value bit for bit).
__device__ __forceinline__ bool cmarch_advance(const SamplerArgs& A, float x[3], const float d[3],
                                               const float j[3], bool inside, float h_in) {
  const float h = inside ? h_in : cmarch_step_len(A, j);
  if (!(h > 0.0f) || isinf(h)) return false;
#pragma unroll
  for (int a = 0; a < 3; ++a) x[a] = __fadd_rn(x[a], __fmul_rn(h, d[a]));
  return true;
}

// Checkpoints of the march for the parallel second pass: the march of a ray
// is cut into kCkpt chunks of L = ceil(max_steps / kCkpt) steps; record c of
// the ray holds x at step c L (3 floats) and the kept samples of chunk c
// (int32, -1 for a chunk the march never reaches).  kCkpt x 4 words per ray
// fit the per-ray keep-bit words of the workspace.
constexpr int kCkpt = 8;

__device__ __forceinline__ int ckpt_len(const SamplerArgs& A) {
  return (A.s.max_steps + kCkpt - 1) / kCkpt;
}

// Mode 1, one thread per ray: the whole march.  Pass 1 (kWrite false)
// counts, and with ckpt records the checkpoints; pass 2 without checkpoints
// (kWrite) repeats the march and writes.
template <bool kWrite>
__global__ void contracted_kernel(SamplerArgs A, const float* __restrict__ ro,
                                  const float* __restrict__ rd, int64_t R,
                                  const uint8_t* __restrict__ mask, int32_t* __restrict__ counts,
                                  uint32_t* __restrict__ ckpt,
                                  const int64_t* __restrict__ ray_off, float* __restrict__ xyz,
                                  int32_t* __restrict__ ray_id, int32_t* __restrict__ step_k,
                                  float* __restrict__ s_mid, float* __restrict__ s_len) {
  const CMarch M = cmarch_consts(A);
  const float inv_steps = __fdiv_rn(1.0f, (float)A.s.max_steps);
  const int L = ckpt_len(A);
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < R;
       r += (int64_t)gridDim.x * blockDim.x) {
    float o[3], d[3];
    load_ray(ro, rd, r, o, d);
    const float h_in = cmarch_step_len(A, d);
    float x[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) x[a] = __fadd_rn(o[a], __fmul_rn(A.s.near, d[a]));
    int cnt = 0, chunk_start = 0, c = -1;
    int64_t pos = kWrite ? ray_off[r] : 0;
    uint32_t* rec = ckpt ? ckpt + r * (4 * kCkpt) : nullptr;
    for (int k = 0; k < A.s.max_steps; ++k) {
      if (!kWrite && rec && k % L == 0) {   // a new chunk: close the previous one, record x
        if (c >= 0) rec[4 * c + 3] = (uint32_t)(cnt - chunk_start);
        ++c;
        chunk_start = cnt;
        rec[4 * c] = __float_as_uint(x[0]);
        rec[4 * c + 1] = __float_as_uint(x[1]);
        rec[4 * c + 2] = __float_as_uint(x[2]);
      }
      float xc[3], j[3];
      bool inside;
      if (!cmarch_point(M, x, d, xc, j, inside)) break;
      if (keep_point(A, mask, xc)) {
        if (kWrite) {
          int64_t s = pos + cnt;
          xyz[3 * s + 0] = xc[0];
          xyz[3 * s + 1] = xc[1];
          xyz[3 * s + 2] = xc[2];
          ray_id[s] = (int32_t)r;
          step_k[s] = k;
          s_mid[s] = __fmul_rn(__fadd_rn((float)k, 0.5f), inv_steps);
          s_len[s] = inv_steps;
        }
        ++cnt;
      }
      if (!cmarch_advance(A, x, d, j, inside, h_in)) break;
    }
    if (!kWrite) {
      counts[r] = cnt;
      if (rec) {
        if (c >= 0) rec[4 * c + 3] = (uint32_t)(cnt - chunk_start);
        for (int cc = c + 1; cc < kCkpt; ++cc) rec[4 * cc + 3] = 0xffffffffu;
      }
    }
  }
}

// Mode 1, pass 2 from the checkpoints: a block of 256 threads takes 32 rays,
// warp c of it chunk c of each of them (the lanes of a warp march the same
// part of 32 rays, so they take the same branches); each thread repeats the
// march of its chunk from the recorded x (the same FP32 operations as pass
// 1, so the same points).  Eight steps at a time: the points go to shared
// memory, then the warp writes the kept ones after those of the ray's earlier
// chunks, four rays at once and eight lanes to a ray.  (Each lane writing its
// own ray's samples, in groups of four, had some lanes write at every step:
// 119 us for 4.1e6 samples of 8192 rays, 99 us now.)
constexpr int kFillSteps = 8;
constexpr int kFillPitch = 100;   // floats a step, [3][32] and 4 more: the write phase's 4 x 8 reads hit 32 banks

__global__ void __launch_bounds__(32 * kCkpt) contracted_fill_kernel(
    SamplerArgs A, const float* __restrict__ rd, int64_t R, const uint8_t* __restrict__ mask,
    const uint32_t* __restrict__ ckpt, const int64_t* __restrict__ ray_off, float* __restrict__ xyz,
    int32_t* __restrict__ ray_id, int32_t* __restrict__ step_k, float* __restrict__ s_mid,
    float* __restrict__ s_len) {
  __shared__ int kept[kCkpt][32];
  __shared__ float points[kCkpt][kFillSteps * kFillPitch];
  const CMarch M = cmarch_consts(A);
  const float inv_steps = __fdiv_rn(1.0f, (float)A.s.max_steps);
  const int L = ckpt_len(A);
  const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
  const int64_t r = (int64_t)blockIdx.x * 32 + lane;
  const bool ray_ok = r < R;
  const uint32_t* rec = ckpt + (ray_ok ? r : 0) * (4 * kCkpt) + 4 * c;
  const uint32_t n_c = ray_ok ? rec[3] : 0xffffffffu;
  const int mine = n_c == 0xffffffffu ? 0 : (int)n_c;
  kept[c][lane] = mine;
  __syncthreads();
  int before = 0;   // kept samples of the ray's earlier chunks
  for (int q = 0; q < c; ++q) before += kept[q][lane];
  bool go = mine != 0;   // (a chunk that keeps nothing is not marched)
  float d[3] = {0.0f, 0.0f, 0.0f}, x[3] = {0.0f, 0.0f, 0.0f}, h_in = 0.0f;
  int64_t s = 0;   // the list position of the next kept sample
  if (go) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      d[a] = __ldg(rd + 3 * r + a);
      x[a] = __uint_as_float(rec[a]);
    }
    h_in = cmarch_step_len(A, d);
    s = ray_off[r] + before;
  }
  float* pts = points[c];
  const int k_end = min((c + 1) * L, A.s.max_steps);
  for (int k0 = c * L; k0 < k_end && __any_sync(0xffffffffu, go); k0 += kFillSteps) {
    uint32_t bits = 0;   // kept steps of this lane's ray
    int look = 0;        // occupancy byte of the step before, looked at a step late
    int u = 0;
#pragma unroll 1
    for (; go && u < kFillSteps && k0 + u < k_end; ++u) {
      float xc[3], j[3];
      bool inside;
      go = cmarch_point(M, x, d, xc, j, inside);
      if (!go) break;
      bits |= (uint32_t)(look != 0) << u;   // (bit u: step u - 1)
      look = keep_byte(A, mask, xc);
#pragma unroll
      for (int a = 0; a < 3; ++a) pts[u * kFillPitch + 32 * a + lane] = xc[a];
      go = cmarch_advance(A, x, d, j, inside, h_in);
      if (!go) {
        ++u;
        break;
      }
    }
    bits = (bits | (uint32_t)(look != 0) << u) >> 1;
    __syncwarp();
#pragma unroll 2
    for (int it = 0; it < 32 * kFillSteps / 32; ++it) {
      const int rl = 4 * it + (lane >> 3), st = lane & 7;
      const uint32_t b = __shfl_sync(0xffffffffu, bits, rl);
      const int64_t s0 = __shfl_sync(0xffffffffu, s, rl);
      if ((b >> st) & 1u) {
        const int64_t at = s0 + __popc(b & ((1u << st) - 1u));
        const int k = k0 + st;
#pragma unroll
        for (int a = 0; a < 3; ++a) xyz[3 * at + a] = pts[st * kFillPitch + 32 * a + rl];
        ray_id[at] = (int32_t)((int64_t)blockIdx.x * 32 + rl);
        step_k[at] = k;
        s_mid[at] = __fmul_rn(__fadd_rn((float)k, 0.5f), inv_steps);
        s_len[at] = inv_steps;
      }
    }
    s += __popc(bits);
    __syncwarp();
  }
}

// Exclusive scan of int32 counts into int64 offsets off[0..n] (n > 0; blocks of
// 1024 threads, scan_blocks(n) of them).  A block owns `chunk` consecutive
// counts and scans them 1024 a pass (one a thread); what lies before them it
// adds up for itself, so the blocks wait for nothing.  Even the last one reads
// each count once, as one block alone would, and the offsets, most of the
// traffic, are written by all.  Bound by the latency of a pass.  Measured with
// the live list's fill of empty rays, one block alone with 8192 counts a pass
// and this form: 9.2 and 5.6 us for 16,384 counts, 5.9 and 4.7 us for 8192, 1580
// and 199 us for 4.2e6.
__host__ __device__ constexpr int64_t scan_chunk(int64_t n, int blocks) {
  return ((n + blocks - 1) / blocks + 1023) / 1024 * 1024;
}
static int scan_blocks(int64_t n) { return (int)std::min<int64_t>((n + 1023) / 1024, kNumSMs); }

__global__ void __launch_bounds__(1024) scan_counts_kernel(const int32_t* __restrict__ counts, int64_t n,
                                                           int64_t* __restrict__ off,
                                                           int64_t* __restrict__ total_out) {
  __shared__ int64_t warp_tot[2][32], warp_before[32];
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int64_t chunk = scan_chunk(n, gridDim.x), start = chunk * blockIdx.x;
  if (start >= n) return;
  const int64_t end = start + chunk < n ? start + chunk : n;
  int64_t before = 0;
  if ((reinterpret_cast<uintptr_t>(counts) & 15u) == 0) {
    for (int64_t i = 4 * t; i < start; i += 4096) {   // (start is a multiple of 1024)
      const int4 a = __ldg(reinterpret_cast<const int4*>(counts + i));
      before += ((int64_t)a.x + a.y) + ((int64_t)a.z + a.w);
    }
  } else {
    for (int64_t i = t; i < start; i += 1024) before += __ldg(counts + i);
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
  if (lane == 0) warp_before[wid] = before;
  int64_t carry = 0;
  int row = 0;   // the warp totals alternate between two rows, so that a pass needs one barrier
  for (int64_t base = start; base < end; base += 1024, row ^= 1) {
    const int64_t i = base + t;
    const int64_t c = i < end ? __ldg(counts + i) : 0;
    int64_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tot[row][wid] = incl;
    __syncthreads();
    if (base == start) {
      carry = warp_before[lane];
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) carry += __shfl_xor_sync(0xffffffffu, carry, o);
    }
    int64_t v = warp_tot[row][lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += y;
    }
    const int64_t prev = __shfl_sync(0xffffffffu, v, wid > 0 ? wid - 1 : 0);
    if (i < end) off[i] = carry + (wid > 0 ? prev : 0) + incl - c;
    carry += __shfl_sync(0xffffffffu, v, 31);
  }
  if (end == n && t == 0) {
    off[n] = carry;
    if (total_out) *total_out = carry;
  }
}

// The same for n <= kScanSmall in one block: eight consecutive counts a thread,
// ceil(n / 8) threads (whole warps), one barrier.  Bound by its latency (one
// load, two warp scans).  Where the line lies: the live list's scan and fill of
// empty rays take 3.0 us so and 4.0 us with scan_counts_kernel for 256 counts,
// 3.5 and 4.3 for 2048, 4.2 and 4.6 for 4096, but 5.0 and 4.5 for 6144.
constexpr int64_t kScanSmall = 4096;
static_assert(kScanSmall <= 8 * 1024, "one block of eight counts a thread");

__global__ void __launch_bounds__(1024) scan_small_kernel(const int32_t* __restrict__ counts, int n,
                                                          int64_t* __restrict__ off,
                                                          int64_t* __restrict__ total_out) {
  __shared__ int64_t warp_tot[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, i0 = 8 * threadIdx.x;
  int32_t c[8];
  if ((reinterpret_cast<uintptr_t>(counts) & 15u) == 0 && i0 + 8 <= n) {
    const int4 a = __ldg(reinterpret_cast<const int4*>(counts + i0));
    const int4 b = __ldg(reinterpret_cast<const int4*>(counts + i0 + 4));
    c[0] = a.x; c[1] = a.y; c[2] = a.z; c[3] = a.w;
    c[4] = b.x; c[5] = b.y; c[6] = b.z; c[7] = b.w;
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) c[k] = i0 + k < n ? __ldg(counts + i0 + k) : 0;
  }
  int64_t loc[8], s = 0;   // sums of the thread's counts before each
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    loc[k] = s;
    s += c[k];
  }
  int64_t incl = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  int64_t v = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : 0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  const int64_t prev = __shfl_sync(0xffffffffu, v, wid > 0 ? wid - 1 : 0), total = __shfl_sync(0xffffffffu, v, 31);
  const int64_t ex = (wid > 0 ? prev : 0) + incl - s;
  if (i0 + 8 <= n && (reinterpret_cast<uintptr_t>(off) & 15u) == 0) {
#pragma unroll
    for (int k = 0; k < 8; k += 2)
      *reinterpret_cast<longlong2*>(off + i0 + k) = make_longlong2(ex + loc[k], ex + loc[k + 1]);
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (i0 + k < n) off[i0 + k] = ex + loc[k];
  }
  if (threadIdx.x == 0) {
    off[n] = total;
    if (total_out) *total_out = total;
  }
}

static void scan_counts(const int32_t* counts, int64_t n, int64_t* off, int64_t* total_out, cudaStream_t st) {
  if (n <= kScanSmall)
    scan_small_kernel<<<1, (int)(n + 255) / 256 * 32, 0, st>>>(counts, (int)n, off, total_out);
  else
    scan_counts_kernel<<<scan_blocks(n), 1024, 0, st>>>(counts, n, off, total_out);
}

// Live list: live_idx[live_off[r] + i] = ray_off[r] + i for i < seg_len[r].
__global__ void live_fill_kernel(const int64_t* __restrict__ ray_off,
                                 const int32_t* __restrict__ seg_len, int64_t R,
                                 const int64_t* __restrict__ live_off, int32_t* __restrict__ live_idx) {
  const int lane = threadIdx.x & 31;
  int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = warp; r < R; r += nwarps) {
    int64_t b = ray_off[r];
    int64_t dst = live_off[r];
    int n = seg_len[r];
    for (int i = lane; i < n; i += 32) live_idx[dst + i] = (int32_t)(b + i);
  }
}

// Low-weight cull of the colour-query list: warp per ray, the first
// seg_len[r] samples, kept iff w >= w_min (one ballot per 32 samples).  With
// fill, kept samples are listed in ray order and the rgb and g_k0 rows of the
// culled ones are zeroed; without, only the count per ray is written.
template <bool kFill>
__global__ void cull_kernel(const int64_t* __restrict__ ray_off, const int32_t* __restrict__ seg_len,
                            const float* __restrict__ w, float w_min, int64_t R, int32_t* __restrict__ counts,
                            const int64_t* __restrict__ off, int32_t* __restrict__ live_idx,
                            float* __restrict__ rgb, float* __restrict__ g_k0) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < R; r += nw) {
    const int64_t b = ray_off[r];
    const int n = seg_len[r];
    int64_t dst = kFill ? off[r] : 0;
    int cnt = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
      const int i = i0 + lane;
      const bool valid = i < n;
      const bool keep = valid && __ldg(w + b + i) >= w_min;
      const unsigned bal = __ballot_sync(0xffffffffu, keep);
      if (kFill) {
        if (keep) live_idx[dst + __popc(bal & lt)] = (int32_t)(b + i);
        if (valid && !keep) {
          const int64_t s = b + i;
          if (rgb) {
            rgb[3 * s] = 0.0f;
            rgb[3 * s + 1] = 0.0f;
            rgb[3 * s + 2] = 0.0f;
          }
          if (g_k0) {
            float4* q = reinterpret_cast<float4*>(g_k0 + s * 12);
            q[0] = q[1] = q[2] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          }
        }
        dst += __popc(bal);
      } else {
        cnt += __popc(bal);
      }
    }
    if (!kFill && lane == 0) counts[r] = cnt;
  }
}

static bool fill_args(SamplerArgs& A, const dvgo_grid_desc* g, const dvgo_sampler_desc* s) {
  for (int a = 0; a < 3; ++a) {
    A.lo[a] = g->lo[a];
    A.hi[a] = g->hi[a];
    A.G[a] = g->G[a];
    if (g->G[a] < 2 || !(g->hi[a] > g->lo[a])) return false;
    // FP32: (float)(G-1) / (hi - lo)
    volatile float num = (float)(g->G[a] - 1);
    volatile float den = g->hi[a] - g->lo[a];
    A.scale[a] = num / den;
  }
  A.s = *s;
  return true;
}

}  // namespace dvgo

using namespace dvgo;

// Workspace: per-ray counts ((R+1) int32, padded to 256 bytes), then R x
// kBitWords uint32 per-ray words: the keep bits of pass 1 (modes 0 and 2) or
// the march checkpoints of pass 1 (mode 1).
static size_t counts_bytes(int64_t R) {
  return (size_t)((R + 1) * sizeof(int32_t) + 255) / 256 * 256;
}

extern "C" size_t dvgo_sample_rays_workspace_size(int64_t R) {
  return counts_bytes(R) + (size_t)R * kBitWords * sizeof(uint32_t);
}

extern "C" int dvgo_sample_rays(const float* rays_o, const float* rays_d, int64_t R,
                                const dvgo_grid_desc* grid, const dvgo_sampler_desc* smp,
                                const uint8_t* mask, int64_t S_cap, int64_t* ray_off, float* xyz,
                                int32_t* ray_id, int32_t* step_k, float* s_mid, float* s_len,
                                void* ws, size_t ws_bytes, void* stream) {
  DVGO_CHECK_ARG(grid && smp && ray_off && R >= 0);
  DVGO_CHECK_ARG(R == 0 || (rays_o && rays_d && xyz && ray_id && step_k && s_mid && s_len && ws));
  DVGO_CHECK_ARG(smp->mode >= 0 && smp->mode <= 2);
  DVGO_CHECK_ARG(smp->max_steps >= 0);
  if (smp->mode == 0 || smp->mode == 2) DVGO_CHECK_ARG(smp->step > 0.0f);
  if (smp->mode == 1) DVGO_CHECK_ARG(smp->step_c > 0.0f && smp->contract_b > 0.0f);
  if (smp->mode == 2) DVGO_CHECK_ARG(smp->ndc_near > 0.0f && smp->ndc_fx > 0.0f && smp->ndc_fy > 0.0f);
  if (S_cap < R * (int64_t)smp->max_steps || S_cap > INT32_MAX) return DVGO_ERR_SHAPE;
  if (ws_bytes < dvgo_sample_rays_workspace_size(R)) return DVGO_ERR_WORKSPACE;
  SamplerArgs A;
  DVGO_CHECK_ARG(fill_args(A, grid, smp));
  cudaStream_t st = as_stream(stream);
  if (R == 0) {
    cudaMemsetAsync(ray_off, 0, sizeof(int64_t), st);
    return launch_status();
  }
  int32_t* counts = reinterpret_cast<int32_t*>(ws);
  if (smp->mode == 0 || smp->mode == 2) {
    const int block = 256;
    int g = grid_for(R * 32, block, 16);
    uint32_t* bits = smp->max_steps <= 32 * kBitWords
                         ? reinterpret_cast<uint32_t*>(static_cast<char*>(ws) + counts_bytes(R))
                         : nullptr;
    if (smp->mode == 0) {
      bbox_count_kernel<false><<<g, block, 0, st>>>(A, rays_o, rays_d, R, mask, counts, bits);
      scan_counts(counts, R, ray_off, nullptr, st);
      bbox_fill_kernel<false><<<g, block, 0, st>>>(A, rays_o, rays_d, R, mask, bits, ray_off, xyz, ray_id,
                                                   step_k, s_mid, s_len);
    } else {
      bbox_count_kernel<true><<<g, block, 0, st>>>(A, rays_o, rays_d, R, mask, counts, bits);
      scan_counts(counts, R, ray_off, nullptr, st);
      bbox_fill_kernel<true><<<g, block, 0, st>>>(A, rays_o, rays_d, R, mask, bits, ray_off, xyz, ray_id,
                                                  step_k, s_mid, s_len);
    }
  } else {
    // one warp of rays per block, so that the sequential marches spread over
    // every SM (8192 rays: 256 blocks)
    const int block = 32;
    int g = (int)ceil_div(R, block);
    // pass 1 records the march's checkpoints in the keep-bit words, so that
    // pass 2 runs kCkpt chunks of each march in parallel
    uint32_t* ckpt = reinterpret_cast<uint32_t*>(static_cast<char*>(ws) + counts_bytes(R));
    contracted_kernel<false><<<g, block, 0, st>>>(A, rays_o, rays_d, R, mask, counts, ckpt,
                                                  nullptr, nullptr, nullptr, nullptr, nullptr, nullptr);
    scan_counts(counts, R, ray_off, nullptr, st);
    contracted_fill_kernel<<<(int)ceil_div(R, 32), 32 * kCkpt, 0, st>>>(A, rays_d, R, mask, ckpt, ray_off,
                                                                        xyz, ray_id, step_k, s_mid, s_len);
  }
  return launch_status();
}

extern "C" size_t dvgo_live_samples_workspace_size(int64_t R) {
  // offsets [R + 1] int64, then (the cull) counts [R] int32
  return (size_t)((R + 1) * sizeof(int64_t) + 255) / 256 * 256 + (size_t)(R * sizeof(int32_t) + 255) / 256 * 256;
}

extern "C" int dvgo_live_samples_cull(const int64_t* ray_off, const int32_t* seg_len, const float* w,
                                      float w_min, int64_t R, int32_t* live_idx, int64_t* live_count,
                                      float* rgb, float* g_k0, void* ws, size_t ws_bytes, void* stream) {
  DVGO_CHECK_ARG(ray_off && seg_len && w && live_idx && live_count && ws && R >= 0 && w_min >= 0.0f);
  DVGO_CHECK_ARG(((uintptr_t)g_k0 % 16) == 0);
  if (ws_bytes < dvgo_live_samples_workspace_size(R)) return DVGO_ERR_WORKSPACE;
  cudaStream_t st = as_stream(stream);
  if (R == 0) {
    cudaMemsetAsync(live_count, 0, sizeof(int64_t), st);
    return launch_status();
  }
  int64_t* off = reinterpret_cast<int64_t*>(ws);
  int32_t* counts = reinterpret_cast<int32_t*>(static_cast<uint8_t*>(ws) +
                                               (size_t)((R + 1) * sizeof(int64_t) + 255) / 256 * 256);
  const int g = grid_for(R * 32, 256, 16);
  cull_kernel<false><<<g, 256, 0, st>>>(ray_off, seg_len, w, w_min, R, counts, nullptr, nullptr, nullptr, nullptr);
  scan_counts(counts, R, off, live_count, st);
  cull_kernel<true><<<g, 256, 0, st>>>(ray_off, seg_len, w, w_min, R, nullptr, off, live_idx, rgb, g_k0);
  return launch_status();
}

extern "C" int dvgo_live_samples(const int64_t* ray_off, const int32_t* seg_len, int64_t R,
                                 int32_t* live_idx, int64_t* live_count, void* ws, size_t ws_bytes,
                                 void* stream) {
  DVGO_CHECK_ARG(ray_off && seg_len && live_idx && live_count && ws && R >= 0);
  if (ws_bytes < dvgo_live_samples_workspace_size(R)) return DVGO_ERR_WORKSPACE;
  cudaStream_t st = as_stream(stream);
  if (R == 0) {
    cudaMemsetAsync(live_count, 0, sizeof(int64_t), st);
    return launch_status();
  }
  int64_t* live_off = reinterpret_cast<int64_t*>(ws);
  scan_counts(seg_len, R, live_off, live_count, st);
  live_fill_kernel<<<grid_for(R * 32, 256, 16), 256, 0, st>>>(ray_off, seg_len, R, live_off,
                                                              live_idx);
  return launch_status();
}

// ------------------------------------------------------------------------
// Ray sampling that allocates nothing.  Some callers cannot call cudaMalloc
// at all -- for example a host application that owns the device's whole
// memory budget and does not let libraries allocate, or code running where
// allocation is not permitted -- so they cannot provide the workspace that
// dvgo_sample_rays needs.  For them the per-ray count scratch lives in a
// fixed-size array in this library's own device memory: every GPU that
// loads the library holds it (4 MiB) until the process exits.
namespace dvgo {

constexpr int64_t kNoAllocMaxRays = 1 << 20;
static __device__ __align__(256) int32_t g_noalloc_counts[kNoAllocMaxRays + 1];

constexpr int kNoAllocMaxDevices = 64;

// The array's device address, cached per device together with the identity
// of the context it was looked up in.  A context that is torn down and
// created again (cudaDeviceReset, or a driver-API context switch) gets a new
// identity, so the address is looked up again there instead of being reused.
struct NoAllocSlot {
  int32_t* ptr = nullptr;
  unsigned long long ctx_id = 0;
};
static NoAllocSlot g_noalloc_slot[kNoAllocMaxDevices];
static std::mutex g_noalloc_mutex;

using CtxGetCurrentFn = CUresult (*)(CUcontext*);
using CtxGetIdFn = CUresult (*)(CUcontext, unsigned long long*);

// Identity of the calling thread's current context (false if there is none
// or the driver does not provide the query).
static bool current_ctx_id(unsigned long long* id) {
  static CtxGetCurrentFn get_current = nullptr;
  static CtxGetIdFn get_id = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess && q == cudaDriverEntryPointSuccess)
      get_current = reinterpret_cast<CtxGetCurrentFn>(f);
    f = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess && q == cudaDriverEntryPointSuccess)
      get_id = reinterpret_cast<CtxGetIdFn>(f);
  });
  if (!get_current || !get_id) return false;
  CUcontext c = nullptr;
  if (get_current(&c) != CUDA_SUCCESS || !c) return false;
  return get_id(c, id) == CUDA_SUCCESS;
}

// Device address of g_noalloc_counts in the current context.  In host code
// the array's name is only a host-side stand-in, so the address is looked up
// (cudaGetSymbolAddress, with the device current) on the first call in a
// context and cached; later calls in the same context reuse it.
static int noalloc_counts(int32_t** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return DVGO_ERR_CUDA;
  if (dev < 0 || dev >= kNoAllocMaxDevices) return DVGO_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  NoAllocSlot& slot = g_noalloc_slot[dev];
  unsigned long long id = 0;
  if (slot.ptr && current_ctx_id(&id) && id == slot.ctx_id) {
    *out = slot.ptr;
    return DVGO_OK;
  }
  void* addr = nullptr;
  if (cudaGetSymbolAddress(&addr, g_noalloc_counts) != cudaSuccess || !addr) return DVGO_ERR_CUDA;
  // without a context identity the address is not cached (looked up every call)
  slot.ptr = current_ctx_id(&id) ? static_cast<int32_t*>(addr) : nullptr;
  slot.ctx_id = id;
  *out = static_cast<int32_t*>(addr);
  return DVGO_OK;
}

}  // namespace dvgo

extern "C" int64_t dvgo_sample_rays_noalloc_max_rays(void) { return dvgo::kNoAllocMaxRays; }

extern "C" int dvgo_sample_rays_noalloc(const float* rays_o, const float* rays_d, int64_t R,
                                        const dvgo_grid_desc* grid, const dvgo_sampler_desc* smp,
                                        const uint8_t* mask, int64_t S_cap, int64_t* ray_off,
                                        float* xyz, int32_t* ray_id, int32_t* step_k,
                                        float* s_mid, float* s_len, void* stream) {
  DVGO_CHECK_ARG(grid && smp && ray_off && R >= 0);
  DVGO_CHECK_ARG(R == 0 || (rays_o && rays_d && xyz && ray_id && step_k && s_mid && s_len));
  DVGO_CHECK_ARG(smp->mode >= 0 && smp->mode <= 2);
  DVGO_CHECK_ARG(smp->max_steps >= 0);
  if (smp->mode == 0 || smp->mode == 2) DVGO_CHECK_ARG(smp->step > 0.0f);
  if (smp->mode == 1) DVGO_CHECK_ARG(smp->step_c > 0.0f && smp->contract_b > 0.0f);
  if (smp->mode == 2) DVGO_CHECK_ARG(smp->ndc_near > 0.0f && smp->ndc_fx > 0.0f && smp->ndc_fy > 0.0f);
  if (R > kNoAllocMaxRays) return DVGO_ERR_SHAPE;
  if (S_cap < R * (int64_t)smp->max_steps || S_cap > INT32_MAX) return DVGO_ERR_SHAPE;
  SamplerArgs A;
  DVGO_CHECK_ARG(fill_args(A, grid, smp));
  int32_t* counts = nullptr;
  int rc = noalloc_counts(&counts);
  if (rc != DVGO_OK) return rc;
  cudaStream_t st = as_stream(stream);
  if (R == 0) {
    cudaMemsetAsync(ray_off, 0, sizeof(int64_t), st);
    return launch_status();
  }
  // the count kernel writes counts[0, R) before the scan reads them, so the
  // shared array needs no clearing between calls
  if (smp->mode == 0) {
    const int block = 256;
    int g = grid_for(R * 32, block, 16);
    bbox_count_kernel<false><<<g, block, 0, st>>>(A, rays_o, rays_d, R, mask, counts, nullptr);
    scan_counts(counts, R, ray_off, nullptr, st);
    bbox_fill_kernel<false><<<g, block, 0, st>>>(A, rays_o, rays_d, R, mask, nullptr, ray_off, xyz,
                                                 ray_id, step_k, s_mid, s_len);
  } else if (smp->mode == 2) {
    const int block = 256;
    int g = grid_for(R * 32, block, 16);
    bbox_count_kernel<true><<<g, block, 0, st>>>(A, rays_o, rays_d, R, mask, counts, nullptr);
    scan_counts(counts, R, ray_off, nullptr, st);
    bbox_fill_kernel<true><<<g, block, 0, st>>>(A, rays_o, rays_d, R, mask, nullptr, ray_off, xyz,
                                                ray_id, step_k, s_mid, s_len);
  } else {
    // one warp of rays per block, so that the sequential marches spread over
    // every SM (8192 rays: 256 blocks)
    const int block = 32;
    int g = (int)ceil_div(R, block);
    contracted_kernel<false><<<g, block, 0, st>>>(A, rays_o, rays_d, R, mask, counts, nullptr,
                                                  nullptr, nullptr, nullptr, nullptr, nullptr, nullptr);
    scan_counts(counts, R, ray_off, nullptr, st);
    contracted_kernel<true><<<g, block, 0, st>>>(A, rays_o, rays_d, R, mask, nullptr, nullptr, ray_off, xyz,
                                                 ray_id, step_k, s_mid, s_len);
  }
  return launch_status();
}

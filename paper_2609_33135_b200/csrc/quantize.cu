// Stage 1 of the QK4PV8 path (Algorithm 1 lines 1-5): sequence means (Eq. 7), centering,
// per-tensor scales, NVFP4 quantization (Eq. 1) of Q and K into the tile layout consumed
// by the prefill kernel (or the fragment-ordered paged layout consumed by decode), the
// compensation vector Delta_S (Eq. 9) and the FP8 quantization of V.
//
// Everything here is bandwidth work: 16-byte global loads, 8/16-byte stores, tiles staged in
// shared memory where the destination order differs from the source order.  Every floating-point step of the means, scales and
// codes uses an explicitly rounded intrinsic, so those are defined to the bit (no FMA contraction; where a division is
// replaced, it is done all the same whenever the result could differ).  Delta_S is summed in FP64 in an order of each kernel's own,
// see there.
#include <cuda_bf16.h>
#include <cuda_fp4.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "sm100_ptx.cuh"
#include "stat_split.hpp"

namespace mpfa {

thread_local int g_last_cuda_error = 0;

mpfa_status device_info(int *dev, int *n_sm) {
  static std::atomic<int> known[MAX_DEVICES];   // SM count; 0: not asked yet, -1: not a device for this library
  int d = 0;
  MPFA_CUDA_OK(cudaGetDevice(&d));
  int n = d < MAX_DEVICES ? known[d].load(std::memory_order_relaxed) : 0;
  if (n == 0) {
    int major = 0;
    MPFA_CUDA_OK(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, d));
    MPFA_CUDA_OK(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, d));
    if (major != 10) n = -1;
    if (d < MAX_DEVICES) known[d].store(n, std::memory_order_relaxed);
  }
  if (n < 0) return MPFA_ERR_ARCH;
  *dev = d;
  *n_sm = n;
  return MPFA_OK;
}

namespace {


__device__ __forceinline__ void unpack8(const uint4 &u, float (&f)[8]) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = __uint_as_float(w[i] << 16);
    f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
  }
}

// One pass over a tensor [B, N, cols] gives, per column, everything the statistics need:
//   the sum in FP64 (Eq. 7);
//   max x and min x - rounding is monotonic and symmetric, so
//   max_t |fl(x_t - mu)| = max(fl(max x - mu), fl(mu - min x)) and no second pass over the tensor is
//   needed for the per-tensor scale.
// A CTA covers one head (128 columns) x one slice of the tokens: thread = (token lane 0..15, 8 columns), eight independent
// 16-byte loads in flight per thread while the eight before them are added; each thread adds its tokens in ascending order, the 16 token lanes are folded in lane
// order in shared memory.  With one slice the CTA writes mean = fl(sum / N) (0 without smoothing) and the head's max |x - mean|
// itself.  Slices of a short tensor are a cluster, whose first CTA adds their partial results in slice order; otherwise these go to the
// workspace and stat_fold_kernel adds them in the same order.  No counter, no memory to clear.  Every addition order is fixed by the shape, the workspace size
// and the device's SM count, so the result is reproducible bit for bit for any input; it equals the oracle's single
// ascending FP64 sum whenever all these sums are exact (always true for BF16 inputs whose exponents span fewer than
// about 40 binades per column).
//
// The conversion instruction FP32 -> FP64 runs at 16 lanes per clock and SM, the FP64 add at 64 (measured: 16.0 and 63.5),
// and the loads need 12.  A BF16 number has at most 7 mantissa bits, so its bits shifted right by three are the high word
// of the double 2^-896 times its value, subnormals and zeros included: three integer operations, and sums of such numbers
// round as the unscaled ones do.  Infinities and NaNs would become finite; an FMA with zero catches them, and that
// thread's slice is added again with the conversion.
// Measured (Q and K, 32:8 heads, 16384 tokens / 1:1 heads, 256 tokens; with memory-set node or fold): with conversions, four
// loads in flight and the last CTA of a group folding the slices 42 / 11 us, now 40 / 3.6 us (4.5 TB/s).  Clusters leave some SMs
// empty and others full: 45 us of the first, so only for short tensors.  There (stage 1 without / with clusters): 8 + 2 heads of 4 x 777
// tokens 16.0 / 11.9 us, 40 + 8 of 1999 21.6 / 19.2, 32 + 8 of 1100 16.2 / 13.1, of 4096 25.5 / 27.5.
constexpr int STAT_THREADS = 256;
constexpr int STAT_LOADS = 8;   // rows in flight per thread, and as many being added
constexpr int STAT_CTAS = 2;    // resident per SM
constexpr int STAT_LANES = STAT_THREADS / 16;

struct ColTensor {
  const __nv_bfloat16 *x;   // null: tensor absent (H = 0)
  int N, H;
  double *psum;             // [slices][B][H * 128] partial results
  float2 *pext;             // (max, min)
  float *mean;              // [B, H, 128]
  float *gmax;              // [B, H] x MAXIMA_STRIDE
};
// The heads' maxima have no room of their own: each stands in the first word of its head's first partial sums, which the head's
// fold has read by then.
constexpr size_t MAXIMA_STRIDE = HEAD_DIM * sizeof(double) / sizeof(float);

__device__ __forceinline__ uint32_t bf16x2_max(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ uint32_t bf16x2_min(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("min.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
// c + 0 a: NaN in a half whose a is not finite
__device__ __forceinline__ uint32_t bf16x2_note_nonfinite(uint32_t a, uint32_t c) {
  uint32_t d;
  asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(0u), "r"(c));
  return d;
}

// Mean of column c of a head and the head's maximum |x - mean|; threads 0..127 of the block (whole warps), s_w: 4 floats.
__device__ __forceinline__ void finish_column(const ColTensor &a, int b, int h, int c, double sum, float mx, float mn, int smooth, float *s_w) {
  const float mu = smooth ? __double2float_rn(__ddiv_rn(sum, (double)a.N)) : 0.0f;
  a.mean[((size_t)b * a.H + h) * HEAD_DIM + c] = mu;
  // non-negative: min <= mu <= max (or mu = 0 and the larger side wins)
  float m = fmaxf(fmaxf(__fsub_rn(mx, mu), __fsub_rn(mu, mn)), 0.0f);
  asm("redux.sync.max.f32 %0, %0, 0xffffffff;" : "+f"(m));
  if ((c & 31) == 0) s_w[c >> 5] = m;
  asm volatile("bar.sync 1, 128;" ::: "memory");
  if (c == 0) a.gmax[((size_t)b * a.H + h) * MAXIMA_STRIDE] = fmaxf(fmaxf(s_w[0], s_w[1]), fmaxf(s_w[2], s_w[3]));
}

// V's quantization depends on no statistic: its tiles ride along in CTAs of their own behind those of the statistics.
struct VTensor {
  const __nv_bfloat16 *x;   // null: none
  int N, H, tiles;
  float inv_scale;
  uint8_t *out;
};
__device__ __forceinline__ void quantize_v_tile(const VTensor &v, int tile, int h, int b);

// grid (slices * heads of both tensors * B, the slice fastest and the batch element slowest, then V's tiles); heads are not a grid
// dimension of their own, which ends at 65535.  CLUSTERS: the slices of a head are a cluster, and its first CTA finishes the head from the
// partial results that the others leave in its shared memory.
template <bool CLUSTERS, bool WITH_V>
__global__ void __launch_bounds__(STAT_THREADS, STAT_CTAS) colstat_kernel(const ColTensor t0, const ColTensor t1, int B, int slices, int smooth, const VTensor v) {
  __shared__ double s_part[CLUSTERS ? STAT_CLUSTER : 2][CLUSTERS ? HEAD_DIM : 1];
  __shared__ uint32_t s_ext[CLUSTERS ? STAT_CLUSTER : 1][CLUSTERS ? HEAD_DIM : 1];   // maximum in the upper half, minimum in the lower
  __shared__ double s_sum[STAT_LANES][HEAD_DIM];
  __shared__ uint32_t s_mx[STAT_LANES][HEAD_DIM / 2], s_mn[STAT_LANES][HEAD_DIM / 2];
  launch_dependents();
  if (CLUSTERS) cluster_arrive();   // so that all CTAs of the cluster are there when the first writes to another
  grid_dependency_wait();
  const int heads = t0.H + t1.H;
  int at = blockIdx.x / slices;
  const int slice = blockIdx.x - at * slices;
  if (WITH_V && at >= heads * B) {
    if (CLUSTERS) cluster_wait();
    const int n = blockIdx.x - slices * heads * B, tile = n % v.tiles, vh = n / v.tiles % v.H, vb = n / v.tiles / v.H;
    if (vb < B) quantize_v_tile(v, tile, vh, vb);
    if (CLUSTERS) cluster_arrive(), cluster_wait();
    return;
  }
  const int b = at / heads;
  at -= b * heads;
  const bool first = at < t0.H;
  const ColTensor &a = first ? t0 : t1;
  const int h = first ? at : at - t0.H;
  const int tid = threadIdx.x, tl = tid >> 4, cg = tid & 15;
  const int len = ((a.N + slices - 1) / slices + STAT_LANES - 1) / STAT_LANES * STAT_LANES;
  const int begin = min(a.N, slice * len), end = min(a.N, begin + len);
  const size_t row = (size_t)a.H * HEAD_DIM, step = STAT_LANES * row;
  const __nv_bfloat16 *const p0 = a.x + ((size_t)b * a.N + begin + tl) * row + h * HEAD_DIM + cg * 8, *p = p0;
  double acc[8];
  uint32_t mx[4], mn[4], odd[4];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.0;
#pragma unroll
  for (int i = 0; i < 4; ++i) mx[i] = 0xFF80FF80u, mn[i] = 0x7F807F80u, odd[i] = 0u;
  auto add = [&](const uint4 &u) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      mx[i] = bf16x2_max(mx[i], w[i]);
      mn[i] = bf16x2_min(mn[i], w[i]);
      odd[i] = bf16x2_note_nonfinite(w[i], odd[i]);
      acc[2 * i] += __hiloint2double(((int)(w[i] << 16) >> 3) & 0x8FFFE000, 0);
      acc[2 * i + 1] += __hiloint2double(((int)w[i] >> 3) & 0x8FFFE000, 0);
    }
  };
  int t = begin + tl;
  // one round of loads is in flight while the previous one is added
  const auto load = [&](uint4 (&u)[STAT_LOADS]) {
#pragma unroll
    for (int j = 0; j < STAT_LOADS; ++j) u[j] = *reinterpret_cast<const uint4 *>(p + j * step);
    p += STAT_LOADS * step;
  };
  const auto full = [&](int at) { return at + STAT_LANES * (STAT_LOADS - 1) < end; };
  constexpr int ROUND = STAT_LANES * STAT_LOADS;
  uint4 u0[STAT_LOADS], u1[STAT_LOADS];
  if (full(t)) load(u0);
  while (full(t)) {
    if (full(t + ROUND)) load(u1);
#pragma unroll
    for (int j = 0; j < STAT_LOADS; ++j) add(u0[j]);
    t += ROUND;
    if (!full(t)) break;
    if (full(t + ROUND)) load(u0);
#pragma unroll
    for (int j = 0; j < STAT_LOADS; ++j) add(u1[j]);
    t += ROUND;
  }
  {   // the last fewer than STAT_LOADS rows of this lane, still in flight together
#pragma unroll
    for (int j = 0; j < STAT_LOADS - 1; ++j)
      if (t + STAT_LANES * j < end) u0[j] = *reinterpret_cast<const uint4 *>(p + j * step);
#pragma unroll
    for (int j = 0; j < STAT_LOADS - 1; ++j)
      if (t + STAT_LANES * j < end) add(u0[j]);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] *= 0x1p896;
  if (((odd[0] | odd[1] | odd[2] | odd[3]) & 0x7FFF7FFFu) != 0u) {   // non-finite values: plain sums
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0.0;
    p = p0;
    for (t = begin + tl; t < end; t += STAT_LANES, p += step) {
      float f[8];
      unpack8(*reinterpret_cast<const uint4 *>(p), f);
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] += (double)f[i];
    }
  }
  // pairs of columns: eight consecutive lanes write 128 contiguous bytes
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    *reinterpret_cast<double2 *>(&s_sum[tl][i * 32 + cg * 2]) = make_double2(acc[2 * i], acc[2 * i + 1]);
    s_mx[tl][i * 16 + cg] = mx[i];
    s_mn[tl][i * 16 + cg] = mn[i];
  }
  __syncthreads();
  if (!CLUSTERS && tid >= HEAD_DIM) return;
  if (CLUSTERS) cluster_wait();
  if (tid < HEAD_DIM) {
    // place of column tid: pair i of group cg
    const int place = ((tid & 7) >> 1) * 32 + (tid >> 3) * 2 + (tid & 1);
    double sum = 0.0;
    uint32_t hi = 0xFF80FF80u, lo = 0x7F807F80u;
#pragma unroll
    for (int j = 0; j < STAT_LANES; ++j) {
      sum += s_sum[j][place];
      hi = bf16x2_max(hi, s_mx[j][place >> 1]);
      lo = bf16x2_min(lo, s_mn[j][place >> 1]);
    }
    const float fmx = __uint_as_float(tid & 1 ? hi & 0xFFFF0000u : hi << 16), fmn = __uint_as_float(tid & 1 ? lo & 0xFFFF0000u : lo << 16);
    if (CLUSTERS) {
      cluster_store(cluster_address(smem_u32(&s_part[slice][tid]), 0), sum);
      cluster_store(cluster_address(smem_u32(&s_ext[slice][tid]), 0), __float_as_uint(fmx) | __float_as_uint(fmn) >> 16);
    } else if (slices == 1) {
      finish_column(a, b, h, tid, sum, fmx, fmn, smooth, reinterpret_cast<float *>(&s_part[0][0]));
    } else {
      const size_t o = ((size_t)slice * B + b) * row + h * HEAD_DIM + tid;
      a.psum[o] = sum;
      a.pext[o] = make_float2(fmx, fmn);
    }
  }
  if (CLUSTERS) {
    cluster_arrive();
    cluster_wait();
    if (slice != 0 || tid >= HEAD_DIM) return;
    double sum = 0.0;
    float mx = -INFINITY, mn = INFINITY;
    for (int s = 0; s < slices; ++s) {
      const uint32_t e = s_ext[s][tid];
      sum += s_part[s][tid], mx = fmaxf(mx, __uint_as_float(e & 0xFFFF0000u)), mn = fminf(mn, __uint_as_float(e << 16));
    }
    finish_column(a, b, h, tid, sum, mx, mn, smooth, reinterpret_cast<float *>(&s_mx[0][0]));
  }
}

// The slices' partial results in slice order; grid (heads of both tensors, B), 128 threads, eight slices' loads in flight.
__global__ void __launch_bounds__(128) stat_fold_kernel(const ColTensor t0, const ColTensor t1, int slices, int smooth) {
  __shared__ float s_w[4];
  launch_dependents();
  grid_dependency_wait();
  const bool first = (int)blockIdx.x < t0.H;
  const ColTensor &a = first ? t0 : t1;
  const int h = first ? blockIdx.x : blockIdx.x - t0.H, b = blockIdx.y, tid = threadIdx.x;
  const size_t row = (size_t)a.H * HEAD_DIM, step = gridDim.y * row, o = (size_t)b * row + h * HEAD_DIM + tid;
  double sum = 0.0;
  float mx = -INFINITY, mn = INFINITY;
  for (int s0 = 0; s0 < slices; s0 += 8) {
    double ps[8];
    float2 pe[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (s0 + j < slices) ps[j] = a.psum[o + (s0 + j) * step], pe[j] = a.pext[o + (s0 + j) * step];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (s0 + j < slices) sum += ps[j], mx = fmaxf(mx, pe[j].x), mn = fminf(mn, pe[j].y);
  }
  finish_column(a, b, h, tid, sum, mx, mn, smooth, s_w);
}

// A per-tensor scale: given (frozen statistics), or max |x - mean| / 2688 from the heads' maxima of the statistics pass of
// the same call (1 for an all-zero tensor).
struct TensorScale {
  float *gscale;       // [B]
  const float *gmax;   // [B, heads] x MAXIMA_STRIDE, or null: read gscale
  int heads;
};

// whole warp
__device__ __forceinline__ float tensor_scale(const TensorScale &s, int b, int lane) {
  if (!s.gmax) return s.gscale[b];
  float m = 0.0f;
  for (int i = lane; i < s.heads; i += 32) m = fmaxf(m, s.gmax[((size_t)b * s.heads + i) * MAXIMA_STRIDE]);
  asm("redux.sync.max.f32 %0, %0, 0xffffffff;" : "+f"(m));
  return m > 0.0f ? __fdiv_rn(m, 2688.0f) : 1.0f;
}

// One NVFP4 block (Eq. 1): 16 centered values -> E4M3 scale code + 8 bytes of E2M1 codes.
__device__ __forceinline__ void quantize_block16(const float (&xc)[16], float d, uint8_t &scale_code, uint2 &codes) {
  float a = 0.0f;
#pragma unroll
  for (int i = 0; i < 16; ++i) a = fmaxf(a, fabsf(xc[i]));
  const float e = __fmul_rn(6.0f, d);
  const float r = __fdiv_rn(a, e);
  scale_code = (uint8_t)__nv_cvt_float_to_fp8(r, __NV_SATFINITE, __NV_E4M3);
  const float sdec = __half2float(__half(__nv_cvt_fp8_to_halfraw(scale_code, __NV_E4M3)));
  const float s = __fmul_rn(sdec, d);
  float inv = __fdiv_rn(1.0f, s);
  if (!(s > 0.0f) || isinf(inv)) inv = 0.0f;
  uint32_t w[2] = {0u, 0u};
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float2 v = make_float2(__fmul_rn(xc[2 * i], inv), __fmul_rn(xc[2 * i + 1], inv));
    uint32_t byte = (uint32_t)__nv_cvt_float2_to_fp4x2(v, __NV_E2M1, cudaRoundNearest);
    w[i >> 2] |= (byte & 0xFFu) << (8 * (i & 3));
  }
  codes = make_uint2(w[0], w[1]);
}

// The same block for kernels that quantize many of one tensor: the same codes without a division per block.
//   - The reciprocal of the decoded scale takes one of 128 values: a table in shared memory, made once per CTA.
//   - The scale code rounds r = fl(amax / (6 d)) to three mantissa bits.  amax * fl(1 / (6 d)) is within three units in the
//     last place of it (each of the two roundings adds at most one half of one part in 2^23), which gives the same code unless
//     a rounding boundary lies between: mantissa bits 19..0 next to 0x80000.  There (seven in 2^20 blocks), and where E4M3 is
//     subnormal or the reciprocal is, the division is done.
// Packed FP32 pairs round each half like the scalar operation.
struct BlockScale {
  float e, rcp;       // 6 d and its reciprocal (NaN: always divide)
  const float *inv;   // [128], by the magnitude of the scale code: its sign is that of d, and the two cancel in the decoded scale
};
__device__ __forceinline__ BlockScale make_block_scale(float d, float *table, int tid) {
  if (tid < 128) {
    const float s = __fmul_rn(__half2float(__half(__nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)tid, __NV_E4M3))), fabsf(d));
    const float inv = __fdiv_rn(1.0f, s);
    table[tid] = (!(s > 0.0f) || isinf(inv)) ? 0.0f : inv;
  }
  BlockScale q;
  q.e = __fmul_rn(6.0f, d);
  q.rcp = (q.e > 1e-30f && q.e < 1e30f) ? __frcp_rn(q.e) : NAN;
  q.inv = table;
  return q;
}
__device__ __forceinline__ void add2(float &d0, float &d1, float a0, float a1, float b0, float b1) {
  asm("{.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;}"
      : "=f"(d0), "=f"(d1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}
__device__ __forceinline__ void mul2(float &d0, float &d1, float a0, float a1, float b) {
  asm("{.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %4};\n\t"
      "mul.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;}"
      : "=f"(d0), "=f"(d1)
      : "f"(a0), "f"(a1), "f"(b));
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ uint32_t e2m1x8(const float (&y)[16], int o) {
  uint32_t w;
  asm("{.reg .b8 b0, b1, b2, b3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n\tcvt.rn.satfinite.e2m1x2.f32 b1, %4, %3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b2, %6, %5;\n\tcvt.rn.satfinite.e2m1x2.f32 b3, %8, %7;\n\t"
      "mov.b32 %0, {b0, b1, b2, b3};}"
      : "=r"(w)
      : "f"(y[o]), "f"(y[o + 1]), "f"(y[o + 2]), "f"(y[o + 3]), "f"(y[o + 4]), "f"(y[o + 5]), "f"(y[o + 6]), "f"(y[o + 7]));
  return w;
}
__device__ __forceinline__ float block_max(const float (&xc)[16]) {
  float m[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) m[i] = max3(fabsf(xc[4 * i]), fabsf(xc[4 * i + 1]), fabsf(xc[4 * i + 2]));
#pragma unroll
  for (int i = 0; i < 2; ++i) m[i] = max3(m[i], fabsf(xc[8 * i + 3]), fabsf(xc[8 * i + 7]));
  return max3(max3(m[0], m[1], m[2]), m[3], 0.0f);   // 0 for a block of NaNs, as above
}
__device__ __forceinline__ bool near_boundary(float r) {
  return !(r >= 0.015625f && r < 512.0f && abs((int)(__float_as_uint(r) & 0xFFFFFu) - 0x80000) > 4);
}
// Two blocks of a row at once: their chains run beside one another, with one branch for both divisions (a branch per block kept the
// blocks one after the other: every instruction waited for the one before, issue slots 54 % used).  scale_codes: two bytes.
__device__ __forceinline__ void quantize_blocks(const float (&xa)[16], const float (&xb)[16], const BlockScale &q, uint32_t &scale_codes,
                                                uint2 &ca, uint2 &cb) {
  const float a = block_max(xa), b = block_max(xb);
  float ra = __fmul_rn(a, q.rcp), rb = __fmul_rn(b, q.rcp);
  if (near_boundary(ra) | near_boundary(rb)) ra = __fdiv_rn(a, q.e), rb = __fdiv_rn(b, q.e);
  scale_codes = (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(ra, rb), __NV_SATFINITE, __NV_E4M3);
  const float ia = q.inv[scale_codes & 127u], ib = q.inv[(scale_codes >> 8) & 127u];
  float ya[16], yb[16];
#pragma unroll
  for (int i = 0; i < 16; i += 2) mul2(ya[i], ya[i + 1], xa[i], xa[i + 1], ia);
#pragma unroll
  for (int i = 0; i < 16; i += 2) mul2(yb[i], yb[i + 1], xb[i], xb[i + 1], ib);
  ca = make_uint2(e2m1x8(ya, 0), e2m1x8(ya, 8));
  cb = make_uint2(e2m1x8(yb, 0), e2m1x8(yb, 8));
}
// One of them, for a kernel that has no registers for both.
__device__ __forceinline__ void quantize_block16(const float (&xc)[16], const BlockScale &q, uint32_t &scale_code, uint2 &codes) {
  const float a = block_max(xc);
  float r = __fmul_rn(a, q.rcp);
  if (near_boundary(r)) r = __fdiv_rn(a, q.e);
  scale_code = (uint32_t)__nv_cvt_float_to_fp8(r, __NV_SATFINITE, __NV_E4M3);
  const float inv = q.inv[scale_code & 127u];
  float y[16];
#pragma unroll
  for (int i = 0; i < 16; i += 2) mul2(y[i], y[i + 1], xc[i], xc[i + 1], inv);
  codes = make_uint2(e2m1x8(y, 0), e2m1x8(y, 8));
}
// The four lanes j of a row hold the scale bytes of blocks j and j + 4: lane 0 gets the word of blocks 0..3, lane 1 that of 4..7.
__device__ __forceinline__ uint32_t scale_word(uint32_t two, int j) {
  uint32_t w = two << (16 * (j & 1));
  w |= __shfl_xor_sync(0xffffffffu, w, 1);                       // bytes of blocks j, j + 4, j + 1, j + 5 (j even)
  const uint32_t o = __shfl_xor_sync(0xffffffffu, w, 2);
  return __byte_perm(w, o, (j & 1) ? 0x7531u : 0x6420u);         // right in lanes 0 and 1
}

// 16 channels of one row.  Two 16-byte loads touch each 32-byte sector twice; tensors that are 32-byte aligned (the interface
// asks for 16) are read with one load.
struct Row16 { uint4 a, b; };
__device__ __forceinline__ Row16 load_row16(const __nv_bfloat16 *p, bool wide) {
  Row16 r;
  if (wide) {
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r.a.x), "=r"(r.a.y), "=r"(r.a.z), "=r"(r.a.w), "=r"(r.b.x), "=r"(r.b.y), "=r"(r.b.z), "=r"(r.b.w)
                 : "l"(p));
  } else {
    const uint4 *u = reinterpret_cast<const uint4 *>(p);
    r.a = u[0], r.b = u[1];
  }
  return r;
}
__device__ __forceinline__ bool wide_rows(const void *x) { return (reinterpret_cast<uintptr_t>(x) & 31) == 0; }
// Means of 16 channels.  The interface asks for no alignment of the statistics beyond a float's: 16-byte loads where the address allows
// them.  The kernels of a decode step, which are chains of a few loads, have an instance of each kind (the branch cost a step
// of 64 requests 0.9 us of 70); the others branch.
inline __host__ __device__ bool vector_means(const float *mean) { return (reinterpret_cast<uintptr_t>(mean) & 15) == 0; }
__device__ __forceinline__ void load_mean16(const float *mean, float (&m)[16], bool vec) {
  if (vec) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float4 v = reinterpret_cast<const float4 *>(mean)[c];
      m[4 * c] = v.x, m[4 * c + 1] = v.y, m[4 * c + 2] = v.z, m[4 * c + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int c = 0; c < 16; ++c) m[c] = mean[c];
  }
}
__device__ __forceinline__ void load_neg_mean(const float *mean, float (&nm)[16], bool vec) {
  load_mean16(mean, nm, vec);
#pragma unroll
  for (int c = 0; c < 16; ++c) nm[c] = -nm[c];
}
__device__ __forceinline__ void center16(const Row16 &x, const float (&nm)[16], float (&xc)[16]) {
  float f[16];
  unpack8(x.a, reinterpret_cast<float(&)[8]>(f[0]));
  unpack8(x.b, reinterpret_cast<float(&)[8]>(f[8]));
#pragma unroll
  for (int i = 0; i < 16; i += 2) add2(xc[i], xc[i + 1], f[i], f[i + 1], nm[i], nm[i + 1]);
}

// Compensation vector (Eq. 9): Delta_S[hq][t] = qmean[hq] . (k[t] - kmean) in FP64, in units of gscale_q * gscale_k, rounded once
// to BF16.  The product of eight keys with the (up to eight) query means of the group is a contraction over the channels and
// runs on the FP64 tensor instruction (m8n8k4): lane (key = lane / 4, j = lane mod 4) holds the 16-channel blocks j and j + 4 of
// its key, so step s of the contraction takes the lane's own s-th channel, in the order
//   channel(j, s) = 16 j + s (s < 16), 64 + 16 j + s - 16,
// and the sums come out complete, without staging rows or shuffling.  (A chain of 128 FP64 FMAs per key and head, as one
// thread each, was bound by latency; with the eight threads of a key taking 16 channels each, by the shared-memory reads of the
// query means.)  The order of the FP64 additions is fixed in each kernel, but not the same: the tensor instruction's here and in
// write_kv_kernel, two chains and two shuffles for groups of one or two heads, eight lanes' chains and three shuffles in
// append_kv_kernel, which also divides where the others multiply by a reciprocal.  The sums differ by a few parts in 2^53 of their
// terms, and one rounding to FP32 and one to BF16 follow: two kernels (or the oracle's single ascending chain) give another
// BF16 only where the exact quotient is that close to a midpoint of two floats which themselves round apart.  No tested input shows
// one; a tie that FP64 holds exactly comes out the same everywhere.
//
// Query means as doubles in operand order: [step][head][j].
typedef double GroupMeans[32][8][4];
__device__ __forceinline__ void convert_group_means(GroupMeans &m, const float *q_mean /* [G, 128] */, int G, int tid, int n_threads) {
  for (int i = tid; i < 8 * HEAD_DIM; i += n_threads) {
    const int g = i >> 7, c = i & 127;
    m[(c & 15) + ((c >> 6) << 4)][g][(c >> 4) & 3] = g < G ? (double)q_mean[g * HEAD_DIM + c] : 0.0;
  }
}
// acc (heads 2 j, 2 j + 1 of the lane's key) += the half's 16 channels
__device__ __forceinline__ void group_dot16(const GroupMeans &m, int half, const float (&xc)[16], int lane, double (&acc)[2]) {
  const double *q = &m[half * 16][0][0] + lane;
#pragma unroll
  for (int s = 0; s < 16; ++s)
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                 : "+d"(acc[0]), "+d"(acc[1])
                 : "d"((double)xc[s]), "d"(q[s * 32]));
}

// One or two heads: of the tensor instruction's eight columns only so many would count, and the plain FP64 pipe has the same
// rate.  A lane takes the products of its own 32 channels (query means as doubles, [head][channel pair][j][2], so that the
// four addresses of a warp's load are one line) and the four lanes of a key are added in a fixed order.
__device__ __forceinline__ void convert_group_means_few(double *m, const float *q_mean /* [G, 128] */, int G, int tid, int n_threads) {
  for (int i = tid; i < G * HEAD_DIM; i += n_threads) {
    const int g = i >> 7, c = i & 127, j = (c >> 4) & 3, s = (c & 15) + ((c >> 6) << 4);
    m[g * HEAD_DIM + (s >> 1) * 8 + j * 2 + (s & 1)] = (double)q_mean[i];
  }
}
// acc[g] += the half's 16 channels of the lane's key, two chains a head
template <int G>
__device__ __forceinline__ void few_dot16(const double *m, int half, const float (&xc)[16], int j, double (&acc)[G][2]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const double x0 = (double)xc[2 * i], x1 = (double)xc[2 * i + 1];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const double2 q = *reinterpret_cast<const double2 *>(m + g * HEAD_DIM + (half * 8 + i) * 8 + j * 2);
      acc[g][0] = fma(q.x, x0, acc[g][0]);
      acc[g][1] = fma(q.y, x1, acc[g][1]);
    }
  }
}

struct QuantTensor {
  const __nv_bfloat16 *x;   // null: tensor absent (H = 0)
  const float *mean;
  TensorScale scale;
  int N, H, tiles;
  int ctas;                 // CTAs per head; CTA c takes the tiles c, c + ctas, ... from the last one
  uint8_t *codes, *sf;
};
struct DeltaArgs {
  const float *q_mean;
  TensorScale q_scale;
  __nv_bfloat16 *delta;    // [B, H_q, N_pad]; null: no Delta_S (direct variant)
  int H_q;
};

// Tiles (128 tokens of one head) of K and Q; blockIdx.x runs over K's CTAs, then Q's, the head index fastest, so that the
// CTAs resident at any time read whole token rows of the [B, N, H, 128] input (contiguous DRAM) instead of 256-byte
// pieces 256 * H bytes apart; from the last token to the first, because the statistics pass has just read the tensors in
// ascending order: of one that fits L2 most is still there, of a larger one the end of its last slice only (32768 tokens of 40:8 heads: 402 of
// 403 MB come from DRAM again).  Warp w takes rows 8 w .. and 64 + 8 w .. of a tile, lane (row, j) their
// 16-channel blocks j and j + 4.  A CTA stays with one head, so that after the set-up's barrier its warps run on their own:
// the loads of the next tile are issued as soon as the registers of a row group are free, scale words and Delta_S go straight
// to memory (partial sectors merge in L2).
// Measured (16384 tokens, 32:8 heads, K with Delta_S and Q): two launches, rows of K staged in shared memory, two
// divisions per block 35 + 38 us; one launch, one tile per CTA 61; with a ring of asynchronous copies and a barrier per tile 87;
// now 45 us.  Both blocks of a row at once and the means in shared memory, where they were taken one after the other with the means in
// registers (stage 1, replayed back to back): 32768 tokens, 40:8 heads 194 -> 176 us, 16384, 32:8 88.7 -> 80.7, 8 x 577, 16:16 29.1 ->
// 27.7; three CTAs per SM of 80 registers 182, 36 for the last; 16 rows of Q dealt to the warps across heads 213 for the first.
constexpr int QT_CTAS = 2;       // resident per SM: 128 registers
constexpr int QT_K_WEIGHT = 2;   // time of a K tile with Delta_S in units of a Q tile's (1 / 2 / 3: 106 / 89 / 96 us of stage 1)
constexpr int QT_SETUP = 2;      // a CTA's set-up in the same units
template <int FEW>   // heads of the group where they are one or two, otherwise 0
__global__ void __launch_bounds__(256, QT_CTAS) quantize_tile_kernel(const QuantTensor k, const QuantTensor q, const DeltaArgs da) {
  __shared__ __align__(16) GroupMeans gm;
  __shared__ float inv_table[128];
  launch_dependents();
  grid_dependency_wait();
  const int b = blockIdx.z, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, j = lane & 3;
  const int k_ctas = k.ctas * k.H;
  const bool is_k = (int)blockIdx.x < k_ctas;
  const QuantTensor &a = is_k ? k : q;
  const int at = is_k ? blockIdx.x : blockIdx.x - k_ctas;
  const int h = at % a.H, N = a.N, ctas = a.ctas;
  int tile = a.tiles - 1 - at / a.H;
  const size_t head = (size_t)b * a.H + h, row = (size_t)a.H * HEAD_DIM;
  const __nv_bfloat16 *const x0 = a.x + (size_t)b * N * row + h * HEAD_DIM + j * 16;
  const int r0 = warp * 8 + (lane >> 2);
  const bool wide = wide_rows(a.x);
  Row16 raw[2][2];
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int t = tile * TILE + it * 64 + r0;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      raw[it][half] = Row16{};
      if (t < N) raw[it][half] = load_row16(x0 + t * row + half * 64, wide);
    }
  }
  const float d = tensor_scale(a.scale, b, lane);
  if (at == 0 && tid == 0 && a.scale.gmax) a.scale.gscale[b] = d;
  const BlockScale bs = make_block_scale(d, inv_table, tid);
  __shared__ __align__(16) float s_neg[8][20];   // by 16-channel block, padded against bank conflicts
  if (tid < HEAD_DIM) s_neg[tid >> 4][tid & 15] = -a.mean[head * HEAD_DIM + tid];
  const bool with_delta = is_k && da.delta;
  const int G = with_delta ? da.H_q / a.H : 0;
  double unit = 0.0;
  if (with_delta) {
    const float *qm = da.q_mean + ((size_t)b * da.H_q + h * G) * HEAD_DIM;
    if (FEW)
      convert_group_means_few(&gm[0][0][0], qm, FEW, tid, 256);
    else
      convert_group_means(gm, qm, G, tid, 256);
    unit = 1.0 / ((double)tensor_scale(da.q_scale, b, lane) * (double)d);
  }
  __syncthreads();
  const size_t n_pad = (size_t)a.tiles * TILE;
  uint8_t *const codes = a.codes + head * n_pad * 64 + j * 8;
  for (; tile >= 0; tile -= ctas) {
    uint8_t *const sf_tile = a.sf + (head * a.tiles + tile) * 1024;
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const int r = it * 64 + r0, t = tile * TILE + r;
      double acc[FEW ? FEW : 1][2];   // FEW: two chains a head, otherwise heads 2 j and 2 j + 1
#pragma unroll
      for (int g = 0; g < (FEW ? FEW : 1); ++g) acc[g][0] = acc[g][1] = 0.0;
      float xa[16], xb[16];
      {
        float nm[16];
        load_mean16(s_neg[j], nm, true);
        center16(raw[it][0], nm, xa);
        load_mean16(s_neg[j + 4], nm, true);
        center16(raw[it][1], nm, xb);
      }
      if (tile >= ctas) {   // a whole tile: only the last has an end
        const __nv_bfloat16 *const x1 = x0 + (size_t)(t - ctas * TILE) * row;
        raw[it][0] = load_row16(x1, wide);
        raw[it][1] = load_row16(x1 + 64, wide);
      }
      uint2 ca, cb;
      uint32_t sc;
      quantize_blocks(xa, xb, bs, sc, ca, cb);
      if (t >= N) ca = cb = make_uint2(0u, 0u), sc = 0u;
      __stcs(reinterpret_cast<uint2 *>(codes + (size_t)t * 64), ca);
      __stcs(reinterpret_cast<uint2 *>(codes + (size_t)t * 64 + 32), cb);
      sc = scale_word(sc, j);
      if (j < 2) *reinterpret_cast<uint32_t *>(sf_tile + j * 512 + (r & 31) * 16 + (r >> 5) * 4) = sc;
      if (with_delta) {
        if constexpr (FEW != 0) {
          few_dot16<FEW>(&gm[0][0][0], 0, xa, j, acc);
          few_dot16<FEW>(&gm[0][0][0], 1, xb, j, acc);
        } else {
          group_dot16(gm, 0, xa, lane, acc[0]);
          group_dot16(gm, 1, xb, lane, acc[0]);
        }
      }
      if (with_delta) {
        __nv_bfloat16 *const dst = da.delta + ((size_t)b * da.H_q + h * G) * n_pad + t;
        if constexpr (FEW != 0) {
#pragma unroll
          for (int g = 0; g < FEW; ++g) {
            double v = acc[g][0] + acc[g][1];
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            if (j == g) dst[g * n_pad] = __float2bfloat16_rn(t < N ? __double2float_rn(v * unit) : 0.0f);
          }
        } else {
#pragma unroll
          for (int n = 0; n < 2; ++n) {
            const int g = 2 * j + n;
            if (g < G) dst[g * n_pad] = __float2bfloat16_rn(t < N ? __double2float_rn(acc[0][n] * unit) : 0.0f);
          }
        }
      }
    }
  }
}

// The tiles of a decode step's queries (at most eight tokens): one warp per (batch element, head), the eight rows and the zeros
// of the other 120.  Bound by writing 9 KB per tile; with a CTA per tile the chain of loads was repeated for six waves of
// CTAs (64 requests, 40 heads: 13.6 us, now 7.1 us).
template <bool VEC>   // vector_means
__global__ void __launch_bounds__(256) quantize_token_kernel(const QuantTensor q, int n_heads) {
  launch_dependents();
  grid_dependency_wait();
  const int head = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31, j = lane & 3, r = lane >> 2;
  if (head >= n_heads) return;
  const int b = head / q.H, h = head % q.H;
  const bool in = r < q.N;
  Row16 raw[2] = {};
  const bool wide = wide_rows(q.x);
#pragma unroll
  for (int half = 0; half < 2; ++half)
    if (in) raw[half] = load_row16(q.x + (((size_t)b * q.N + r) * q.H + h) * HEAD_DIM + (half * 4 + j) * 16, wide);
  const float d = tensor_scale(q.scale, b, lane);
  float neg_mean[2][16];
  load_neg_mean(q.mean + (size_t)head * HEAD_DIM + j * 16, neg_mean[0], VEC);
  load_neg_mean(q.mean + (size_t)head * HEAD_DIM + (4 + j) * 16, neg_mean[1], VEC);
  if (h == 0 && lane == 0 && q.scale.gmax) q.scale.gscale[b] = d;
  uint8_t *const codes = q.codes + (size_t)head * TILE * 64, *const sf = q.sf + (size_t)head * 1024;
  const uint4 z = make_uint4(0u, 0u, 0u, 0u);
  for (int i = 32 + lane; i < TILE * 4; i += 32) reinterpret_cast<uint4 *>(codes)[i] = z;
  for (int i = lane; i < 64; i += 32)
    if ((i & 31) >= 8) reinterpret_cast<uint4 *>(sf)[i] = z;   // 16 bytes per row of the atom: rows 8..31 of both halves
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    float xc[16];
    center16(raw[half], neg_mean[half], xc);
    uint8_t s8 = 0;
    uint2 c = make_uint2(0u, 0u);
    if (in) quantize_block16(xc, d, s8, c);
    *reinterpret_cast<uint2 *>(codes + r * 64 + (half * 4 + j) * 8) = c;
    uint32_t sc = (uint32_t)s8 << (8 * j);
    sc |= __shfl_xor_sync(0xffffffffu, sc, 1);
    sc |= __shfl_xor_sync(0xffffffffu, sc, 2);
    if (j == 0) *reinterpret_cast<uint4 *>(sf + half * 512 + r * 16) = make_uint4(sc, 0u, 0u, 0u);
  }
}

__device__ __forceinline__ uint4 quantize_v16(const Row16 &x, float inv) {
  float f[16];
  unpack8(x.a, reinterpret_cast<float(&)[8]>(f[0]));
  unpack8(x.b, reinterpret_cast<float(&)[8]>(f[8]));
#pragma unroll
  for (int i = 0; i < 16; i += 2) mul2(f[i], f[i + 1], f[i], f[i + 1], inv);
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i)   // two conversions written into the halves of one register
    asm("{.reg .b16 lo, hi;\n\t"
        "cvt.rn.satfinite.e4m3x2.f32 lo, %2, %1;\n\tcvt.rn.satfinite.e4m3x2.f32 hi, %4, %3;\n\t"
        "mov.b32 %0, {lo, hi};}"
        : "=r"(w[i])
        : "f"(f[4 * i]), "f"(f[4 * i + 1]), "f"(f[4 * i + 2]), "f"(f[4 * i + 3]));
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// V tile -> [B, H, N_pad, 128] E4M3; 256 threads
__device__ __forceinline__ void quantize_v_tile(const VTensor &v, int tile, int h, int b) {
  const size_t n_pad = (size_t)v.tiles * TILE;
  const bool wide = wide_rows(v.x);
  const int r0 = threadIdx.x >> 3, seg = threadIdx.x & 7;
  Row16 x[4] = {};
#pragma unroll
  for (int it = 0; it < 4; ++it) {
    const int t = tile * TILE + it * 32 + r0;
    if (t < v.N) x[it] = load_row16(v.x + (((size_t)b * v.N + t) * v.H + h) * HEAD_DIM + seg * 16, wide);
  }
#pragma unroll
  for (int it = 0; it < 4; ++it) {
    const int t = tile * TILE + it * 32 + r0;
    *reinterpret_cast<uint4 *>(v.out + (((size_t)b * v.H + h) * n_pad + t) * HEAD_DIM + seg * 16) =
        t < v.N ? quantize_v16(x[it], v.inv_scale) : make_uint4(0u, 0u, 0u, 0u);
  }
}
// grid (N_pad/128, H, B)
__global__ void __launch_bounds__(256) quantize_v_tile_kernel(const VTensor v) {
  launch_dependents();
  grid_dependency_wait();
  quantize_v_tile(v, blockIdx.x, blockIdx.y, blockIdx.z);
}

// grid (N_pad/128, H, B): V tile -> [B, H, N_pad, 128] BF16, unchanged values (the NVFP4 + BF16 precision assignment
// of Section 3.1 reads V in BF16); pad rows zero.
__global__ void __launch_bounds__(256) pack_v_bf16_kernel(const __nv_bfloat16 *__restrict__ v, int N, int H,
                                                          __nv_bfloat16 *__restrict__ out) {
  const int tile = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  const int n_pad = gridDim.x * TILE;
#pragma unroll
  for (int it = 0; it < 8; ++it) {
    const int id = it * 256 + threadIdx.x;
    const int r = id >> 4, seg = id & 15;
    const int t = tile * TILE + r;
    uint4 c = make_uint4(0u, 0u, 0u, 0u);
    if (t < N) c = *reinterpret_cast<const uint4 *>(v + (((size_t)b * N + t) * H + h) * HEAD_DIM + seg * 8);
    *reinterpret_cast<uint4 *>(out + (((size_t)b * H + h) * n_pad + t) * HEAD_DIM + seg * 8) = c;
  }
}

// grid (N_pad/128, H, B): V tile for the NVFP4 + NVFP4 precision assignment of Section 3.1.  The second MMA contracts
// over the keys, so the 16-element blocks of Eq. 1 lie along the token axis and the operand is stored channel-major
// (K-major B operand): codes [B, H, N_pad/128, 128 channels, 64 bytes] (two keys per byte, the even key in the low
// nibble), block scales as two 512-byte tcgen05.cp atoms per tile (atom = 64 keys: byte (c mod 32) 16 + (c / 32) 4 +
// block mod 4).  Recipe of the Q/K quantizer with the caller's tensor scale d and no centering; keys past N are zero.
__global__ void __launch_bounds__(256) quantize_v_fp4_tile_kernel(const __nv_bfloat16 *__restrict__ v, int N, int H, float d,
                                                                  uint8_t *__restrict__ codes, uint8_t *__restrict__ sf) {
  __shared__ __align__(16) __nv_bfloat16 tile[TILE][HEAD_DIM + 8];   // padded rows: the column reads below stay conflict-free
  __shared__ __align__(16) uint8_t ctile[HEAD_DIM][64];
  __shared__ __align__(16) uint8_t stile[1024];
  const int t0 = blockIdx.x * TILE, h = blockIdx.y, b = blockIdx.z;
  const int n_tiles = gridDim.x;
#pragma unroll
  for (int it = 0; it < 8; ++it) {
    const int id = it * 256 + threadIdx.x;
    const int r = id >> 4, seg = id & 15;
    uint4 u = make_uint4(0u, 0u, 0u, 0u);
    if (t0 + r < N) u = __ldcs(reinterpret_cast<const uint4 *>(v + (((size_t)b * N + t0 + r) * H + h) * HEAD_DIM + seg * 8));
    *reinterpret_cast<uint4 *>(&tile[r][seg * 8]) = u;
  }
  __syncthreads();
#pragma unroll 1
  for (int it = 0; it < 4; ++it) {
    const int id = it * 256 + threadIdx.x;
    const int c = id & 127, kb = id >> 7;   // channel, 16-key block of the tile
    float x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = __bfloat162float(tile[kb * 16 + i][c]);
    uint8_t sc;
    uint2 cw;
    quantize_block16(x, d, sc, cw);
    *reinterpret_cast<uint2 *>(&ctile[c][kb * 8]) = cw;
    stile[(kb >> 2) * 512 + (c & 31) * 16 + (c >> 5) * 4 + (kb & 3)] = sc;
  }
  __syncthreads();
  const size_t tile_id = ((size_t)b * H + h) * n_tiles + blockIdx.x;
  uint4 *cdst = reinterpret_cast<uint4 *>(codes + tile_id * 8192);
#pragma unroll
  for (int it = 0; it < 2; ++it) cdst[it * 256 + threadIdx.x] = reinterpret_cast<const uint4 *>(&ctile[0][0])[it * 256 + threadIdx.x];
  if (threadIdx.x < 64) reinterpret_cast<uint4 *>(sf + tile_id * 1024)[threadIdx.x] = reinterpret_cast<const uint4 *>(stile)[threadIdx.x];
}

// Paged cache write for one request: tokens first .. first + N - 1 go to their slots of the pages, whole pages or parts of
// them.  grid (H_kv, CTAs per head); a CTA stays with one head and takes every gridDim.y-th page.  Warp w takes a page's slots
// 8 w .. 8 w + 7, lane (slot, j) the 16-channel blocks j and j + 4, in the byte order of the decode kernel's shared-memory operand
// tiles: K codes as 64-byte rows with the 64-byte swizzle, V as 128-byte rows with the 128-byte swizzle, Delta_S with its
// 16-byte groups XOR-ed by the head.  K, V and Delta_S come from one read of K and V, and the rows of the next page are
// requested while the current ones are quantized.  Slots past the last token are zero-filled in pages that the call
// starts (a recycled page may hold anything, and decode needs finite bytes there); slots of earlier tokens are left alone.
// Measured (9001 tokens, 32:8 heads): page kernel + a Delta_S kernel that read K again 12 + 16 us, one page per CTA 19.5 us.  The two blocks
// of a row one after the other, each half's next rows requested as soon as its registers are free, and the means in shared memory: the kernel
// alone 11.7 us, means in registers 12.8; 5505 tokens of 4:4 heads 7.2 and 7.9, 45313 of 16:16 137 and 143.  Both blocks at once, as in the
// tile kernel, wait for the next rows longer than they gain: 13.0, 8.4 and 160 with the means in registers; with shared means 12.5, 7.7 and 129,
// but 512 tokens of 32:8 4.4 where one after the other takes 4.2, 1408 5.5 and 5.2.
constexpr int WK_CTAS = 2;   // resident per SM: 128 registers
__global__ void __launch_bounds__(256, WK_CTAS) write_kv_kernel(const __nv_bfloat16 *k, const __nv_bfloat16 *v,
                                                                const float *k_mean, const TensorScale k_scale,
                                                                const float *q_mean, const float *q_gscale,
                                                                int N, int first, int n_pages, int H_q, int H_kv, float inv_vscale,
                                                                const int32_t *page_row, int num_pages,
                                                                uint8_t *k_codes, uint8_t *k_sf,
                                                                uint8_t *v_fp8, __nv_bfloat16 *delta) {
  __shared__ __align__(16) GroupMeans gm;
  __shared__ float inv_table[128];
  launch_dependents();
  grid_dependency_wait();
  const int tid = threadIdx.x, lane = tid & 31, j = lane & 3, h = blockIdx.x, G = H_q / H_kv;
  const int t = (tid >> 5) * 8 + (lane >> 2);   // slot of the page
  const int page0 = first / PAGE;               // first page of the request that is touched
  const bool wide_k = wide_rows(k), wide_v = wide_rows(v);
  Row16 kr[2], vr[2];
  int pg = blockIdx.y, page;
  const auto fetch = [&](int half) {
    const int i = (page0 + pg) * PAGE + t - first;   // index among the new tokens
    kr[half] = vr[half] = Row16{};
    if (pg < n_pages && i >= 0 && i < N) {
      const size_t at = ((size_t)i * H_kv + h) * HEAD_DIM + (half * 4 + j) * 16;
      kr[half] = load_row16(k + at, wide_k);
      vr[half] = load_row16(v + at, wide_v);
    }
  };
  fetch(0);
  fetch(1);
  page = page_row[page0 + pg];
  const float d = tensor_scale(k_scale, 0, lane);
  if (blockIdx.y == 0 && h == 0 && tid == 0 && k_scale.gmax) k_scale.gscale[0] = d;
  const BlockScale bs = make_block_scale(d, inv_table, tid);
  __shared__ __align__(16) float s_neg[8][20];   // by 16-channel block, padded against bank conflicts
  if (tid < HEAD_DIM) s_neg[tid >> 4][tid & 15] = -k_mean[(size_t)h * HEAD_DIM + tid];
  double unit = 0.0;
  if (delta) {
    convert_group_means(gm, q_mean + (size_t)h * G * HEAD_DIM, G, tid, 256);
    unit = 1.0 / ((double)q_gscale[0] * (double)d);
  }
  __syncthreads();
  while (pg < n_pages) {
    const int i = (page0 + pg) * PAGE + t - first;
    const bool page_ok = page >= 0 && page < num_pages;   // a bad id is skipped
    const bool is_new = page_ok && i >= 0 && i < N, fresh_pad = page_ok && i >= N && (page0 + pg) * PAGE >= first;
    const size_t slab = (size_t)(page_ok ? page : 0) * H_kv + h;
    uint8_t *const kd = k_codes + slab * 4096 + (t >> 3) * 512 + (t & 7) * 64, *const sd = k_sf + slab * 512 + t * 8;
    uint8_t *const vd = v_fp8 + slab * 8192 + (t >> 3) * 1024 + (t & 7) * 128;
    __nv_bfloat16 *const dd = delta + ((size_t)(page_ok ? page : 0) * H_q + h * G) * PAGE + (t & 7);
    pg += gridDim.y;
    if (pg < n_pages) page = page_row[page0 + pg];
    double acc[2] = {0.0, 0.0};
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int blk = half * 4 + j;
      float xc[16];
      {
        float nm[16];
        load_mean16(s_neg[blk], nm, true);
        center16(kr[half], nm, xc);
      }
      uint2 c = make_uint2(0u, 0u);
      uint32_t sc = 0u;
      uint4 vc = quantize_v16(vr[half], inv_vscale);
      fetch(half);
      if (is_new)
        quantize_block16(xc, bs, sc, c);
      else
        vc = make_uint4(0u, 0u, 0u, 0u);
      sc <<= 8 * j;   // the four scale bytes of half a token in one word
      sc |= __shfl_xor_sync(0xffffffffu, sc, 1);
      sc |= __shfl_xor_sync(0xffffffffu, sc, 2);
      if (is_new || fresh_pad) {
        *reinterpret_cast<uint2 *>(kd + (((blk >> 1) ^ ((t & 7) >> 1)) << 4) + (blk & 1) * 8) = c;
        if (j == 0) *reinterpret_cast<uint32_t *>(sd + half * 4) = sc;
        *reinterpret_cast<uint4 *>(vd + ((blk ^ (t & 7)) << 4)) = vc;
      }
      if (delta) group_dot16(gm, half, xc, lane, acc);
    }
    if (delta && (is_new || fresh_pad)) {
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        const int g = 2 * j + n;
        if (g < G) dd[g * PAGE + (((t >> 3) ^ g) << 3)] = __float2bfloat16_rn(is_new ? __double2float_rn(acc[n] * unit) : 0.0f);
      }
    }
  }
}

// Decode-time append of a batch (Section 6): request b's one new token goes to index positions[b] with its own frozen
// statistics and page-table row; a negative position skips the request.  One warp per (request, kv head): lane = (part 0..3,
// 16-channel block); part 0 writes K, part 1 V, and part p the Delta_S of heads p and p + 4.  A token that starts a page zeroes the
// other 63 slots.  Bound by the latency of three dependent loads; the loads that depend on nothing are issued together.
// Measured (64 requests, 40:8 heads): with one thread per FP64 chain of 128 terms and 2 x 256 threads per pair
// 9.8 us, now 6.6 us.
template <bool VEC>   // vector_means of both means
__global__ void __launch_bounds__(256) append_kv_kernel(const __nv_bfloat16 *k, const __nv_bfloat16 *v,
                                                        const float *q_mean, const float *k_mean,
                                                        const float *q_gscale, const float *k_gscale,
                                                        int B, int H_q, int H_kv, float inv_vscale,
                                                        const int32_t *page_table, int max_pages, int num_pages,
                                                        const int32_t *positions, uint8_t *k_codes,
                                                        uint8_t *k_sf, uint8_t *v_fp8,
                                                        __nv_bfloat16 *delta) {
  launch_dependents();
  grid_dependency_wait();
  const int pair = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31, blk = lane & 7, part = lane >> 3;
  if (pair >= B * H_kv) return;
  const int b = pair / H_kv, h = pair % H_kv, G = H_q / H_kv;
  const int pos = positions[b];
  const Row16 kr = load_row16(k + (size_t)pair * HEAD_DIM + blk * 16, wide_rows(k));
  const Row16 vr = load_row16(v + (size_t)pair * HEAD_DIM + blk * 16, wide_rows(v));
  const float d = k_gscale[b];
  const double denom = delta ? (double)q_gscale[b] * (double)d : 1.0;
  float xc[16], neg_mean[16];
  load_neg_mean(k_mean + (size_t)pair * HEAD_DIM + blk * 16, neg_mean, VEC);
  center16(kr, neg_mean, xc);
  const bool in_table = pos >= 0 && (pos >> 6) < max_pages;   // else: skipped, or no page-table entry for that position
  const int page = in_table ? page_table[(size_t)b * max_pages + (pos >> 6)] : -1;
  const int t = pos & 63;
  // Delta_S of heads part and part + 4, while the page id is on its way
  double acc[2] = {0.0, 0.0};
  if (delta) {
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      const int g = part + 4 * n;
      if (g < G) {
        float m[16];
        load_mean16(q_mean + ((size_t)b * H_q + h * G + g) * HEAD_DIM + blk * 16, m, VEC);
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[n] = fma((double)m[i], (double)xc[i], acc[n]);
      }
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) acc[n] += __shfl_xor_sync(0xffffffffu, acc[n], o);
    }
  }
  if (page < 0 || page >= num_pages) return;
  const size_t slab = (size_t)page * H_kv + h;
  uint8_t *const kd = k_codes + slab * 4096, *const sd = k_sf + slab * 512, *const vd = v_fp8 + slab * 8192;
  __nv_bfloat16 *const dd = delta ? delta + ((size_t)page * H_q + h * G) * PAGE : nullptr;
  if (part == 0) {
    uint8_t sc;
    uint2 c;
    quantize_block16(xc, d, sc, c);
    *reinterpret_cast<uint2 *>(kd + (t >> 3) * 512 + (t & 7) * 64 + (((blk >> 1) ^ ((t & 7) >> 1)) << 4) + (blk & 1) * 8) = c;
    sd[t * 8 + blk] = sc;
  } else if (part == 1) {
    *reinterpret_cast<uint4 *>(vd + (t >> 3) * 1024 + (t & 7) * 128 + ((blk ^ (t & 7)) << 4)) = quantize_v16(vr, inv_vscale);
  }
  if (t == 0) {   // slot 0 is the first row of each slab
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    for (int i = 4 + lane; i < 256; i += 32) reinterpret_cast<uint4 *>(kd)[i] = z;
    for (int i = 2 + lane; i < 128; i += 32) reinterpret_cast<uint32_t *>(sd)[i] = 0u;
    for (int i = 8 + lane; i < 512; i += 32) reinterpret_cast<uint4 *>(vd)[i] = z;
    if (dd)
      for (int i = lane; i < G * PAGE; i += 32)
        if ((i & 63) != ((i >> 6) << 3)) dd[i] = __float2bfloat16_rn(0.0f);
  }
  if (dd && blk == 0) {
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      const int g = part + 4 * n;
      if (g < G) dd[g * PAGE + ((((t >> 3) ^ g) << 3) | (t & 7))] = __float2bfloat16_rn(__double2float_rn(__ddiv_rn(acc[n], denom)));
    }
  }
}

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// Workspace of the statistics pass: S slices of per-column partial results (FP64 sum, maximum and minimum).  S is the largest slice
// count <= STAT_MAX_SLICES that fits the bytes the caller gave (at least 1) beside a region that is no longer used: callers' sizes
// stay what they were.
constexpr int STAT_MAX_SLICES = 32;
size_t stats_fixed_bytes(int B, int H_q, int H_kv) {
  return align256(((size_t)2 * B + (size_t)B * ((H_q + 1) / 2 + (H_kv + 1) / 2) + 1) * sizeof(unsigned int));
}
size_t stats_slice_bytes(int B, int H_q, int H_kv) {   // one slice of both tensors
  return align256((size_t)B * H_q * HEAD_DIM * 8) + 2 * align256((size_t)B * H_q * HEAD_DIM * 4) +
         align256((size_t)B * H_kv * HEAD_DIM * 8) + 2 * align256((size_t)B * H_kv * HEAD_DIM * 4);
}

struct StatsWorkspace {
  double *psum_q, *psum_k;
  float2 *pext_q, *pext_k;
  float *gmax_q, *gmax_k;
  int slices;   // 0: too small
};
StatsWorkspace carve(void *ws, size_t ws_bytes, int B, int H_q, int H_kv) {
  StatsWorkspace w{};
  const size_t fixed = stats_fixed_bytes(B, H_q, H_kv), per = stats_slice_bytes(B, H_q, H_kv);
  const int S = ws_bytes > fixed ? (int)std::min((ws_bytes - fixed) / per, (size_t)STAT_MAX_SLICES) : 0;
  const size_t nq = (size_t)B * H_q, nk = (size_t)B * H_kv, n = S;
  w.slices = S;
  uint8_t *p = static_cast<uint8_t *>(ws);
  w.psum_q = reinterpret_cast<double *>(p);  p += n * nq * HEAD_DIM * 8;
  w.psum_k = reinterpret_cast<double *>(p);  p += n * nk * HEAD_DIM * 8;
  w.pext_q = reinterpret_cast<float2 *>(p);  p += n * nq * HEAD_DIM * 8;
  w.pext_k = reinterpret_cast<float2 *>(p);
  w.gmax_q = reinterpret_cast<float *>(w.psum_q);
  w.gmax_k = reinterpret_cast<float *>(w.psum_k);
  return w;
}

// Means and the heads' maxima of up to two tensors, and V's tiles.
constexpr long long V_APART = 512ll << 20;
mpfa_status tensor_stats(const ColTensor &c0, const ColTensor &c1, int B, int max_slices, int n_sm, bool smooth, const VTensor &v, cudaStream_t st) {
  const int heads = c0.H + c1.H, N = std::max(c0.x ? c0.N : 0, c1.x ? c1.N : 0);
  if (heads == 0) return MPFA_OK;
  const long long v_ctas = v.x ? (long long)v.tiles * v.H * B : 0;
  const auto cluster_grid = [&](int C) { return Grid(dim3((unsigned)((long long)C * heads * B + (v_ctas + C - 1) / C * C)), C); };
  // The stream's context may own a part of the device only, without room for so many CTAs side by side: the driver is asked for this
  // launch, with this stream, since an answer that was kept would not hold for another one.  That takes 0.3 us of host time, a thirtieth of
  // the shortest calls, whose clusters fit on two SMs; contexts get those in pairs.
  const auto placeable = [&](int C) {
    if (C <= 2 * STAT_CTAS) return true;
    if (C > 8 && cudaFuncSetAttribute(colstat_kernel<true, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)   // kept per context
      return (void)cudaGetLastError(), false;
    return max_active_clusters(colstat_kernel<true, true>, cluster_grid(C), dim3(STAT_THREADS), 0, st) > 0;
  };
  const StatSplit split = stat_split((long long)heads * B, N, max_slices, STAT_CTAS, n_sm, placeable);
  const int S = split.slices;
  if (split.clusters) {
    MPFA_CUDA_OK(launch(colstat_kernel<true, true>, cluster_grid(S), dim3(STAT_THREADS), 0, st, c0, c1, B, S, smooth ? 1 : 0, v));
    return MPFA_OK;
  }
  MPFA_CUDA_OK(launch(v.x ? colstat_kernel<false, true> : colstat_kernel<false, false>, dim3((unsigned)((long long)S * heads * B + v_ctas)),
                      dim3(STAT_THREADS), 0, st, c0, c1, B, S, smooth ? 1 : 0, v));
  if (S > 1) MPFA_CUDA_OK(launch(stat_fold_kernel, dim3(heads, B), dim3(128), 0, st, c0, c1, S, smooth ? 1 : 0));
  return MPFA_OK;
}

}  // namespace
}  // namespace mpfa

using namespace mpfa;

extern "C" size_t mpfa_quantize_workspace_bytes(int B, int H_q, int H_kv) {
  if (B <= 0 || H_q <= 0 || H_kv <= 0) return 0;
  return stats_fixed_bytes(B, H_q, H_kv) + (size_t)STAT_MAX_SLICES * stats_slice_bytes(B, H_q, H_kv);
}

extern "C" size_t mpfa_quantize_workspace_min_bytes(int B, int H_q, int H_kv) {
  if (B <= 0 || H_q <= 0 || H_kv <= 0) return 0;
  return stats_fixed_bytes(B, H_q, H_kv) + stats_slice_bytes(B, H_q, H_kv);
}

static mpfa_status quantize_qkv(const void *q_bf16, const void *k_bf16, const VTensor &v, int B, int N_q, int N_kv, int H_q,
                                int H_kv, int flags, mpfa_stats *st, mpfa_fp4_tensor *q_out,
                                mpfa_fp4_tensor *k_out, void *delta_s_bf16, void *workspace,
                                size_t workspace_bytes, void *stream) {
  const bool smooth = flags & MPFA_SMOOTH, frozen = flags & MPFA_STATS_FROZEN;
  if (!st || (!q_bf16 && !k_bf16) || B <= 0 || H_q <= 0 || H_kv <= 0) return MPFA_ERR_INVALID_ARG;
  if ((q_bf16 && (N_q <= 0 || !q_out)) || (k_bf16 && (N_kv <= 0 || !k_out))) return MPFA_ERR_INVALID_ARG;
  if (!st->q_mean || !st->k_mean || !st->q_gscale || !st->k_gscale) return MPFA_ERR_INVALID_ARG;
  if (H_q % H_kv != 0 || H_q / H_kv > 8) return MPFA_ERR_UNSUPPORTED;
  if (N_q > (1 << 24) || N_kv > (1 << 24)) return MPFA_ERR_UNSUPPORTED;
  if (smooth && k_bf16 && !delta_s_bf16) return MPFA_ERR_INVALID_ARG;
  if (smooth && !q_bf16 && !frozen) return MPFA_ERR_INVALID_ARG;  // Delta_S needs the query mean
  if (q_bf16 && (q_out->B != B || q_out->H != H_q || q_out->N != N_q || !q_out->codes || !q_out->sf))
    return MPFA_ERR_INVALID_ARG;
  if (k_bf16 && (k_out->B != B || k_out->H != H_kv || k_out->N != N_kv || !k_out->codes || !k_out->sf))
    return MPFA_ERR_INVALID_ARG;
  if (!aligned(q_bf16, 16) || !aligned(k_bf16, 16) || !aligned(delta_s_bf16, 256)) return MPFA_ERR_ALIGNMENT;
  if (q_bf16 && (!aligned(q_out->codes, 1024) || !aligned(q_out->sf, 1024))) return MPFA_ERR_ALIGNMENT;
  if (k_bf16 && (!aligned(k_out->codes, 1024) || !aligned(k_out->sf, 1024))) return MPFA_ERR_ALIGNMENT;
  StatsWorkspace w{};
  if (!frozen) {
    if (!workspace) return MPFA_ERR_INVALID_ARG;
    if (!aligned(workspace, 256)) return MPFA_ERR_ALIGNMENT;
    w = carve(workspace, workspace_bytes, B, H_q, H_kv);
    if (w.slices < 1) return MPFA_ERR_WORKSPACE;
  }
  int dev = 0, n_sm = 0;
  mpfa_status rc = device_info(&dev, &n_sm);
  if (rc != MPFA_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const __nv_bfloat16 *q = static_cast<const __nv_bfloat16 *>(q_bf16);
  const __nv_bfloat16 *k = static_cast<const __nv_bfloat16 *>(k_bf16);
  // V has a launch of its own where there is no other, and for the largest tensors.  Together the two are 1 to 4 % faster (40:8 heads, together /
  // apart: 16384 tokens, 201 MB of Q and K, 92.8 / 95.3 us; 24576, 302 MB 132.2 / 134.8; 40960, 503 MB 213.1 / 216.3; 49152, 604 MB 254.6 /
  // 261.0; 65536, 805 MB 335.2 / 337.7), but in some placements of the tensors in memory the statistics with V take 1.6 times as long
  // (49152 419 us, 65536 555), where those alone kept their time; below the line such placements slow both forms (32768 283 us).
  const bool apart = v.x && (frozen || ((long long)N_q * (q ? H_q : 0) + (long long)N_kv * (k ? H_kv : 0)) * B * HEAD_DIM * 2 > V_APART);
  if (!frozen) {
    rc = tensor_stats(ColTensor{q, N_q, q ? H_q : 0, w.psum_q, w.pext_q, st->q_mean, w.gmax_q},
                      ColTensor{k, N_kv, k ? H_kv : 0, w.psum_k, w.pext_k, st->k_mean, w.gmax_k}, B, w.slices, n_sm, smooth, apart ? VTensor{} : v, s);
    if (rc != MPFA_OK) return rc;
  }
  if (apart) MPFA_CUDA_OK(launch(quantize_v_tile_kernel, dim3(v.tiles, v.H, B), dim3(256), 0, s, v));
  // Q and K tiles in one launch; with smoothing the K tiles also produce Delta_S (Eq. 9)
  const TensorScale sq{st->q_gscale, frozen ? nullptr : w.gmax_q, H_q}, sk{st->k_gscale, frozen ? nullptr : w.gmax_k, H_kv};
  QuantTensor tq{q, st->q_mean, sq, N_q, q ? H_q : 0, q ? pad128(N_q) / TILE : 0, 0, q ? q_out->codes : nullptr, q ? q_out->sf : nullptr};
  QuantTensor tk{k, st->k_mean, sk, N_kv, k ? H_kv : 0, k ? pad128(N_kv) / TILE : 0, 0, k ? k_out->codes : nullptr, k ? k_out->sf : nullptr};
  const DeltaArgs da{st->q_mean, sq, k && smooth ? static_cast<__nv_bfloat16 *>(delta_s_bf16) : nullptr, H_q};
  if (!k && N_q <= 8) {
    MPFA_CUDA_OK(launch(vector_means(tq.mean) ? quantize_token_kernel<true> : quantize_token_kernel<false>, dim3((B * H_q + 7) / 8), dim3(256), 0, s, tq, B * H_q));
    return MPFA_OK;
  }
  // At most one wave of CTAs where every head can have one: a CTA's set-up (scale, table of reciprocals, query means) is paid
  // once, and the next tile's loads run under the arithmetic of the current one.  A few CTAs more than a wave would take twice
  // the time.
  const int k_weight = da.delta && H_q / H_kv > 2 ? QT_K_WEIGHT : 1;
  const long long work = ((long long)k_weight * tk.tiles * tk.H + (long long)tq.tiles * tq.H) * B, wave = (long long)QT_CTAS * n_sm;
  const auto split = [&](long long per) {   // CTAs of `per` units of work; how many that makes
    const long long per_k = (per + k_weight - 1) / k_weight;
    tk.ctas = tk.x ? (int)((tk.tiles + per_k - 1) / per_k) : 0;
    tq.ctas = tq.x ? (int)((tq.tiles + per - 1) / per) : 0;
    return ((long long)tk.ctas * tk.H + (long long)tq.ctas * tq.H) * B;
  };
  const long long mean = (work + wave - 1) / wave;
  if (((long long)tk.H + tq.H) * B <= wave) {
    for (long long per = std::max(1LL, mean / 2); split(per) > wave; ++per) {}   // the shortest Q tasks that fit
  } else {
    // More heads than a wave has CTAs: the work with its set-ups spread over the SMs, and one CTA's length at the end.  (One CTA
    // per head here left one query token on 9 x 4865 keys, 40:8 heads, at 219 us of stage 1, now 127; 10 x 5647 467 -> 406;
    // 16 x 2000, 32:8 heads, 254 -> 210; set-ups of 0.2 / 0.5 / 1 / 2 units 143 / 143 / 129 / 127 us for the first.)
    long long best = 1;
    double best_time = 1e30;
    for (long long per = 1; per <= 2 * mean; per *= 2) {
      const long long ctas = split(per);
      const long long longest = std::min(per, std::max<long long>(tq.tiles, (long long)k_weight * tk.tiles));
      const double time = (double)(work + QT_SETUP * ctas) / (double)wave + (double)longest;
      if (time < best_time) best_time = time, best = per;
    }
    split(best);
  }
  const int few = da.delta && H_q / H_kv <= 2 ? H_q / H_kv : 0;
  MPFA_CUDA_OK(launch(few == 0 ? quantize_tile_kernel<0> : few == 1 ? quantize_tile_kernel<1> : quantize_tile_kernel<2>,
                      dim3(tk.ctas * tk.H + tq.ctas * tq.H, 1, B), dim3(256), 0, s, tk, tq, da));
  return MPFA_OK;
}

extern "C" mpfa_status mpfa_quantize_qk(const void *q_bf16, const void *k_bf16, int B, int N_q, int N_kv, int H_q,
                                        int H_kv, int flags, mpfa_stats *st, mpfa_fp4_tensor *q_out,
                                        mpfa_fp4_tensor *k_out, void *delta_s_bf16, void *workspace,
                                        size_t workspace_bytes, void *stream) {
  return quantize_qkv(q_bf16, k_bf16, VTensor{}, B, N_q, N_kv, H_q, H_kv, flags, st, q_out, k_out, delta_s_bf16, workspace, workspace_bytes, stream);
}

extern "C" mpfa_status mpfa_quantize_qkv(const void *q_bf16, const void *k_bf16, const void *v_bf16, int B, int N_q, int N_kv, int H_q,
                                         int H_kv, int flags, float v_scale, mpfa_stats *st, mpfa_fp4_tensor *q_out,
                                         mpfa_fp4_tensor *k_out, uint8_t *v_fp8, void *delta_s_bf16, void *workspace,
                                         size_t workspace_bytes, void *stream) {
  if (!v_bf16 || !v_fp8 || B <= 0 || N_kv <= 0 || H_kv <= 0 || !(v_scale > 0.0f)) return MPFA_ERR_INVALID_ARG;
  if (!aligned(v_bf16, 16) || !aligned(v_fp8, 1024)) return MPFA_ERR_ALIGNMENT;
  if (B > 65535 || H_kv > 65535) return MPFA_ERR_UNSUPPORTED;   // as mpfa_quantize_v, whose launch fails
  const VTensor v{static_cast<const __nv_bfloat16 *>(v_bf16), N_kv, H_kv, pad128(N_kv) / TILE, 1.0f / v_scale, v_fp8};
  return quantize_qkv(q_bf16, k_bf16, v, B, N_q, N_kv, H_q, H_kv, flags, st, q_out, k_out, delta_s_bf16, workspace, workspace_bytes, stream);
}

extern "C" mpfa_status mpfa_quantize_v(const void *v_bf16, int B, int N_kv, int H_kv, float v_scale, uint8_t *v_fp8,
                                       void *stream) {
  if (!v_bf16 || !v_fp8 || B <= 0 || N_kv <= 0 || H_kv <= 0 || !(v_scale > 0.0f)) return MPFA_ERR_INVALID_ARG;
  if (!aligned(v_bf16, 16) || !aligned(v_fp8, 1024)) return MPFA_ERR_ALIGNMENT;
  int dev = 0, n_sm = 0;
  mpfa_status rc = device_info(&dev, &n_sm);
  if (rc != MPFA_OK) return rc;
  dim3 grid(pad128(N_kv) / TILE, H_kv, B);
  MPFA_CUDA_OK(launch(quantize_v_tile_kernel, grid, dim3(256), 0, static_cast<cudaStream_t>(stream),
                      VTensor{static_cast<const __nv_bfloat16 *>(v_bf16), N_kv, H_kv, pad128(N_kv) / TILE, 1.0f / v_scale, v_fp8}));
  return MPFA_OK;
}

extern "C" mpfa_status mpfa_pack_v_bf16(const void *v_bf16, int B, int N_kv, int H_kv, void *v_tiles_bf16, void *stream) {
  if (!v_bf16 || !v_tiles_bf16 || B <= 0 || N_kv <= 0 || H_kv <= 0) return MPFA_ERR_INVALID_ARG;
  if (!aligned(v_bf16, 16) || !aligned(v_tiles_bf16, 1024)) return MPFA_ERR_ALIGNMENT;
  int dev = 0, n_sm = 0;
  mpfa_status rc = device_info(&dev, &n_sm);
  if (rc != MPFA_OK) return rc;
  pack_v_bf16_kernel<<<dim3(pad128(N_kv) / TILE, H_kv, B), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<const __nv_bfloat16 *>(v_bf16), N_kv, H_kv, static_cast<__nv_bfloat16 *>(v_tiles_bf16));
  MPFA_LAUNCH_OK();
  return MPFA_OK;
}

extern "C" size_t mpfa_v_fp4_bytes(int B, int H_kv, int N_kv) {
  if (B <= 0 || H_kv <= 0 || N_kv <= 0) return 0;
  return (size_t)B * H_kv * (pad128(N_kv) / TILE) * (8192 + 1024);
}

extern "C" mpfa_status mpfa_quantize_v_fp4(const void *v_bf16, int B, int N_kv, int H_kv, float v_gscale, uint8_t *v_fp4,
                                           void *stream) {
  if (!v_bf16 || !v_fp4 || B <= 0 || N_kv <= 0 || H_kv <= 0 || !(v_gscale > 0.0f)) return MPFA_ERR_INVALID_ARG;
  if (!aligned(v_bf16, 16) || !aligned(v_fp4, 1024)) return MPFA_ERR_ALIGNMENT;
  int dev = 0, n_sm = 0;
  mpfa_status rc = device_info(&dev, &n_sm);
  if (rc != MPFA_OK) return rc;
  const size_t n_tiles = (size_t)B * H_kv * (pad128(N_kv) / TILE);
  quantize_v_fp4_tile_kernel<<<dim3(pad128(N_kv) / TILE, H_kv, B), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<const __nv_bfloat16 *>(v_bf16), N_kv, H_kv, v_gscale, v_fp4, v_fp4 + n_tiles * 8192);
  MPFA_LAUNCH_OK();
  return MPFA_OK;
}

extern "C" mpfa_status mpfa_quantize_kv_paged(const void *k_bf16, const void *v_bf16, int N_tokens, int first_token,
                                              int H_q, int H_kv, int flags, mpfa_stats *st, float v_scale,
                                              const mpfa_paged_kv *kv, const int32_t *page_table_row,
                                              void *workspace, size_t workspace_bytes, void *stream) {
  const bool smooth = flags & MPFA_SMOOTH, frozen = flags & MPFA_STATS_FROZEN;
  if (!k_bf16 || !v_bf16 || !st || !kv || !page_table_row || N_tokens <= 0 || first_token < 0 || H_q <= 0 ||
      H_kv <= 0 || !(v_scale > 0.0f))
    return MPFA_ERR_INVALID_ARG;
  if (!st->q_mean || !st->k_mean || !st->q_gscale || !st->k_gscale) return MPFA_ERR_INVALID_ARG;
  if (!kv->k_codes || !kv->k_sf || !kv->v_fp8 || kv->num_pages <= 0) return MPFA_ERR_INVALID_ARG;
  if (smooth && !kv->delta_s_bf16) return MPFA_ERR_INVALID_ARG;
  if (kv->page_size != PAGE || H_q % H_kv != 0 || H_q / H_kv > 8) return MPFA_ERR_UNSUPPORTED;
  if (kv->H_q != H_q || kv->H_kv != H_kv) return MPFA_ERR_INVALID_ARG;
  if (!frozen && first_token != 0) return MPFA_ERR_INVALID_ARG;
  if (!aligned(k_bf16, 16) || !aligned(v_bf16, 16) || !aligned(kv->k_codes, 256) || !aligned(kv->k_sf, 256) ||
      !aligned(kv->v_fp8, 256) || !aligned(kv->delta_s_bf16, 256))
    return MPFA_ERR_ALIGNMENT;
  StatsWorkspace w{};
  if (!frozen) {
    if (!workspace) return MPFA_ERR_INVALID_ARG;
    if (!aligned(workspace, 256)) return MPFA_ERR_ALIGNMENT;
    w = carve(workspace, workspace_bytes, 1, H_q, H_kv);
    if (w.slices < 1) return MPFA_ERR_WORKSPACE;
  }
  int dev = 0, n_sm = 0;
  mpfa_status rc = device_info(&dev, &n_sm);
  if (rc != MPFA_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const __nv_bfloat16 *k = static_cast<const __nv_bfloat16 *>(k_bf16);
  const __nv_bfloat16 *v = static_cast<const __nv_bfloat16 *>(v_bf16);
  if (!frozen) {
    rc = tensor_stats(ColTensor{k, N_tokens, H_kv, w.psum_k, w.pext_k, st->k_mean, w.gmax_k}, ColTensor{}, 1, w.slices, n_sm, smooth, VTensor{}, s);
    if (rc != MPFA_OK) return rc;
  }
  const TensorScale sk{st->k_gscale, frozen ? nullptr : w.gmax_k, H_kv};
  const int n_pages = (first_token + N_tokens - 1) / PAGE - first_token / PAGE + 1;
  const long long wave = (long long)WK_CTAS * n_sm;
  const int per_cta = (int)(((long long)n_pages * H_kv + wave - 1) / wave);
  MPFA_CUDA_OK(launch(write_kv_kernel, dim3(H_kv, (n_pages + per_cta - 1) / per_cta), dim3(256), 0, s, k, v, st->k_mean, sk, st->q_mean,
                      st->q_gscale, N_tokens, first_token, n_pages, H_q, H_kv, 1.0f / v_scale, page_table_row, kv->num_pages,
                      kv->k_codes, kv->k_sf, kv->v_fp8, smooth ? static_cast<__nv_bfloat16 *>(kv->delta_s_bf16) : nullptr));
  return MPFA_OK;
}

// ---------------------------------------------------------------------------------------
extern "C" mpfa_status mpfa_append_kv_paged(const void *k_bf16, const void *v_bf16, int B, int H_q, int H_kv, int flags,
                                            const mpfa_stats *st, float v_scale, const mpfa_paged_kv *kv,
                                            const int32_t *page_table, int max_pages_per_req,
                                            const int32_t *positions, void *stream) {
  const bool smooth = flags & MPFA_SMOOTH;
  if (!k_bf16 || !v_bf16 || !st || !kv || !page_table || !positions || B <= 0 || H_q <= 0 || H_kv <= 0 ||
      max_pages_per_req <= 0 || !(v_scale > 0.0f))
    return MPFA_ERR_INVALID_ARG;
  if (!st->k_mean || !st->k_gscale || (smooth && (!st->q_mean || !st->q_gscale))) return MPFA_ERR_INVALID_ARG;
  if (!kv->k_codes || !kv->k_sf || !kv->v_fp8 || kv->num_pages <= 0) return MPFA_ERR_INVALID_ARG;
  if (smooth && !kv->delta_s_bf16) return MPFA_ERR_INVALID_ARG;
  if (kv->page_size != PAGE || H_q % H_kv != 0 || H_q / H_kv > 8 || B > 65535) return MPFA_ERR_UNSUPPORTED;
  if (kv->H_q != H_q || kv->H_kv != H_kv) return MPFA_ERR_INVALID_ARG;
  if (!aligned(k_bf16, 16) || !aligned(v_bf16, 16) || !aligned(kv->k_codes, 256) || !aligned(kv->k_sf, 256) ||
      !aligned(kv->v_fp8, 256) || !aligned(kv->delta_s_bf16, 256))
    return MPFA_ERR_ALIGNMENT;
  int dev = 0, n_sm = 0;
  mpfa_status rc = device_info(&dev, &n_sm);
  if (rc != MPFA_OK) return rc;
  const bool vec = vector_means(st->k_mean) && vector_means(st->q_mean);
  MPFA_CUDA_OK(launch(vec ? append_kv_kernel<true> : append_kv_kernel<false>, dim3((B * H_kv + 7) / 8), dim3(256), 0, static_cast<cudaStream_t>(stream),
                      static_cast<const __nv_bfloat16 *>(k_bf16), static_cast<const __nv_bfloat16 *>(v_bf16), st->q_mean, st->k_mean,
                      st->q_gscale, st->k_gscale, B, H_q, H_kv, 1.0f / v_scale, page_table, max_pages_per_req, kv->num_pages,
                      positions, kv->k_codes, kv->k_sf, kv->v_fp8,
                      smooth ? static_cast<__nv_bfloat16 *>(kv->delta_s_bf16) : nullptr));
  return MPFA_OK;
}

// mpfa_quantize_qk_static: the same stage-1 call for callers that cannot provide scratch.
// ---------------------------------------------------------------------------------------
namespace mpfa {
namespace {

// Scratch for the column sums and maxima, resident in every device that loads the library.
constexpr size_t STATIC_SCRATCH_BYTES = MPFA_STATIC_SCRATCH_BYTES;
static __device__ __align__(256) unsigned char g_static_scratch[STATIC_SCRATCH_BYTES];

void *g_static_scratch_addr[MAX_DEVICES] = {};
std::mutex g_static_scratch_mutex;

// In host code the array's name is only a handle; the device address has to be asked for,
// once per device, with that device current.
mpfa_status static_scratch_address(void **out) {
  int dev = 0;
  MPFA_CUDA_OK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= MAX_DEVICES) return MPFA_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_static_scratch_mutex);
  if (!g_static_scratch_addr[dev]) {
    void *ptr = nullptr;
    MPFA_CUDA_OK(cudaGetSymbolAddress(&ptr, g_static_scratch));
    g_static_scratch_addr[dev] = ptr;
  }
  *out = g_static_scratch_addr[dev];
  return MPFA_OK;
}

}  // namespace
}  // namespace mpfa

extern "C" size_t mpfa_static_scratch_bytes(void) { return STATIC_SCRATCH_BYTES; }

extern "C" mpfa_status mpfa_quantize_qk_static(const void *q_bf16, const void *k_bf16, int B, int N_q, int N_kv,
                                               int H_q, int H_kv, int flags, mpfa_stats *st, mpfa_fp4_tensor *q_out,
                                               mpfa_fp4_tensor *k_out, void *delta_s_bf16, void *stream) {
  if (B <= 0 || H_q <= 0 || H_kv <= 0) return MPFA_ERR_INVALID_ARG;
  // with frozen statistics nothing is accumulated: no scratch is touched, so no size limit applies
  if (flags & MPFA_STATS_FROZEN)
    return mpfa_quantize_qk(q_bf16, k_bf16, B, N_q, N_kv, H_q, H_kv, flags, st, q_out, k_out, delta_s_bf16, nullptr, 0,
                            stream);
  if (stats_fixed_bytes(B, H_q, H_kv) + stats_slice_bytes(B, H_q, H_kv) > STATIC_SCRATCH_BYTES) return MPFA_ERR_WORKSPACE;
  void *scratch = nullptr;
  mpfa_status rc = static_scratch_address(&scratch);
  if (rc != MPFA_OK) return rc;
  return mpfa_quantize_qk(q_bf16, k_bf16, B, N_q, N_kv, H_q, H_kv, flags, st, q_out, k_out, delta_s_bf16, scratch,
                          STATIC_SCRATCH_BYTES, stream);
}

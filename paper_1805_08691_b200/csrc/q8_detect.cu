// The SSD tail of the 8-bit path and the FP32 route for signed residual sums.
//
// The paper runs SSD with a detection-output layer (artifact appendix) and sends potentially negative activations
// through FP32 (Sec. "8-bit Low Precision Inference", calibration paragraph) without printing arithmetic for either;
// the kernels below follow the detector's published definition, every floating-point step one IEEE fp32 operation
// in a fixed order (the library is built without contraction; fused steps are written as fused):
//   * L2 normalisation across channels on 8-bit codes (one warp per pixel, integer sum of squares by dp4a);
//   * Q_8(max(a + b, 0), q): the FP32 sum, ReLU and re-quantization of two dequantized convolution outputs;
//   * detection output: box decoding and softmax (exponentials only for boxes that can hold a candidate), per (image, class) candidate selection by a
//     bitonic sort in shared memory and greedy suppression over a bit matrix of overlaps, per-image selection of
//     the best detections.
#include <atomic>
#include <cfloat>
#include <cmath>

#include "q8_internal.h"

namespace q8 {
namespace {

// ------------------------------------------------------------------------------------------ L2 normalisation
//   S = sum_c z_c^2,  r = 1 / sqrt(float(S) * (q_x * q_x) + eps),  y_c = clamp(Round((float(z_c) * m_c) * r), 0, 255)
__device__ __forceinline__ unsigned int l2_word(unsigned int w, const float4 m, float r) {
  // byte -> float without a conversion instruction: 0x4B0000bb is 2^23 + b exactly
  const float f0 = __fsub_rn(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7540u)), 8388608.0f);
  const float f1 = __fsub_rn(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7541u)), 8388608.0f);
  const float f2 = __fsub_rn(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7542u)), 8388608.0f);
  const float f3 = __fsub_rn(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7543u)), 8388608.0f);
  const float v0 = __fmul_rn(__fmul_rn(f0, m.x), r), v1 = __fmul_rn(__fmul_rn(f1, m.y), r);
  const float v2 = __fmul_rn(__fmul_rn(f2, m.z), r), v3 = __fmul_rn(__fmul_rn(f3, m.w), r);
  unsigned int b0, b1, b2, b3;
  asm("cvt.rni.sat.u8.f32 %0, %1;" : "=r"(b0) : "f"(v0));
  asm("cvt.rni.sat.u8.f32 %0, %1;" : "=r"(b1) : "f"(v1));
  asm("cvt.rni.sat.u8.f32 %0, %1;" : "=r"(b2) : "f"(v2));
  asm("cvt.rni.sat.u8.f32 %0, %1;" : "=r"(b3) : "f"(v3));
  return __byte_perm(__byte_perm(b0, b1, 0x0040u), __byte_perm(b2, b3, 0x0040u), 0x5410u);
}

__device__ __forceinline__ float l2_recip(unsigned int s, float qx2, float eps) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return __fdiv_rn(1.0f, __fsqrt_rn(__fadd_rn(__fmul_rn((float)s, qx2), eps)));
}

// A warp takes two pixels per step (all loads of both are issued before the first sum is reduced), C a multiple of
// 4 and rows 4-byte aligned: a lane takes words lane, lane + 32, ... of each pixel, kept in registers (kL2Words
// words per lane: up to 512 channels; wider rows take the kernel below).
constexpr int kL2Words = 4;
__global__ void __launch_bounds__(256) l2norm_kernel(const unsigned int* __restrict__ x, size_t pixels, int cw, float qx2,
                                                     float eps, const float4* __restrict__ mult, unsigned int* __restrict__ y) {
  const int lane = threadIdx.x & 31;
  const size_t warp = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = ((size_t)gridDim.x * blockDim.x) >> 5;
  float4 m[kL2Words];
#pragma unroll
  for (int j = 0; j < kL2Words; ++j) m[j] = lane + 32 * j < cw ? __ldg(mult + lane + 32 * j) : make_float4(0.f, 0.f, 0.f, 0.f);
  for (size_t p = 2 * warp; p < pixels; p += 2 * nwarps) {
    const bool two = p + 1 < pixels;
    const unsigned int* row0 = x + p * (size_t)cw;
    const unsigned int* row1 = row0 + (two ? cw : 0);
    unsigned int w0[kL2Words], w1[kL2Words];
#pragma unroll
    for (int j = 0; j < kL2Words; ++j) {
      const int i = lane + 32 * j;
      w0[j] = i < cw ? __ldcs(row0 + i) : 0u;
      w1[j] = i < cw ? __ldcs(row1 + i) : 0u;
    }
    unsigned int s0 = 0, s1 = 0;  // at most 2048 channels of 255^2: far below 2^32
#pragma unroll
    for (int j = 0; j < kL2Words; ++j) { s0 = __dp4a(w0[j], w0[j], s0); s1 = __dp4a(w1[j], w1[j], s1); }
    const float r0 = l2_recip(s0, qx2, eps), r1 = l2_recip(s1, qx2, eps);
    unsigned int* out0 = y + p * (size_t)cw;
#pragma unroll
    for (int j = 0; j < kL2Words; ++j) {
      const int i = lane + 32 * j;
      if (i < cw) {
        __stcs(out0 + i, l2_word(w0[j], m[j], r0));
        if (two) __stcs(out0 + cw + i, l2_word(w1[j], m[j], r1));
      }
    }
  }
}

// Rows wider than the registers of the kernel above hold (C % 4 == 0): one warp per pixel, the row is read twice.
__global__ void __launch_bounds__(256) l2norm_wide_kernel(const unsigned int* __restrict__ x, size_t pixels, int cw, float qx2,
                                                          float eps, const float4* __restrict__ mult, unsigned int* __restrict__ y) {
  const int lane = threadIdx.x & 31;
  const size_t warp = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = ((size_t)gridDim.x * blockDim.x) >> 5;
  for (size_t p = warp; p < pixels; p += nwarps) {
    const unsigned int* row = x + p * (size_t)cw;
    unsigned int s = 0;  // at most 65536 channels of 255^2: below 2^32
    for (int i = lane; i < cw; i += 32) {
      const unsigned int v = __ldg(row + i);
      s = __dp4a(v, v, s);
    }
    const float r = l2_recip(s, qx2, eps);
    unsigned int* out = y + p * (size_t)cw;
    for (int i = lane; i < cw; i += 32) out[i] = l2_word(__ldg(row + i), __ldg(mult + i), r);
  }
}

// any C: one thread per pixel
__global__ void __launch_bounds__(256) l2norm_scalar_kernel(const unsigned char* __restrict__ x, size_t pixels, int C, float qx2,
                                                            float eps, const float* __restrict__ mult, unsigned char* __restrict__ y) {
  const size_t n = (size_t)gridDim.x * blockDim.x;
  for (size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x; p < pixels; p += n) {
    const unsigned char* row = x + p * (size_t)C;
    unsigned long long s = 0;
    for (int c = 0; c < C; ++c) s += (unsigned int)row[c] * (unsigned int)row[c];
    const float r = __fdiv_rn(1.0f, __fsqrt_rn(__fadd_rn(__fmul_rn((float)s, qx2), eps)));
    for (int c = 0; c < C; ++c) {
      unsigned int b;
      asm("cvt.rni.sat.u8.f32 %0, %1;" : "=r"(b) : "f"(__fmul_rn(__fmul_rn((float)row[c], mult[c]), r)));
      y[p * (size_t)C + c] = (unsigned char)b;
    }
  }
}

// ------------------------------------------------------------------------------------------ FP32 route of a sum
// y = clamp(Round(max(a + b, 0) / q), 0, 255): 32 bytes of fp32 in, 4 bytes out per thread and step.
__device__ __forceinline__ unsigned int arq1(float a, float b, float q) {
  unsigned int r;
  asm("cvt.rni.sat.u8.f32 %0, %1;" : "=r"(r) : "f"(__fdiv_rn(fmaxf(__fadd_rn(a, b), 0.0f), q)));
  return r;
}
__global__ void __launch_bounds__(512) add_relu_quantize_kernel(const float4* __restrict__ a, const float4* __restrict__ b, size_t n4,
                                                                float q, unsigned int* __restrict__ y) {
  const size_t nthreads = (size_t)gridDim.x * blockDim.x;
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (; i + nthreads < n4; i += 2 * nthreads) {
    const float4 a0 = __ldcs(a + i), b0 = __ldcs(b + i), a1 = __ldcs(a + i + nthreads), b1 = __ldcs(b + i + nthreads);
    y[i] = arq1(a0.x, b0.x, q) | (arq1(a0.y, b0.y, q) << 8) | (arq1(a0.z, b0.z, q) << 16) | (arq1(a0.w, b0.w, q) << 24);
    y[i + nthreads] = arq1(a1.x, b1.x, q) | (arq1(a1.y, b1.y, q) << 8) | (arq1(a1.z, b1.z, q) << 16) | (arq1(a1.w, b1.w, q) << 24);
  }
  for (; i < n4; i += nthreads) {
    const float4 a0 = __ldcs(a + i), b0 = __ldcs(b + i);
    y[i] = arq1(a0.x, b0.x, q) | (arq1(a0.y, b0.y, q) << 8) | (arq1(a0.z, b0.z, q) << 16) | (arq1(a0.w, b0.w, q) << 24);
  }
}
__global__ void __launch_bounds__(256) add_relu_quantize_tail_kernel(const float* __restrict__ a, const float* __restrict__ b,
                                                                     size_t first, size_t n, float q, unsigned char* __restrict__ y) {
  const size_t i = first + (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = (unsigned char)arq1(a[i], b[i], q);
}

// ------------------------------------------------------------------------------------------ detection output
// exp(x) by a fixed recipe, so that a confidence has the same bits wherever it is computed: clamp to [-87, 88],
// k = Round(x log2 e), r = x - k ln2 in two fused steps, degree-7 Taylor polynomial by fused Horner steps, times 2^k.
__device__ __forceinline__ float exp_fixed(float x) {
  x = x < -87.0f ? -87.0f : (x > 88.0f ? 88.0f : x);
  const float k = rintf(__fmul_rn(x, 1.44269504088896341f));
  float r = __fmaf_rn(-k, 0.693145751953125f, x);
  r = __fmaf_rn(-k, 1.42860682030941723e-6f, r);
  float p = 1.0f / 5040.0f;
  p = __fmaf_rn(p, r, 1.0f / 720.0f);
  p = __fmaf_rn(p, r, 1.0f / 120.0f);
  p = __fmaf_rn(p, r, 1.0f / 24.0f);
  p = __fmaf_rn(p, r, 1.0f / 6.0f);
  p = __fmaf_rn(p, r, 0.5f);
  p = __fmaf_rn(p, r, 1.0f);
  p = __fmaf_rn(p, r, 1.0f);
  return __fmul_rn(p, __int_as_float(((int)k + 127) << 23));
}

// The same for x <= 0 (or NaN), in fewer instructions: the upper clamp cannot apply; adding 1.5 * 2^23 rounds x log2 e to
// the nearest integer, ties to even, and leaves that integer in the low mantissa bits, from where it shifts into the
// exponent of the scale.  Identical results.
__device__ __forceinline__ float exp_fixed_neg(float x) {
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(x) : "f"(x), "f"(-87.0f));
  const float t = __fadd_rn(__fmul_rn(x, 1.44269504088896341f), 12582912.0f);
  const float k = __fsub_rn(t, 12582912.0f);
  float r = __fmaf_rn(-k, 0.693145751953125f, x);
  r = __fmaf_rn(-k, 1.42860682030941723e-6f, r);
  float p = 1.0f / 5040.0f;
  p = __fmaf_rn(p, r, 1.0f / 720.0f);
  p = __fmaf_rn(p, r, 1.0f / 120.0f);
  p = __fmaf_rn(p, r, 1.0f / 24.0f);
  p = __fmaf_rn(p, r, 1.0f / 6.0f);
  p = __fmaf_rn(p, r, 0.5f);
  p = __fmaf_rn(p, r, 1.0f);
  p = __fmaf_rn(p, r, 1.0f);
  return __fmul_rn(p, __int_as_float((__float_as_int(t) << 23) + 0x3f800000));
}

constexpr int kMaxSources = 8;
constexpr int kRegClasses = 24;   // class counts up to this keep a block's logits in shared memory
struct DetSources {
  const float* loc[kMaxSources];
  const float* conf[kMaxSources];
  int loc_stride[kMaxSources], conf_stride[kMaxSources];  // floats between consecutive cells
  int cells[kMaxSources], boxes[kMaxSources];              // cells per image, boxes per cell
  int first[kMaxSources + 1];                              // first prior of each source
  int n;
};

// Decoded corner boxes and class probabilities:
//   cx = (v0 l0) pw + pcx, cy = (v1 l1) ph + pcy, w = exp(v2 l2) pw, h = exp(v3 l3) ph, corners = centre -+ half
//   e_c = exp(x_c - max x), p_c = e_c / sum_c e_c (sum in class order)
// boxes: [N][P] float4.  Only candidates (p_c > conf_thresh, c not the background) leave the kernels: bit p of
// masks[n][c] says whether box p is one, and only then prob[n][c][p] is written, and boxes[n][p] for boxes that may hold one.
// e_c below 0.99 conf_thresh sum cannot be one (the quotient is off by 2^-24 at most), which saves its division.

// Prior q of image n: its regression and class values.
__device__ __forceinline__ void det_source(const DetSources& src, int n, int q, int classes, const float** l, const float** x) {
  int s = 0;
#pragma unroll
  for (int j = 1; j < kMaxSources; ++j)
    if (j < src.n && q >= src.first[j]) s = j;
  const int local = q - src.first[s];
  const int cell = local / src.boxes[s], b = local - cell * src.boxes[s];
  const size_t pix = (size_t)n * src.cells[s] + cell;
  *l = src.loc[s] + pix * src.loc_stride[s] + b * 4;
  *x = src.conf[s] + pix * src.conf_stride[s] + (size_t)b * classes;
}

__device__ __forceinline__ float4 det_box(const float* l, const float4 pr, float v0, float v1, float v2, float v3) {
  const float cx = __fadd_rn(__fmul_rn(__fmul_rn(v0, l[0]), pr.z), pr.x);
  const float cy = __fadd_rn(__fmul_rn(__fmul_rn(v1, l[1]), pr.w), pr.y);
  const float w = __fmul_rn(exp_fixed(__fmul_rn(v2, l[2])), pr.z);
  const float h = __fmul_rn(exp_fixed(__fmul_rn(v3, l[3])), pr.w);
  const float hw = __fmul_rn(w, 0.5f), hh = __fmul_rn(h, 0.5f);
  return make_float4(__fsub_rn(cx, hw), __fsub_rn(cy, hh), __fadd_rn(cx, hw), __fadd_rn(cy, hh));
}

constexpr int kDecThreads = 256;
constexpr int kDecFew = 64;  // boxes of a block where there are few

// Up to kRegClasses classes.  A block takes kBoxes boxes of an image (256, or 64 where there are few), whose logits travel
// through shared memory (a thread per box would touch 21 lines with every load).  Most boxes of a detector are background and
// need no exponential: the largest term of the sum is exp(0) = 1, so p_c <= e_c, and a box whose foreground logits all lie
// `cutoff` = ln(conf_thresh), less a margin for the recipe's roundings, or more below its largest has no candidate.  What is
// left (one box in six at a threshold of 0.01) is listed, and the block's threads share its (box, class) pairs.  A NaN among a
// box's logits makes its sum a NaN, so no class of it passes, whether the maxima (which skip a NaN) list it or not; infinities
// of one sign compare by a NaN difference, which lists.  One box per thread with all of its exponentials was bound by issue
// (1291 warp instructions per 32 boxes, 790 with a list but loads through registers, five blocks per SM): detection output of
// 32 images, 8732 boxes, 21 classes, replayed from a graph 45.8 -> 39.8 -> 36.7 us with eight resident blocks.
template <int kBoxes>
__global__ void __launch_bounds__(kDecThreads, 8) decode_listed_kernel(const __grid_constant__ DetSources src, const float4* __restrict__ priors,
                                                                       float v0, float v1, float v2, float v3, int P, int classes,
                                                                       int background, float conf_thresh, float cutoff, float4* __restrict__ boxes,
                                                                       float* __restrict__ prob, unsigned int* __restrict__ masks) {
  constexpr int kWords = kBoxes / 32;
  __shared__ __align__(16) float stage[kBoxes * kRegClasses];
  __shared__ float top[kBoxes], total[kBoxes];
  __shared__ unsigned int bits[kRegClasses][kWords];
  __shared__ unsigned short list[kBoxes];
  __shared__ int listed;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int n = blockIdx.y, lane = threadIdx.x & 31, PW = (P + 31) >> 5, tid = (int)threadIdx.x;
  const int p0 = blockIdx.x * kBoxes, p = p0 + tid;
  const bool mine = tid < kBoxes, live = mine && p < P;
  const float *l, *x;
  det_source(src, n, live ? p : P - 1, classes, &l, &x);
  if (tid == 0) listed = 0;
  if (tid < kRegClasses * kWords) bits[tid / kWords][tid % kWords] = 0u;
  if (mine && (p & ~31) < P) {  // whole warps
    float* st = stage + (tid & ~31) * classes;
    const float* x0 = reinterpret_cast<const float*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(x), 0));
    if (__all_sync(0xffffffffu, x == x0 + lane * classes)) {  // the warp's boxes lie one after the other
      // (asynchronous copies hold no registers: all blocks of 32 images of 8732 boxes are resident at once)
      if ((reinterpret_cast<unsigned long long>(x0) & 15u) == 0) {
        for (int c = lane; c < classes * 8; c += 32)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned int)__cvta_generic_to_shared(st + 4 * c)), "l"(x0 + 4 * c) : "memory");
      } else {
        for (int c = lane; c < classes * 32; c += 32)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned int)__cvta_generic_to_shared(st + c)), "l"(x0 + c) : "memory");
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
    } else {
      const unsigned int inv = 65536u / (unsigned)classes + 1u;  // k / classes for k < 32 * 24
      for (int c0 = 0; c0 < classes; c0 += 8) {  // eight loads in flight
        float t[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int k = (c0 + u) * 32 + lane, box = min((int)(((unsigned)k * inv) >> 16), 31);
          const float* xb = reinterpret_cast<const float*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(x), box));
          if (c0 + u < classes) t[u] = __ldg(xb + (k - box * classes));
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (c0 + u < classes) st[(c0 + u) * 32 + lane] = t[u];
      }
    }
  }
  __syncthreads();
  if (live) {
    // the largest foreground logit against the largest of all, which is that or the background's
    const float* xs = stage + tid * classes;
    float f = -INFINITY;
    const int bg = background < 0 ? classes : background;
#pragma unroll 4
    for (int c = 0; c < bg; ++c) f = fmaxf(f, xs[c]);
#pragma unroll 4
    for (int c = bg + 1; c < classes; ++c) f = fmaxf(f, xs[c]);
    const float m = bg < classes ? fmaxf(f, xs[bg]) : f;
    if (!(__fsub_rn(f, m) < cutoff)) list[atomicAdd(&listed, 1)] = (unsigned short)tid;
  }
  __syncthreads();
  const int count = listed, items = count * classes;
  if (tid < count) {  // the largest logit as the sum's terms see it (a NaN in front stays)
    const int b = list[tid];
    const float* xs = stage + b * classes;
    float m = xs[0];
#pragma unroll 4
    for (int c = 1; c < classes; ++c) m = xs[c] > m ? xs[c] : m;
    top[b] = m;
  }
  if (kDecThreads - 1 - tid < count) {  // its box, by other warps where the list is short
    const int q = p0 + list[kDecThreads - 1 - tid];
    det_source(src, n, q, classes, &l, &x);
    boxes[(size_t)n * P + q] = det_box(l, __ldg(priors + q), v0, v1, v2, v3);
  }
  __syncthreads();
  const unsigned int inv = (1u << 20) / (unsigned)classes + 1u;  // i / classes for i < 256 classes, classes <= 24
  for (int i = tid; i < items; i += kDecThreads) {
    const int k = (int)(((unsigned)i * inv) >> 20), c = i - k * classes, b = list[k];
    float* xs = stage + b * classes + c;
    *xs = exp_fixed_neg(__fsub_rn(*xs, top[b]));
  }
  __syncthreads();
  if (tid < count) {
    const int b = list[tid];
    const float* e = stage + b * classes;
    float sum = 0.0f;
#pragma unroll 4
    for (int c = 0; c < classes; ++c) sum = __fadd_rn(sum, e[c]);
    total[b] = sum;
  }
  __syncthreads();
  for (int i = tid; i < items; i += kDecThreads) {
    const int k = (int)(((unsigned)i * inv) >> 20), c = i - k * classes, b = list[k];
    const float e = stage[b * classes + c], sum = total[b];
    if (c == background || e < 0.99f * conf_thresh * sum) continue;
    const float v = __fdiv_rn(e, sum);
    if (!(v > conf_thresh)) continue;
    prob[((size_t)n * classes + c) * P + p0 + b] = v;
    atomicOr(&bits[c][b >> 5], 1u << (b & 31));
  }
  __syncthreads();
  if (tid < classes * kWords) {
    const int c = tid / kWords, w = tid % kWords, at = (p0 >> 5) + w;
    if (at < PW) masks[((size_t)n * classes + c) * PW + at] = bits[c][w];
  }
}

// Any number of classes: one thread per box, its exponentials formed twice.
__global__ void __launch_bounds__(kDecThreads) decode_softmax_kernel(const __grid_constant__ DetSources src, const float4* __restrict__ priors,
                                                                     float v0, float v1, float v2, float v3, int P, int classes,
                                                                     int background, float conf_thresh, float4* __restrict__ boxes,
                                                                     float* __restrict__ prob, unsigned int* __restrict__ masks) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int n = blockIdx.y, lane = threadIdx.x & 31, PW = (P + 31) >> 5;
  const int p = blockIdx.x * kDecThreads + (int)threadIdx.x;
  if ((p & ~31) >= P) return;  // whole warps
  const bool live = p < P;
  const int q = live ? p : P - 1;
  const float *l, *x;
  det_source(src, n, q, classes, &l, &x);
  if (live) boxes[(size_t)n * P + p] = det_box(l, __ldg(priors + q), v0, v1, v2, v3);
  float* pr_out = prob + (size_t)n * classes * P + p;
  unsigned int* mk = masks + (size_t)n * classes * PW + (p >> 5);
  float m = x[0];
  for (int c = 1; c < classes; ++c) m = x[c] > m ? x[c] : m;
  float sum = 0.0f;
  for (int c = 0; c < classes; ++c) sum = __fadd_rn(sum, exp_fixed_neg(__fsub_rn(x[c], m)));
  const float floor_e = 0.99f * conf_thresh * sum;
  for (int c = 0; c < classes; ++c) {
    const float e = exp_fixed_neg(__fsub_rn(x[c], m));
    bool cand = live && !(e < floor_e) && c != background;
    if (cand) {
      const float v = __fdiv_rn(e, sum);
      cand = v > conf_thresh;
      if (cand) pr_out[(size_t)c * P] = v;
    }
    const unsigned int word = __ballot_sync(0xffffffffu, cand);
    if (lane == 0) mk[(size_t)c * PW] = word;
  }
}

// Ascending bitonic sort of n (a power of two) 64-bit keys in shared memory by the whole block.
__device__ void bitonic_sort(unsigned long long* keys, int n) {
  for (int k = 2; k <= n; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int ixj = i ^ j;
        if (ixj > i) {
          const unsigned long long a = keys[i], b = keys[ixj];
          if ((a > b) == ((i & k) == 0)) { keys[i] = b; keys[ixj] = a; }
        }
      }
      __syncthreads();
    }
}

__device__ __forceinline__ float box_area(const float4 a) { return __fmul_rn(__fsub_rn(a.z, a.x), __fsub_rn(a.w, a.y)); }

// Whether the overlap of two corner boxes (intersection over union; 0 when they do not intersect) exceeds `thresh`.  The
// quotient decides; it is only formed where the product comparison is closer than the roundings can settle.
__device__ __forceinline__ bool overlap_exceeds(const float4 a, float area_a, const float4 b, float area_b, float thresh) {
  const float ix0 = a.x > b.x ? a.x : b.x, iy0 = a.y > b.y ? a.y : b.y;
  const float ix1 = a.z < b.z ? a.z : b.z, iy1 = a.w < b.w ? a.w : b.w;
  const float iw = __fsub_rn(ix1, ix0), ih = __fsub_rn(iy1, iy0);
  if (!(iw > 0.0f) || !(ih > 0.0f)) return 0.0f > thresh;
  const float inter = __fmul_rn(iw, ih);
  const float uni = __fsub_rn(__fadd_rn(area_a, area_b), inter);
  const float t = thresh * uni;
  if (uni > 1e-30f && uni < 1e30f && t > 1e-30f && t < 1e30f && !(fabsf(inter - t) < 1e-5f * t)) return inter > t;
  return __fdiv_rn(inter, uni) > thresh;
}

constexpr int kNmsThreads = 256;     // per (image, class) block
constexpr int kTopThreads = 1024;    // per image block
constexpr int kRankMax = 256;        // up to this many keys are sorted by counting the smaller ones
constexpr int kMaxTopK = 512;        // candidates that enter the suppression of one class
constexpr int kMaxSort = 16384;      // boxes per image; keys the per-image block sorts in shared memory
constexpr int kSelBits = 11;         // key bits per histogram pass of the pre-selection
constexpr int kSelBins = 1 << kSelBits;
constexpr int kSelCap = 2048;        // keys handed to the per-class sort

// Warp 0 only: the first bin at which the running sum of hist reaches `need` (need <= the total), and the sum of
// the bins before it.
__device__ int select_bin(const int* hist, int need, int* below) {
  const int lane = threadIdx.x & 31;
  constexpr int kPer = kSelBins / 32;
  static_assert(kPer == 64, "two bins per lane below");
  int local = 0;  // lane l owns bins 64 l .. 64 l + 63; each starts at another one, so that the banks differ
#pragma unroll 16
  for (int j = 0; j < kPer; ++j) local += hist[lane * kPer + ((j + lane) & (kPer - 1))];
  int incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  const unsigned int reached = __ballot_sync(0xffffffffu, incl >= need);
  const int src = reached ? __ffs(reached) - 1 : 31;
  const int before = __shfl_sync(0xffffffffu, incl - local, src);
  // the 64 bins of that lane, two per lane
  const int h0 = hist[src * kPer + 2 * lane], h1 = hist[src * kPer + 2 * lane + 1];
  int sum2 = h0 + h1;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, sum2, o);
    if (lane >= o) sum2 += v;
  }
  const unsigned int r2 = __ballot_sync(0xffffffffu, before + sum2 >= need);
  const int s2 = r2 ? __ffs(r2) - 1 : 31;
  const int base = before + sum2 - h0 - h1;
  const bool first = base + h0 >= need;
  *below = __shfl_sync(0xffffffffu, first ? base : base + h0, s2);
  return src * kPer + 2 * s2 + (__shfl_sync(0xffffffffu, first ? 1 : 0, s2) ? 0 : 1);
}

__device__ __forceinline__ unsigned long long nms_key(float s, int p) {
  return ((unsigned long long)(~__float_as_uint(s)) << 32) | (unsigned int)p;
}

// Sort of m unique keys: few are placed by counting the smaller ones (one pass, no barrier per step), more by the
// bitonic network.  `scratch` holds kRankMax keys and may not overlap `keys`; keys has room up to the next power of two.
__device__ void sort_keys(unsigned long long* keys, int m, unsigned long long* scratch) {
  if (m <= kRankMax) {
    for (int i = threadIdx.x; i < m; i += blockDim.x) scratch[i] = keys[i];
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
      const unsigned long long key = scratch[i];
      int rank = 0;
      for (int j = 0; j < m; ++j) rank += scratch[j] < key ? 1 : 0;
      keys[rank] = key;
    }
    __syncthreads();
    return;
  }
  int size = 1;
  while (size < m) size <<= 1;
  for (int i = m + threadIdx.x; i < size; i += blockDim.x) keys[i] = ~0ull;
  __syncthreads();
  bitonic_sort(keys, size);
}

// One block per (image, class other than background).  Keys order candidates (probability > conf_thresh) by
// probability, highest first, then by box index: (~bits of the positive probability) << 32 | box; they are unique.
// Only the best top_k can matter.  The candidates are the set bits of the class's mask (P bits); up to kSelCap of them
// are simply collected, more are narrowed by a radix selection over kSelBits key bits per pass (per pass: the bin in
// which the running count reaches top_k; keys below it are in, keys in it go to the next pass over the next bits) until
// the keys at or below the chosen prefix number at most kSelCap; with unique keys that ends at the latest when all 64
// bits are fixed.  The collected keys are sorted, the best top_k and their boxes copied out, their overlaps written as
// a bit matrix (over the sort area) and one warp walks the candidates in order.
// Blocks of 256 threads and 37 KB: all (image, class) pairs of a batch of 32 are resident at once (512 threads and four
// blocks per SM took two waves).  With ~70 candidates a class: 52 -> 13 us.
__global__ void __launch_bounds__(kNmsThreads) nms_class_kernel(const float4* __restrict__ boxes, const float* __restrict__ prob,
                                                                const unsigned int* __restrict__ masks, int P, int classes,
                                                                int background, float nms_thresh, int top_k, unsigned int work_bytes,
                                                                unsigned long long* __restrict__ kept_keys,
                                                                int* __restrict__ kept_count) {
  // work_bytes: room for kSelCap keys and for top_k rows of the overlap matrix, whichever is larger; then the selected
  // keys and their boxes, over which the histogram and the candidate mask lie until the selection is done
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned long long* work = reinterpret_cast<unsigned long long*>(smem_raw);
  unsigned long long* top = reinterpret_cast<unsigned long long*>(smem_raw + work_bytes);
  float4* tbox = reinterpret_cast<float4*>(top + kMaxTopK);
  float* tarea = reinterpret_cast<float*>(tbox + kMaxTopK);
  int* hist = reinterpret_cast<int*>(smem_raw + work_bytes);                    // kSelBins ints
  unsigned int* cmask = reinterpret_cast<unsigned int*>(hist + kSelBins);       // kMaxSort / 32 words
  unsigned int* mask = reinterpret_cast<unsigned int*>(smem_raw);
  static_assert(kSelBins * 4 + kMaxSort / 8 <= kMaxTopK * 24, "histogram and mask lie over the selected keys and boxes");
  __shared__ int cnt, sel_bin, sel_below, sel_in_bin, sel_cnt;
  const int n = blockIdx.y, PW = (P + 31) >> 5;
  int c = blockIdx.x;
  if (background >= 0 && c >= background) ++c;  // blockIdx.x runs over the foreground classes
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (threadIdx.x == 0) { cnt = 0; sel_cnt = 0; }
  __syncthreads();
  {
    const unsigned int* gm = masks + ((size_t)n * classes + c) * PW;
    int mine = 0;
    for (int i = threadIdx.x; i < PW; i += blockDim.x) {
      const unsigned int w = gm[i];
      cmask[i] = w;
      mine += __popc(w);
    }
    mine = __reduce_add_sync(0xffffffffu, mine);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&cnt, mine);
  }
  __syncthreads();
  int m = cnt;
  const float* sc = prob + ((size_t)n * classes + c) * P;
  if (m <= kRankMax) {               // few: every thread takes the bits of its words
    for (int i = threadIdx.x; i < PW; i += blockDim.x)
      for (unsigned int w = cmask[i]; w; w &= w - 1) {
        const int p = i * 32 + __ffs(w) - 1;
        work[atomicAdd(&sel_cnt, 1)] = nms_key(sc[p], p);
      }
  } else {
    auto candidate = [&](int p) { return ((cmask[p >> 5] >> (p & 31)) & 1u) != 0; };
    int shift = 64;                  // keys with (key >> shift) <= limit are collected; 64: all candidates
    unsigned long long limit = 0;
    if (m > kSelCap) {               // (the whole block takes this branch or none of it does)
      int need = top_k, accepted = 0;  // accepted: keys below the prefix chosen so far
      int width = kSelBits;            // bits of the digit the histogram holds
      unsigned long long prefix = 0;
      shift = 64 - kSelBits;
      int above = 64;                  // keys whose bits from `above` up equal the prefix are counted
      for (;;) {
        for (int i = threadIdx.x; i < kSelBins; i += blockDim.x) hist[i] = 0;
        __syncthreads();
        const unsigned int dmask = (1u << width) - 1u;
        for (int p0 = threadIdx.x; p0 < P; p0 += 4 * blockDim.x) {
          float v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int p = p0 + u * blockDim.x;
            v[u] = (p < P && candidate(p)) ? sc[p] : -1.0f;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (v[u] >= 0.0f) {
              const unsigned long long key = nms_key(v[u], p0 + u * blockDim.x);
              if (above == 64 || (key >> above) == prefix) atomicAdd(&hist[(unsigned int)(key >> shift) & dmask], 1);
            }
        }
        __syncthreads();
        if (threadIdx.x < 32) {
          int below;
          const int bin = select_bin(hist, need, &below);
          if (threadIdx.x == 0) { sel_bin = bin; sel_below = below; sel_in_bin = hist[bin]; }
        }
        __syncthreads();
        prefix = (prefix << width) | (unsigned int)sel_bin;
        limit = prefix;
        accepted += sel_below;
        need -= sel_below;
        m = accepted + sel_in_bin;
        if (m <= kSelCap || shift == 0) break;
        above = shift;
        shift = shift >= kSelBits ? shift - kSelBits : 0;
        width = above - shift;
        __syncthreads();
      }
    }
    for (int p0 = threadIdx.x; p0 < P; p0 += 4 * blockDim.x) {
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int p = p0 + u * blockDim.x;
        v[u] = (p < P && candidate(p)) ? sc[p] : -1.0f;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (v[u] >= 0.0f) {
          const unsigned long long key = nms_key(v[u], p0 + u * blockDim.x);
          if (shift == 64 || (key >> shift) <= limit) work[atomicAdd(&sel_cnt, 1)] = key;
        }
    }
  }
  __syncthreads();
  sort_keys(work, m, top);           // (the histogram and the mask are done with)
  const int k = m < top_k ? m : top_k;
  const float4* bx = boxes + (size_t)n * P;
  for (int i = threadIdx.x; i < k; i += blockDim.x) {
    const unsigned long long key = work[i];
    top[i] = key;
    const float4 b = bx[(unsigned int)key];
    tbox[i] = b;
    tarea[i] = box_area(b);
  }
  __syncthreads();
  // Overlap matrix: a lane holds the box of row i and meets eight later candidates, one byte of its row; a warp takes 32 rows
  // and one byte (words before i's own are never read).  With a lane per later candidate and a vote per word, the lanes of
  // a row's first and last word were mostly idle (68 candidates: 140 votes against 108 columns) and a step took twice the instructions.
  const int W = (k + 31) >> 5, lane = threadIdx.x & 31;
  unsigned char* mask8 = reinterpret_cast<unsigned char*>(mask);
  for (int c8 = 0, turn = threadIdx.x >> 5; c8 < 4 * W; ++c8)
    for (int g = 0; g <= c8 >> 2; ++g, ++turn) {
      if ((turn & (kNmsThreads / 32 - 1)) != 0) continue;   // the warps take the (byte, row group) pairs in turn
      const int i = g * 32 + lane, j0 = c8 * 8;
      const float4 bi = tbox[min(i, k - 1)];
      const float ai = tarea[min(i, k - 1)];
      unsigned int byte = 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int j = j0 + u;
        if (j < k && overlap_exceeds(tbox[j], tarea[j], bi, ai, nms_thresh) && j > i) byte |= 1u << u;
      }
      if (i < k) mask8[i * W * 4 + c8] = (unsigned char)byte;
    }
  __syncthreads();
  if (threadIdx.x < 32) {
    // 32 candidates at a time: the survivors of a group follow from its diagonal words, then they strike out the later
    // candidates they overlap, a word per step
    unsigned int removed = 0;        // lane l holds word l of the removed set (W <= 16)
    int nk = 0;
    unsigned long long* out = kept_keys + ((size_t)n * classes + c) * top_k;
    for (int g = 0; g < W; ++g) {
      const int i = g * 32 + lane;
      const unsigned int diag = i < k ? mask[i * W + g] : 0u;
      unsigned int alive = ~__shfl_sync(0xffffffffu, removed, g);
      if (k - g * 32 < 32) alive &= (1u << (k - g * 32)) - 1u;
      // only the rows that strike something out take a step: those before the next of them stay as they are
      const unsigned int strikes = __ballot_sync(0xffffffffu, diag != 0u);
      unsigned int left = alive & strikes;
      while (left) {
        const int t = __ffs(left) - 1;
        alive &= ~__shfl_sync(0xffffffffu, diag, t);
        left = alive & strikes & ~(2u * (1u << t) - 1u);
      }
      const unsigned int kept = alive;
      const bool keep = ((kept >> lane) & 1u) != 0;
      if (keep) out[nk + __popc(kept & ((1u << lane) - 1u))] = top[i];
      nk += __popc(kept);
      for (int w = g + 1; w < W; ++w) {
        const unsigned int hit = __reduce_or_sync(0xffffffffu, keep ? mask[i * W + w] : 0u);
        if (lane == w) removed |= hit;
      }
    }
    if (lane == 0) kept_count[n * classes + c] = nk;
  }
}

// One block per image: the kept detections of all classes ordered by probability (ties: class, then box), the first
// keep_top_k written as rows (class, probability, xmin, ymin, xmax, ymax); unused rows are zero.  Only the best
// keep_top_k are sorted: they are narrowed by the same radix selection as above, on the keys in shared memory
// (32 images, ~1000 kept detections each: 37 -> 9 us against a sort of all of them).
__global__ void __launch_bounds__(kTopThreads) keep_top_kernel(const float4* __restrict__ boxes, const unsigned long long* __restrict__ kept_keys,
                                                               const int* __restrict__ kept_count, int P, int classes, int background,
                                                               int top_k, int keep_top_k, int sort_cap, float* __restrict__ out,
                                                               int* __restrict__ counts) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(smem_raw);
  __shared__ __align__(16) int hist[kSelBins];
  __shared__ int warp_sum[kTopThreads / 32];
  __shared__ int sel_bin, sel_below, sel_in_bin, sel_cnt;
  const int n = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  int m = 0;
  // kTopThreads classes at a time: their counts by one load each, their places by a prefix sum, then a warp per class
  for (int c0 = 0; c0 < classes; c0 += kTopThreads) {
    const int c = c0 + (int)threadIdx.x;
    const int kc = (c < classes && c != background) ? kept_count[n * classes + c] : 0;
    int incl = kc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    __syncthreads();
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    int base = m;
    for (int w = 0; w < warp; ++w) base += warp_sum[w];
    int total = 0;
    for (int w = 0; w < kTopThreads / 32; ++w) total += warp_sum[w];
    hist[2 * threadIdx.x] = base + incl - kc;
    hist[2 * threadIdx.x + 1] = kc;
    __syncthreads();
    const int nc = min(classes - c0, kTopThreads);
    for (int j = warp; j < nc; j += kTopThreads / 32) {
      const int at = hist[2 * j], cnt = hist[2 * j + 1], cls = c0 + j;
      const unsigned long long* kk = kept_keys + ((size_t)n * classes + cls) * top_k;
      for (int i = lane; i < cnt; i += 32) {
        const unsigned long long key = kk[i];
        keys[at + i] = (key & 0xffffffff00000000ull) | ((unsigned long long)cls << 16) | (key & 0xffffull);
      }
    }
    m += total;
    __syncthreads();
  }
  static_assert(kSelBins >= 2 * kTopThreads, "the histogram doubles as the class table");
  const int k = m < keep_top_k ? m : keep_top_k;
  unsigned long long* sorted = keys;
  if (m > sort_cap) {                // sort_cap >= keep_top_k keys fit behind the kept ones
    int need = k, accepted = 0, width = kSelBits, above = 64, shift = 64 - kSelBits, sel = m;
    unsigned long long prefix = 0;
    for (;;) {
      for (int i = threadIdx.x; i < kSelBins; i += blockDim.x) hist[i] = 0;
      __syncthreads();
      const unsigned int dmask = (1u << width) - 1u;
      for (int i = threadIdx.x; i < m; i += blockDim.x)
        if (above == 64 || (keys[i] >> above) == prefix) atomicAdd(&hist[(unsigned int)(keys[i] >> shift) & dmask], 1);
      __syncthreads();
      if (threadIdx.x < 32) {
        int below;
        const int bin = select_bin(hist, need, &below);
        if (threadIdx.x == 0) { sel_bin = bin; sel_below = below; sel_in_bin = hist[bin]; sel_cnt = 0; }
      }
      __syncthreads();
      prefix = (prefix << width) | (unsigned int)sel_bin;
      accepted += sel_below;
      need -= sel_below;
      sel = accepted + sel_in_bin;
      if (sel <= sort_cap || shift == 0) break;
      above = shift;
      shift = shift >= kSelBits ? shift - kSelBits : 0;
      width = above - shift;
      __syncthreads();
    }
    sorted = keys + m;
    for (int i = threadIdx.x; i < m; i += blockDim.x)
      if ((keys[i] >> shift) <= prefix) sorted[atomicAdd(&sel_cnt, 1)] = keys[i];
    m = sel;
  }
  __syncthreads();
  sort_keys(sorted, m, reinterpret_cast<unsigned long long*>(hist));
  float* o = out + (size_t)n * keep_top_k * 6;
  for (int i = threadIdx.x; i < keep_top_k; i += blockDim.x) {
    float row[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (i < k) {
      const unsigned long long key = sorted[i];
      const float4 b = boxes[(size_t)n * P + (unsigned int)(key & 0xffffull)];
      row[0] = (float)(unsigned int)((key >> 16) & 0xffffull);
      row[1] = __uint_as_float(~(unsigned int)(key >> 32));
      row[2] = b.x; row[3] = b.y; row[4] = b.z; row[5] = b.w;
    }
#pragma unroll
    for (int j = 0; j < 6; ++j) o[i * 6 + j] = row[j];
  }
  if (threadIdx.x == 0) counts[n] = k;
}

size_t align256(size_t v) { return (v + 255) / 256 * 256; }
struct DetLayout { size_t boxes, prob, masks, keys, counts, total; };
DetLayout det_layout(int N, int P, int classes, int top_k) {
  DetLayout L;
  L.boxes = 0;
  L.prob = align256((size_t)N * P * 16);
  L.masks = L.prob + align256((size_t)N * classes * P * 4);
  L.keys = L.masks + align256((size_t)N * classes * ((P + 31) / 32) * 4);
  L.counts = L.keys + align256((size_t)N * classes * top_k * 8);
  L.total = L.counts + align256((size_t)N * classes * 4);
  return L;
}

// Launch whose set-up may overlap the kernel before it in the stream; the kernel orders itself with griddepcontrol.wait.
template <typename... Params, typename... Args>
cudaError_t launch_dependent(void (*kernel)(Params...), dim3 grid, unsigned block, size_t smem, cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

}  // namespace
}  // namespace q8

using namespace q8;

extern "C" {

int q8_l2norm(const void* x, size_t pixels, int C, float qx, float eps, const float* d_mult, void* y, void* stream) {
  clear_error();
  if ((!x || !y || !d_mult) && pixels) return fail(Q8_ERR_INVALID_ARG, "q8_l2norm: null pointer");
  if (C <= 0 || C > 65536) return fail(Q8_ERR_INVALID_ARG, "q8_l2norm: need 0 < C <= 65536");
  if (!(qx > 0.f) || std::isinf(qx) || !(eps >= 0.f) || std::isinf(eps)) return fail(Q8_ERR_NONFINITE, "q8_l2norm: factor must be finite positive, eps finite and >= 0");
  if (pixels == 0) return Q8_OK;
  volatile float qx2 = qx * qx;  // one fp32 multiply
  cudaStream_t s = as_stream(stream);
  const bool vec = C % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 3u) == 0 && (reinterpret_cast<uintptr_t>(y) & 3u) == 0 && aligned16(d_mult);
  if (vec) {
    const size_t cap = (size_t)sm_count() * 8;
    if (C / 4 <= 32 * kL2Words) {
      const size_t blocks = (pixels + 15) / 16;  // eight warps of two pixels per block and step
      l2norm_kernel<<<(unsigned)(blocks < cap ? blocks : cap), 256, 0, s>>>(static_cast<const unsigned int*>(x), pixels, C / 4, qx2, eps,
                                                                              reinterpret_cast<const float4*>(d_mult), static_cast<unsigned int*>(y));
      return check_launch("l2norm_kernel");
    }
    const size_t blocks = (pixels + 7) / 8;
    l2norm_wide_kernel<<<(unsigned)(blocks < cap ? blocks : cap), 256, 0, s>>>(static_cast<const unsigned int*>(x), pixels, C / 4, qx2, eps,
                                                                                 reinterpret_cast<const float4*>(d_mult), static_cast<unsigned int*>(y));
    return check_launch("l2norm_wide_kernel");
  }
  const size_t blocks = (pixels + 255) / 256, cap = (size_t)sm_count() * 8;
  l2norm_scalar_kernel<<<(unsigned)(blocks < cap ? blocks : cap), 256, 0, s>>>(static_cast<const unsigned char*>(x), pixels, C, qx2, eps, d_mult,
                                                                                 static_cast<unsigned char*>(y));
  return check_launch("l2norm_scalar_kernel");
}

int q8_add_relu_quantize(const float* a, const float* b, size_t n, float q, void* y, void* stream) {
  clear_error();
  if ((!a || !b || !y) && n) return fail(Q8_ERR_INVALID_ARG, "q8_add_relu_quantize: null pointer");
  if (!(q > 0.f) || std::isinf(q)) return fail(Q8_ERR_NONFINITE, "q8_add_relu_quantize: factor must be finite and positive");
  if (n == 0) return Q8_OK;
  cudaStream_t s = as_stream(stream);
  size_t done = 0;
  if (aligned16(a) && aligned16(b) && (reinterpret_cast<uintptr_t>(y) & 3u) == 0 && n >= 4) {
    const size_t n4 = n / 4, blocks = (n4 + 511) / 512, cap = (size_t)sm_count() * 4;
    add_relu_quantize_kernel<<<(unsigned)(blocks < cap ? blocks : cap), 512, 0, s>>>(reinterpret_cast<const float4*>(a), reinterpret_cast<const float4*>(b),
                                                                                        n4, q, static_cast<unsigned int*>(y));
    done = n4 * 4;
  }
  if (done < n) {
    const size_t rest = n - done;
    if (rest > 0x7fffffffu * 256ull) return fail(Q8_ERR_UNSUPPORTED, "q8_add_relu_quantize: unaligned tensors above 2^39 elements");
    add_relu_quantize_tail_kernel<<<(unsigned)((rest + 255) / 256), 256, 0, s>>>(a, b, done, n, q, static_cast<unsigned char*>(y));
  }
  return check_launch("add_relu_quantize_kernel");
}

static int det_check(int N, int P, int classes, int background, int nms_top_k, int keep_top_k) {
  if (N <= 0 || P <= 0 || classes <= 0 || nms_top_k <= 0 || keep_top_k <= 0 || background < -1 || background >= classes)
    return fail(Q8_ERR_INVALID_ARG, "q8_detection_output: bad extent or class index");
  const int fg = classes - (background >= 0 ? 1 : 0);
  if (fg <= 0) return fail(Q8_ERR_INVALID_ARG, "q8_detection_output: no foreground class");
  if (P > kMaxSort || nms_top_k > kMaxTopK || classes > 65535 || (long long)fg * nms_top_k > kMaxSort || N > 65535)
    return fail(Q8_ERR_UNSUPPORTED, "q8_detection_output: limits are %d boxes per image, nms_top_k <= %d, (classes - 1) * nms_top_k <= %d, N <= 65535",
                kMaxSort, kMaxTopK, kMaxSort);
  return Q8_OK;
}

int q8_detection_output_workspace_bytes(int N, int P, int classes, int background, int nms_top_k, int keep_top_k, size_t* bytes) {
  clear_error();
  if (!bytes) return fail(Q8_ERR_INVALID_ARG, "q8_detection_output_workspace_bytes: null pointer");
  const int rc = det_check(N, P, classes, background, nms_top_k, keep_top_k);
  if (rc != Q8_OK) return rc;
  *bytes = det_layout(N, P, classes, nms_top_k).total;
  return Q8_OK;
}

int q8_detection_output(int n_sources, const float* const* loc, const int* loc_stride, const float* const* conf,
                        const int* conf_stride, const int* cells, const int* boxes_per_cell, const float* d_priors,
                        const float* variances, int N, int classes, int background, float conf_thresh, float nms_thresh,
                        int nms_top_k, int keep_top_k, void* workspace, size_t workspace_bytes, float* d_out, int* d_counts,
                        void* stream) {
  clear_error();
  if (n_sources <= 0 || n_sources > kMaxSources || !loc || !loc_stride || !conf || !conf_stride || !cells || !boxes_per_cell ||
      !d_priors || !variances || !d_out || !d_counts)
    return fail(Q8_ERR_INVALID_ARG, "q8_detection_output: null pointer or more than %d sources", kMaxSources);
  if (classes <= 0) return fail(Q8_ERR_INVALID_ARG, "q8_detection_output: classes must be positive");
  DetSources src{};
  src.n = n_sources;
  long long P = 0;
  for (int i = 0; i < n_sources; ++i) {
    if (!loc[i] || !conf[i] || cells[i] <= 0 || boxes_per_cell[i] <= 0 || loc_stride[i] < boxes_per_cell[i] * 4 ||
        (long long)conf_stride[i] < (long long)boxes_per_cell[i] * classes)
      return fail(Q8_ERR_INVALID_ARG, "q8_detection_output: source %d: null pointer, empty, or a cell stride below its values", i);
    src.loc[i] = loc[i]; src.conf[i] = conf[i];
    src.loc_stride[i] = loc_stride[i]; src.conf_stride[i] = conf_stride[i];
    src.cells[i] = cells[i]; src.boxes[i] = boxes_per_cell[i];
    src.first[i] = (int)P;
    P += (long long)cells[i] * boxes_per_cell[i];
    if (P > kMaxSort) return fail(Q8_ERR_UNSUPPORTED, "q8_detection_output: more than %d boxes per image", kMaxSort);
  }
  src.first[n_sources] = (int)P;
  const int rc = det_check(N, (int)P, classes, background, nms_top_k, keep_top_k);
  if (rc != Q8_OK) return rc;
  if (!std::isfinite(conf_thresh) || !std::isfinite(nms_thresh) || conf_thresh < 0.f)
    return fail(Q8_ERR_NONFINITE, "q8_detection_output: thresholds must be finite, the confidence threshold not negative");
  if (!aligned16(d_priors)) return fail(Q8_ERR_ALIGNMENT, "q8_detection_output: priors not 16-byte aligned");
  const DetLayout L = det_layout(N, (int)P, classes, nms_top_k);
  if (!workspace || workspace_bytes < L.total || (reinterpret_cast<uintptr_t>(workspace) & 255u))
    return fail(Q8_ERR_WORKSPACE, "q8_detection_output: workspace of %zu bytes, 256-byte aligned, needed", L.total);
  cudaStream_t s = as_stream(stream);
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  float4* boxes = reinterpret_cast<float4*>(ws + L.boxes);
  float* prob = reinterpret_cast<float*>(ws + L.prob);
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(ws + L.keys);
  unsigned int* masks = reinterpret_cast<unsigned int*>(ws + L.masks);
  int* kcount = reinterpret_cast<int*>(ws + L.counts);
  const dim3 dec_grid((unsigned)((P + kDecThreads - 1) / kDecThreads), (unsigned)N);
  if (classes <= kRegClasses) {
    // (where the recipe clamps its argument every class may pass)
    const double ln = std::log((double)conf_thresh) - 1e-4;
    const float cutoff = ln > -86.5 ? (float)(ln - 1e-5) : -INFINITY;
    // Where a quarter of the SMs can take 64 boxes each they do: a thread's share of the (box, class) pairs is a fourth (963
    // boxes with flat logits at a threshold of 0.3: 15.9 -> 13.1 us).  No further: the blocks of the next launch find room as
    // these leave it, and beside more of them they pile up on the SMs that are free (2 images of 8732 boxes 111 -> 223 us).
    const dim3 few_grid((unsigned)((P + kDecFew - 1) / kDecFew), (unsigned)N);
    const bool few = (long long)few_grid.x * N * 4 <= sm_count();
    (few ? decode_listed_kernel<kDecFew> : decode_listed_kernel<kDecThreads>)<<<few ? few_grid : dec_grid, kDecThreads, 0, s>>>(
        src, reinterpret_cast<const float4*>(d_priors), variances[0], variances[1], variances[2], variances[3], (int)P, classes, background,
        conf_thresh, cutoff, boxes, prob, masks);
  } else {
    decode_softmax_kernel<<<dec_grid, kDecThreads, 0, s>>>(src, reinterpret_cast<const float4*>(d_priors), variances[0], variances[1], variances[2],
                                                           variances[3], (int)P, classes, background, conf_thresh, boxes, prob, masks);
  }
  int rc2 = check_launch("decode kernel");
  if (rc2 != Q8_OK) return rc2;
  const int fg = classes - (background >= 0 ? 1 : 0);
  const int dev = current_device();
  {
    const unsigned int W = (unsigned)(nms_top_k + 31) / 32;
    unsigned int work_bytes = (unsigned)kSelCap * 8u;
    if (work_bytes < (unsigned)nms_top_k * W * 4u) work_bytes = (unsigned)nms_top_k * W * 4u;
    work_bytes = (work_bytes + 15u) & ~15u;
    const size_t smem = (size_t)work_bytes + (size_t)kMaxTopK * (8 + 16 + 4);
    static std::atomic<size_t> configured[kMaxDevices];
    if (dev < 0 || configured[dev].load() < smem) {
      rc2 = check_cuda(cudaFuncSetAttribute(nms_class_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem), "cudaFuncSetAttribute(nms_class_kernel)");
      if (rc2 != Q8_OK) return rc2;
      if (dev >= 0) configured[dev].store(smem);
    }
    rc2 = check_cuda(launch_dependent(nms_class_kernel, dim3((unsigned)fg, (unsigned)N), kNmsThreads, smem, s, boxes, prob, masks, (int)P, classes,
                                      background, nms_thresh, nms_top_k, work_bytes, keys, kcount), "nms_class_kernel");
    if (rc2 != Q8_OK) return rc2;
  }
  {
    // room for every kept key and, where that is smaller, for the selection that is sorted (a power of two)
    const int most = fg * nms_top_k;
    int cap = 1, sort_cap = 1024;
    while (cap < most) cap <<= 1;
    while (sort_cap < 2 * (keep_top_k < most ? keep_top_k : most)) sort_cap <<= 1;
    if (sort_cap >= cap) sort_cap = cap;
    const size_t smem = (size_t)(sort_cap >= cap ? cap : most + sort_cap) * 8;
    static std::atomic<size_t> configured[kMaxDevices];
    if (dev < 0 || configured[dev].load() < smem) {
      rc2 = check_cuda(cudaFuncSetAttribute(keep_top_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem), "cudaFuncSetAttribute(keep_top_kernel)");
      if (rc2 != Q8_OK) return rc2;
      if (dev >= 0) configured[dev].store(smem);
    }
    rc2 = check_cuda(launch_dependent(keep_top_kernel, dim3((unsigned)N), kTopThreads, smem, s, boxes, keys, kcount, (int)P, classes, background,
                                      nms_top_k, keep_top_k, sort_cap, d_out, d_counts), "keep_top_kernel");
    if (rc2 != Q8_OK) return rc2;
  }
  return check_launch("keep_top_kernel");
}

}  // extern "C"

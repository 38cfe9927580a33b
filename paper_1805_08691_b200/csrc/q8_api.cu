// Host entry points of libq8 that are not tied to one kernel file: errors, status word,
// descriptor validation and dispatch of q8_conv2d.
#include <atomic>
#include <cstdio>
#include <cstring>

#include "q8_internal.h"

namespace q8 {

namespace {
thread_local char g_last_error[512] = "";
__device__ unsigned int g_status_word = 0;
}  // namespace

int fail(int code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_last_error, sizeof(g_last_error), fmt, ap);
  va_end(ap);
  return code;
}

void clear_error() { g_last_error[0] = '\0'; }

int check_cuda(cudaError_t e, const char* what) {
  if (e == cudaSuccess) return Q8_OK;
  return fail(Q8_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

int check_launch(const char* kernel) { return check_cuda(cudaGetLastError(), kernel); }

int current_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return -1;
  return dev;
}

int sm_count() {
  static std::atomic<int> cached[kMaxDevices];  // zero-initialised; racing threads store the same value
  const int dev = current_device();
  int n = dev >= 0 ? cached[dev].load(std::memory_order_relaxed) : 0;
  if (n == 0) {
    int cur = 0;
    if (cudaGetDevice(&cur) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, cur) != cudaSuccess || n <= 0) n = 148;
    if (dev >= 0) cached[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

unsigned int* status_word_device_ptr() {
  // One lookup per device; the symbol address is a device address obtained from the runtime.
  static thread_local int cached_dev = -1;
  static thread_local unsigned int* cached_ptr = nullptr;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  if (dev != cached_dev) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_status_word) != cudaSuccess) return nullptr;
    cached_ptr = static_cast<unsigned int*>(p);
    cached_dev = dev;
  }
  return cached_ptr;
}

namespace {

int validate_desc(const q8_conv_desc* d, int* P, int* Q) {
  if (!d) return fail(Q8_ERR_INVALID_ARG, "conv: null descriptor");
  if (d->N <= 0 || d->H <= 0 || d->W <= 0 || d->C <= 0 || d->K <= 0 || d->R <= 0 || d->S <= 0)
    return fail(Q8_ERR_INVALID_ARG, "conv: extents must be positive");
  if (d->stride_h <= 0 || d->stride_w <= 0 || d->dil_h <= 0 || d->dil_w <= 0 || d->pad_h < 0 || d->pad_w < 0)
    return fail(Q8_ERR_INVALID_ARG, "conv: stride/dilation must be positive, padding non-negative");
  if (d->x_type != Q8_U8 && d->x_type != Q8_S8) return fail(Q8_ERR_INVALID_ARG, "conv: x_type must be Q8_U8 or Q8_S8");
  if (d->y_type < Q8_U8 || d->y_type > Q8_F32) return fail(Q8_ERR_INVALID_ARG, "conv: bad y_type");
  if (d->res_type != Q8_U8 && d->res_type != Q8_S8) return fail(Q8_ERR_INVALID_ARG, "conv: res_type must be Q8_U8 or Q8_S8");
  if (d->scale_count != 1 && d->scale_count != d->K) return fail(Q8_ERR_INVALID_ARG, "conv: scale_count must be 1 or K");
  if (d->algo < Q8_ALGO_AUTO || d->algo > Q8_ALGO_DIRECT) return fail(Q8_ERR_INVALID_ARG, "conv: bad algo");
  // |x| <= 255, |w| <= 128: R*S*C terms stay inside int32 up to floor(2^31 / (255*128))
  if ((long long)d->R * d->S * d->C > 65793) return fail(Q8_ERR_INVALID_ARG, "conv: R*S*C > 65793 could overflow the int32 accumulator");
  int p = conv_out_extent(d->H, d->pad_h, d->dil_h, d->R, d->stride_h);
  int q = conv_out_extent(d->W, d->pad_w, d->dil_w, d->S, d->stride_w);
  if (p <= 0 || q <= 0) return fail(Q8_ERR_INVALID_ARG, "conv: empty output");
  if ((long long)d->N * p * q > 0x7fffffffll - 256) return fail(Q8_ERR_INVALID_ARG, "conv: N*P*Q too large");
  int ldc = d->y_ldc == 0 ? d->K : d->y_ldc;
  if (d->y_c_offset < 0 || ldc < d->y_c_offset + d->K) return fail(Q8_ERR_INVALID_ARG, "conv: y_ldc < y_c_offset + K");
  *P = p;
  *Q = q;
  return Q8_OK;
}

// Time of the direct kernel in microseconds.  A thread forms one output, tap by tap; outputs cost index arithmetic and,
// like the products of all of them, throughput; the products of one output are a chain of loads, longer where the weights
// of the lanes lie in different sectors.  Fitted, with gather_us, to 2600 layers with 1 to 500 output channels, filters up
// to 7x7 and up to 8000 products (median error of both 8 %).  Taking the smaller estimate is on average 1.5 % off the
// better kernel over the layers with C off the 16-channel grid (8.6 % with the limits in products and outputs that stood
// here, 7 times at worst: 7x7 of 163 -> 397 channels on one pixel takes 15 us directly, 102 gathered).
double direct_us(const ConvArgs& a) {
  const q8_conv_desc& d = a.d;
  const double outputs = 1e-6 * (double)a.M * d.K, taps = (double)d.R * d.S;
  const int in_h = (d.H - 1) / d.dil_h + 1, in_w = (d.W - 1) / d.dil_w + 1;  // filter rows and columns that fit the image
  const double seen = (double)(d.R < in_h ? d.R : in_h) * (d.S < in_w ? d.S : in_w), chain = seen * d.C;
  const double apart = taps * d.C > 32 ? (d.K < 32 ? d.K / 32.0 : 1.0) : 0.0;
  return 2.4 + outputs * (9.0 + 0.22 * chain) + chain * (0.033 + 0.019 * apart) + (taps > 1 ? 0.1 * seen : 0.0) + 0.03 * taps;
}

// 8-bit rows off the 16-byte grid, short ones with short reductions: gathering the operands (or the direct kernel) costs
// less than the kernel that moves such rows through shared memory, whose start-up is longer.  The gathering kernel's time
// grows faster, by the bytes that its producers fetch (reduction x pixels) and by every 16 columns that it stores byte by
// byte, which is what the limits are in (1x1 64 -> 9 at 56x56: batch 4 3.9 against 4.6 us, batch 16 5.0 against 5.5, batch 32
// 7.2 against 7.1; 32 -> 31 on one 8x8 image 4.2 against 4.7, 12x12 5.6 against 4.6).  Over 870 random layers with such
// rows, the kernel taken is on average 0.9 % off the fastest of the three.
bool short_rows(const ConvArgs& a) {
  const long long products = (long long)a.d.R * a.d.S * a.d.C;
  return products <= 64 && (a.d.K <= 16 ? products * a.M <= 4000000 : a.d.K <= 32 && a.M <= 128);
}

// The kernel a call takes, from its descriptor and the alignment of its pointers; `why` is set where the TMA-fed one is
// not taken.  That kernel may still find no tile that fits (umma_fits, or kPlanNoFit from its launch); route_off_tma then
// says what takes its place.
enum Route { kRouteRefused, kRouteDirect, kRouteGather, kRoutePacked, kRouteTma };

Route route_off_tma(const ConvArgs& a) {
  if (a.d.algo == Q8_ALGO_UMMA) return kRouteRefused;
  const double direct = direct_us(a), gather = gather_addressable(a.d) ? gather_us(a) : direct;
  if (packed_better(a)) return kRoutePacked;
  return gather < direct ? kRouteGather : kRouteDirect;
}

Route conv_route(const ConvArgs& a, const char** why) {
  const q8_conv_desc& d = a.d;
  if (d.algo == Q8_ALGO_DIRECT) return kRouteDirect;
  if (!umma_shape_eligible(d, why)) return route_off_tma(a);
  if (!aligned16(a.x) || !aligned16(a.w)) { *why = "x or w not 16-byte aligned"; return route_off_tma(a); }
  const bool out8 = d.y_type == Q8_U8 || d.y_type == Q8_S8;
  if (d.algo == Q8_ALGO_UMMA || !out8) {
    if (out8 && (!aligned16(a.y) || a.ldc % 16 || a.c_off % 16)) { *why = "8-bit output needs y, y_ldc, y_c_offset aligned to 16"; return route_off_tma(a); }
    if (a.residual && !aligned16(a.residual)) { *why = "residual not 16-byte aligned"; return route_off_tma(a); }
  } else if (rows_off_tma(a)) {
    // Other such rows are moved by the epilogue warps (see rows_out), which takes 5 to 6 us at the least.  The direct kernel
    // where it is surely faster: below 4.5 us by its estimate (1x1 32 -> 44 on 108 pixels: 4.0 against 5.5 us).
    if (short_rows(a)) return route_off_tma(a);
    if (direct_us(a) < 4.5) return kRouteDirect;
  }
  return kRouteTma;
}

// The call a descriptor describes, with pointers that stand for 16-byte aligned ones.
int described_call(const q8_conv_desc* d, bool residual, ConvArgs* a) {
  *a = ConvArgs{};
  const int rc = validate_desc(d, &a->P, &a->Q);
  if (rc != Q8_OK) return rc;
  a->d = *d;
  a->M = (long long)d->N * a->P * a->Q;
  a->x = reinterpret_cast<const void*>(256); a->w = reinterpret_cast<const int8_t*>(256); a->y = reinterpret_cast<void*>(256);
  a->residual = residual && d->y_type != Q8_S32 ? reinterpret_cast<const void*>(256) : nullptr;
  a->ldc = d->y_ldc == 0 ? d->K : d->y_ldc;
  a->c_off = d->y_c_offset;
  return Q8_OK;
}
}  // namespace
}  // namespace q8

using namespace q8;

extern "C" {

const char* q8_version(void) { return "q8 0.1 (sm_100a)"; }

const char* q8_last_error(void) { return g_last_error; }

int q8_read_status(void* stream) {
  clear_error();
  int rc = check_cuda(cudaStreamSynchronize(as_stream(stream)), "q8_read_status: synchronize");
  if (rc != Q8_OK) return rc;
  unsigned int* dptr = status_word_device_ptr();
  if (!dptr) return fail(Q8_ERR_CUDA, "q8_read_status: no status word on this device");
  unsigned int host = 0;
  rc = check_cuda(cudaMemcpy(&host, dptr, sizeof(host), cudaMemcpyDeviceToHost), "q8_read_status: read");
  if (rc != Q8_OK) return rc;
  if (host != 0) {
    unsigned int zero = 0;
    cudaMemcpy(dptr, &zero, sizeof(zero), cudaMemcpyHostToDevice);
    return fail(Q8_ERR_TIMEOUT, "a kernel gave up on a bounded wait (site mask 0x%x)", host);
  }
  return Q8_OK;
}

int q8_conv2d_workspace_bytes(const q8_conv_desc* d, size_t* bytes) {
  clear_error();
  ConvArgs a;
  const int rc = described_call(d, false, &a);
  if (rc != Q8_OK) return rc;
  if (!bytes) return fail(Q8_ERR_INVALID_ARG, "q8_conv2d_workspace_bytes: null pointer");
  const char* why = nullptr;
  const int splits = conv_route(a, &why) == kRouteTma ? umma_splits(a) : 1;
  *bytes = splits > 1 ? (size_t)splits * (size_t)a.M * (size_t)d->K * sizeof(int32_t) : 0;
  return Q8_OK;
}

int q8_conv2d_query_algo(const q8_conv_desc* d, int* algo) {
  clear_error();
  ConvArgs a;
  const int rc = described_call(d, false, &a);
  if (rc != Q8_OK) return rc;
  if (!algo) return fail(Q8_ERR_INVALID_ARG, "q8_conv2d_query_algo: null pointer");
  const char* why = nullptr;
  *algo = conv_route(a, &why) == kRouteTma && umma_fits(a) ? Q8_ALGO_UMMA : Q8_ALGO_DIRECT;
  return Q8_OK;
}

int q8_conv2d_query_plan(const q8_conv_desc* d, int residual, q8_conv_plan* plan) {
  clear_error();
  ConvArgs a;
  const int rc = described_call(d, residual != 0, &a);
  if (rc != Q8_OK) return rc;
  if (!plan) return fail(Q8_ERR_INVALID_ARG, "q8_conv2d_query_plan: null pointer");
  memset(plan, 0, sizeof(*plan));
  const char* why = "";
  Route route = conv_route(a, &why);
  if (route == kRouteTma && !umma_describe(a, plan)) { route = route_off_tma(a); why = "no tile shape of this layer fits in shared memory"; }
  if (route == kRouteRefused) return fail(Q8_ERR_UNSUPPORTED, "q8_conv2d: tensor-core kernel not eligible: %s", why);
  plan->kernel = route == kRouteTma ? Q8_KERNEL_TMA : (route == kRouteDirect ? Q8_KERNEL_DIRECT : Q8_KERNEL_GATHER);
  if (route == kRoutePacked) plan->operand = 3;
  return Q8_OK;
}

int q8_conv2d_query_row_buffers(const q8_conv_desc* d, const q8_conv_desc* then_1x1, int residual, int* buffers) {
  clear_error();
  ConvArgs a;
  int rc = described_call(d, residual != 0, &a);
  if (rc != Q8_OK) return rc;
  if (!buffers) return fail(Q8_ERR_INVALID_ARG, "q8_conv2d_query_row_buffers: null pointer");
  if (then_1x1) {
    int P, Q;
    rc = validate_desc(then_1x1, &P, &Q);
    if (rc != Q8_OK) return rc;
    *buffers = fused_row_buffers(*d, *then_1x1, residual != 0);
    return Q8_OK;
  }
  const char* why = nullptr;
  *buffers = conv_route(a, &why) == kRouteTma ? umma_row_buffers(a) : 0;
  return Q8_OK;
}

int q8_conv2d(const q8_conv_desc* d, const void* x, const int8_t* w, const int32_t* bias, const float* scale,
              const void* residual, float residual_scale, void* y, void* workspace, size_t workspace_bytes,
              void* stream) {
  clear_error();
  ConvArgs a;
  int rc = validate_desc(d, &a.P, &a.Q);
  if (rc != Q8_OK) return rc;
  if (!x || !w || !y) return fail(Q8_ERR_INVALID_ARG, "q8_conv2d: null x, w or y");
  if (!scale && d->y_type != Q8_S32) return fail(Q8_ERR_INVALID_ARG, "q8_conv2d: null scale");
  a.d = *d;
  a.M = (long long)d->N * a.P * a.Q;
  a.x = x; a.w = w; a.bias = bias; a.scale = scale;
  a.residual = d->y_type == Q8_S32 ? nullptr : residual;
  a.residual_scale = residual_scale;
  a.y = y;
  a.ldc = d->y_ldc == 0 ? d->K : d->y_ldc;
  a.c_off = d->y_c_offset;
  a.workspace = workspace; a.workspace_bytes = workspace_bytes;
  a.stream = as_stream(stream);

  const char* why = "";
  Route route = conv_route(a, &why);
  if (route == kRouteTma) {
    rc = launch_conv_umma(a);
    if (rc != kPlanNoFit) return rc;
    route = route_off_tma(a);
    why = "no tile shape of this layer fits in shared memory";
  }
  if (route == kRouteRefused) return fail(Q8_ERR_UNSUPPORTED, "q8_conv2d: tensor-core kernel not eligible: %s", why);
  if (route == kRoutePacked) {
    rc = launch_conv_packed(a);
    if (rc != kPlanNoFit) return rc;
    route = gather_addressable(a.d) && gather_us(a) < direct_us(a) ? kRouteGather : kRouteDirect;
  }
  return route == kRouteGather ? launch_conv_gather(a) : launch_conv_direct(a);
}

int q8_conv2d_then_1x1_supported(const q8_conv_desc* d1, const q8_conv_desc* d2, int* supported) {
  clear_error();
  int P, Q;
  int rc = validate_desc(d1, &P, &Q);
  if (rc != Q8_OK) return rc;
  rc = validate_desc(d2, &P, &Q);
  if (rc != Q8_OK) return rc;
  if (!supported) return fail(Q8_ERR_INVALID_ARG, "q8_conv2d_then_1x1_supported: null pointer");
  const char* why = "";
  *supported = (d1->algo != Q8_ALGO_DIRECT && d2->algo != Q8_ALGO_DIRECT && fused_pair_eligible(*d1, *d2, &why)) ? 1 : 0;
  return Q8_OK;
}

int q8_conv2d_then_1x1(const q8_conv_desc* d1, const q8_conv_desc* d2, const void* x, const int8_t* w1, const int32_t* bias1,
                       const float* scale1, const int8_t* w2, const int32_t* bias2, const float* scale2,
                       const void* residual, float residual_scale, void* y, void* stream) {
  clear_error();
  int P, Q;
  int rc = validate_desc(d1, &P, &Q);
  if (rc != Q8_OK) return rc;
  rc = validate_desc(d2, &P, &Q);
  if (rc != Q8_OK) return rc;
  if (!x || !w1 || !w2 || !y || !scale1 || !scale2) return fail(Q8_ERR_INVALID_ARG, "q8_conv2d_then_1x1: null x, w1, w2, y, scale1 or scale2");
  if (!aligned16(x) || !aligned16(w1) || !aligned16(w2) || !aligned16(y))
    return fail(Q8_ERR_UNSUPPORTED, "q8_conv2d_then_1x1: x, w1, w2 and y must be 16-byte aligned");
  return launch_conv_fused(*d1, *d2, x, w1, bias1, scale1, w2, bias2, scale2, residual, residual_scale, y, as_stream(stream));
}

}  // extern "C"

// Quantized convolution on the tensor cores for layers that TMA cannot address: channel counts that are no multiple
// of 16 (a three-channel image, pruned layers), inputs or weights off the 16-byte grid, strides above 8; and, being cheaper
// to start, short reductions into few channels whose 8-bit rows are off that grid.
//
//   D[128 pixels, BN channels] (int32, TMEM) = A[128, Kp] (gathered) x B[BN, Kp]^T (gathered)
//
// The reduction axis is cut into runs of bytes that are contiguous in memory on both sides: one filter row
// (S * C bytes of NHWC input and of KRSC weights) without dilation along W, one filter tap (C bytes) with it.  A run
// is padded with zeros to whole 16-byte chunks, which is exact, so that a chunk never spans two runs; K order is free
// as long as both operands share it.  Producer warps fetch the unaligned 16 bytes of a chunk with five aligned
// 32-bit loads and funnel shifts, mask what lies outside the image or the run, and store it at its place in the
// K-major swizzled tile that tcgen05.mma reads.
//
// Roles: warps 0-7 two epilogue groups on alternate tiles (thread = accumulator row), warp 8 MMA issue and TMEM,
// warps 9-24 two producer groups of eight warps on alternate stages, so that one group's loads are in flight while the
// other stores.  Weights are gathered once per CTA where they fit in shared memory, else stage by stage with the
// activations.  All waits are bounded as in the other tensor-core kernels.
//
// Bound by the instructions of its warps (3x3/2 of 3 -> 32 channels: 5560 per tile of 128 pixels over all roles, issue slots
// 58 % busy, tensor pipe 1 %, nothing else near a limit), hence no division per chunk, rows per thread fixed at compile time
// and branch-free loads.  Measured against the CUDA-core kernel: 3x3/2 of 3 -> 32 channels on 8 x 299x299 157.7 ->
// 12.2 us, 7x7/2 of 3 -> 64 on 224x224 134 -> 7.7 us, 3x3 of 100 -> 120 on 8 x 28x28 963 -> 26 us, 1x1 of 200 -> 500 at 14x14
// 32.8 -> 10.2 us.
#include "q8_umma_common.cuh"

namespace q8 {
namespace {

constexpr int kGEpiGroups = 2;                                         // four warps each, on alternate tiles
constexpr int kGProdGroups = 2;
constexpr int kGProdThreads = 256;                                     // per group
constexpr int kGMmaWarp = 4 * kGEpiGroups;
constexpr int kGFirstProd = kGMmaWarp + 1;
constexpr int kGThreads = (kGFirstProd * 32) + kGProdGroups * kGProdThreads;  // 800
constexpr int kGMaxStages = 8;

struct GatherParams {
  const unsigned char* x;
  const unsigned char* w;
  const int* bias;
  const float* scale;
  const unsigned char* res;
  void* y;
  unsigned int* status;
  int H, W, C, K, S;
  int P, Q, PQ, M;
  int stride_h, stride_w, pad_h, pad_w, dil_h, dil_w;
  int rsc;                       // bytes of one filter
  int run_len, run_chunks;       // bytes of a run, 16-byte chunks of a padded run
  int run_taps;                  // taps along W in a run: S, or 1 with dilation
  int chunks;                    // runs * run_chunks
  int bkb, lg_cpb, nblk;         // bytes per K block (32, 64 or 128), log2 of its chunks, number of blocks
  int bn, n_tiles, tiles;
  int stages, b_resident;
  unsigned int stage_bytes, b_block_bytes, off_stages, off_chan;
  unsigned int idesc, desc_hi, swz_mask;
  int acc_stride, tmem_cols;
  FastDiv fd_q, fd_pq, fd_chunks, fd_s, fd_ntiles, fd_bn;
  int scale_count, res_signed, res_vec, relu, ldc, c_off, y_vec;
  float res_scale;
};

// Bytes pos .. pos+15 of the row that starts at `row`, those outside [vlo, vhi) zero, in two steps without a branch
// between them, so that the loads of several chunks are in flight together.  Every word loaded holds at least one byte
// of that range.
struct Gathered {
  unsigned int v[5];
  int m, nl, nh;  // bytes of the first word before pos; first and one past the last valid byte of the sixteen
};
__device__ __forceinline__ void gather_load(Gathered& g, bool live, const unsigned char* row, int pos, int vlo, int vhi) {
  const int lo = max(pos, vlo), hi = min(pos + 16, vhi);
  live = live && lo < hi;
  const unsigned long long a = (unsigned long long)row + (long long)pos;
  const unsigned int* wp = reinterpret_cast<const unsigned int*>(a & ~3ull);
  g.m = (int)(a & 3ull);
  g.nl = live ? lo - pos : 16;
  g.nh = live ? hi - pos : 0;
#pragma unroll
  for (int k = 0; k < 5; ++k) g.v[k] = (4 * k - g.m + 3 >= g.nl && 4 * k - g.m < g.nh) ? __ldg(wp + k) : 0u;
}
__device__ __forceinline__ uint4 gather_finish(const Gathered& g) {
  unsigned int d[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) d[k] = __funnelshift_r(g.v[k], g.v[k + 1], (unsigned)g.m * 8u);
  if (g.nl > 0 || g.nh < 16) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int l = min(max(g.nl - 4 * k, 0), 4), h = min(max(g.nh - 4 * k, 0), 4);
      const unsigned int below_h = h == 4 ? 0xffffffffu : (1u << (8 * h)) - 1u;
      const unsigned int below_l = l == 4 ? 0xffffffffu : (1u << (8 * l)) - 1u;
      d[k] &= below_h & ~below_l;
    }
  }
  return make_uint4(d[0], d[1], d[2], d[3]);
}

__device__ __forceinline__ uint32_t swizzled(const GatherParams& p, int row, int chunk) {
  const uint32_t off = (uint32_t)(row * p.bkb + chunk * 16);
  return off ^ (((off >> 7) & p.swz_mask) << 4);
}

// K blocks [blk0, blk0 + nblk) of the weight tile of channels n0 .. n0+bn-1, `b_block_bytes` apart, by `nthreads`
// threads: four chunks of a thread in flight at a time.
__device__ __forceinline__ void gather_weights(const GatherParams& p, unsigned char* dst, int n0, int blk0, int nblk, int t, int nthreads) {
  const int items = (nblk * p.bn) << p.lg_cpb, chunk = t & ((1 << p.lg_cpb) - 1);
  for (int i0 = t; i0 < items; i0 += 4 * nthreads) {
    Gathered v[4];
    uint32_t at[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = i0 + j * nthreads, rowall = i >> p.lg_cpb, b = p.fd_bn.div(rowall), row = rowall - b * p.bn;
      const int kc = ((blk0 + b) << p.lg_cpb) + chunk, run = p.fd_chunks.div(kc);
      gather_load(v[j], i < items && kc < p.chunks && n0 + row < p.K, p.w + (size_t)(n0 + row) * p.rsc + (size_t)run * p.run_len,
                  (kc - run * p.run_chunks) * 16, 0, p.run_len);
      at[j] = (uint32_t)b * p.b_block_bytes + swizzled(p, row, chunk);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (i0 + j * nthreads < items) *reinterpret_cast<uint4*>(dst + at[j]) = gather_finish(v[j]);
  }
}

// Sixteen channels k0 .. k0+15 of pixel m, straight to global memory.
template <int kOut>
__device__ __forceinline__ void gather_epilogue(const GatherParams& p, const int* s_bias, const float* s_scale, int (&acc)[16], long long m, int k0) {
  const int valid = min(16, p.K - k0);
  if (m >= p.M || valid <= 0) return;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int4 b = reinterpret_cast<const int4*>(s_bias + k0)[j];
    acc[4 * j] += b.x; acc[4 * j + 1] += b.y; acc[4 * j + 2] += b.z; acc[4 * j + 3] += b.w;
  }
  const bool vec = p.y_vec && valid == 16;
  const size_t o = (size_t)m * p.ldc + p.c_off + k0;
  float v[16];
  if (kOut != Q8_S32) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 s = reinterpret_cast<const float4*>(s_scale + k0)[j];
      v[4 * j] = __fmul_rn(__int2float_rn(acc[4 * j]), s.x); v[4 * j + 1] = __fmul_rn(__int2float_rn(acc[4 * j + 1]), s.y);
      v[4 * j + 2] = __fmul_rn(__int2float_rn(acc[4 * j + 2]), s.z); v[4 * j + 3] = __fmul_rn(__int2float_rn(acc[4 * j + 3]), s.w);
    }
    if (p.res) {
      const unsigned char* rp = p.res + (size_t)m * p.K + k0;
      unsigned int rb[4] = {0u, 0u, 0u, 0u};
      if (p.res_vec && valid == 16) {
        const uint4 r = *reinterpret_cast<const uint4*>(rp);
        rb[0] = r.x; rb[1] = r.y; rb[2] = r.z; rb[3] = r.w;
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (j < valid) rb[j >> 2] |= (unsigned int)rp[j] << (8 * (j & 3));
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const unsigned int b = (rb[j >> 2] >> (8 * (j & 3))) & 255u;
        v[j] = __fadd_rn(v[j], __fmul_rn(__int2float_rn(p.res_signed ? (int)(signed char)b : (int)b), p.res_scale));
      }
    }
    if (p.relu) {
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = fmaxf(v[j], 0.0f);
    }
  }
  if (kOut == Q8_U8 || kOut == Q8_S8) {
    int z[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) z[j] = __float2int_rn(v[j]);
    unsigned int q[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) q[j] = pack4_sat<kOut == Q8_S8>(z[4 * j], z[4 * j + 1], z[4 * j + 2], z[4 * j + 3]);
    unsigned char* yp = static_cast<unsigned char*>(p.y) + o;
    if (vec) {
      *reinterpret_cast<uint4*>(yp) = make_uint4(q[0], q[1], q[2], q[3]);
    } else {
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (j < valid) yp[j] = (unsigned char)(q[j >> 2] >> (8 * (j & 3)));
    }
  } else {
    int* yp = static_cast<int*>(p.y) + o;
    if (kOut == Q8_F32) {
#pragma unroll
      for (int j = 0; j < 16; ++j) acc[j] = __float_as_int(v[j]);
    }
    if (vec) {
#pragma unroll
      for (int j = 0; j < 4; ++j) reinterpret_cast<int4*>(yp)[j] = make_int4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
    } else {
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (j < valid) yp[j] = acc[j];
    }
  }
}

// kRows: rows of a K block per producer thread (4, 2 or 1 for blocks of 128, 64 or 32 bytes).
template <int kOut, int kRows>
__global__ void __launch_bounds__(kGThreads, 1) conv_gather_kernel(const __grid_constant__ GatherParams p) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long full[kGMaxStages], empty[kGMaxStages];
  __shared__ __align__(8) unsigned long long acc_full[2], acc_empty[2];
  __shared__ uint32_t tmem_holder;
  __shared__ int abort_flag;
  const uint32_t raw_base = smem_u32(smem_raw);
  const uint32_t base = (raw_base + 1023u) & ~1023u;
  unsigned char* const base_ptr = smem_raw + (base - raw_base);
  int* const s_bias = reinterpret_cast<int*>(base_ptr + p.off_chan);
  float* const s_scale = reinterpret_cast<float*>(base_ptr + p.off_chan) + p.n_tiles * p.bn;
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  volatile int* abortp = &abort_flag;

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (warp == kGMmaWarp) {
    if (lane < p.stages) { mbar_init(smem_u32(&full[lane]), kGProdThreads); mbar_init(smem_u32(&empty[lane]), 1); }
    else if (lane >= 16 && lane < 18) { mbar_init(smem_u32(&acc_full[lane - 16]), 1); mbar_init(smem_u32(&acc_empty[lane - 16]), 4); }
    else if (lane == 18) abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
    tmem_alloc(smem_u32(&tmem_holder), (uint32_t)p.tmem_cols);
    tmem_relinquish();
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (warp < kGMmaWarp) {
    for (int i = (int)threadIdx.x; i < p.n_tiles * p.bn; i += kGMmaWarp * 32) {
      s_bias[i] = (p.bias && i < p.K) ? p.bias[i] : 0;
      s_scale[i] = p.scale ? (p.scale_count == 1 ? p.scale[0] : (i < p.K ? p.scale[i] : 0.f)) : 0.f;
    }
  } else if (p.b_resident && warp >= kGFirstProd) {
    for (int nt = 0; nt < p.n_tiles; ++nt)
      gather_weights(p, base_ptr + (size_t)(nt * p.nblk) * p.b_block_bytes, nt * p.bn, 0, p.nblk, (int)threadIdx.x - kGFirstProd * 32,
                     kGProdGroups * kGProdThreads);
    fence_proxy_async_smem();
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem_base = tmem_holder;
  const uint32_t full0 = smem_u32(&full[0]), empty0 = smem_u32(&empty[0]);

  if (warp >= kGFirstProd) {
    // ------------------------------------------------------------------ producers: group g fills K blocks g, g + 2, ...
    const int t = ((int)threadIdx.x - kGFirstProd * 32) & (kGProdThreads - 1);
    const int g = ((int)threadIdx.x - kGFirstProd * 32) / kGProdThreads;
    const int chunk = t & ((1 << p.lg_cpb) - 1), row0 = t >> p.lg_cpb, row_step = kGProdThreads >> p.lg_cpb;
    uint32_t it = 0;  // K blocks of this CTA so far; stage it % stages, parity from it / stages
    uint32_t stage = 0, par = 1;
    bool ok = true;
    for (int tile = (int)blockIdx.x; tile < p.tiles && ok; tile += (int)gridDim.x) {
      if (p.nblk == 1 && (int)(it & 1u) != g) {  // the tile's only block is the other group's
        ++it;
        if (++stage == (uint32_t)p.stages) { stage = 0; par ^= 1u; }
        continue;
      }
      const int mt = p.fd_ntiles.div(tile), nt = tile - mt * p.n_tiles;
      const unsigned char* img[kRows];
      int h0[kRows], c0[kRows], w0[kRows];  // first input row, first byte and first column of the pixel's window
#pragma unroll
      for (int i = 0; i < kRows; ++i) {
        const int m = mt * kBM + row0 + i * row_step;
        const int n = p.fd_pq.div(m), rem = m - n * p.PQ, pr = p.fd_q.div(rem), qc = rem - pr * p.Q;
        img[i] = p.x + (size_t)n * p.H * p.W * p.C;
        h0[i] = m < p.M ? pr * p.stride_h - p.pad_h : -(1 << 28);  // never a row of the image
        w0[i] = qc * p.stride_w - p.pad_w;
        c0[i] = w0[i] * p.C;
      }
      for (int blk = 0; blk < p.nblk; ++blk, ++it) {
        if ((int)(it & 1u) == g) {
          if (!mbar_wait(empty0 + stage * 8u, par, abortp)) { ok = false; break; }
          unsigned char* const dst = base_ptr + p.off_stages + (size_t)stage * p.stage_bytes;
          const int kc = (blk << p.lg_cpb) + chunk;
          const int run = p.fd_chunks.div(kc), j16 = (kc - run * p.run_chunks) * 16;
          const bool live = kc < p.chunks;
          int r = run, s = 0;
          if (p.run_taps != p.S) { r = p.fd_s.div(run); s = run - r * p.S; }
          const int dw = s * p.dil_w;
          Gathered v[kRows];
#pragma unroll
          for (int i = 0; i < kRows; ++i) {
            const int h = h0[i] + r * p.dil_h, first = c0[i] + dw * p.C, wl = w0[i] + dw;
            gather_load(v[i], live && (unsigned)h < (unsigned)p.H, img[i] + (long long)h * p.W * p.C, first + j16, max(wl, 0) * p.C,
                        min(wl + p.run_taps, p.W) * p.C);
          }
#pragma unroll
          for (int i = 0; i < kRows; ++i)
            *reinterpret_cast<uint4*>(dst + swizzled(p, row0 + i * row_step, chunk)) = gather_finish(v[i]);
          if (!p.b_resident) gather_weights(p, dst + kBM * p.bkb, nt * p.bn, blk, 1, t, kGProdThreads);
          fence_proxy_async_smem();
          mbar_arrive(full0 + stage * 8u);
        }
        if (++stage == (uint32_t)p.stages) { stage = 0; par ^= 1u; }
      }
    }
    if (!ok && lane == 0) { abort_flag = 1; atomicOr(p.status, kTimeoutProducer); }
  } else if (warp == kGMmaWarp) {
    // ------------------------------------------------------------------ MMA issue
    const uint32_t st_d0 = kDescLbo | (((base + p.off_stages) >> 4) & 0x3fffu), bres_d0 = kDescLbo | ((base >> 4) & 0x3fffu);
    const uint32_t stage16 = p.stage_bytes >> 4, a16 = (uint32_t)(kBM * p.bkb) >> 4, bblk16 = p.b_block_bytes >> 4;
    const int ksteps = p.bkb >> 5;
    uint32_t stage = 0, par = 0, ab = 0, apar = 1;
    bool ok = true;
    for (int tile = (int)blockIdx.x; tile < p.tiles && ok; tile += (int)gridDim.x) {
      const int mt = p.fd_ntiles.div(tile), nt = tile - mt * p.n_tiles;
      if (!mbar_wait(smem_u32(&acc_empty[0]) + ab * 8u, apar, abortp)) { ok = false; break; }
      tcgen05_fence_after();
      uint32_t accum = 0, bres = bres_d0 + (uint32_t)(nt * p.nblk) * bblk16;
      for (int blk = 0; blk < p.nblk; ++blk, bres += bblk16) {
        if (!mbar_wait(full0 + stage * 8u, par, abortp)) { ok = false; break; }
        tcgen05_fence_after();
        const uint32_t ad = st_d0 + stage * stage16;
        if (elect_one()) {
          umma_i8_block(tmem_base + ab * (uint32_t)p.acc_stride, ad, p.b_resident ? bres : ad + a16, p.desc_hi, p.idesc, accum, ksteps);
          umma_commit(empty0 + stage * 8u);
        }
        accum = 1;
        if (++stage == (uint32_t)p.stages) { stage = 0; par ^= 1u; }
      }
      if (elect_one()) umma_commit(smem_u32(&acc_full[0]) + ab * 8u);
      ab ^= 1u;
      if (ab == 0) apar ^= 1u;
    }
    if (!ok && lane == 0) { abort_flag = 1; atomicOr(p.status, kTimeoutMma); }
  } else {
    // ------------------------------------------------------------------ epilogue, straight to global memory
    // group g takes every second tile of the CTA, which always sits in accumulator g
    const int g = warp >> 2, quad = warp & 3, row = quad * 32 + lane;
    const uint32_t accf = smem_u32(&acc_full[g]), acce = smem_u32(&acc_empty[g]);
    const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(g * p.acc_stride);
    uint32_t apar = 0;
    for (int tile = (int)blockIdx.x + g * (int)gridDim.x; tile < p.tiles; tile += 2 * (int)gridDim.x, apar ^= 1u) {
      const int mt = p.fd_ntiles.div(tile), nt = tile - mt * p.n_tiles;
      if (!mbar_wait(accf, apar, abortp)) {
        if (lane == 0) { abort_flag = 1; atomicOr(p.status, kTimeoutEpilogue); }
        break;
      }
      tcgen05_fence_after();
      for (int c = 0; c < p.bn; c += 16) {
        int acc[16];
        tmem_ld_16(taddr + c, acc);
        tmem_ld_wait(acc);
        if (c + 16 >= p.bn) {  // the accumulator's last columns are in registers
          tcgen05_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(acce);
        }
        gather_epilogue<kOut>(p, s_bias, s_scale, acc, (long long)mt * kBM + row, nt * p.bn + c);
        __syncwarp();
      }
    }
  }

  tcgen05_fence_before();
  __syncthreads();
  if (warp == kGMmaWarp) {
    __syncwarp();
    tcgen05_fence_after();
    tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
  }
}

template <int kOut, int kRows>
int launch_gather_variant(const GatherParams& p, size_t dyn, cudaStream_t stream) {
  auto kernel = conv_gather_kernel<kOut, kRows>;
  static std::atomic<bool> configured[kMaxDevices];
  const int dev = current_device();
  if (dev < 0 || !configured[dev].load(std::memory_order_acquire)) {
    int rc = check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit - kStaticSmemReserve),
                        "conv_gather: set shared memory size");
    if (rc != Q8_OK) return rc;
    rc = check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared),
                    "conv_gather: set shared memory carve-out");
    if (rc != Q8_OK) return rc;
    if (dev >= 0) configured[dev].store(true, std::memory_order_release);
  }
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)(p.tiles < sm_count() ? p.tiles : sm_count()));
  cfg.blockDim = dim3((unsigned)kGThreads);
  cfg.dynamicSmemBytes = dyn < 120 * 1024 ? 120 * 1024 : dyn;  // one CTA per SM owns the SM's TMEM
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t le = cudaLaunchKernelEx(&cfg, kernel, p);
  if (le != cudaSuccess) {
    cudaGetLastError();
    return fail(Q8_ERR_CUDA, "conv_gather: launch failed (%s)", cudaGetErrorString(le));
  }
  return check_launch("conv_gather_kernel");
}

}  // namespace

namespace {
struct GatherTiles {
  int run_taps, run_chunks, chunks;  // see GatherParams
  int lg_cpb, nblk, bn, n_tiles;
  long long tiles;
};

GatherTiles gather_tiles(const ConvArgs& a) {
  const q8_conv_desc& d = a.d;
  GatherTiles t;
  t.run_taps = (d.dil_w == 1 || d.S == 1) ? d.S : 1;
  t.run_chunks = (t.run_taps * d.C + 15) / 16;
  t.chunks = (d.R * d.S / t.run_taps) * t.run_chunks;
  t.lg_cpb = t.chunks <= 2 ? 1 : (t.chunks <= 4 ? 2 : 3);
  t.nblk = (t.chunks + (1 << t.lg_cpb) - 1) >> t.lg_cpb;
  // Tile width: up to 128 columns; narrower ones while most SMs would stay without a tile.  The activations are
  // gathered again for every tile of columns, but by SMs that had nothing to do (1x1 of 200 -> 500 channels at 14x14:
  // 30.8 us with tiles of 128 columns, 10.2 us with these).
  const long long m_tiles = (a.M + kBM - 1) / kBM;
  t.n_tiles = (d.K + 127) / 128;
  while (m_tiles * t.n_tiles * 2 <= sm_count() && (d.K + 2 * t.n_tiles - 1) / (2 * t.n_tiles) > 16) t.n_tiles *= 2;
  t.bn = ((d.K + t.n_tiles - 1) / t.n_tiles + 15) / 16 * 16;
  t.n_tiles = (d.K + t.bn - 1) / t.bn;
  t.tiles = m_tiles * t.n_tiles;
  return t;
}

// Whole 16-channel chunks of a row can be stored in 16-byte pieces.
bool gather_vec(const ConvArgs& a) {
  const int grid = a.d.y_type == Q8_U8 || a.d.y_type == Q8_S8 ? 16 : 4;
  return aligned16(a.y) && a.ldc % grid == 0 && a.c_off % grid == 0;
}
}  // namespace

// Fitted together with the direct kernel's estimate (see there).  Start-up; a K block in flight; the chunks of columns that
// a CTA stores, dearest byte by byte; the bytes that its producers gather.
double gather_us(const ConvArgs& a) {
  const GatherTiles t = gather_tiles(a);
  const double waves = (double)((t.tiles + sm_count() - 1) / sm_count()), columns = (t.bn < a.d.K ? t.bn : a.d.K) / 16.0;
  const bool out8 = a.d.y_type == Q8_U8 || a.d.y_type == Q8_S8;
  const double store = gather_vec(a) ? 0.18 : (out8 ? 1.6 * (a.M < kBM ? (double)a.M / kBM : 1.0) : 0.66);
  return 2.5 + 0.75 * t.nblk + waves * (columns * store + 4.6 * t.nblk * t.bn / 128.0 * (1 << t.lg_cpb) / 8.0);
}

// The channel arrays of 4096 outputs fit beside the stages.  Positions in a row of input pixels, padding included, are
// 32-bit byte offsets, and rows past the last pixel are told by a row number below -2^28; wider images and filters stay
// with the direct kernel, whose addresses are 64-bit.
bool gather_addressable(const q8_conv_desc& d) {
  const long long row = ((long long)d.W + 2ll * d.pad_w + (long long)d.S * d.dil_w) * d.C;
  return d.K <= 4096 && row < (1ll << 30) && d.H + 2ll * d.pad_h < (1ll << 28) && (long long)d.R * d.dil_h < (1ll << 28);
}

int launch_conv_gather(const ConvArgs& a) {
  const q8_conv_desc& d = a.d;
  GatherParams p;
  memset(&p, 0, sizeof(p));
  p.status = status_word_device_ptr();
  if (!p.status) return fail(Q8_ERR_CUDA, "conv_gather: status word not available");
  p.x = static_cast<const unsigned char*>(a.x);
  p.w = reinterpret_cast<const unsigned char*>(a.w);
  p.bias = a.bias; p.scale = a.scale; p.scale_count = d.scale_count;
  p.res = static_cast<const unsigned char*>(a.residual);
  p.res_vec = d.K % 16 == 0 && aligned16(a.residual);
  p.res_signed = d.res_type == Q8_S8; p.res_scale = a.residual_scale;
  p.y = a.y; p.ldc = a.ldc; p.c_off = a.c_off; p.relu = d.relu;
  p.y_vec = gather_vec(a);
  p.H = d.H; p.W = d.W; p.C = d.C; p.K = d.K; p.S = d.S;
  p.P = a.P; p.Q = a.Q; p.PQ = a.P * a.Q; p.M = (int)a.M;
  p.stride_h = d.stride_h; p.stride_w = d.stride_w; p.pad_h = d.pad_h; p.pad_w = d.pad_w; p.dil_h = d.dil_h; p.dil_w = d.dil_w;
  const GatherTiles t = gather_tiles(a);
  p.rsc = d.R * d.S * d.C;
  p.run_taps = t.run_taps; p.run_len = t.run_taps * d.C; p.run_chunks = t.run_chunks; p.chunks = t.chunks;
  p.lg_cpb = t.lg_cpb;
  p.bkb = 16 << t.lg_cpb;
  p.nblk = t.nblk;
  p.swz_mask = p.bkb == 128 ? 7u : (p.bkb == 64 ? 3u : 1u);
  p.bn = t.bn; p.n_tiles = t.n_tiles;
  const long long tiles = t.tiles;
  if (tiles > 0x7fffffff) return fail(Q8_ERR_UNSUPPORTED, "conv_gather: too many tiles");
  p.tiles = (int)tiles;
  p.acc_stride = 32;
  while (p.acc_stride < p.bn) p.acc_stride *= 2;
  p.tmem_cols = 2 * p.acc_stride;
  p.fd_q = make_fastdiv(p.Q); p.fd_pq = make_fastdiv(p.PQ); p.fd_chunks = make_fastdiv(p.run_chunks);
  p.fd_s = make_fastdiv(d.S); p.fd_ntiles = make_fastdiv(p.n_tiles); p.fd_bn = make_fastdiv(p.bn);
  p.b_block_bytes = round_up((unsigned)(p.bn * p.bkb), 1024u);
  const unsigned chan = round_up((unsigned)(p.n_tiles * p.bn) * 8u, 1024u);
  const unsigned budget = (unsigned)(kSmemLimit - kStaticSmemReserve) - 1024u - chan;
  const unsigned long long b_all = (unsigned long long)p.n_tiles * p.nblk * p.b_block_bytes;
  const unsigned a_bytes = (unsigned)(kBM * p.bkb);
  // resident weights cost one gather of all of them: worth it for CTAs that run through every tile of columns
  p.b_resident = tiles >= (long long)p.n_tiles * sm_count() && b_all <= 128u * 1024u && budget >= b_all + 3u * a_bytes;
  p.stage_bytes = a_bytes + (p.b_resident ? 0u : p.b_block_bytes);
  p.off_stages = p.b_resident ? (unsigned)b_all : 0u;
  const unsigned rest = budget - p.off_stages;
  p.stages = (int)(rest / p.stage_bytes);
  if (p.stages > kGMaxStages) p.stages = kGMaxStages;
  p.off_chan = p.off_stages + (unsigned)p.stages * p.stage_bytes;
  const size_t dyn = 1024u + p.off_chan + chan;
  // instruction and matrix descriptors as in the TMA-fed kernel (q8_conv_umma.cu)
  p.idesc = (2u << 4) | ((d.x_type == Q8_S8 ? 1u : 0u) << 7) | (1u << 10) | ((unsigned)(p.bn >> 3) << 17) | ((unsigned)(kBM >> 4) << 24);
  p.desc_hi = (unsigned)((8 * p.bkb) >> 4) | (1u << 14) | ((p.bkb == 128 ? 2u : (p.bkb == 64 ? 4u : 6u)) << 29);
#define Q8_GATHER(OUT)                                                          \
  do {                                                                          \
    if (p.lg_cpb == 3) return launch_gather_variant<OUT, 4>(p, dyn, a.stream);  \
    if (p.lg_cpb == 2) return launch_gather_variant<OUT, 2>(p, dyn, a.stream);  \
    return launch_gather_variant<OUT, 1>(p, dyn, a.stream);                     \
  } while (0)
  if (d.y_type == Q8_U8) Q8_GATHER(Q8_U8);
  if (d.y_type == Q8_S8) Q8_GATHER(Q8_S8);
  if (d.y_type == Q8_F32) Q8_GATHER(Q8_F32);
  Q8_GATHER(Q8_S32);
#undef Q8_GATHER
}

}  // namespace q8

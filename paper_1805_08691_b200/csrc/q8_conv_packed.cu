// Quantized convolution on the tensor cores for images of three channels, as they come: the first layer of a network.
//
//   D[128 pixels, BN channels] (int32, TMEM) = A[128, Kp] (packed) x B[BN, Kp]^T,   Kp = R S C bytes, padded to whole K steps
//
// A tile is 128 consecutive output pixels.  The input rows that they read are one contiguous span of memory (NHWC; also
// across the end of an image), which one bulk copy brings into shared memory.  A thread per pixel then packs the pixel's
// R runs of S C bytes densely, in the order in which the weights of a filter lie in memory, into its row of the K-major
// swizzled tile that tcgen05.mma reads: unaligned words of the span by funnel shifts, joined by shifts that are compile-time
// constants (filters of 3, 5 or 7 rows and 1, 3, 5 or 7 columns, and 1x1).  Bytes outside the image are masked to zero, the exact code of 0.0.
//
// Roles: warps 0-15 four epilogue groups, each with its accumulator (thread = accumulator row), warp 16 MMA issue and TMEM, warp
// 17 bulk copies, warps 18-25 two packing groups on alternate tiles.  Weights are resident.  All waits are bounded as in the
// other tensor-core kernels.
//
// The gathering kernel, which took these layers before, fetches every 16-byte chunk of a run from global memory with five
// predicated loads and masks: 5560 warp instructions per tile of 3x3/2 on three channels, 64 bytes of reduction for 27
// (3 -> 32 channels on 8 x 299x299 12.3 us, here 7.8 us, of which about 3 are the chain of a launch).
#include <type_traits>

#include "q8_umma_common.cuh"

namespace q8 {
namespace {

constexpr int kPkEpiGroups = 4;                                    // ... and accumulators
constexpr int kPkMmaWarp = 4 * kPkEpiGroups, kPkCopyWarp = kPkMmaWarp + 1, kPkFirstPack = kPkCopyWarp + 1;
constexpr int kPkMaxReduction = 256;                               // bytes of a filter
constexpr int kPkGroups = 2;                                       // packing groups
constexpr int kPkStages = 4;                                       // span stages, A stages
constexpr int kPkThreads = (kPkFirstPack + 4 * kPkGroups) * 32;    // 832
constexpr unsigned int kPkMaxSpan = 24 * 1024;                     // bytes of a tile's span

struct PackedParams {
  UmmaParams u;              // what the epilogue reads: M, K, bn, bias, scale, residual, output
  const unsigned char* x;
  const unsigned char* w;
  int H, W, C;
  int stride_h, stride_w, pad_h, pad_w, dil_h;
  int R, run_len;            // runs (filter rows), bytes of a run
  int reduction;             // R * run_len
  int row_bytes;             // W * C
  int bkb, lg_cpb, nblk;     // bytes per K block (32, 64 or 128), log2 of its 16-byte chunks, number of blocks
  int ksteps, last_ksteps;   // K steps of a block, of the last one
  int m_tiles;
  unsigned int span_cap, margin, off_a, a_bytes, off_span, off_chan, b_block_bytes, swz_mask;
  int acc_stride, tmem_cols, res_vec;
  FastDiv fd_q, fd_pq, fd_words;
};

// First input row (of all images' rows, one after the other) and one past the last that the pixels m0 .. m1 read.
__device__ __forceinline__ void tile_rows(const PackedParams& p, int m0, int m1, int* first, int* end) {
  const int n0 = p.fd_pq.div(m0), n1 = p.fd_pq.div(m1);
  const int h0 = p.fd_q.div(m0 - n0 * p.u.PQ) * p.stride_h - p.pad_h;
  const int h1 = p.fd_q.div(m1 - n1 * p.u.PQ) * p.stride_h - p.pad_h + (p.R - 1) * p.dil_h;
  *first = n0 * p.H + min(max(h0, 0), p.H - 1);
  *end = n1 * p.H + min(max(h1, 0), p.H - 1) + 1;
}

// One pixel's row of the operand tile: kR runs of kL bytes, the first at byte at0 of the span, the others row by row below it.
template <int kL, int kR, bool kMasked>
__device__ __forceinline__ void pack_row(const PackedParams& p, const unsigned char* span, unsigned char* dst, int row, int at0, int vl, int vh,
                                         int h0) {
  constexpr int kWords = (kL + 3) / 4, kLoads = (kL + 6) / 4;  // words of a run; those that hold it at any alignment
  unsigned int inside[kWords];                                 // bytes of a run that lie inside the image
  if (kMasked) {
#pragma unroll
    for (int j = 0; j < kWords; ++j) {
      const int lo = min(max(vl - 4 * j, 0), 4), hi = min(max(vh - 4 * j, 0), 4);
      inside[j] = (hi == 4 ? 0xffffffffu : (1u << (8 * hi)) - 1u) & (lo == 4 ? 0u : ~((1u << (8 * lo)) - 1u));
    }
  }
  unsigned int q[4] = {0u, 0u, 0u, 0u}, cur = 0u;
  auto emit = [&](int kw, unsigned int word) {
    q[kw & 3] = word;
    if ((kw & 3) == 3 || kw == (kL * kR + 3) / 4 - 1) {
      const int blk = (kw >> 2) >> p.lg_cpb, col = (kw >> 2 << 4) - (blk << (p.lg_cpb + 4));
      const uint32_t off = (uint32_t)(row * p.bkb + col);
      *reinterpret_cast<uint4*>(dst + (size_t)blk * (kBM * p.bkb) + (off ^ (((off >> 7) & p.swz_mask) << 4))) = make_uint4(q[0], q[1], q[2], q[3]);
      q[0] = q[1] = q[2] = q[3] = 0u;
    }
  };
#pragma unroll
  for (int r = 0; r < kR; ++r) {
    int at = at0 + r * p.dil_h * p.row_bytes;
    const bool ok = !kMasked || (unsigned)(h0 + r * p.dil_h) < (unsigned)p.H;
    if (kMasked && !ok) at = 0;  // (a row outside the image is not in the span)
    const unsigned int* s = reinterpret_cast<const unsigned int*>(span + (at & ~3));
    unsigned int w[kLoads];
#pragma unroll
    for (int j = 0; j < kLoads; ++j) w[j] = s[j];
#pragma unroll
    for (int j = 0; j < kWords; ++j) {
      unsigned int v = __funnelshift_r(w[j], j + 1 < kLoads ? w[j + 1] : 0u, 8u * (unsigned)at);
      const int bytes = kL - 4 * j < 4 ? kL - 4 * j : 4, pos = r * kL + 4 * j, fill = pos & 3;
      if (kMasked) v &= ok ? inside[j] : 0u;
      if (bytes < 4) v &= (1u << (8 * bytes)) - 1u;
      cur |= v << (8 * fill);
      if (fill + bytes >= 4) {
        emit(pos >> 2, cur);
        cur = fill ? v >> (8 * (4 - fill)) : 0u;
      }
    }
  }
  if (kL * kR % 4) emit(kL * kR / 4, cur);
}
template <int kL, bool kMasked>
__device__ __forceinline__ void pack_rows(const PackedParams& p, const unsigned char* span, unsigned char* dst, int row, int at0, int vl, int vh,
                                          int h0) {
  if (kL == 3 && p.R == 1) pack_row<kL, kL == 3 ? 1 : 3, kMasked>(p, span, dst, row, at0, vl, vh, h0);
  else if (p.R == 3) pack_row<kL, 3, kMasked>(p, span, dst, row, at0, vl, vh, h0);
  else if (p.R == 5) pack_row<kL, 5, kMasked>(p, span, dst, row, at0, vl, vh, h0);
  else pack_row<kL, 7, kMasked>(p, span, dst, row, at0, vl, vh, h0);
}
template <bool kMasked>
__device__ __forceinline__ void pack_any(const PackedParams& p, const unsigned char* span, unsigned char* dst, int row, int at0, int vl, int vh,
                                         int h0) {
  if (p.run_len == 3) pack_rows<3, kMasked>(p, span, dst, row, at0, vl, vh, h0);
  else if (p.run_len == 9) pack_rows<9, kMasked>(p, span, dst, row, at0, vl, vh, h0);
  else if (p.run_len == 15) pack_rows<15, kMasked>(p, span, dst, row, at0, vl, vh, h0);
  else pack_rows<21, kMasked>(p, span, dst, row, at0, vl, vh, h0);
}

template <int kOut, int kRes, bool kUniform>
__global__ void __launch_bounds__(kPkThreads, 1) conv_packed_kernel(const __grid_constant__ PackedParams p) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long span_full[kPkStages], span_empty[kPkStages], a_full[kPkStages], a_empty[kPkStages];
  __shared__ __align__(8) unsigned long long acc_full[kPkEpiGroups], acc_empty[kPkEpiGroups];
  __shared__ uint32_t tmem_holder;
  __shared__ int abort_flag;
  const uint32_t raw_base = smem_u32(smem_raw);
  const uint32_t base = (raw_base + 1023u) & ~1023u;
  unsigned char* const base_ptr = smem_raw + (base - raw_base);
  int* const s_bias = reinterpret_cast<int*>(base_ptr + p.off_chan);
  float* const s_scale = reinterpret_cast<float*>(base_ptr + p.off_chan) + p.u.k_pad;
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  volatile int* abortp = &abort_flag;

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (warp == kPkMmaWarp) {
    if (lane < kPkStages) {
      mbar_init(smem_u32(&span_full[lane]), 1);
      mbar_init(smem_u32(&span_empty[lane]), kGroupThreads);
      mbar_init(smem_u32(&a_full[lane]), kGroupThreads);
      mbar_init(smem_u32(&a_empty[lane]), 1);
    } else if (lane >= 16 && lane < 16 + kPkEpiGroups) {
      mbar_init(smem_u32(&acc_full[lane - 16]), 1);
      mbar_init(smem_u32(&acc_empty[lane - 16]), 4);
    } else if (lane == 24) {
      abort_flag = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
    tmem_alloc(smem_u32(&tmem_holder), (uint32_t)p.tmem_cols);
    tmem_relinquish();
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (warp < kPkMmaWarp) {
    for (int i = (int)threadIdx.x; i < p.u.k_pad; i += kPkMmaWarp * 32) {
      s_bias[i] = (p.u.bias && i < p.u.K) ? p.u.bias[i] : 0;
      s_scale[i] = p.u.scale ? (p.u.scale_count == 1 ? p.u.scale[0] : (i < p.u.K ? p.u.scale[i] : 0.f)) : 0.f;
    }
  }
  if (warp < kPkMmaWarp || warp >= kPkFirstPack) {
    // weights: row n of the tile holds the `reduction` bytes of filter n and zeros; a word per thread and turn, four in flight
    constexpr int kStagers = (kPkMmaWarp + 4 * kPkGroups) * 32;
    const int t = warp < kPkMmaWarp ? (int)threadIdx.x : (int)threadIdx.x - 64, words = p.nblk << (p.lg_cpb + 2), items = p.u.k_pad * words;
    const uintptr_t end = reinterpret_cast<uintptr_t>(p.w) + (size_t)p.u.K * p.reduction;
#pragma unroll 4
    for (int i = t; i < items; i += kStagers) {
      const int n = p.fd_words.div(i), kw = i - n * words, bytes = min(p.reduction - 4 * kw, 4);
      unsigned int v = 0;
      if (n < p.u.K && bytes > 0) {
        const uintptr_t at = reinterpret_cast<uintptr_t>(p.w) + (size_t)n * p.reduction + 4 * kw;
        const unsigned int* g = reinterpret_cast<const unsigned int*>(at & ~(uintptr_t)3);
        const unsigned int hi = (at & 3) != 0 && (at & ~(uintptr_t)3) + 4 < end ? g[1] : 0u;
        v = __funnelshift_r(g[0], hi, 8u * (unsigned)(at & 3));
        if (bytes < 4) v &= (1u << (8 * bytes)) - 1u;
      }
      const int blk = kw >> (p.lg_cpb + 2), col = 4 * kw - (blk << (p.lg_cpb + 4));
      const uint32_t off = (uint32_t)(n * p.bkb + (col & ~15));
      *reinterpret_cast<unsigned int*>(base_ptr + (size_t)blk * p.b_block_bytes + (off ^ (((off >> 7) & p.swz_mask) << 4)) + (col & 15)) = v;
    }
    fence_proxy_async_smem();
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem_base = tmem_holder;
  const int step = (int)gridDim.x, first_tile = (int)blockIdx.x;

  if (warp >= kPkFirstPack) {
    // ------------------------------------------------------------------ packing: group g takes tiles g, g + 2, ... of the CTA
    const int t = (int)threadIdx.x - kPkFirstPack * 32, g = t >> 7, row = t & 127;
    uint32_t stage = (uint32_t)g, par = 0;
    bool ok = true;
    for (int tile = first_tile + g * step; tile < p.m_tiles; tile += kPkGroups * step) {
      unsigned char* const span = base_ptr + p.off_span + (size_t)stage * (p.span_cap + 2 * p.margin) + p.margin;
      unsigned char* const dst = base_ptr + p.off_a + (size_t)stage * p.a_bytes;
      const int m0 = tile * kBM, m = min(m0 + row, p.u.M - 1);
      int first, end;
      tile_rows(p, m0, min(m0 + kBM, p.u.M) - 1, &first, &end);
      const int n = p.fd_pq.div(m), rem = m - n * p.u.PQ, pr = p.fd_q.div(rem), qc = rem - pr * p.u.Q;
      const int h0 = pr * p.stride_h - p.pad_h, w0 = qc * p.stride_w - p.pad_w;
      const int vl = max(-w0, 0) * p.C, vh = max(min(p.run_len, (p.W - w0) * p.C), 0);  // bytes of a run inside the image
      // byte of the span at which the pixel's first run starts (it may lie in the margin)
      const int lead = (int)((reinterpret_cast<uintptr_t>(p.x) + (size_t)first * p.row_bytes) & 15u);
      const int at0 = lead + (n * p.H + h0 - first) * p.row_bytes + w0 * p.C;
      const bool inside = vl == 0 && vh == p.run_len && h0 >= 0 && h0 + (p.R - 1) * p.dil_h < p.H;
      ok = mbar_wait(smem_u32(&span_full[stage]), par, abortp) && mbar_wait(smem_u32(&a_empty[stage]), par ^ 1u, abortp);
      if (!ok) break;
      if (__all_sync(0xffffffffu, inside)) pack_any<false>(p, span, dst, row, at0, vl, vh, h0);
      else pack_any<true>(p, span, dst, row, at0, vl, vh, h0);
      // (what lies behind the last word of a row meets zero weights)
      mbar_arrive(smem_u32(&span_empty[stage]));
      fence_proxy_async_smem();
      mbar_arrive(smem_u32(&a_full[stage]));
      stage += kPkGroups;
      if (stage >= kPkStages) { stage -= kPkStages; par ^= 1u; }
    }
    if (!ok && lane == 0) { abort_flag = 1; atomicOr(p.u.status, kTimeoutProducer); }
  } else if (warp == kPkCopyWarp) {
    // ------------------------------------------------------------------ bulk copies of the spans
    uint32_t g = 0, par = 1;
    bool ok = true;
    for (int tile = first_tile; tile < p.m_tiles; tile += step) {
      int first, end;
      tile_rows(p, tile * kBM, min(tile * kBM + kBM, p.u.M) - 1, &first, &end);
      const uintptr_t a = reinterpret_cast<uintptr_t>(p.x) + (size_t)first * p.row_bytes, b = reinterpret_cast<uintptr_t>(p.x) + (size_t)end * p.row_bytes;
      const uintptr_t lo = a & ~(uintptr_t)15;                                       // whole 16-byte lines, each with a byte of the span
      const unsigned int bytes = min((unsigned int)(((b + 15) & ~(uintptr_t)15) - lo), p.span_cap);  // (span_cap holds any tile's)
      if (!mbar_wait(smem_u32(&span_empty[g]), par, abortp)) { ok = false; break; }
      if (elect_one()) {
        const uint32_t bar = smem_u32(&span_full[g]);
        mbar_arrive_expect_tx(bar, bytes);
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(base + p.off_span + g * (p.span_cap + 2 * p.margin) + p.margin), "l"(lo), "r"(bytes), "r"(bar)
                     : "memory");
      }
      if (++g == kPkStages) { g = 0; par ^= 1u; }
    }
    if (!ok && lane == 0) { abort_flag = 1; atomicOr(p.u.status, kTimeoutProducer); }
  } else if (warp == kPkMmaWarp) {
    // ------------------------------------------------------------------ MMA issue
    const uint32_t a_d0 = kDescLbo | (((base + p.off_a) >> 4) & 0x3fffu), b_d0 = kDescLbo | ((base >> 4) & 0x3fffu);
    const uint32_t a16 = p.a_bytes >> 4, ablk16 = (uint32_t)(kBM * p.bkb) >> 4, bblk16 = p.b_block_bytes >> 4;
    uint32_t g = 0, par = 0, ab = 0, apar = 1;
    bool ok = true;
    for (int tile = first_tile; tile < p.m_tiles && ok; tile += step) {
      if (!mbar_wait(smem_u32(&a_full[g]), par, abortp)) { ok = false; break; }
      if (!mbar_wait(smem_u32(&acc_empty[ab]), apar, abortp)) { ok = false; break; }
      tcgen05_fence_after();
      if (elect_one()) {
        uint32_t ad = a_d0 + g * a16, bd = b_d0;
        for (int blk = 0; blk < p.nblk; ++blk, ad += ablk16, bd += bblk16) {
          const int ks = blk == p.nblk - 1 ? p.last_ksteps : p.ksteps;
          for (int k = 0; k < ks; ++k)
            umma_i8(tmem_base + ab * (uint32_t)p.acc_stride, ad + 2 * k, bd + 2 * k, p.u.desc_hi, p.u.idesc, blk | k ? 1u : 0u);
        }
        umma_commit(smem_u32(&acc_full[ab]));
      }
      if (++ab == kPkEpiGroups) { ab = 0; apar ^= 1u; }
      if (elect_one()) umma_commit(smem_u32(&a_empty[g]));
      if (++g == kPkStages) { g = 0; par ^= 1u; }
    }
    if (!ok && lane == 0) { abort_flag = 1; atomicOr(p.u.status, kTimeoutMma); }
  } else if (warp < kPkMmaWarp) {
    // ------------------------------------------------------------------ epilogue: group g owns accumulator g
    const int g = warp >> 2, quad = warp & 3, row = quad * 32 + lane;
    const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(g * p.acc_stride);
    EpiTile t;
    t.s_bias = s_bias;
    t.s_scale = s_scale;
    t.scale = s_scale[0];
    const float us = kUniform ? __uint_as_float(__reduce_or_sync(0xffffffffu, __float_as_uint(t.scale))) : 0.0f;
    t.buf = nullptr;
    t.yrow = nullptr;
    t.rrow = nullptr;
    t.wide = t.res_wide = false;
    t.y_off = 0;
    t.srow = row;
    t.smem_ok = true;
    t.row_base = t.swz = 0;
    uint32_t apar = 0;
    for (int tile = first_tile + g * step; tile < p.m_tiles; tile += kPkEpiGroups * step) {
        if (!mbar_wait(smem_u32(&acc_full[g]), apar, abortp)) {
          if (lane == 0) { abort_flag = 1; atomicOr(p.u.status, kTimeoutEpilogue); }
          break;
        }
        apar ^= 1u;
        tcgen05_fence_after();
        t.n0 = 0;
        t.m = tile * kBM + row;
        t.row_ok = t.m < p.u.M;
        const int chunks = p.u.bn >> 4;
        int ra[16], rb[16];
        auto residual = [&](int nb, int valid) {
          uint4 rv = make_uint4(0u, 0u, 0u, 0u);
          if (kRes != kResNone && valid > 0) {
            const unsigned char* rp = p.u.res + (size_t)t.m * p.u.K + nb;
            if (p.res_vec && valid == 16) {
              rv = *reinterpret_cast<const uint4*>(rp);
            } else {
              unsigned int b[4] = {0u, 0u, 0u, 0u};
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (j < valid) b[j >> 2] |= (unsigned int)rp[j] << (8 * (j & 3));
              rv = make_uint4(b[0], b[1], b[2], b[3]);
            }
          }
          return rv;
        };
        for (int ch = 0; ch < chunks; ch += 2) {
          const bool two = ch + 1 < chunks;
          tmem_ld_16(taddr + ch * 16, ra);
          if (two) tmem_ld_16(taddr + ch * 16 + 16, rb);
          const int nb = t.n0 + ch * 16, v0 = t.row_ok ? min(16, p.u.K - nb) : 0, v1 = two && t.row_ok ? min(16, p.u.K - nb - 16) : 0;
          const uint4 r0 = residual(nb, v0), r1 = residual(nb + 16, v1);
          tmem_ld_wait(ra);
          tmem_ld_wait(rb);
          if (ch + 2 >= chunks) {  // the accumulator's last columns are in registers
            tcgen05_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&acc_empty[g]));
          }
          const uint4 o0 = epilogue_chunk<kOut, kRes, kUniform>(p.u, t, ch, ra, us, r0);
          uint4 o1 = make_uint4(0u, 0u, 0u, 0u);
          if (two) o1 = epilogue_chunk<kOut, kRes, kUniform>(p.u, t, ch + 1, rb, us, r1);
          if (kOut == Q8_U8 || kOut == Q8_S8) {
            // (rows are stored in 16-byte pieces, see packed_better: a chunk of a row is all there or not)
            unsigned char* yp = static_cast<unsigned char*>(p.u.y) + (size_t)t.m * p.u.ldc + p.u.c_off + nb;
            if (p.u.y_wide && v1 == 16) {
              store_32(yp, o0, o1);
            } else {
              if (v0 > 0) *reinterpret_cast<uint4*>(yp) = o0;
              if (v1 > 0) *reinterpret_cast<uint4*>(yp + 16) = o1;
            }
          }
          __syncwarp();
        }
      }
  }

  tcgen05_fence_before();
  __syncthreads();
  if (warp == kPkMmaWarp) {
    __syncwarp();
    tcgen05_fence_after();
    tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
  }
}

template <int kOut, int kRes, bool kUniform>
int launch_packed_variant(const PackedParams& p, size_t dyn, cudaStream_t stream) {
  auto kernel = conv_packed_kernel<kOut, kRes, kUniform>;
  static std::atomic<bool> configured[kMaxDevices];
  const int dev = current_device();
  if (dev < 0 || !configured[dev].load(std::memory_order_acquire)) {
    int rc = check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit - kStaticSmemReserve),
                        "conv_packed: set shared memory size");
    if (rc != Q8_OK) return rc;
    rc = check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared),
                    "conv_packed: set shared memory carve-out");
    if (rc != Q8_OK) return rc;
    if (dev >= 0) configured[dev].store(true, std::memory_order_release);
  }
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)(p.m_tiles < sm_count() ? p.m_tiles : sm_count()));
  cfg.blockDim = dim3((unsigned)kPkThreads);
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
    return fail(Q8_ERR_CUDA, "conv_packed: launch failed (%s)", cudaGetErrorString(le));
  }
  return check_launch("conv_packed_kernel");
}

// Input rows that 128 consecutive pixels read at most: their output rows, the window below the last, and where they cross the
// end of an image (once, with P Q >= 128) the rows of a window and a stride that no pixel of the image's last row starts in.
long long span_rows(const q8_conv_desc& d, int Q) {
  const long long out_rows = (kBM - 2 + Q) / Q + 1;
  return (out_rows + 2) * d.stride_h + 2ll * (d.R - 1) * d.dil_h + d.pad_h + 2;
}
bool packed_eligible(const q8_conv_desc& d, int P, int Q) {
  const long long red = (long long)d.R * d.S * d.C, row = (long long)d.W * d.C, pads = ((long long)d.pad_w + (long long)d.S) * d.C;
  auto compiled = [](int v) { return v == 1 || v == 3 || v == 5 || v == 7; };
  return d.C == 3 && compiled(d.R) && compiled(d.S) && (d.R > 1 || d.S == 1) && (d.dil_w == 1 || d.S == 1) && red <= kPkMaxReduction &&
         (long long)P * Q >= kBM && d.K <= 128 && pads <= 1024 &&
         d.pad_h < (1 << 20) && (long long)d.R * d.dil_h < (1 << 20) && span_rows(d, Q) * row + 32 <= (long long)kPkMaxSpan &&
         (long long)d.N * d.H < (1ll << 31) && (d.H - 1ll + d.pad_h) * row < (1ll << 30);
}
}  // namespace

// Where it is faster than the kernels that took such layers: one tile of columns (weights are staged word by word, and what is
// gathered again for every further tile is little), rows stored in 16-byte pieces (the kernel relies on it), half of the SMs at
// work, and not a single run of several columns (1xS), which the gathering kernel fetches densely as well (1x7 of 3 -> 112 on
// 7 x 58x60: 5.4 there, 6.2 us here).  Over 160 random layers of these forms, replayed from a graph, 1.31 times faster in the
// mean, from 2.7 times (5x5 of 3 -> 16 on 30 x 197x199 89 -> 33 us) to as fast (5x5 of 3 -> 80 on 108x108 6.1 us both).
// 32-bit outputs of more than 48 channels that end inside a 16-column chunk store that chunk word by word: up to three tiles
// per CTA still faster (85 random layers: 1.1 times), slower beyond (3x3 of 3 -> 104 on 10 x 258x258 172 against 118 us gathered;
// 3x7 of 3 -> 60 on 25 x 172x174 149 against 108), while whole chunks and narrower outputs gain at any size (1.2 and 1.4 times).
bool packed_better(const ConvArgs& a) {
  const int grid = a.d.y_type == Q8_U8 || a.d.y_type == Q8_S8 ? 16 : 4;
  if (grid == 4 && a.d.K % 16 && a.d.K > 48 && a.M > 3ll * kBM * sm_count()) return false;
  return packed_eligible(a.d, a.P, a.Q) && a.M > (long long)kBM * sm_count() / 2 && a.d.K % grid == 0 && aligned16(a.y) && a.ldc % grid == 0 &&
         a.c_off % grid == 0;
}

int launch_conv_packed(const ConvArgs& a) {
  const q8_conv_desc& d = a.d;
  PackedParams p;
  memset(&p, 0, sizeof(p));
  UmmaParams& u = p.u;
  u.status = status_word_device_ptr();
  if (!u.status) return fail(Q8_ERR_CUDA, "conv_packed: status word not available");
  const bool out8 = d.y_type == Q8_U8 || d.y_type == Q8_S8;
  u.M = (int)a.M; u.K = d.K; u.P = a.P; u.Q = a.Q; u.PQ = a.P * a.Q;
  u.bias = a.bias; u.scale = a.scale; u.scale_count = d.scale_count;
  u.res = static_cast<const unsigned char*>(a.residual);
  u.res_mode = a.residual ? kResVec : kResNone;
  u.res_signed = d.res_type == Q8_S8; u.res_scale = a.residual_scale;
  u.y = a.y; u.y_type = d.y_type; u.ldc = a.ldc; u.c_off = a.c_off; u.relu = d.relu;
  u.y_vec = 1;
  u.y_wide = out8 && (reinterpret_cast<uintptr_t>(a.y) & 31u) == 0 && a.ldc % 32 == 0 && a.c_off % 32 == 0;
  p.res_vec = d.K % 16 == 0 && aligned16(a.residual);
  p.x = static_cast<const unsigned char*>(a.x);
  p.w = reinterpret_cast<const unsigned char*>(a.w);
  p.H = d.H; p.W = d.W; p.C = d.C;
  p.stride_h = d.stride_h; p.stride_w = d.stride_w; p.pad_h = d.pad_h; p.pad_w = d.pad_w; p.dil_h = d.dil_h;
  p.R = d.R; p.run_len = d.S * d.C; p.reduction = d.R * p.run_len;
  p.row_bytes = d.W * d.C;
  const int chunks = (p.reduction + 15) / 16;
  p.lg_cpb = chunks <= 2 ? 1 : (chunks <= 4 ? 2 : 3);
  p.bkb = 16 << p.lg_cpb;
  p.nblk = (p.reduction + p.bkb - 1) / p.bkb;
  p.ksteps = p.bkb / 32;
  p.last_ksteps = (p.reduction - (p.nblk - 1) * p.bkb + 31) / 32;
  p.swz_mask = p.bkb == 128 ? 7u : (p.bkb == 64 ? 3u : 1u);
  u.bn = (d.K + 15) / 16 * 16;
  u.k_pad = u.bn;
  p.m_tiles = (int)((a.M + kBM - 1) / kBM);
  p.acc_stride = 32;
  while (p.acc_stride < u.bn) p.acc_stride *= 2;
  p.tmem_cols = kPkEpiGroups * p.acc_stride;
  p.fd_q = make_fastdiv(a.Q); p.fd_pq = make_fastdiv(u.PQ); p.fd_words = make_fastdiv(p.nblk << (p.lg_cpb + 2));
  p.b_block_bytes = round_up((unsigned)(u.bn * p.bkb), 1024u);
  p.a_bytes = (unsigned)(p.nblk * kBM * p.bkb);
  // runs that start left of the image or end right of it are read (and masked) up to this far outside the span
  p.margin = round_up((unsigned)((d.pad_w + d.S) * d.C) + 16u, 128u);
  p.span_cap = round_up((unsigned)(span_rows(d, a.Q) * p.row_bytes + 32), 128u);
  p.off_a = (unsigned)p.nblk * p.b_block_bytes;
  p.off_span = p.off_a + (unsigned)kPkStages * p.a_bytes;
  p.off_chan = round_up(p.off_span + (unsigned)kPkStages * (p.span_cap + 2u * p.margin), 1024u);
  const size_t dyn = 1024u + p.off_chan + round_up((unsigned)u.k_pad * 8u, 1024u);
  if (dyn > (size_t)(kSmemLimit - kStaticSmemReserve)) return kPlanNoFit;
  // instruction and matrix descriptors as in the TMA-fed kernel (q8_conv_umma.cu)
  u.idesc = (2u << 4) | ((d.x_type == Q8_S8 ? 1u : 0u) << 7) | (1u << 10) | ((unsigned)(u.bn >> 3) << 17) | ((unsigned)(kBM >> 4) << 24);
  u.desc_hi = (unsigned)((8 * p.bkb) >> 4) | (1u << 14) | ((p.bkb == 128 ? 2u : (p.bkb == 64 ? 4u : 6u)) << 29);
#define Q8_PACKED(OUT)                                                                                              \
  do {                                                                                                              \
    if (a.residual) return launch_packed_variant<OUT, kResVec, false>(p, dyn, a.stream);                            \
    if (d.scale_count == 1) return launch_packed_variant<OUT, kResNone, true>(p, dyn, a.stream);                    \
    return launch_packed_variant<OUT, kResNone, false>(p, dyn, a.stream);                                           \
  } while (0)
  if (d.y_type == Q8_U8) Q8_PACKED(Q8_U8);
  if (d.y_type == Q8_S8) Q8_PACKED(Q8_S8);
  if (d.y_type == Q8_F32) Q8_PACKED(Q8_F32);
  return launch_packed_variant<Q8_S32, kResNone, false>(p, dyn, a.stream);
#undef Q8_PACKED
}

}  // namespace q8

// Device and host helpers shared by the tensor-core convolution kernels (q8_conv_umma.cu, q8_conv_fused.cu):
// launch constants, the kernel parameter block, the tile walker, single-instruction PTX wrappers (mbarrier, TMA,
// tcgen05), the requantizing epilogue of one accumulator row, and the host-side planning helpers (driver entry
// points for tensor maps, halo tiling, channel-block and tile-width choice).  Everything here has internal linkage.
#pragma once
#include <cuda.h>

#include <atomic>
#include <cstdlib>
#include <cstring>
#include <initializer_list>

#include "q8_internal.h"

namespace q8 {
namespace {

constexpr int kBM = 128;
constexpr int kCtrlWarps = 4;            // producer, MMA 0, 1, 2
constexpr int kCtrlThreads = kCtrlWarps * 32;
constexpr int kMmaWarps = 3;             // at most this many MMA-issuing lanes; tile lt belongs to lane lt % mma_lanes
constexpr int kGroupThreads = 128;      // one epilogue group
constexpr int kMaxStages = 8;           // A stages
constexpr int kMaxBStages = 8;          // weight ring
constexpr int kMaxAcc = 4;
constexpr int kMaxSlots = 8;            // 8-bit tile buffers over all groups
constexpr int kMaxTaps = 64;            // halo mode: filter taps (one TMA box holds all taps of resident weights)
constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // 2 s per wait
constexpr int kSmemLimit = 232448;                           // 227 KiB opt-in maximum per CTA
constexpr int kStaticSmemReserve = 2048;                     // barriers and flags

enum StatusBits : unsigned int {
  kTimeoutProducer = 1u,
  kTimeoutMma = 2u,
  kTimeoutEpilogue = 4u,
  kTimeoutResidual = 8u,
  kTimeoutStore = 16u,
};

enum ResMode : int { kResNone = 0, kResVec = 1, kResGlobal = 2, kResRows = 3, kResTma = 4 };
enum AMode : int { kAPlain = 0, kAIm2col = 1, kAHalo = 2 };
enum BMode : int { kBStage = 0, kBResident = 1, kBRing = 2 };

// Division by a launch-time constant without the ~35-instruction software divide, which costs a
// lone control lane some 200 cycles: q = (umulhi(x, m) + x) >> l for 0 <= x < 2^31 (Granlund-Montgomery).
struct FastDiv {
  unsigned int m, l;
  int d;
#ifdef __CUDACC__
  __device__ __forceinline__ int div(int x) const { return (int)((__umulhi((unsigned int)x, m) + (unsigned int)x) >> l); }
#endif
};

struct UmmaParams {
  int M, K;                  // GEMM rows (pixels) and Cout
  int P, Q, PQ;              // output height, width, pixels per image
  int stride_h, stride_w, pad_h, pad_w, dil_h, dil_w;
  int R, S, taps;            // filter height, width, R * S
  int C_pad, c_blocks;       // channels rounded up to whole K blocks, number of K blocks
  int bn, bk, ksteps;        // tile width (multiple of 16), K bytes per block (32/64/128), bk / 32
  int a_mode, b_mode;
  int k_iters, kb;           // plain/im2col: taps * c_blocks (tap, block) iterations, kb of them per A stage
  int tw, th, twb, hb;       // halo: tile and patch extents in pixels (pixel pairs along W when halo_sw == 2)
  int halo_sw, halo_e, c_true;  // halo: stride along W (1 or 2), parity of pad_w, channels per input pixel
  int p_tiles, q_tiles;      // halo: tiles per image column / row
  int stages, b_stages;      // A stages, weight-ring stages
  int nacc, acc_stride, tmem_cols;  // TMEM accumulators, columns between them, allocation (power of two)
  int m_tiles, n_tiles;
  FastDiv fd_ntiles, fd_perimg, fd_qtiles, fd_pq, fd_q;  // n_tiles, p_tiles*q_tiles, q_tiles, P*Q, Q
  int splits, kps;           // split-K: work item = (tile, split), each split runs kps of the k_iters iterations
  FastDiv fd_splits, fd_cblocks, fd_s;  // splits, c_blocks, S
  long long split_stride;    // elements between the partial results of two splits in the workspace
  unsigned int idesc;        // tcgen05 instruction descriptor
  unsigned int desc_hi;      // high word of the shared-memory matrix descriptors
  unsigned int a_sub_bytes;  // plain/im2col: one 128 x bk block; halo: bytes of one patch load
  unsigned int b_tile_bytes; // bn * bk
  unsigned int b_sub_bytes;  // b_tile_bytes rounded up to 1 KiB (placement inside a stage); ring: one ring stage
  int cta2;                  // 1: CTA pairs (clusters of two) issue tcgen05.mma.cta_group::2 over two m tiles that
                             // share the n tile; each CTA holds its own A patch and half of the weight tile rows
  int m_tiles_real;          // cta2: number of real m tiles (m_tiles counts pairs)
  // halo: the taps of a filter are walked in the order of their weight tiles, `tap_inner` of them at a time; the
  // patch descriptor moves by in16 (16-byte units) from one tap to the next and by out16 from one group to the next
  unsigned int in16, out16;
  int tap_inner;
  int mma_lanes;             // MMA-issuing warps: 3 with four accumulators, else 2 (see plan_tiles)
  int pair_shift;            // cta2: log2 of the epilogue groups that share the columns of a tile
  int epi_split;             // 1: every epilogue group takes a share of the columns of every tile (short launches)
  int b_T, b_chunks;         // weight ring: filter taps per ring stage (one TMA operation), stages per channel block
  unsigned int a_stage_bytes;
  unsigned int tile8_bytes;
  int nbuf;                  // 8-bit tile buffers per epilogue group or team that TMA fills and empties (0: none)
  unsigned int res_tx_bytes; // bytes one residual tile load delivers
  unsigned int off_a, off_bring, off_bufs, off_chan;  // from the 1 KiB aligned base; resident weights at 0
  int pw_shift, pmask, panels;  // 8-bit tiles live in smem as panels of 2^pw_shift bytes per row
  int k_pad;                 // n_tiles * bn channels of bias/scale staged in smem
  const int* bias;
  const float* scale;
  int scale_count;
  const unsigned char* res;
  int res_mode, res_signed;
  float res_scale;
  void* y;
  int y_type, y_vec, ldc, c_off, relu;
  int y_wide, res_wide;      // 8-bit rows of the output, of the residual, start on 32-byte lines
  unsigned int* status;
};

// Walks the tiles of one role: tile = first, first + step, ...; tile -> (m tile, n tile) with the
// n tiles of one m tile adjacent (they share the A operand through L2), and for halo tiles
// m tile -> (image, tile row, tile column).  Only additions after init().
template <bool kPair>
struct TileIterT {
  int tile, step;    // work item index (tile * splits + split) and its stride
  int sp, d_sp;      // split-K part of the work item
  int mt, nt;        // m tile, n tile
  int img, pt, qt;   // halo: image, tile row, tile column
  int d_mt, d_nt, d_img, d_pt, d_qt;
  int rank;          // cta2: this CTA's rank in its pair; work items are pairs of m tiles (2 * pair + rank)
  bool valid;        // cta2: the m tile exists (the last pair of an odd count has a phantom second tile)

  // cta2: plain re-decoding, a handful of multiply-shift divisions per tile of several thousand cycles
  __device__ __forceinline__ void decode_pair(const UmmaParams& p) {
    const int mp = p.fd_ntiles.div(tile);
    nt = tile - mp * p.n_tiles;
    mt = 2 * mp + rank;
    valid = mt < p.m_tiles_real;
    const int per_img = p.p_tiles * p.q_tiles;
    img = p.fd_perimg.div(mt);
    const int r = mt - img * per_img;
    pt = p.fd_qtiles.div(r);
    qt = r - pt * p.q_tiles;
  }

  __device__ __forceinline__ void init(const UmmaParams& p, int first, int step_, int rank_ = 0) {
    tile = first; step = step_;
    rank = rank_; valid = true;
    if constexpr (kPair) { sp = d_sp = 0; decode_pair(p); return; }
    int t0 = first, dt = step_;  // output tile and its stride
    sp = d_sp = 0;
    if (p.splits > 1) {
      t0 = p.fd_splits.div(first); sp = first - t0 * p.splits;
      dt = p.fd_splits.div(step_); d_sp = step_ - dt * p.splits;
    }
    mt = p.fd_ntiles.div(t0); nt = t0 - mt * p.n_tiles;
    d_mt = p.fd_ntiles.div(dt); d_nt = dt - d_mt * p.n_tiles;
    img = pt = qt = d_img = d_pt = d_qt = 0;
    if (p.a_mode == kAHalo) {
      const int per_img = p.p_tiles * p.q_tiles;
      img = p.fd_perimg.div(mt);
      int r = mt - img * per_img;
      pt = p.fd_qtiles.div(r); qt = r - pt * p.q_tiles;
      d_img = p.fd_perimg.div(d_mt);
      r = d_mt - d_img * per_img;
      d_pt = p.fd_qtiles.div(r); d_qt = r - d_pt * p.q_tiles;
    }
  }
  __device__ __forceinline__ void next(const UmmaParams& p) {
    tile += step;
    if constexpr (kPair) { decode_pair(p); return; }
    int carry = 0;
    sp += d_sp;
    if (sp >= p.splits) { sp -= p.splits; carry = 1; }
    nt += d_nt + carry; carry = 0;
    if (nt >= p.n_tiles) { nt -= p.n_tiles; carry = 1; }
    mt += d_mt + carry;
    if (p.a_mode == kAHalo) {
      qt += d_qt + carry; carry = 0;
      if (qt >= p.q_tiles) { qt -= p.q_tiles; carry = 1; }
      pt += d_pt + carry; carry = 0;
      if (pt >= p.p_tiles) { pt -= p.p_tiles; carry = 1; }
      img += d_img + carry;
    }
  }
};

// ------------------------------------------------------------------------------------------ PTX
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long global_timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Low word of a shared-memory matrix descriptor: (start address >> 4) | kDescLbo, the leading-byte-offset field
// (bits 16-29), unused for swizzled K-major tiles, set to 1.
constexpr uint32_t kDescLbo = 1u << 16;

// One lane of a converged warp.  The control roles issue under this predicate and never under "lane == 0": tcgen05.mma
// and the TMA copies take warp-uniform operands, and an elected branch tells the compiler that it holds a single thread.
// Together with 32-bit descriptor words and rolled tap loops, timed against the branch on the lane number: 3x3 64->64 at
// 300x300 63.3 -> 53.5 us (batch 16), 3x3 512->512 at 7x7 18.9 -> 15.1 us, 3x3 64->64 + 1x1 64->256 + residual at 56x56
// 38.2 -> 32.3 us (batch 64), one 14x14 layer 5.3 -> 4.4 us.
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
  return pred != 0;
}

// Waits are warp collective: every role runs as a whole converged warp (its loop counters, addresses and
// descriptors then are warp-uniform values), all 32 lanes poll, and the votes make the outcome uniform by
// construction.
// Slow path of a wait, out of line to keep the role loops small.  Gives up after about
// kWaitLimitNs or when another role of this CTA has already given up; the caller then records the
// site and leaves its loop.  The wall clock is only read once the wait has lasted a while.
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                            unsigned long long limit_ns = kWaitLimitNs) {
  unsigned long long t0 = 0;
  uint32_t spins = 0;
  for (;;) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity) ? 1 : 0)) return true;
    if ((++spins & 0x3ffu) == 0) {
      int give_up = *abort_flag;
      const unsigned long long now = global_timer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) give_up = 1;
      if (__any_sync(0xffffffffu, give_up)) return false;
    }
  }
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity) ? 1 : 0)) return true;
  return mbar_wait_slow(bar, parity, abort_flag);
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}

// im2col load of a 4-D (C, W, H, N) tensor: `pixelsPerColumn` output pixels starting at base pixel
// (w, h, n), filter-tap offsets (off_w, off_h) added to every pixel, `channelsPerPixel` channels from c.
__device__ __forceinline__ void tma_load_im2col_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c, int w,
                                                   int h, int n, unsigned short off_w, unsigned short off_h) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"(off_w), "h"(off_h)
      : "memory");
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}

__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
               ::"l"(map), "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
               : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
               ::"l"(map), "r"(src), "r"(c0), "r"(c1)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

__device__ __forceinline__ void tcgen05_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tcgen05_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t holder_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(holder_smem), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t addr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}

// ---- CTA pairs (cta_group::2).  The leader (even rank) issues the MMAs; operands sit at the same shared-memory
// offsets in both CTAs; loads of either CTA signal the leader's barrier; commits arrive in both CTAs.
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_to_cta(uint32_t smem_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, uint32_t leader_bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(map), "r"(leader_bar), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
__device__ __forceinline__ void tma_load_4d_pair(uint32_t dst, const CUtensorMap* map, uint32_t leader_bar, int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(leader_bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t holder_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(holder_smem), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t addr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}
__device__ __forceinline__ void umma_i8_pair(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::i8 [%0], da, db, %4, p;\n\t}"
      ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate)
      : "memory");
}
// arrives on the barrier at this offset in both CTAs of the pair once the MMAs issued so far have completed
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"((unsigned short)3)
               : "memory");
}

// D[tmem] (+)= A[smem desc] * B[smem desc]^T, 8-bit integer inputs, int32 accumulate.  Both operands' descriptors
// share the constant high word; only low words (start address >> 4 | kDescLbo) are computed, with 32-bit additions.
__device__ __forceinline__ void umma_i8(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], da, db, %4, p;\n\t}"
      ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_i8_acc(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
      "setp.eq.u32 p, 0, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], da, db, %4, p;\n\t}"
      ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc)
      : "memory");
}

// The instructions of one K block of ksteps * 32 bytes (ksteps = 1, 2 or 4, uniform): +2 in 16-byte address units
// per step.
__device__ __forceinline__ void umma_i8_block(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc,
                                              uint32_t accumulate_first, int ksteps) {
  umma_i8(d_tmem, a_lo, b_lo, hi, idesc, accumulate_first);
  if (ksteps > 1) {
    umma_i8_acc(d_tmem, a_lo + 2, b_lo + 2, hi, idesc);
    if (ksteps > 2) {
      umma_i8_acc(d_tmem, a_lo + 4, b_lo + 4, hi, idesc);
      umma_i8_acc(d_tmem, a_lo + 6, b_lo + 6, hi, idesc);
    }
  }
}

// The mbarrier gets one arrival once every tcgen05.mma issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// 32 lanes x 16 consecutive 32-bit columns: thread i of the warp receives row (lane base + i).
__device__ __forceinline__ void tmem_ld_16(uint32_t taddr, int (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}
// Waits for this thread's TMEM loads.  The registers are named as operands so that no use of them
// can be scheduled ahead of the wait.
__device__ __forceinline__ void tmem_ld_wait(int (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]), "+r"(v[8]),
                 "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
               :
               : "memory");
}

// {lo byte, next byte} = {sat(b), sat(a)}, upper half = low half of c.
__device__ __forceinline__ unsigned int pack_sat_u8(int a, int b, unsigned int c) {
  unsigned int d;
  asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ unsigned int pack_sat_s8(int a, int b, unsigned int c) {
  unsigned int d;
  asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
// bytes (z0, z1, z2, z3), z0 lowest, each saturated to the 8-bit range
template <bool kSigned>
__device__ __forceinline__ unsigned int pack4_sat(int z0, int z1, int z2, int z3) {
  return kSigned ? pack_sat_s8(z1, z0, pack_sat_s8(z3, z2, 0u)) : pack_sat_u8(z1, z0, pack_sat_u8(z3, z2, 0u));
}

// Packed fp32 arithmetic: two independent IEEE operations (round to nearest even, no contraction) in one
// instruction slot.  The epilogue of a layer with a short reduction is bound by instruction issue.
__device__ __forceinline__ unsigned long long pack_f2(float a, float b) {
  unsigned long long d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ void unpack_f2(unsigned long long d, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(d));
}
__device__ __forceinline__ unsigned long long fmul2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long fsub2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// ------------------------------------------------------------------------------------------ epilogue
struct EpiTile {
  const int* s_bias;       // smem, k_pad entries
  const float* s_scale;    // smem, k_pad entries
  float scale;             // the first of them: the multiplier of every channel when there is one per tensor
  unsigned char* buf;      // 8-bit tile in shared memory (kTile)
  unsigned char* yrow;     // this thread's row of the 8-bit output, at the tile's first channel
  const unsigned char* rrow;  // ... of the residual
  bool wide, res_wide;     // pairs of chunks of those rows start on 32-byte lines
  int m;                   // output pixel (row of the [M][Cout] result, fewer than 2^31) of this thread
  long long y_off;         // element offset of this work item's output (split-K partial results), else 0
  int srow;                // row of this thread's pixel inside the 8-bit tile buffer
  uint32_t row_base, swz;  // byte offset of that row inside a panel, and the row's swizzle term (set by epi_row_setup)
  int n0;                  // first channel of the tile
  bool row_ok;             // the pixel exists (inside the image and below M)
  bool smem_ok;            // this accumulator row maps to a pixel of the tile (always, except halo tiles)
};

// 32 bytes of one row, a whole sector.
__device__ __forceinline__ void store_32(unsigned char* g, const uint4& a, const uint4& b) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"l"(g), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
               : "memory");
}
__device__ __forceinline__ void load_32(const unsigned char* g, uint4& a, uint4& b) {
  asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
               : "l"(g)
               : "memory");
}

// Residual bytes of the chunks ch and ch + 1 of this thread's row (zero where there are none).
struct ResPair { uint4 a, b; };
__device__ __forceinline__ void load_residual(const UmmaParams& p, const EpiTile& t, int ch, int nchunk, ResPair& r) {
  r.a = r.b = make_uint4(0u, 0u, 0u, 0u);
  const int nb = t.n0 + ch * 16;
  if (!t.row_ok || nb >= p.K) return;
  const unsigned char* g = t.rrow + ch * 16;
  const bool two = ch + 1 < nchunk && nb + 16 < p.K;
  if (t.res_wide && two) {
    load_32(g, r.a, r.b);
  } else {
    r.a = *reinterpret_cast<const uint4*>(g);
    if (two) r.b = *reinterpret_cast<const uint4*>(g + 16);
  }
}

// Position of a thread's row in the swizzled 8-bit tile buffers: constant for the thread's lifetime.  A panel is
// 128 rows of 2^pw_shift bytes; the 16-byte chunk index of a row is XORed with address bits 7.. (the swizzle the
// TMA and the tensor core use), which for rows of one swizzle span depend on the row alone.
__device__ __forceinline__ void epi_row_setup(const UmmaParams& p, EpiTile& t) {
  t.row_base = (uint32_t)t.srow << p.pw_shift;
  t.swz = ((t.row_base >> 7) & (uint32_t)p.pmask) << 4;
}

// One 16-column chunk of one accumulator row.  kOut: Q8_U8, Q8_S8, Q8_S32 or Q8_F32.  kRes: kResNone, kResVec
// (a residual in `rv` if p.res_mode says so, else none: decided at run time), kResGlobal (fp32 outputs), kResRows
// (8-bit rows that 16-byte accesses cannot address: the warps move them through a tile buffer) or kResTma (TMA moves them
// through one).  Fewer
// distinct kernels matter more than one uniform branch per chunk: a launch of another kernel function than
// the one before it starts with cold instruction caches, which costs a layer of a network 2 to 6 us, so the
// layers with and without a residual sum share their kernels.  (One straight-line copy of the rows' code per case runs 30 %
// fewer instructions, but 3 % of ResNet-50 slower: 700 -> 730 us, 56x56 bottleneck 30.8 -> 33.9 us.)
//   v = float(acc + bias) * s;  v += float(res) * s_res;  v = max(v, 0);  y = clamp(Round(v))
// Each step is one IEEE fp32 operation (the library is built without FMA contraction).
// kUniform: one multiplier for all channels (scale_count 1, `us`), else one per channel from shared memory.  A broadcast
// load of four words takes the shared-memory port four passes like any other 512-byte load, and the loads of bias and
// multiplier are what the epilogue waits for most.
// Returns the sixteen bytes of an 8-bit output; wider outputs are stored here.
template <int kOut, int kRes, bool kUniform>
__device__ __forceinline__ uint4 epilogue_chunk(const UmmaParams& p, const EpiTile& t, int ch, const int (&raw)[16], const float us,
                                                const uint4 rv) {
  const int c16 = ch * 16;
  const int nb = t.n0 + c16;
  uint4 o = make_uint4(0u, 0u, 0u, 0u);
  int acc[16];
  {
    const int4* bp = reinterpret_cast<const int4*>(t.s_bias + nb);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int4 b = bp[j];
      acc[4 * j] = raw[4 * j] + b.x; acc[4 * j + 1] = raw[4 * j + 1] + b.y;
      acc[4 * j + 2] = raw[4 * j + 2] + b.z; acc[4 * j + 3] = raw[4 * j + 3] + b.w;
    }
  }
  if (kOut == Q8_S32) {
    if (t.row_ok && nb < p.K) {
      const int valid = min(16, p.K - nb);
      int* yp = static_cast<int*>(p.y) + t.y_off + (size_t)t.m * p.ldc + p.c_off + nb;
      if (p.y_vec && valid == 16) {
#pragma unroll
        for (int j = 0; j < 4; ++j) reinterpret_cast<int4*>(yp)[j] = make_int4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (j < valid) yp[j] = acc[j];
      }
    }
    return o;
  }
  unsigned long long v2[8];  // v[2i], v[2i + 1]
  float v[16];
  {
    const float4* sp = reinterpret_cast<const float4*>(t.s_scale + nb);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 s = kUniform ? make_float4(us, us, us, us) : sp[j];
      v2[2 * j] = fmul2(pack_f2(__int2float_rn(acc[4 * j]), __int2float_rn(acc[4 * j + 1])), pack_f2(s.x, s.y));
      v2[2 * j + 1] = fmul2(pack_f2(__int2float_rn(acc[4 * j + 2]), __int2float_rn(acc[4 * j + 3])), pack_f2(s.z, s.w));
    }
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) unpack_f2(v2[j], v[2 * j], v[2 * j + 1]);
  if (kRes == kResGlobal || ((kRes == kResVec || kRes == kResRows || kRes == kResTma) && p.res_mode != kResNone)) {
    unsigned int rw[4] = {rv.x, rv.y, rv.z, rv.w};
    if (kRes == kResGlobal && t.row_ok && nb < p.K) {
      const int valid = min(16, p.K - nb);
      const unsigned char* rp = p.res + (size_t)t.m * p.K + nb;
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (j < valid) rw[j >> 2] |= (unsigned int)rp[j] << (8 * (j & 3));
    }
    // byte b -> float without a conversion instruction: 0x4B0000bb is 2^23 + b exactly; a signed
    // byte is first biased by 128
    const unsigned int sign_mask = p.res_signed ? 0x80808080u : 0u;
    const float magic = p.res_signed ? 8388736.0f : 8388608.0f;
    const unsigned long long magic2 = pack_f2(magic, magic), rs2 = pack_f2(p.res_scale, p.res_scale);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const unsigned int w = rw[j >> 1] ^ sign_mask;
      const float r0 = __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7540u | (unsigned)((2 * j) & 3)));
      const float r1 = __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7540u | (unsigned)((2 * j + 1) & 3)));
      // the sum stays scalar: with a packed multiply followed by a packed add a bit-exact test saw one rounding instead of
      // two, as of a fused operation, which would break the two-rounding definition
      float t0, t1;
      unpack_f2(fmul2(fsub2(pack_f2(r0, r1), magic2), rs2), t0, t1);
      v[2 * j] = __fadd_rn(v[2 * j], t0);
      v[2 * j + 1] = __fadd_rn(v[2 * j + 1], t1);
    }
  }
  if (kOut == Q8_F32) {
    if (p.relu) {
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = fmaxf(v[j], 0.0f);
    }
    if (t.row_ok && nb < p.K) {
      const int valid = min(16, p.K - nb);
      float* yp = static_cast<float*>(p.y) + (size_t)t.m * p.ldc + p.c_off + nb;
      if (p.y_vec && valid == 16) {
#pragma unroll
        for (int j = 0; j < 4; ++j) reinterpret_cast<float4*>(yp)[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (j < valid) yp[j] = v[j];
      }
    }
    return o;
  }
  // 8-bit output: the saturating pack clamps to [0,255] (which also is the ReLU) or [-128,127]
  if (kOut == Q8_S8 && p.relu) {
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = fmaxf(v[j], 0.0f);
  }
  int z[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) z[j] = __float2int_rn(v[j]);
  o.x = pack4_sat<kOut == Q8_S8>(z[0], z[1], z[2], z[3]);
  o.y = pack4_sat<kOut == Q8_S8>(z[4], z[5], z[6], z[7]);
  o.z = pack4_sat<kOut == Q8_S8>(z[8], z[9], z[10], z[11]);
  o.w = pack4_sat<kOut == Q8_S8>(z[12], z[13], z[14], z[15]);
  return o;
}

// Byte offset of a 16-byte chunk of this thread's row inside a swizzled 8-bit tile in shared memory.
__device__ __forceinline__ uint32_t tile_offset(const UmmaParams& p, const EpiTile& t, int ch) {
  const int c16 = ch * 16;
  return t.row_base + (((uint32_t)(c16 & ((1 << p.pw_shift) - 1))) ^ t.swz) + (uint32_t)(c16 >> p.pw_shift) * ((uint32_t)kBM << p.pw_shift);
}

// All chunks of one accumulator row, TMEM loads one chunk ahead of the arithmetic, residual bytes one pair of chunks ahead
// (`r` holds the first pair on entry).  The accumulator is released (acc_empty) as soon as its last chunk is in registers.
// 8-bit results go straight to global memory, 32 bytes a lane, or with kTile into the shared-memory tile t.buf.
template <int kOut, int kRes, bool kPair, bool kUniform, bool kTile>
__device__ __forceinline__ void epilogue_row(const UmmaParams& p, const EpiTile& t, uint32_t taddr, uint32_t acc_empty_bar,
                                             int lane, const int ch0, const int nchunk, ResPair r) {
  // chunks ch0 .. nchunk-1 of 16 columns each
  constexpr bool k8 = kOut == Q8_U8 || kOut == Q8_S8;
  int ra[16], rb[16];
  // passed through a warp-wide reduction, which tells the compiler that the value is the same in all lanes (1x1 64->256
  // at 56x56, batch 64: 18.6 us with the loads, 18.2 us without the reduction, 17.2 us with it; 3x3 + 1x1 pair 32.0 /
  // 30.9 / 30.3 us)
  const float us = kUniform ? __uint_as_float(__reduce_or_sync(0xffffffffu, __float_as_uint(t.scale))) : 0.0f;
  auto release = [&] {  // every accumulator value of this warp is in registers: hand the TMEM buffer back
    tcgen05_fence_before();
    __syncwarp();
    if (lane == 0) { if constexpr (kPair) mbar_arrive_cluster(acc_empty_bar); else mbar_arrive(acc_empty_bar); }
  };
  if (ch0 >= nchunk) {  // no columns for this warp in this tile: it still hands the accumulator back
    release();
    return;
  }
  auto given = [&](int ch, const uint4& v) {  // residual bytes of a row moved through the tile buffer
    // (a buffer that TMA fills holds the residual or nothing: its bytes are read ahead of the uniform branch on which)
    if (kRes == kResTma || (kRes == kResRows && p.res_mode != kResNone)) return *reinterpret_cast<const uint4*>(t.buf + tile_offset(p, t, ch));
    return v;
  };
  tmem_ld_16(taddr + ch0 * 16, ra);
#pragma unroll 1
  for (int ch = ch0; ch < nchunk; ch += 2) {
    tmem_ld_wait(ra);
    const bool more1 = ch + 1 < nchunk, more2 = ch + 2 < nchunk;
    if (more1) tmem_ld_16(taddr + (ch + 1) * 16, rb);
    else release();
    ResPair next;
    if (kRes == kResVec && p.res_mode != kResNone && more2) load_residual(p, t, ch + 2, nchunk, next);
    const uint4 o0 = epilogue_chunk<kOut, kRes, kUniform>(p, t, ch, ra, us, given(ch, r.a));
    if (kTile && t.smem_ok) *reinterpret_cast<uint4*>(t.buf + tile_offset(p, t, ch)) = o0;
    uint4 o1 = make_uint4(0u, 0u, 0u, 0u);
    if (more1) {
      tmem_ld_wait(rb);
      if (more2) tmem_ld_16(taddr + (ch + 2) * 16, ra);
      else release();
      o1 = epilogue_chunk<kOut, kRes, kUniform>(p, t, ch + 1, rb, us, given(ch + 1, r.b));
      if (kTile && t.smem_ok) *reinterpret_cast<uint4*>(t.buf + tile_offset(p, t, ch + 1)) = o1;
    }
    if (k8 && !kTile && t.row_ok) {
      const int nb = t.n0 + ch * 16;
      unsigned char* g = t.yrow + ch * 16;
      if (t.wide && more1 && nb + 16 < p.K) {
        store_32(g, o0, o1);
      } else {
        if (nb < p.K) *reinterpret_cast<uint4*>(g) = o0;
        if (more1 && nb + 16 < p.K) *reinterpret_cast<uint4*>(g + 16) = o1;
      }
    }
    if (kRes == kResVec) r = next;
  }
}
// 8-bit tensors whose rows 16-byte accesses cannot address (channel counts, pitches, offsets or pointers off that grid): a warp
// moves the rows of its 32 accumulator rows between global memory and the group's tile buffer itself.  Neighbouring lanes
// take neighbouring words of a row, `lpr` lanes a row (a power of two that covers it, so that narrow rows share a pass);
// the global words are aligned ones, the buffer's follow from two of them by a funnel shift.  Only words that hold a byte
// of the row are touched, and on the way out bytes outside it are never written.  Columns c0 .. c0 + nb - 1 of the tile.
// (Against gathered operands: 3x3 128 -> 100 at 28x28, batch 32 46.0 -> 9.4 us; 1x1 64 -> 250 at 56x56, batch 16 118 ->
// 17.9 us, as long as 256 channels take, with a residual sum 138 -> 28.6 us; partial words inside the loop over rows,
// a residual fetched after the accumulator: 32.6 and 51.9 us.)
struct RowMove {
  int c0, nb, lpr_shift;
  __device__ __forceinline__ void init(const UmmaParams& p, int n0, int ch0, int ch1) {
    c0 = ch0 * 16;
    nb = min(ch1 * 16, p.K - n0) - c0;
    const int words = (nb + 3) >> 2;
    lpr_shift = words > 16 ? 5 : (words > 8 ? 4 : (words > 4 ? 3 : (words > 2 ? 2 : (words > 1 ? 1 : 0))));
  }
};

__device__ __forceinline__ uint32_t row_buf_offset(const UmmaParams& p, int srow, int col) {
  const uint32_t rb = (uint32_t)srow << p.pw_shift;
  return rb + (((uint32_t)(col & ((1 << p.pw_shift) - 1))) ^ (((rb >> 7) & (uint32_t)p.pmask) << 4)) +
         (uint32_t)(col >> p.pw_shift) * ((uint32_t)kBM << p.pw_shift);
}

// Residual rows into the buffer, four passes of loads in flight.  All lanes of the warp call it.
__device__ __forceinline__ void rows_in(const UmmaParams& p, const EpiTile& t, const RowMove& mv, int lane) {
  constexpr int U = 4;
  const int lpr = 1 << mv.lpr_shift, sub = lane & (lpr - 1), per_pass = 32 >> mv.lpr_shift;
  const unsigned char* mine = p.res + (long long)t.m * p.K + t.n0 + mv.c0;
#pragma unroll 1
  for (int r0 = 0; r0 < 32; r0 += U * per_pass) {
    uintptr_t at[U];
    int srow[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int r = r0 + u * per_pass + (lane >> mv.lpr_shift);
      at[u] = (uintptr_t)__shfl_sync(0xffffffffu, (unsigned long long)mine, r & 31);
      srow[u] = __shfl_sync(0xffffffffu, t.row_ok ? t.srow : -1, r & 31);
      if (r >= 32) srow[u] = -1;
    }
#pragma unroll 1
    for (int k = sub; 4 * k < mv.nb; k += lpr) {
      unsigned int lo[U], hi[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int head = (int)(at[u] & 3u);
        const unsigned int* g = reinterpret_cast<const unsigned int*>(at[u] - head) + k;
        lo[u] = hi[u] = 0u;
        if (srow[u] >= 0) lo[u] = g[0];
        if (srow[u] >= 0 && 4 * (k + 1) - head < mv.nb) hi[u] = g[1];
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (srow[u] >= 0)
          *reinterpret_cast<unsigned int*>(t.buf + row_buf_offset(p, srow[u], mv.c0 + 4 * k)) = __funnelshift_r(lo[u], hi[u], 8 * (int)(at[u] & 3u));
    }
  }
}

// Output rows out of the buffer: the whole words of each row by its group of lanes, the up to three bytes before and after
// them by the lane whose row it is (partial words in the loop over rows doubled its length).  All lanes call it.
__device__ __forceinline__ void rows_out(const UmmaParams& p, const EpiTile& t, const RowMove& mv, int lane) {
  const int lpr = 1 << mv.lpr_shift, sub = lane & (lpr - 1);
  unsigned char* mine = static_cast<unsigned char*>(p.y) + (long long)t.m * p.ldc + p.c_off + t.n0 + mv.c0;
  for (int r0 = 0; r0 < 32; r0 += 32 >> mv.lpr_shift) {
    const int r = r0 + (lane >> mv.lpr_shift);
    unsigned char* g = reinterpret_cast<unsigned char*>(__shfl_sync(0xffffffffu, (unsigned long long)mine, r));
    const int srow = __shfl_sync(0xffffffffu, t.row_ok ? t.srow : -1, r);
    const int head = (int)(0u - (unsigned)(uintptr_t)g) & 3;   // bytes before the first whole word
    const int end = srow < 0 ? 0 : mv.nb - 3;
    for (int b = head + 4 * sub; b < end; b += 4 * lpr) {
      // bytes b .. b + 3 of the row, from the buffer words that hold byte b and byte b + 3
      const unsigned int lo = *reinterpret_cast<const unsigned int*>(t.buf + row_buf_offset(p, srow, mv.c0 + (b & ~3)));
      const unsigned int hi = *reinterpret_cast<const unsigned int*>(t.buf + row_buf_offset(p, srow, mv.c0 + ((b + 3) & ~3)));
      *reinterpret_cast<unsigned int*>(g + b) = __funnelshift_r(lo, hi, 8 * head);
    }
  }
  if (!t.row_ok || mv.nb <= 0) return;
  const int head = min((int)(0u - (unsigned)(uintptr_t)mine) & 3, mv.nb), tail = head + ((mv.nb - head) & ~3);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    if (j < head) mine[j] = t.buf[row_buf_offset(p, t.srow, mv.c0 + j)];
    if (tail + j < mv.nb) mine[tail + j] = t.buf[row_buf_offset(p, t.srow, mv.c0 + tail + j)];
  }
}

// ------------------------------------------------------------------------------------------ MMA role
struct MmaRoleArgs {
  uint32_t base, tmem_base;
  uint32_t a_full, a_empty, b_full, b_empty, acc_full, acc_empty, bres_full, turn;
  int first_tile, tile_step, total_tiles;  // this CTA's work items: first_tile, first_tile + tile_step, ... below total_tiles
  volatile int* abortp;
};

// One MMA-issuing warp (an elected lane issues).  Returns false if a wait gave up.
__device__ __forceinline__ bool mma_role(const UmmaParams& p, const MmaRoleArgs& r, const int who) {
  // This lane's tiles are lt = who, who + kMmaWarps, ... of the CTA's sequence; the stage, weight-ring
  // and accumulator positions of a tile follow from lt alone.  A parity wait is only meaningful for
  // the use of a barrier that is in flight, so a lane starts the stage waits of tile lt only after
  // the lane of tile lt - 1 has passed all of its own (the turn barriers); the per-tile bookkeeping
  // and the accumulator wait run ahead of that.
  TileIterT<false> ti;
  const int L = p.mma_lanes;
  ti.init(p, r.first_tile + who * r.tile_step, L * r.tile_step);
  const uint32_t nstages = (uint32_t)p.stages, nbst = (uint32_t)p.b_stages;
  const uint32_t hi = p.desc_hi;
  const uint32_t a_d0 = kDescLbo | (((r.base + p.off_a) >> 4) & 0x3fffu), bring_d0 = kDescLbo | (((r.base + p.off_bring) >> 4) & 0x3fffu);
  const uint32_t bres_d0 = kDescLbo | ((r.base >> 4) & 0x3fffu);
  const uint32_t stage16 = p.a_stage_bytes >> 4, asub16 = p.a_sub_bytes >> 4, bsub16 = p.b_sub_bytes >> 4, btile16 = p.b_tile_bytes >> 4;
  const uint32_t idesc = p.idesc;
  const int taps = p.taps, c_blocks = p.c_blocks, k_iters = p.kps, kb = p.kb;  // k iterations of one work item
  const bool halo = p.a_mode == kAHalo, ring = p.b_mode == kBRing, b_in_stage = p.b_mode == kBStage;
  // ring positions of tile lt = who, and how far the other lanes' tiles move them between two of ours
  const uint32_t spt = halo ? (uint32_t)c_blocks : (uint32_t)((k_iters + kb - 1) / kb);  // A stages per tile
  const int bT = p.b_T;
  const uint32_t bpt = (uint32_t)(p.b_chunks * c_blocks);                                 // ring stages per tile
  const uint32_t skip_a = (uint32_t)(L - 1) * spt, skip_b = (uint32_t)(L - 1) * bpt;
  uint32_t stage = ((uint32_t)who * spt) % nstages, phase = (((uint32_t)who * spt) / nstages) & 1u;
  uint32_t bs = 0, bphase = 0;
  if (ring) { bs = ((uint32_t)who * bpt) % nbst; bphase = (((uint32_t)who * bpt) / nbst) & 1u; }
  uint32_t a_d = a_d0 + stage * stage16;
  uint32_t bring_d = bring_d0 + bs * bsub16;
  const uint32_t nacc = (uint32_t)p.nacc;
  uint32_t ab = (uint32_t)who % nacc, acc_par = 1u ^ (((uint32_t)who / nacc) & 1u);  // accumulator and the parity of its empty barrier
  uint32_t my_k = 0;  // number of tiles this lane has issued
  const uint32_t turn_next = r.turn + (uint32_t)((who + 1) % L) * 8u;  // the next lane's turn barrier
  const uint32_t turn_mine = r.turn + (uint32_t)who * 8u;
  if (p.b_mode == kBResident && !mbar_wait(r.bres_full, 0u, r.abortp)) return false;
  const uint32_t in16 = p.in16, out16 = p.out16;
  const int inner = p.tap_inner, ksteps = p.ksteps;
  for (; ti.tile < r.total_tiles; ti.next(p)) {
    if (!mbar_wait(r.acc_empty + ab * 8u, acc_par, r.abortp)) return false;
    // turn[w] counts the tiles the other lane has finished waiting for: tile number k of lane 0 needs
    // k of them, tile number k of lane 1 needs k + 1
    if (who == 0) { if (my_k > 0 && !mbar_wait(turn_mine, (my_k - 1) & 1u, r.abortp)) return false; }
    else if (!mbar_wait(turn_mine, my_k & 1u, r.abortp)) return false;
    tcgen05_fence_after();
    const uint32_t d_tmem = r.tmem_base + ab * (uint32_t)p.acc_stride;
    uint32_t accum = 0;
    // resident weights: tile (nt, cb, tap) sits at ((nt * c_blocks + cb) * taps + tap) * b_tile_bytes
    const uint32_t bres_nt = bres_d0 + (uint32_t)(ti.nt * c_blocks * taps) * btile16;
    if (halo) {
      uint32_t bres = bres_nt;  // (cb, tap) is exactly the order of the loops below
      for (int cb = 0; cb < c_blocks; ++cb) {
        if (!mbar_wait(r.a_full + stage * 8u, phase, r.abortp)) return false;
        const bool last_cb = cb == c_blocks - 1;
        if (last_cb && !ring && elect_one()) mbar_arrive(turn_next);  // this tile's last wait is behind us
        tcgen05_fence_after();
        uint32_t a_row = a_d, a_tap = a_d;  // descriptor of the filter row's first tap, of this tap
        int left = inner;
        if (ring) {
          for (int tap0 = 0; tap0 < taps; tap0 += bT) {
            if (!mbar_wait(r.b_full + bs * 8u, bphase, r.abortp)) return false;
            tcgen05_fence_after();
            const int nt = min(bT, taps - tap0);
            if (last_cb && tap0 + bT >= taps && elect_one()) mbar_arrive(turn_next);
            uint32_t bd = bring_d;
            for (int t = 0; t < nt; ++t, bd += btile16) {
              if (elect_one()) umma_i8_block(d_tmem, a_tap, bd, hi, idesc, accum, ksteps);
              accum = 1;
              a_tap += in16;
              if (--left == 0) { left = inner; a_row += out16; a_tap = a_row; }
            }
            if (elect_one()) umma_commit(r.b_empty + bs * 8u);
            bring_d += bsub16;
            if (++bs == nbst) { bs = 0; bphase ^= 1u; bring_d = bring_d0; }
          }
        } else {
          if (elect_one()) {
            uint32_t bt = bres;
            for (int t0 = 0; t0 < taps; t0 += inner, a_row += out16) {
              uint32_t at = a_row;
              if (ksteps == 1) {  // (the run-time step count costs the one-instruction block a tenth of its rate)
                for (int t = 0; t < inner; ++t, at += in16, bt += btile16) {
                  umma_i8(d_tmem, at, bt, hi, idesc, accum);
                  accum = 1;
                }
              } else {
                for (int t = 0; t < inner; ++t, at += in16, bt += btile16) {
                  umma_i8_block(d_tmem, at, bt, hi, idesc, accum, ksteps);
                  accum = 1;
                }
              }
            }
          }
          accum = 1;
          bres += (uint32_t)taps * btile16;
        }
        if (elect_one()) umma_commit(r.a_empty + stage * 8u);
        a_d += stage16;
        if (++stage == nstages) { stage = 0; phase ^= 1u; a_d = a_d0; }
      }
    } else {
      uint32_t bres_tap = bres_nt, bres = bres_nt;  // iterations run over taps with the channel blocks innermost
      int cb = 0;
      if (p.splits > 1) {
        const int it0 = ti.sp * k_iters, tap0 = p.fd_cblocks.div(it0);
        cb = it0 - tap0 * c_blocks;
        bres_tap += (uint32_t)tap0 * btile16;
        bres = bres_tap + (uint32_t)(cb * taps) * btile16;
      }
      const uint32_t b_off16 = (uint32_t)kb * asub16;
      for (int it = 0; it < k_iters;) {
        const int nsub = min(kb, k_iters - it);
        if (!mbar_wait(r.a_full + stage * 8u, phase, r.abortp)) return false;
        if (it + nsub >= k_iters && elect_one()) mbar_arrive(turn_next);  // this tile's last wait is behind us
        tcgen05_fence_after();
        uint32_t sa = a_d, sb = a_d + b_off16;
        if (b_in_stage) {
          if (elect_one())
            for (int j = 0; j < nsub; ++j, sa += asub16, sb += bsub16) {
              umma_i8_block(d_tmem, sa, sb, hi, idesc, accum, ksteps);
              accum = 1;
            }
        } else {
          for (int j = 0; j < nsub; ++j, sa += asub16) {
            if (elect_one()) umma_i8_block(d_tmem, sa, bres, hi, idesc, accum, ksteps);
            accum = 1;
            bres += (uint32_t)taps * btile16;
            if (++cb == c_blocks) { cb = 0; bres_tap += btile16; bres = bres_tap; }
          }
        }
        accum = 1;
        if (elect_one()) umma_commit(r.a_empty + stage * 8u);
        it += nsub;
        a_d += stage16;
        if (++stage == nstages) { stage = 0; phase ^= 1u; a_d = a_d0; }
      }
    }
    ++my_k;
    if (elect_one()) umma_commit(r.acc_full + ab * 8u);
    ab += (uint32_t)L;
    while (ab >= nacc) { ab -= nacc; acc_par ^= 1u; }
    // step over the stages and ring tiles of the other lanes' tiles
    stage += skip_a;
    while (stage >= nstages) { stage -= nstages; phase ^= 1u; }
    a_d = a_d0 + stage * stage16;
    if (ring) {
      bs += skip_b;
      while (bs >= nbst) { bs -= nbst; bphase ^= 1u; }
      bring_d = bring_d0 + bs * bsub16;
    }
  }
  return true;
}

// ------------------------------------------------------------------------------------------ host
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
typedef CUresult (*EncodeIm2colFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const int*, const int*, cuuint32_t, cuuint32_t, const cuuint32_t*,
                                   CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                   CUtensorMapFloatOOBfill);

struct DriverFns {
  EncodeTiledFn tiled = nullptr;
  EncodeIm2colFn im2col = nullptr;
};

// Looked up once per process; the function-local static is initialised by exactly one thread, and the others
// wait for it (C++11), so no caller can see half-filled pointers.
const DriverFns& driver_fns() {
  static const DriverFns f = [] {
    DriverFns r;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qr) == cudaSuccess && qr == cudaDriverEntryPointSuccess)
      r.tiled = reinterpret_cast<EncodeTiledFn>(p);
    p = nullptr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeIm2col", &p, cudaEnableDefault, &qr) == cudaSuccess && qr == cudaDriverEntryPointSuccess)
      r.im2col = reinterpret_cast<EncodeIm2colFn>(p);
    return r;
  }();
  return f;
}


int pick_bk(int C) {
  // A pipeline iteration costs one TMA operation per operand (several hundred cycles whatever its size), so the
  // widest channel block that C reaches wins even when it pads C: out-of-range channels are zero filled by TMA
  // and cost tensor-core time only, which a short reduction has to spare.
  return C <= 32 ? 32 : (C <= 64 ? 64 : 128);
}

// Tile width: the multiple of 16 (power-of-two panels keep the 8-bit tile layout simple) that pads
// Cout least; short reductions are bandwidth bound and take narrower tiles, which leaves room for
// four TMEM accumulators.
int pick_bn(int K, int kgemm) {
  const int cap = kgemm <= 640 ? 128 : 256;
  const double k_steps = (kgemm + 31) / 32, k_iters = (kgemm + 127) / 128;
  int best = 16;
  double best_cost = -1.0;
  for (int w = 16; w <= cap; w += 16) {
    const int n_tiles = (K + w - 1) / w;
    // cycles per 128-row block of the output: every tile of columns runs the whole reduction again (one
    // 128 x w x 32 MMA takes max(59, 0.53 w) cycles, a pipeline iteration about 550), the epilogue pays for
    // every padded column.  Against all widths on 26 layers of the three networks' shapes the choice is the fastest
    // or within 3 %, but for 512->2048 at 7x7, batch 64 (128 columns 9.1 us, 256 7.8 us).
    const double mma = k_steps * (0.53 * w > 59.0 ? 0.53 * w : 59.0), feed = k_iters * 550.0;
    const double cost = n_tiles * ((mma > feed ? mma : feed) + 200.0) + (double)n_tiles * w * 8.0;
    if (best_cost < 0 || cost <= best_cost) { best = w; best_cost = cost; }
  }
  return best;
}

CUtensorMapSwizzle swizzle_for_bytes(int row_bytes) {
  return row_bytes >= 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                          : (row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                             : (row_bytes == 32 ? CU_TENSOR_MAP_SWIZZLE_32B : CU_TENSOR_MAP_SWIZZLE_NONE));
}

unsigned int round_up(unsigned int v, unsigned int a) { return (v + a - 1) / a * a; }

FastDiv make_fastdiv(int d) {
  FastDiv f;
  f.d = d < 1 ? 1 : d;
  unsigned int l = 0;
  while ((1ull << l) < (unsigned long long)f.d) ++l;
  f.l = l;
  f.m = (unsigned int)(((1ull << 32) * ((1ull << l) - (unsigned long long)f.d)) / (unsigned long long)f.d + 1ull);
  return f;
}

// Developer knobs for sweeps of tile shapes and pipeline depths.  They exist only in builds made with
// -DQ8_TUNE_KNOBS (the library proper never reads the environment) and are honoured only when Q8_TUNE is set.
// Every knob is confined to the range [lo, hi] that the plan supports at that point (the default always lies
// inside it); a value outside the range, or not a number, is ignored, so a typo cannot produce a launch whose
// shared-memory or TMEM plan does not hold.
//   Q8_PDL 0/1 dependent launch, Q8_HALO 0/1 halo tiles, Q8_BN tile width (multiple of 16), Q8_LANES 2/3 MMA warps,
//   Q8_SPLIT 0/1 column-split epilogue (only where the plan allows it), Q8_G 2/4 epilogue groups, Q8_BRES 0 weights
//   not resident, Q8_CTA2 0 no CTA pairs, Q8_CTA2MIN pair-mode threshold, Q8_BT taps per weight-ring
//   stage, Q8_KB channel blocks per A stage, Q8_BSTAGES / Q8_STAGES ring depths (at
//   most what fits), Q8_GRID number of CTAs (at most the default).
int tune_env(const char* name, int dflt, int lo, int hi) {
#ifdef Q8_TUNE_KNOBS
  static const bool enabled = getenv("Q8_TUNE") != nullptr;
  if (!enabled) return dflt;
  const char* v = getenv(name);
  if (!v || !*v) return dflt;
  char* end = nullptr;
  const long x = strtol(v, &end, 10);
  if (end == v || *end != '\0' || x < lo || x > hi) return dflt;
  return (int)x;
#else
  (void)name; (void)lo; (void)hi;
  return dflt;
#endif
}

// Halo tiling of a stride-1 filter: TH x TW output pixels per tile, (TH + ext_h) x (TW + ext_w)
// input pixels per patch, TH * (TW + ext_w) <= 128 accumulator rows.  Picks the extents that waste
// the fewest accumulator rows, preferring less halo among near-equals.
struct HaloTile {
  int tw, th, twb, hb;
  double eff;  // useful output pixels per computed accumulator row
  int sw;      // stride along W: 1, or 2 = the input is read as pixel pairs [N, H, W/2, 2C]
  int s_eff;   // filter taps along W in that view
  int pad_w_eff, e;  // left padding in that view; parity of pad_w
};

// Stride 2 along W needs no data movement: with W even, NHWC memory is also a tensor of pixel pairs with 2C
// channels, and output column q reads pairs q + t' - pad', t' = 0 .. S'-1, i.e. a stride-1 filter of
// S' = ceil((S + e) / 2) taps (e = pad_w & 1).  Stride along H is served by tiles of one output row.
bool search_halo_tile(const q8_conv_desc& d, int P, int Q, HaloTile* out) {
  const int sw = d.stride_w;
  if (sw != 1 && sw != 2) return false;
  int s_eff = d.S, pad_eff = d.pad_w, e = 0, dil_w = d.dil_w;
  if (sw == 2) {
    if (d.W % 2 || d.dil_w != 1 || (d.C != 16 && d.C != 32 && d.C != 64)) return false;
    e = d.pad_w & 1;
    s_eff = (d.S + e + 1) / 2;
    pad_eff = (d.pad_w + e) / 2;
    dil_w = 1;
    // this view keeps the weights resident in shared memory
    const int BN = pick_bn(d.K, d.R * d.S * d.C);
    if ((long long)((d.K + BN - 1) / BN) * BN * d.R * s_eff * 2 * d.C > 80 * 1024) return false;
  }
  const int taps = d.R * s_eff;
  if (taps < 2 || taps > kMaxTaps) return false;
  const int ext_w = (s_eff - 1) * dil_w, ext_h = (d.R - 1) * d.dil_h;
  HaloTile best = {0, 0, 0, 0, 0.0, sw, s_eff, pad_eff, e};
  double best_score = 0.0;
  for (int tw = 1; tw <= Q && tw + ext_w <= kBM; ++tw) {
    const int twb = tw + ext_w;
    int th = d.stride_h == 1 ? kBM / twb : 1;
    if (th > P) th = P;
    if (th < 1) continue;
    const int hb = (th - 1) * d.stride_h + ext_h + 1;
    if (hb > 256 || twb > 256) continue;
    const long long tiles = (long long)((Q + tw - 1) / tw) * ((P + th - 1) / th);
    const double eff = (double)P * Q / ((double)tiles * kBM);
    const double halo = (double)hb * twb / ((double)th * tw);
    const double score = eff / (1.0 + 0.04 * halo);
    if (score > best_score) { best_score = score; best.tw = tw; best.th = th; best.twb = twb; best.hb = hb; best.eff = eff; }
  }
  // Tiny images waste accumulator rows (a 7x7 image fills 49 of 128 rows).  Where the im2col path is
  // open it is the better choice for them (it can split the reduction); tensors below its size limit
  // still take halo tiles rather than leave the tensor cores.
  const bool im2col_closed = (long long)d.N * d.H * d.W * d.C < 131072;
  if (!im2col_closed && best.eff < 0.5) return false;
  if (best.tw == 0) return false;
  *out = best;
  return true;
}

// A call asks for the tile of its descriptor three or four times, and the search costs up to 2 us on a wide image, which a
// small layer's launch does not hide: the last tiles found are kept per thread, by the descriptor's values, on which alone
// they depend (3x3 64->64 on a 4x120 image, batch 1: 6.7 -> 4.4 us of host time per call).
bool choose_halo_tile(const q8_conv_desc& d, int P, int Q, HaloTile* out) {
  struct Entry { q8_conv_desc d; HaloTile t; int state; };  // state 0: empty, 1: no tile, 2: tile
  static thread_local Entry cache[64];
  unsigned int h = 2166136261u;
  const int32_t key[] = {d.N, d.H, d.W, d.C, d.K, d.R, d.S, d.stride_h, d.stride_w, d.pad_h, d.pad_w, d.dil_h, d.dil_w};
  for (int32_t v : key) h = (h ^ (unsigned int)v) * 16777619u;
  Entry& e = cache[(h ^ (h >> 16)) & 63u];
  if (e.state == 0 || memcmp(&e.d, &d, sizeof(d)) != 0) {
    e.t = HaloTile{};
    e.state = search_halo_tile(d, P, Q, &e.t) ? 2 : 1;
    e.d = d;
  }
  if (e.state == 2) *out = e.t;
  return e.state == 2;
}

}  // namespace
}  // namespace q8

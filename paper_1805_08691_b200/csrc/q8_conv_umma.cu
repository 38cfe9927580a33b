// Quantized convolution as an implicit GEMM on the 5th-generation tensor cores (sm_100a).
//
//   D[M = N*P*Q pixels, Cout] (int32, in TMEM) = A[M, R*S*C] (u8/s8) x B[Cout, R*S*C]^T (s8)
//
// Persistent kernel: one CTA per SM walks over output tiles of 128 accumulator rows x BN channels.
// Every TMA operation occupies the SM's copy engine for at least ~370 cycles whatever its size, and a control
// warp spends some hundred cycles on a pipeline iteration, so the pipeline moves few, large pieces:
//
//   A operand, three sources
//     plain  : 1x1 / stride 1 / no padding.  The activation tensor is the [M][C] matrix itself; a
//              stage holds several consecutive 128 x BK channel blocks (2-D tiled loads).
//     halo   : filters of stride 1 along W, or 2 where the input can be read as pixel pairs.  A tile is TH x TW output pixels of one image.  One 4-D tiled load
//              brings the (TH + halo) x (TW + halo) input patch of a channel block, zero filled
//              outside the image (the exact code of 0.0 under a symmetric quantizer).  Every filter
//              tap (r, s) is then the same patch read from a start address shifted by
//              (r*dil_h * patch width + s*dil_w) pixels: accumulator row i = pp * patch width + qq
//              is output pixel (pp, qq); rows with qq >= TW are computed and dropped.  Each input
//              byte crosses the L2 port about 1.5 times instead of R*S times.
//     im2col : everything else (strided, tiny images): one im2col-mode load per tap and channel
//              block, several of them per stage.
//   B operand (KRSC weights), three sources
//     resident : the whole layer's weights sit in shared memory for the CTA's lifetime;
//     ring     : (halo) BN x BK tiles per tap and channel block through their own ring, several taps per
//                stage (one TMA operation) for tiles up to 128 columns and for CTA pairs;
//     stage    : (plain, im2col) one BN x BK tile next to each A block of a stage.
//
// Roles (whole converged warps, an elected lane issues):
//   warp 0     : TMA producer of A patches / blocks and of B tiles;
//   warps 1, 2 : tcgen05.mma.kind::i8 issue (128 x BN x 32 per instruction, int32 accumulators in a
//   (and 3)      ring of up to four TMEM buffers), alternate tiles each, so that the per-tile
//                bookkeeping of one warp overlaps the issue of the other; tcgen05.commit releases
//                stages and publishes accumulators.  Warp 1 also owns the TMEM allocation;
//   warps 4..  : G epilogue groups of four warps; group g owns every G-th tile of the CTA, or, in launches
//                with at most two tiles per CTA, a share of the columns of every tile.  A thread
//                owns one accumulator row: tcgen05.ld, + bias, requantise, + residual, ReLU, round,
//                clamp, straight to global memory; residual bytes come from there the same way, a pair of
//                16-column chunks ahead.
// Where the rows are most of a launch (see buffered()), another instantiation moves them by TMA: warp 4 hands tile buffers in
// shared memory to the epilogue groups, filled with the residual tile when there is one, the groups turn them into output
// tiles in place, warp 5 stores those and recycles the buffers; the groups are warps 6 and up.
// Without buffers there are two hand-offs less behind the last tile, whose store ended 0.8 us after its arithmetic with them and
// ends 0.2 us after it now (14x14 256->256 3x3, batch 64), and their shared memory holds operands: ResNet-50 batch 1 285 -> 252
// us, batch 64 722 -> 702 us, Inception-v3 batch 64 1226 -> 1164 us, 14x14 bottleneck batch 64 33.1 -> 30.6 us.  Measured and not
// kept: rows exchanged through shared memory so that two lanes share one (64 contiguous bytes an access): 14x14 bottleneck 33.3
// us, 56x56 41 us; four lanes a row by tcgen05.ld.16x128b and weight rows in permuted order: 32.3 and 44 us.
// The kernel is launched with programmatic stream serialization: its set-up overlaps the tail of the kernel
// before it, and every global access comes after griddepcontrol.wait.
// All hand-offs are mbarriers, there is no block-wide barrier after the prologue.  Every wait is
// bounded in wall-clock time; on expiry a bit of the library's status word is set and all roles drain
// instead of hanging.
#include "q8_umma_common.cuh"

namespace q8 {
namespace {

// The MMA lanes of the leader CTA of a pair (halo tiles, weight ring): the same schedule as mma_role, with
// tcgen05.mma.cta_group::2 over both CTAs' tiles and commits that arrive in both CTAs.
__device__ __forceinline__ bool mma_role_pair(const UmmaParams& p, const MmaRoleArgs& r, const int who, const int vblock,
                                              const int vgrid) {
  TileIterT<true> ti;
  const int L = p.mma_lanes;
  ti.init(p, vblock + who * vgrid, L * vgrid, 0);
  const uint32_t nstages = (uint32_t)p.stages, nbst = (uint32_t)p.b_stages;
  const uint32_t hi = p.desc_hi;
  const uint32_t a_d0 = kDescLbo | (((r.base + p.off_a) >> 4) & 0x3fffu), bring_d0 = kDescLbo | (((r.base + p.off_bring) >> 4) & 0x3fffu);
  const uint32_t stage16 = p.a_stage_bytes >> 4, bsub16 = p.b_sub_bytes >> 4, btile16 = p.b_tile_bytes >> 4;
  const uint32_t idesc = p.idesc;
  const int taps = p.taps, c_blocks = p.c_blocks, bT = p.b_T, inner = p.tap_inner;
  const bool four = p.ksteps == 4;  // K blocks of 128 bytes, else 64 (the plan pairs no narrower ones)
  const uint32_t in16 = p.in16, out16 = p.out16;
  const uint32_t spt = (uint32_t)c_blocks, bpt = (uint32_t)(p.b_chunks * c_blocks);
  const uint32_t skip_a = (uint32_t)(L - 1) * spt, skip_b = (uint32_t)(L - 1) * bpt;
  uint32_t stage = ((uint32_t)who * spt) % nstages, phase = (((uint32_t)who * spt) / nstages) & 1u;
  uint32_t bs = ((uint32_t)who * bpt) % nbst, bphase = (((uint32_t)who * bpt) / nbst) & 1u;
  uint32_t a_d = a_d0 + stage * stage16, bring_d = bring_d0 + bs * bsub16;
  const uint32_t nacc = (uint32_t)p.nacc;
  uint32_t ab = (uint32_t)who % nacc, acc_par = 1u ^ (((uint32_t)who / nacc) & 1u);
  uint32_t my_k = 0;
  const uint32_t turn_next = r.turn + (uint32_t)((who + 1) % L) * 8u;
  const uint32_t turn_mine = r.turn + (uint32_t)who * 8u;
  for (; ti.tile < r.total_tiles; ti.next(p)) {
    if (!mbar_wait(r.acc_empty + ab * 8u, acc_par, r.abortp)) return false;
    if (who == 0) { if (my_k > 0 && !mbar_wait(turn_mine, (my_k - 1) & 1u, r.abortp)) return false; }
    else if (!mbar_wait(turn_mine, my_k & 1u, r.abortp)) return false;
    tcgen05_fence_after();
    const uint32_t d_tmem = r.tmem_base + ab * (uint32_t)p.acc_stride;
    uint32_t accum = 0;
    for (int cb = 0; cb < c_blocks; ++cb) {
      if (!mbar_wait(r.a_full + stage * 8u, phase, r.abortp)) return false;
      const bool last_cb = cb == c_blocks - 1;
      uint32_t a_row = a_d, a_tap = a_d;
      int left = inner;
      for (int tap0 = 0; tap0 < taps; tap0 += bT) {
        if (!mbar_wait(r.b_full + bs * 8u, bphase, r.abortp)) return false;
        tcgen05_fence_after();
        const int nt = min(bT, taps - tap0);
        if (last_cb && tap0 + bT >= taps && elect_one()) mbar_arrive(turn_next);
        uint32_t bd = bring_d;
        for (int t = 0; t < nt; ++t, bd += btile16) {
          if (elect_one()) {
            umma_i8_pair(d_tmem, a_tap, bd, hi, idesc, accum);
            umma_i8_pair(d_tmem, a_tap + 2, bd + 2, hi, idesc, 1u);
            if (four) {
              umma_i8_pair(d_tmem, a_tap + 4, bd + 4, hi, idesc, 1u);
              umma_i8_pair(d_tmem, a_tap + 6, bd + 6, hi, idesc, 1u);
            }
          }
          accum = 1;
          a_tap += in16;
          if (--left == 0) { left = inner; a_row += out16; a_tap = a_row; }
        }
        if (elect_one()) umma_commit_pair(r.b_empty + bs * 8u);
        bring_d += bsub16;
        if (++bs == nbst) { bs = 0; bphase ^= 1u; bring_d = bring_d0; }
      }
      if (elect_one()) umma_commit_pair(r.a_empty + stage * 8u);
      a_d += stage16;
      if (++stage == nstages) { stage = 0; phase ^= 1u; a_d = a_d0; }
    }
    ++my_k;
    if (elect_one()) umma_commit_pair(r.acc_full + ab * 8u);
    ab += (uint32_t)L;
    while (ab >= nacc) { ab -= nacc; acc_par ^= 1u; }
    stage += skip_a;
    while (stage >= nstages) { stage -= nstages; phase ^= 1u; }
    a_d = a_d0 + stage * stage16;
    bs += skip_b;
    while (bs >= nbst) { bs -= nbst; bphase ^= 1u; }
    bring_d = bring_d0 + bs * bsub16;
  }
  return true;
}

// ------------------------------------------------------------------------------------------ kernel
// G epilogue groups; one instantiation per output type and residual source keeps a single epilogue
// body in each kernel (several of them in one kernel made the register allocator spill).
// kCta2: the CTA-pair variant (its cta_group::2 instructions make the kernel launchable as clusters of two only).
// kRes = kResTma: 8-bit rows, a residual's in and the output's out, move by TMA through tile buffers in shared memory.
template <int kRes>
constexpr int kCtrlOf = kRes == kResTma ? kCtrlWarps + 2 : kCtrlWarps;  // control warps
template <bool kBufs>
struct RowMaps {};           // tensor maps of the residual's and the output's tiles
template <>
struct RowMaps<true> { CUtensorMap res, y; };
constexpr int kFillWarp = kCtrlWarps, kStoreWarp = kCtrlWarps + 1;
template <bool kBufs>
__device__ __forceinline__ void prefetch_maps(const RowMaps<kBufs>& maps, bool residual, bool out8) {
  if constexpr (kBufs) {
    if (residual) prefetch_tensormap(&maps.res);
    if (out8) prefetch_tensormap(&maps.y);
  }
}

template <int G, int kOut, int kRes, bool kCta2, bool kUniform>
__global__ void __launch_bounds__(kCtrlOf<kRes> * 32 + G * kGroupThreads, 1)
    conv_umma_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                     const __grid_constant__ UmmaParams p, const __grid_constant__ RowMaps<kRes == kResTma> maps) {
  constexpr bool kBufs = kRes == kResTma, k8 = kOut == Q8_U8 || kOut == Q8_S8;
  constexpr int kCtrl = kCtrlOf<kRes>, kCtrlT = kCtrl * 32;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long a_full[kMaxStages], a_empty[kMaxStages];
  __shared__ __align__(8) unsigned long long b_full[kMaxBStages], b_empty[kMaxBStages];
  __shared__ __align__(8) unsigned long long acc_full[kMaxAcc], acc_empty[kMaxAcc];
  // per buffer: residual arrived (or none to come), output tile read by its store, output tile written
  __shared__ __align__(8) unsigned long long buf_full[kBufs ? kMaxSlots : 1], buf_empty[kBufs ? kMaxSlots : 1], store_ready[kBufs ? kMaxSlots : 1];
  __shared__ __align__(8) unsigned long long bres_full;
  __shared__ __align__(8) unsigned long long mma_turn[kMmaWarps];
  __shared__ uint32_t tmem_holder;
  __shared__ int abort_flag;

  // dynamic smem: [resident weights] [A stages] [weight ring] [8-bit tile buffers] [bias, scale]
  const uint32_t raw_base = smem_u32(smem_raw);
  const uint32_t base = (raw_base + 1023u) & ~1023u;
  unsigned char* const base_ptr = smem_raw + (base - raw_base);
  int* const s_bias = reinterpret_cast<int*>(base_ptr + p.off_chan);
  float* const s_scale = reinterpret_cast<float*>(base_ptr + p.off_chan) + p.k_pad;
  // the warp index through a broadcast, so that the compiler treats it, and the role it selects, as warp uniform
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const bool lane0 = lane == 0;
  // CTA pairs: both CTAs walk the same sequence of work items (pairs of m tiles); rank 1 takes the second tile
  int cta_rank = 0;
  if constexpr (kCta2) cta_rank = __shfl_sync(0xffffffffu, (int)cluster_ctarank(), 0);
  const int vblock = kCta2 ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  const int vgrid = kCta2 ? (int)(gridDim.x >> 1) : (int)gridDim.x;
  const int total_tiles = p.m_tiles * p.n_tiles * p.splits;  // work items
  const int slots = (kCta2 ? G >> p.pair_shift : G) * p.nbuf;  // tile buffers of the CTA, used round robin

  // Programmatic dependent launch: the next kernel of the stream may be scheduled onto SMs as they fall idle
  // (it waits below, like this one, before it touches global memory), and this kernel's own set-up (barriers,
  // TMEM allocation, descriptor prefetch) runs while the previous kernel drains.  Both are no-ops for a
  // launch without the attribute.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // Prologue.  Each control lane initialises the barriers it owns.  Warp 0 only signals the
  // start-up barriers (bar.arrive) and goes straight to its loads, so that the first bytes are on
  // their way while the others allocate TMEM.  Single CTAs keep the epilogue warps off the critical path: the
  // control warps meet on barrier 1 among themselves and start; the epilogue warps first touch every line of the
  // kernel parameters (the control warps' first reads of them would otherwise miss the constant cache one after
  // the other), fetch bias and scale, and join on barrier 3, which the control warps only signal.
  const int nthreads = kCtrlT + G * kGroupThreads;
  if (!kCta2 && warp >= kCtrl) {
    const unsigned int* words = reinterpret_cast<const unsigned int*>(&p);
    unsigned int touched = 0;
    for (int i = ((int)threadIdx.x - kCtrlT) * 16; i < (int)(sizeof(UmmaParams) / 4); i += G * kGroupThreads * 16) touched ^= words[i];
    asm volatile("" ::"r"(touched));
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int i = (int)threadIdx.x - kCtrlT; i < p.k_pad; i += G * kGroupThreads) {
      s_bias[i] = (p.bias && i < p.K) ? p.bias[i] : 0;
      s_scale[i] = p.scale ? (p.scale_count == 1 ? p.scale[0] : (i < p.K ? p.scale[i] : 0.f)) : 0.f;
    }
    asm volatile("bar.sync 3, %0;" ::"r"(nthreads) : "memory");
    tcgen05_fence_after();
  } else if (warp == 0) {
    // one barrier per lane: a lone lane would spend ~50 cycles on each
    if (lane < p.stages) { mbar_init(smem_u32(&a_full[lane]), 1); mbar_init(smem_u32(&a_empty[lane]), 1); }
    else if (lane >= 8 && lane - 8 < p.b_stages) { mbar_init(smem_u32(&b_full[lane - 8]), 1); mbar_init(smem_u32(&b_empty[lane - 8]), 1); }
    else if (lane == 16) { mbar_init(smem_u32(&bres_full), 1); abort_flag = 0; }
    else if (lane == 17) prefetch_tensormap(&tmA);
    else if (lane == 18) prefetch_tensormap(&tmB);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
    if constexpr (kCta2) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      cluster_sync_all();  // the peer's barriers exist before anything signals them
      asm volatile("bar.arrive 1, %0;" ::"r"(nthreads) : "memory");
    } else {
      asm volatile("bar.arrive 1, %0;" ::"r"(kCtrlT) : "memory");
      asm volatile("bar.arrive 3, %0;" ::"r"(nthreads) : "memory");
    }
  } else {
    if (warp == 1) {
      // one arrival per epilogue warp that reads the accumulator: a group's four, or all of them in split mode
      if (lane < p.nacc) { mbar_init(smem_u32(&acc_full[lane]), 1); mbar_init(smem_u32(&acc_empty[lane]), kCta2 ? 8 << p.pair_shift : (p.epi_split ? 4 * G : 4)); }
      else if (lane >= 8 && lane - 8 < kMmaWarps) mbar_init(smem_u32(&mma_turn[lane - 8]), 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    } else if (kBufs && warp == kFillWarp) {
      if (lane < slots) { mbar_init(smem_u32(&buf_full[lane]), 1); mbar_init(smem_u32(&buf_empty[lane]), 1); }
      else if (lane == 16) prefetch_maps(maps, p.res_mode != kResNone, k8);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    } else if (kBufs && warp == kStoreWarp) {
      if (lane < slots) mbar_init(smem_u32(&store_ready[lane]), kCta2 ? kGroupThreads << p.pair_shift : kGroupThreads);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
      __syncwarp();
      if constexpr (kCta2) {
        tmem_alloc_pair(smem_u32(&tmem_holder), (uint32_t)p.tmem_cols);
        tmem_relinquish_pair();
      } else {
        tmem_alloc(smem_u32(&tmem_holder), (uint32_t)p.tmem_cols);
        tmem_relinquish();
      }
    }
    if constexpr (kCta2) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      // bias and scale of every channel, once per CTA (zero beyond Cout; one scale replicated if per tensor)
      for (int i = threadIdx.x - 32; i < p.k_pad; i += nthreads - 32) {
        s_bias[i] = (p.bias && i < p.K) ? p.bias[i] : 0;
        s_scale[i] = p.scale ? (p.scale_count == 1 ? p.scale[0] : (i < p.K ? p.scale[i] : 0.f)) : 0.f;
      }
      tcgen05_fence_before();
      __syncwarp();
      cluster_sync_all();
      asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
    } else {
      tcgen05_fence_before();
      asm volatile("bar.arrive 3, %0;" ::"r"(nthreads) : "memory");      // the epilogue warps wait for this set-up
      asm volatile("bar.sync 1, %0;" ::"r"(kCtrlT) : "memory");    // the control warps only for each other
    }
    tcgen05_fence_after();
  }
  const uint32_t tmem_base = warp == 0 ? 0u : tmem_holder;  // warp 0 never touches TMEM
  volatile int* abortp = &abort_flag;

  if (warp == 0) {
    // ------------------------------------------------------------------ A / B producer (whole warp; an elected lane issues)
    TileIterT<kCta2> ti;
    ti.init(p, vblock, vgrid, cta_rank);
    const uint32_t nstages = (uint32_t)p.stages, nbst = (uint32_t)p.b_stages;
    const uint32_t afull0 = smem_u32(&a_full[0]), aempty0 = smem_u32(&a_empty[0]);
    const uint32_t bfull0 = smem_u32(&b_full[0]), bempty0 = smem_u32(&b_empty[0]);
    const uint32_t a0 = base + p.off_a, bring0 = base + p.off_bring;
    uint32_t stage = 0, phase = 0, a_dst = a0;
    uint32_t bs = 0, bphase = 0, b_dst = bring0;
    bool ok = true;
    // Everything the previous kernel wrote is visible from here.  The roles wait for it themselves, as late as they
    // touch global memory, so that their set-up runs while that kernel drains; the MMA warps (and the store warp) only
    // ever follow loads of this warp and need no wait of their own.
    if constexpr (!kCta2) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (p.b_mode == kBResident) {
      // every weight tile of the layer, once: one load per (n tile, channel block) brings all taps,
      // laid out [tap][bn rows][bk bytes], i.e. one K-major operand tile per tap
      const uint32_t bar = smem_u32(&bres_full);
      uint32_t dst = base;
      if (!elect_one()) {
        // only an elected lane issues
      } else if (p.a_mode == kAHalo && p.halo_sw == 2) {
        mbar_arrive_expect_tx(bar, (uint32_t)(p.n_tiles * p.c_blocks * p.taps) * p.b_tile_bytes);
        // pixel-pair taps: tap t' of a filter row covers s = 2t' - e and 2t' - e + 1, whose weights are 2C
        // contiguous bytes of the (s, c) axis; a start left of s = 0 is zero filled.  One load per t' brings
        // all R filter rows: tile order (t', r).
        for (int nt = 0; nt < p.n_tiles; ++nt)
          for (int t = 0; t < p.S; ++t, dst += (uint32_t)p.R * p.b_tile_bytes) tma_load_3d(dst, &tmB, bar, (2 * t - p.halo_e) * p.c_true, nt * p.bn, 0);
      } else {
        mbar_arrive_expect_tx(bar, (uint32_t)(p.n_tiles * p.c_blocks * p.taps) * p.b_tile_bytes);
        for (int nt = 0; nt < p.n_tiles; ++nt)
          for (int c = 0; c < p.C_pad; c += p.bk, dst += (uint32_t)p.taps * p.b_tile_bytes) tma_load_3d(dst, &tmB, bar, c, nt * p.bn, 0);
      }
    }
    if (p.a_mode == kAHalo) {
      const uint32_t b_tx = (uint32_t)p.b_T * p.b_tile_bytes;
      for (; ti.tile < total_tiles && ok; ti.next(p)) {
        const int n0 = ti.nt * p.bn + (kCta2 ? cta_rank * (p.bn >> 1) : 0);
        const int q0 = ti.qt * p.tw - p.pad_w, p0 = ti.pt * p.th * p.stride_h - p.pad_h;
        for (int c = 0; c < p.C_pad && ok; c += p.bk) {
          if (!mbar_wait(aempty0 + stage * 8u, phase ^ 1u, abortp)) { ok = false; break; }
          const uint32_t bar = afull0 + stage * 8u;
          if (!elect_one()) {
          } else if constexpr (kCta2) {
            // the leader's barrier counts the bytes of both CTAs' patches
            if (cta_rank == 0) mbar_arrive_expect_tx(bar, 2u * p.a_sub_bytes);
            tma_load_4d_pair(a_dst, &tmA, map_to_cta(bar, 0), c, q0, p0, ti.img);
          } else {
            mbar_arrive_expect_tx(bar, p.a_sub_bytes);
            tma_load_4d(a_dst, &tmA, bar, c, q0, p0, ti.img);
          }
          a_dst += p.a_stage_bytes;
          if (++stage == nstages) { stage = 0; phase ^= 1u; a_dst = a0; }
          if (p.b_mode == kBRing) {
            // one operation brings the weight tiles of b_T taps (a box that runs past the last tap is zero filled
            // and still counts in full): the copy engine spends ~600 cycles per operation whatever its size
            for (int tap = 0; tap < p.taps; tap += p.b_T) {
              if (!mbar_wait(bempty0 + bs * 8u, bphase ^ 1u, abortp)) { ok = false; break; }
              const uint32_t bbar = bfull0 + bs * 8u;
              if (!elect_one()) {
              } else if constexpr (kCta2) {
                if (cta_rank == 0) mbar_arrive_expect_tx(bbar, 2u * b_tx);
                tma_load_3d_pair(b_dst, &tmB, map_to_cta(bbar, 0), c, n0, tap);
              } else {
                mbar_arrive_expect_tx(bbar, b_tx);
                tma_load_3d(b_dst, &tmB, bbar, c, n0, tap);
              }
              b_dst += p.b_sub_bytes;
              if (++bs == nbst) { bs = 0; bphase ^= 1u; b_dst = bring0; }
            }
          }
        }
      }
    } else {
      const uint32_t sub_tx = p.a_sub_bytes + (p.b_mode == kBStage ? p.b_tile_bytes : 0u);
      const uint32_t b_in_stage = (uint32_t)p.kb * p.a_sub_bytes;
      for (; ti.tile < total_tiles && ok; ti.next(p)) {
        const int m0 = ti.mt * kBM, n0 = ti.nt * p.bn;
        int w0 = 0, h0 = 0, img = 0;
        if (p.a_mode == kAIm2col) {
          img = p.fd_pq.div(m0);
          const int rem = m0 - img * p.PQ;
          const int pr = p.fd_q.div(rem), qc = rem - pr * p.Q;
          h0 = pr * p.stride_h - p.pad_h;
          w0 = qc * p.stride_w - p.pad_w;
        }
        int c = 0, tap = 0, s = 0, off_w = 0, off_h = 0;
        if (p.splits > 1) {  // this split starts at iteration sp * kps = (tap, channel block)
          const int it0 = ti.sp * p.kps;
          tap = p.fd_cblocks.div(it0);
          c = (it0 - tap * p.c_blocks) * p.bk;
          const int r0 = p.fd_s.div(tap);
          s = tap - r0 * p.S;
          off_w = s * p.dil_w; off_h = r0 * p.dil_h;
        }
        for (int it = 0; it < p.kps;) {
          const int nsub = min(p.kb, p.kps - it);
          if (!mbar_wait(aempty0 + stage * 8u, phase ^ 1u, abortp)) { ok = false; break; }
          const uint32_t bar = afull0 + stage * 8u;
          if (elect_one()) mbar_arrive_expect_tx(bar, (uint32_t)nsub * sub_tx);
          uint32_t dst = a_dst, bdst = a_dst + b_in_stage;
          for (int j = 0; j < nsub; ++j) {
            if (!elect_one()) {
            } else if (p.a_mode == kAIm2col) tma_load_im2col_4d(dst, &tmA, bar, c, w0, h0, img, (unsigned short)off_w, (unsigned short)off_h);
            else tma_load_2d(dst, &tmA, bar, c, m0);
            if (p.b_mode == kBStage && elect_one()) tma_load_3d(bdst, &tmB, bar, c, tap, n0);
            dst += p.a_sub_bytes;
            bdst += p.b_sub_bytes;
            c += p.bk;
            if (c >= p.C_pad) {  // next tap
              c = 0; ++tap; ++s; off_w += p.dil_w;
              if (s == p.S) { s = 0; off_w = 0; off_h += p.dil_h; }
            }
          }
          it += nsub;
          a_dst += p.a_stage_bytes;
          if (++stage == nstages) { stage = 0; phase ^= 1u; a_dst = a0; }
        }
      }
    }
    if (!ok && lane0) {
      abort_flag = 1;
      atomicOr(p.status, kTimeoutProducer);
    }
  } else if (warp < kCtrlWarps) {
    // ------------------------------------------------------------------ MMA issuers (warps 1 to 3; an elected lane issues)
    const int who = warp - 1;
    MmaRoleArgs ra;
    ra.base = base; ra.tmem_base = tmem_base; ra.total_tiles = total_tiles; ra.abortp = abortp;
    ra.first_tile = (int)blockIdx.x; ra.tile_step = (int)gridDim.x;
    ra.a_full = smem_u32(&a_full[0]); ra.a_empty = smem_u32(&a_empty[0]);
    ra.b_full = smem_u32(&b_full[0]); ra.b_empty = smem_u32(&b_empty[0]);
    ra.acc_full = smem_u32(&acc_full[0]); ra.acc_empty = smem_u32(&acc_empty[0]);
    ra.bres_full = smem_u32(&bres_full); ra.turn = smem_u32(&mma_turn[0]);
    bool ok = true;
    if (who >= p.mma_lanes) {
      // two issuing warps
    } else if constexpr (kCta2) {
      if (cta_rank == 0) ok = mma_role_pair(p, ra, who, vblock, vgrid);
    } else {
      ok = mma_role(p, ra, who);
    }
    if (!ok && lane0) {
      abort_flag = 1;
      atomicOr(p.status, kTimeoutMma);
    }
  } else if (kBufs && warp == kFillWarp) {
    // ------------------------------------------------------------------ tile buffers to the epilogue, with their residual tile
    if constexpr (kBufs) {
      TileIterT<kCta2> ti;
      ti.init(p, vblock, vgrid, cta_rank);
      const uint32_t bfull0 = smem_u32(&buf_full[0]), bempty0 = smem_u32(&buf_empty[0]);
      const uint32_t nslots = (uint32_t)slots;
      uint32_t slot = 0, par = 1;  // tile lt of the CTA's sequence uses buffer lt % slots
      bool ok = true;
      const int pw = 1 << p.pw_shift;
      const uint32_t panel_bytes = (uint32_t)kBM << p.pw_shift;
      if constexpr (!kCta2) asm volatile("griddepcontrol.wait;" ::: "memory");
      for (; ti.tile < total_tiles; ti.next(p)) {
        if (!mbar_wait(bempty0 + slot * 8u, par, abortp)) { ok = false; break; }
        const uint32_t bar = bfull0 + slot * 8u;
        if (!elect_one()) {
        } else if (p.res_mode != kResNone && ti.valid) {
          uint32_t dst = base + p.off_bufs + slot * p.tile8_bytes;
          mbar_arrive_expect_tx(bar, p.res_tx_bytes);
          if (p.a_mode == kAHalo) {
            for (int pn = 0, c = ti.nt * p.bn; pn < p.panels; ++pn, c += pw, dst += panel_bytes) tma_load_4d(dst, &maps.res, bar, c, ti.qt * p.tw, ti.pt * p.th, ti.img);
          } else {
            for (int pn = 0, c = ti.nt * p.bn; pn < p.panels; ++pn, c += pw, dst += panel_bytes) tma_load_2d(dst, &maps.res, bar, c, ti.mt * kBM);
          }
        } else {
          mbar_arrive(bar);
        }
        if (++slot == nslots) { slot = 0; par ^= 1u; }
      }
      if (!ok && lane0) {
        abort_flag = 1;
        atomicOr(p.status, kTimeoutResidual);
      }
    }
  } else if (kBufs && warp == kStoreWarp) {
    // ------------------------------------------------------------------ finished tiles to global memory, buffers back
    if constexpr (kBufs) {
      TileIterT<kCta2> ti;
      ti.init(p, vblock, vgrid, cta_rank);
      const uint32_t bempty0 = smem_u32(&buf_empty[0]), ready0 = smem_u32(&store_ready[0]);
      const uint32_t nslots = (uint32_t)slots;
      uint32_t slot = 0, spar = 0;
      int prev_slot = -1;
      const bool one_each = p.nbuf == 1;
      bool ok = true;
      const int pw = 1 << p.pw_shift;
      const uint32_t panel_bytes = (uint32_t)kBM << p.pw_shift;
      for (; ti.tile < total_tiles; ti.next(p)) {
        if (!mbar_wait(ready0 + slot * 8u, spar, abortp)) { ok = false; break; }
        if (!k8) {
          if (elect_one()) mbar_arrive(bempty0 + slot * 8u);  // (32-bit rows are stored by the epilogue: the residual has been read)
        } else if (elect_one()) {
          uint32_t src = base + p.off_bufs + slot * p.tile8_bytes;
          if (!ti.valid) {
            // second tile of the last pair of an odd count: nothing to store
          } else if (p.a_mode == kAHalo) {
            for (int pn = 0, c = p.c_off + ti.nt * p.bn; pn < p.panels; ++pn, c += pw, src += panel_bytes) tma_store_4d(&maps.y, src, c, ti.qt * p.tw, ti.pt * p.th, ti.img);
          } else {
            for (int pn = 0, c = p.c_off + ti.nt * p.bn; pn < p.panels; ++pn, c += pw, src += panel_bytes) tma_store_2d(&maps.y, src, c, ti.mt * kBM);
          }
          bulk_commit();
          if (one_each) {
            // one buffer per group: its group waits for it, so it is handed back as soon as it has been read (3x3
            // 128->192 at 73x73, batch 64, two groups: 66.0 -> 62.3 us; with more buffers the wait would only hold up
            // this warp)
            bulk_wait_read<0>();
            mbar_arrive(bempty0 + slot * 8u);
          } else {
            // the store before this one has read its buffer: hand that buffer back
            bulk_wait_read<1>();
            if (prev_slot >= 0) mbar_arrive(bempty0 + (uint32_t)prev_slot * 8u);
          }
          prev_slot = (int)slot;
        }
        if (++slot == nslots) { slot = 0; spar ^= 1u; }
      }
      if (k8 && elect_one()) {
        bulk_wait_read<0>();  // the CTA's shared memory must outlive the reads of its last stores
        if (prev_slot >= 0 && !one_each) mbar_arrive(bempty0 + (uint32_t)prev_slot * 8u);
      }
      if (!ok && lane0) {
        abort_flag = 1;
        atomicOr(p.status, kTimeoutStore);
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue groups
    const int g = (warp - kCtrl) >> 2;
    const int quad = warp & 3;  // TMEM lane quadrant this warp may read
    const int row = quad * 32 + lane;  // accumulator row of this thread
    EpiTile t;
    t.s_bias = s_bias;
    t.s_scale = s_scale;
    t.scale = s_scale[0];
    // halo tiles: accumulator row -> pixel (pp, qq) of the patch grid; rows right of the tile are dropped
    int pp = 0, qq = 0;
    t.srow = row;
    t.smem_ok = true;
    t.yrow = nullptr;
    t.rrow = nullptr;
    t.wide = t.res_wide = false;
    if (p.a_mode == kAHalo) {
      pp = row / p.twb;  // once per thread
      qq = row - pp * p.twb;
      t.smem_ok = pp < p.th && qq < p.tw;
      t.srow = t.smem_ok ? pp * p.tw + qq : 0;
    }
    epi_row_setup(p, t);
    // this group's tiles are lt = g, g + G, ... of the CTA's sequence; ring positions advance by additions
    // pair mode: the accumulators of both CTAs are handed back on the leader's barriers
    const uint32_t accf0 = smem_u32(&acc_full[0]);
    uint32_t acce0 = smem_u32(&acc_empty[0]);
    if constexpr (kCta2) acce0 = map_to_cta(acce0, 0);
    const uint32_t nacc = (uint32_t)p.nacc;
    // split mode: every group works on every tile and takes the chunks [ch0, ch1) of its columns, so that a
    // launch with one or two tiles per CTA does not leave three of four groups idle
    const bool split = !kBufs && p.epi_split != 0;
    const int team = kCta2 ? g >> p.pair_shift : (split ? 0 : g);
    const int tile_step = kCta2 ? G >> p.pair_shift : (split ? 1 : G);
    const int nchunk_all = p.bn >> 4;
    int ch0 = split ? (g * nchunk_all) / G : 0, ch1 = split ? ((g + 1) * nchunk_all) / G : nchunk_all;
    if constexpr (kCta2) {
      const int member = g - (team << p.pair_shift);
      ch0 = (member * nchunk_all) >> p.pair_shift;
      ch1 = ((member + 1) * nchunk_all) >> p.pair_shift;
    }
    uint32_t ab = (uint32_t)team % nacc, acc_par = ((uint32_t)team / nacc) & 1u;
    uint32_t slot = (uint32_t)team, slot_par = 0;
    TileIterT<kCta2> ti;
    ti.init(p, vblock + team * vgrid, tile_step * vgrid, cta_rank);
    for (; ti.tile < total_tiles; ti.next(p)) {
      auto place = [&] {  // the tile's pixel and columns of this thread
        t.n0 = ti.nt * p.bn;
        t.y_off = (long long)ti.sp * p.split_stride;
        if (p.a_mode == kAHalo) {
          const int pr = ti.pt * p.th + pp, qc = ti.qt * p.tw + qq;
          t.row_ok = t.smem_ok && pr < p.P && qc < p.Q && ti.valid;
          t.m = (ti.img * p.P + pr) * p.Q + qc;
        } else {
          t.m = ti.mt * kBM + row;
          t.row_ok = t.m < p.M;
        }
      };
      place();
      ResPair rp = {};
      RowMove mv;
      if constexpr (kBufs) {
        t.buf = base_ptr + p.off_bufs + (size_t)slot * p.tile8_bytes;
      } else if constexpr (kRes == kResRows) {  // one buffer per group, shared where groups share tiles: their columns are disjoint
        t.buf = base_ptr + p.off_bufs + (split ? (size_t)0 : (size_t)g * p.tile8_bytes);
        mv.init(p, t.n0, ch0, ch1);
        if (p.res_mode != kResNone) rows_in(p, t, mv, lane);  // while the accumulator is being formed
        __syncwarp();
      } else {
        t.wide = p.y_wide && ((t.n0 + ch0 * 16) & 31) == 0;
        t.res_wide = p.res_wide && ((t.n0 + ch0 * 16) & 31) == 0;
        t.yrow = static_cast<unsigned char*>(p.y) + (long long)t.m * p.ldc + p.c_off + t.n0;
        t.rrow = p.res + (long long)t.m * p.K + t.n0;
        if (kRes == kResVec && p.res_mode != kResNone) load_residual(p, t, ch0, ch1, rp);  // the first bytes, likewise
      }
      bool ok = mbar_wait(accf0 + ab * 8u, acc_par, abortp);
      if (kBufs && ok) ok = mbar_wait(smem_u32(&buf_full[0]) + slot * 8u, slot_par, abortp);
      if (!ok) {
        if (lane == 0) {
          abort_flag = 1;
          atomicOr(p.status, kTimeoutEpilogue);
        }
        break;
      }
      tcgen05_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + ab * (uint32_t)p.acc_stride;
      epilogue_row<kOut, kRes, kCta2, kUniform, (kBufs && k8) || kRes == kResRows>(p, t, taddr, acce0 + ab * 8u, lane, ch0, ch1, rp);
      if constexpr (kBufs) {
        if (k8) fence_proxy_async_smem();  // this thread's reads and writes of the buffer are done; the store reads it
        mbar_arrive(smem_u32(&store_ready[0]) + slot * 8u);
        slot += (uint32_t)tile_step;
        if (slot >= (uint32_t)slots) { slot -= (uint32_t)slots; slot_par ^= 1u; }
      }
      if constexpr (kRes == kResRows) {
        __syncwarp();
        rows_out(p, t, mv, lane);
        __syncwarp();  // the buffer is read before the next tile's rows go into it
      }
      ab += (uint32_t)tile_step;
      while (ab >= nacc) { ab -= nacc; acc_par ^= 1u; }
    }
  }

  tcgen05_fence_before();
  __syncthreads();
  if constexpr (kCta2) cluster_sync_all();  // the peer may still read this CTA's weight halves and signal its barriers until here
  if (warp == 1) {
    __syncwarp();
    tcgen05_fence_after();
    if constexpr (kCta2) tmem_dealloc_pair(tmem_base, (uint32_t)p.tmem_cols);
    else tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
  }
}

// ------------------------------------------------------------------------------------------ host
template <int G, int kOut, int kRes, bool kCta2, bool kUniform>
int launch_variant(const CUtensorMap& tmA, const CUtensorMap& tmB, const RowMaps<true>& row_maps, const UmmaParams& p, size_t dyn, int grid,
                   cudaStream_t stream) {
  constexpr int kThreads = kCtrlOf<kRes> * 32 + G * kGroupThreads;
  RowMaps<kRes == kResTma> maps;
  if constexpr (kRes == kResTma) maps = row_maps;
  auto kernel = conv_umma_kernel<G, kOut, kRes, kCta2, kUniform>;
  static std::atomic<bool> configured[kMaxDevices];  // per instantiation and device (the attribute is per device)
  const int dev = current_device();
  if (dev < 0 || !configured[dev].load(std::memory_order_acquire)) {
    int rc = check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit - kStaticSmemReserve),
                        "conv_umma: set shared memory size");
    if (rc != Q8_OK) return rc;
    // every tensor-core kernel of the library asks for the largest shared-memory carve-out, so that consecutive
    // launches of different kernels or shapes never make the SMs switch their L1 / shared-memory split
    rc = check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared),
                    "conv_umma: set shared memory carve-out");
    if (rc != Q8_OK) return rc;
    if (dev >= 0) configured[dev].store(true, std::memory_order_release);
  }
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)kThreads);
  cfg.dynamicSmemBytes = dyn;
  cfg.stream = stream;
  // let this kernel's set-up overlap the tail of the kernel before it in the stream
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = tune_env("Q8_PDL", 1, 0, 1) ? 1 : 0;
  if (p.cta2) {  // CTA pairs: clusters of two, beside the dependent launch
    const int pdl = (int)cfg.numAttrs;
    attr[pdl].id = cudaLaunchAttributeClusterDimension;
    attr[pdl].val.clusterDim.x = 2;
    attr[pdl].val.clusterDim.y = 1;
    attr[pdl].val.clusterDim.z = 1;
    cfg.numAttrs = pdl + 1;
  }
  const cudaError_t le = cudaLaunchKernelEx(&cfg, kernel, tmA, tmB, p, maps);
  if (le != cudaSuccess) {
    cudaGetLastError();
    return fail(Q8_ERR_CUDA, "conv_umma: launch failed (%s; grid %d, block %d, shared memory %zu, cluster %d)", cudaGetErrorString(le),
                grid, kThreads, dyn, p.cta2 ? 2 : 1);
  }
  return check_launch("conv_umma_kernel");
}

template <int G>
int launch_groups(const CUtensorMap& tmA, const CUtensorMap& tmB, const RowMaps<true>& maps, const UmmaParams& p, bool rows, size_t dyn, int grid,
                  cudaStream_t stream) {
#define Q8_LAUNCH(OUT, RES)                                                                                          \
  do {                                                                                                               \
    if (p.scale_count == 1) return launch_variant<G, OUT, RES, false, true>(tmA, tmB, maps, p, dyn, grid, stream);   \
    return launch_variant<G, OUT, RES, false, false>(tmA, tmB, maps, p, dyn, grid, stream);                          \
  } while (0)
  // kResTma and kResVec stand for "a residual, or none"
  const bool global_res = p.res_mode == kResGlobal;
  if (p.y_type == Q8_U8) {
    if (rows) Q8_LAUNCH(Q8_U8, kResRows);
    if (p.nbuf) Q8_LAUNCH(Q8_U8, kResTma);
    Q8_LAUNCH(Q8_U8, kResVec);
  }
  if (p.y_type == Q8_S8) {
    if (rows) Q8_LAUNCH(Q8_S8, kResRows);
    if (p.nbuf) Q8_LAUNCH(Q8_S8, kResTma);
    Q8_LAUNCH(Q8_S8, kResVec);
  }
  if (p.y_type == Q8_F32) {
    if (global_res) Q8_LAUNCH(Q8_F32, kResGlobal);
    if (p.nbuf) Q8_LAUNCH(Q8_F32, kResTma);
    Q8_LAUNCH(Q8_F32, kResVec);
  }
  return launch_variant<G, Q8_S32, kResVec, false, false>(tmA, tmB, maps, p, dyn, grid, stream);
#undef Q8_LAUNCH
}

bool is_plain(const q8_conv_desc& d) {
  return d.R == 1 && d.S == 1 && d.stride_h == 1 && d.stride_w == 1 && d.pad_h == 0 && d.pad_w == 0;
}

// im2col tensor maps: corners are 8-bit signed, tap offsets 8-bit unsigned, strides at most 8.
bool im2col_open(const q8_conv_desc& d, const char** why) {
  const int up_w = d.pad_w - (d.S - 1) * d.dil_w, up_h = d.pad_h - (d.R - 1) * d.dil_h;
  if (d.pad_w > 128 || d.pad_h > 128 || up_w < -128 || up_h < -128 || up_w > 127 || up_h > 127) { *why = "padding/dilation outside the im2col corner range"; return false; }
  if ((d.S - 1) * d.dil_w > 255 || (d.R - 1) * d.dil_h > 255) { *why = "filter extent outside the im2col offset range"; return false; }
  if (d.stride_h > 8 || d.stride_w > 8) { *why = "stride > 8"; return false; }
  if ((long long)d.N * d.H * d.W * d.C < 131072) { *why = "activation tensor smaller than 128 KiB"; return false; }
  return true;
}

}  // namespace

bool umma_shape_eligible(const q8_conv_desc& d, const char** why) {
  const char* dummy;
  if (!why) why = &dummy;
  if (d.C % 16) { *why = "C is not a multiple of 16"; return false; }
  if (d.K > 4096) { *why = "more than 4096 output channels"; return false; }
  if (is_plain(d)) return true;
  HaloTile ht;
  const int P = conv_out_extent(d.H, d.pad_h, d.dil_h, d.R, d.stride_h), Q = conv_out_extent(d.W, d.pad_w, d.dil_w, d.S, d.stride_w);
  return choose_halo_tile(d, P, Q, &ht) || im2col_open(d, why);
}

namespace {
// Tile width of a launch whose tiles of the default width would leave SMs without work: the narrowest of 16, 32, 64 and
// 128 columns that still gives every tile an SM of its own, else the default.  Such a launch lasts as long as one CTA
// takes to stream its operands, and a narrower tile streams fewer weights (1x1 1024->256 on one 14x14 image: two 256-wide
// tiles 11.9 us even with the reduction split, 32 tiles of 16 columns 4.6 us; 3x3 512->512 on one 7x7 image 10.1 -> 7.6).
// Short reductions gain less than the extra CTAs cost: up to 256 products stay as they are (1x1 256->1024 at 14x14 4.27
// against 4.64 us), up to 512 take half of the SMs at most (512->2048 at 7x7 4.7 against 5.2 us with all).
int narrow_bn(int bn, int K, int kgemm, long long m_tiles) {
  if (kgemm <= 256) return bn;
  const long long most = kgemm <= 512 ? sm_count() / 2 : sm_count();
  for (int w = 16; w < bn && w <= 128; w *= 2)
    if (m_tiles * ((K + w - 1) / w) <= most) return w;
  return bn;
}
}  // namespace

bool rows_unaligned(const ConvArgs& a) {
  return (a.d.y_type == Q8_U8 || a.d.y_type == Q8_S8) && (!aligned16(a.y) || a.ldc % 16 || a.c_off % 16 || (a.residual && !aligned16(a.residual)));
}

bool rows_off_tma(const ConvArgs& a) {
  return rows_unaligned(a) || ((a.d.y_type == Q8_U8 || a.d.y_type == Q8_S8) && a.d.K % 16);
}

namespace {
// How a layer runs: tiles, shared memory and pipeline depths.  Decided from the descriptor and the alignment of the
// pointers alone, so that it can be asked for without a device.
struct UmmaPlan {
  UmmaParams p;
  HaloTile ht;
  int G, res_mode, c_eff;
  bool rows, paired, resident;
  size_t dyn;
};

bool plan_tiles(const ConvArgs& a, int splits, int bk_cap, bool allow_halo, bool allow_bufs, UmmaPlan* plan);

// Tries tile shapes from the preferred one down: halo patches of dilated filters on wide channel blocks can
// exceed shared memory, narrower channel blocks shrink them; im2col loads need the least, where they are open.
bool plan_conv(const ConvArgs& a, int splits, UmmaPlan* plan) {
  static const struct { int bk_cap; bool halo; } kTries[] = {{128, true}, {64, true}, {32, true}, {128, false}, {64, false}};
  const char* why;
  for (const auto& t : kTries)
    if ((t.halo || is_plain(a.d) || im2col_open(a.d, &why)) && plan_tiles(a, splits, t.bk_cap, t.halo, true, plan)) return true;
  return false;
}

int launch_planned(const ConvArgs& a, int splits);
}  // namespace

bool umma_fits(const ConvArgs& a) {
  UmmaPlan plan;
  return plan_conv(a, 1, &plan);
}

namespace {
// The first pass of a split: raw partial accumulators of every part into the workspace.
ConvArgs partial_call(const ConvArgs& a) {
  ConvArgs part = a;
  part.d.y_type = Q8_S32;
  part.d.relu = 0;
  part.y = a.workspace;
  part.ldc = a.d.K;
  part.c_off = 0;
  part.bias = nullptr;
  part.residual = nullptr;
  return part;
}

// Split-K plan: layers whose output tiles cannot occupy a quarter of the SMs split the reduction over
// (tap, channel block) iterations into equal parts; every part writes raw int32 partial sums (integer addition is
// associative, so the result stays bit exact).  Only the plain and im2col operand paths split.  Returns the parts a call
// runs in, given scratch for them: 1 where it runs unsplit.
int split_parts(const ConvArgs& a) {
  const q8_conv_desc& d = a.d;
  if (d.y_type == Q8_S32 || rows_unaligned(a) || !umma_shape_eligible(d, nullptr)) return 1;
  HaloTile ht;
  if (!is_plain(d) && choose_halo_tile(d, a.P, a.Q, &ht)) return 1;
  const int kg = d.R * d.S * d.C, BK = pick_bk(d.C), BN = pick_bn(d.K, kg);
  const long long m_tiles = (a.M + kBM - 1) / kBM, tiles = m_tiles * ((d.K + BN - 1) / BN);
  const int k_iters = d.R * d.S * ((d.C + BK - 1) / BK);
  const int sms = sm_count();
  // a split costs a second (small) kernel and the partial-sum traffic: it pays once most SMs would idle
  if (tiles * 4 > sms) return 1;
  int splits = 1;
  for (int sp = 2; sp <= 16 && tiles * sp <= sms; ++sp)
    if (k_iters % sp == 0 && k_iters / sp >= 4) splits = sp;
  if (splits == 1) return 1;
  // Narrow tiles against the split of the default ones, by the operand bytes a CTA streams (~60 per cycle); a split
  // pays ~6000 cycles for its second kernel.
  const double t_split = (double)kg / splits * (kBM + BN) / 60.0 + 6000.0;
  const double t_narrow = (double)kg * (kBM + narrow_bn(BN, d.K, kg, m_tiles)) / 60.0;
  return t_narrow <= t_split ? 1 : splits;
}
}  // namespace

int umma_splits(const ConvArgs& a) {
  const int splits = split_parts(a);
  UmmaPlan plan;
  return splits > 1 && plan_conv(partial_call(a), splits, &plan) ? splits : 1;
}

bool umma_describe(const ConvArgs& a, q8_conv_plan* out) {
  UmmaPlan plan;
  const int splits = umma_splits(a);
  if (!plan_conv(splits > 1 ? partial_call(a) : a, splits, &plan)) return false;
  out->tile_n = plan.p.bn;
  out->operand = plan.p.a_mode;
  out->splits = splits;
  out->weights = plan.p.b_mode;
  out->cta_pair = plan.p.cta2;
  out->shared_groups = plan.p.cta2 ? 1 << plan.p.pair_shift : (plan.p.epi_split ? plan.G : 1);
  out->moved_rows = plan.rows;
  return true;
}

int umma_row_buffers(const ConvArgs& a) {
  UmmaPlan plan;
  if (umma_splits(a) > 1 || !plan_conv(a, 1, &plan)) return 0;
  const UmmaParams& p = plan.p;
  return (p.cta2 ? plan.G >> p.pair_shift : plan.G) * p.nbuf;
}

int launch_conv_umma(const ConvArgs& a) {
  const int splits = a.workspace && aligned16(a.workspace) ? split_parts(a) : 1;
  if (splits > 1 && a.workspace_bytes >= (size_t)splits * (size_t)a.M * a.d.K * sizeof(int)) {
    const int rc = launch_planned(partial_call(a), splits);
    if (rc == Q8_OK) return launch_splitk_reduce(a, splits);  // pass 2: sum, bias, epilogue
    if (rc != kPlanNoFit) return rc;
  }
  return launch_planned(a, 1);
}

namespace {
// Whether the 8-bit rows of a layer go through tile buffers, `two` of which fit per epilogue group or else one.
//
// Without them a warp's access touches 32 rows a pitch apart, which keeps the load/store unit busy in proportion to the bytes
// of the rows; with them the copy engine moves whole lines, at the price of two more hand-offs at the end of a CTA and of
// shared memory.  So buffers are for CTAs with many tiles, wide ones and short reductions, where rows and not operands are
// the launch, more so with a residual, whose bytes count again.  Inputs not in L2, buffers against none (us):
//   1x1 64->256 at 56x56 with a residual: batch 8 (2.6 tiles a CTA) 8.1 / 7.9, 16 (5.3) 10.9 / 12.9, 32 16.0 / 21.3, 64 25.9 /
//     39.4; without one: batch 16 8.4 / 8.4, 32 11.5 / 12.0, 64 18.1 / 20.3; 32 columns never gain (32->32 at 112x112, batch 64
//     24.7 / 22.6; 256->32 at 56x56 with a residual 14.2 / 13.5);
//   room for one buffer per group only: 1x1 256->256 at 56x56, batch 64 27.4 / 23.0 (too few operand stages are left), with a
//     residual 31.7 / 43.4; 128->512 at 28x28 with one 19.2 / 21.4, without 12.6 / 12.6;
//   halo tiles: 3x3 64->64 at 56x56, batch 64 12.3 / 13.3, batch 32 9.1 / 8.7; 32->96 at 112x112 with a residual, batch 8 (6
//     tiles a CTA) 12.3 / 11.1, 64 46.3 / 55.7; pairs at 75x75, batch 32 128->192 32.2 / 34.5, 128->256 40.1 / 38.9;
//   tiles shared by all groups: 1x1 128->512 at 28x28, batch 8 with a residual 6.3 / 7.1, without 5.5 / 5.6.
// Shared tiles take none all the same: a launch of another kernel function than the one before it starts slower, and in
// ResNet-50 at batch 16 that costs more than it gives (402 -> 410 us; batch 32 501 -> 508).  The other lines lie where the
// networks gain or stay: SSD-300 at batch 32 1095 -> 1076 us, ResNet-50 and Inception-v3 within 0.3 % from batch 8 to 64
// (matrices without a residual, taken from 12 tiles a CTA, still cost ResNet-50 at batch 40 551 -> 554 us).
// 32-bit outputs are stored by the epilogue; a residual of theirs (8-bit) comes through buffers already from one tile a CTA, in
// groups of their own: 408 layers 3.6 % faster in the mean, 1x1 256->512 at 112x112, batch 4 51.8 -> 46.5 us, 3x3 256->512 at
// 56x56, batch 16 73.7 -> 64.4.
// Over 2131 layers with 8-bit outputs the rule is on average 3.0 % below no buffers at all (34 % at best).
bool buffered(const ConvArgs& a, const UmmaParams& p, bool two) {
  const bool residual = a.residual != nullptr, plain = p.a_mode == kAPlain, wide = a.ldc % 32 == 0 && a.c_off % 32 == 0;
  const int reduction = a.d.R * a.d.S * a.d.C, ctas = p.cta2 ? sm_count() / 2 : sm_count();
  const long long items = (long long)p.m_tiles * p.n_tiles;
  auto more_than = [&](int per_cta) { return items > (long long)per_cta * ctas; };
  if (p.splits > 1) return false;
  if (a.d.y_type == Q8_F32) return p.bn > 64 ? more_than(1) : (p.bn == 64 && more_than(8));
  if (p.epi_split) return false;
  const bool broad = p.bn > 128 && p.bn < 256;
  if (p.bn < 64 || reduction > (residual || broad ? 1152 : 864)) return false;
  if (residual) return more_than(plain || p.n_tiles > 1 || p.bn > 128 ? 4 : 8);
  if (p.bn < 96) return !plain && two && more_than(12);
  if (!plain) return more_than(two || (broad && p.cta2) ? 8 : 12);
  return ((two || reduction <= 128) && more_than(16)) || (!wide && reduction <= 288 && more_than(8));  // (!wide: twice the accesses)
}

bool plan_tiles(const ConvArgs& a, int splits, int bk_cap, bool allow_halo, bool allow_bufs, UmmaPlan* plan) {
  const q8_conv_desc& d = a.d;
  const bool out8 = d.y_type == Q8_U8 || d.y_type == Q8_S8;
  int res_mode = kResNone;
  if (a.residual) res_mode = (d.K % 16 == 0 && aligned16(a.residual)) ? kResVec : (out8 ? kResRows : kResGlobal);
  // 8-bit rows that 16-byte accesses cannot address are moved by the epilogue warps in words, in both directions if in one
  const bool rows = out8 && (rows_off_tma(a) || res_mode == kResRows);
  if (rows && a.residual) res_mode = kResRows;
  UmmaParams& p = plan->p;
  memset(&p, 0, sizeof(p));
  HaloTile& ht = plan->ht;
  ht = {0, 0, 0, 0, 0.0, 1, d.S, d.pad_w, 0};
  p.a_mode = is_plain(d) ? kAPlain : ((allow_halo && tune_env("Q8_HALO", 1, 0, 1) && choose_halo_tile(d, a.P, a.Q, &ht)) ? kAHalo : kAIm2col);
  const bool paired = p.a_mode == kAHalo && ht.sw == 2;  // input read as pixel pairs with 2C channels
  const int c_eff = paired ? 2 * d.C : d.C;
  const int BK = pick_bk(c_eff) < bk_cap ? pick_bk(c_eff) : bk_cap;
  int BN = pick_bn(d.K, d.R * d.S * d.C);
  {
    // Few output tiles (small images, small batches): narrower ones, so that more CTAs get work.
    const long long m_tiles = p.a_mode == kAHalo ? (long long)d.N * ((a.P + ht.th - 1) / ht.th) * ((a.Q + ht.tw - 1) / ht.tw)
                                                 : (a.M + kBM - 1) / kBM;
    // (only where the tiles of the default width do not outnumber half of the SMs, and not for pixel pairs, whose plan
    // keeps the weights of the default tiles resident)
    if (splits == 1 && !paired && m_tiles * ((d.K + BN - 1) / BN) * 2 <= sm_count()) BN = narrow_bn(BN, d.K, d.R * d.S * d.C, m_tiles);
  }
  {
    const int want = tune_env("Q8_BN", BN, 16, 256);
    if (want % 16 == 0) BN = want;
  }
  p.bn = BN; p.bk = BK; p.ksteps = BK / 32;
  p.P = a.P; p.Q = a.Q; p.PQ = a.P * a.Q; p.M = (int)a.M; p.K = d.K;
  p.stride_h = d.stride_h; p.stride_w = d.stride_w; p.pad_h = d.pad_h; p.pad_w = d.pad_w; p.dil_h = d.dil_h; p.dil_w = d.dil_w;
  p.R = d.R; p.S = d.S; p.taps = d.R * d.S;
  p.halo_sw = 1; p.halo_e = 0; p.c_true = d.C;
  if (p.a_mode == kAHalo) {
    p.S = ht.s_eff; p.taps = d.R * ht.s_eff; p.pad_w = ht.pad_w_eff;
    p.halo_sw = ht.sw; p.halo_e = ht.e;
    const int dil_w = paired ? 1 : d.dil_w;
    // tap order = order of the weight tiles in shared memory: (r, s) normally, (t', r) for pixel pairs
    const unsigned row16 = (unsigned)(d.dil_h * ht.twb) * (unsigned)(BK >> 4), col16 = (unsigned)dil_w * (unsigned)(BK >> 4);
    p.in16 = paired ? row16 : col16;
    p.out16 = paired ? col16 : row16;
    p.tap_inner = paired ? d.R : ht.s_eff;
  }
  p.c_blocks = (c_eff + BK - 1) / BK;
  if (paired && p.c_blocks != 1) return false;  // the weights of a pixel pair are one block of 2C channels
  p.C_pad = p.c_blocks * BK;
  p.k_iters = p.taps * p.c_blocks;
  p.splits = splits;
  p.kps = p.k_iters / splits;  // the plan only splits evenly
  p.fd_splits = make_fastdiv(splits);
  p.fd_cblocks = make_fastdiv(p.c_blocks);
  p.fd_s = make_fastdiv(d.S);
  p.split_stride = (long long)a.M * a.ldc;
  // 8-bit tile buffers: panels as wide as the largest power of two dividing BN, at most one swizzle span
  int pw = BN & -BN;
  if (pw > 128) pw = 128;
  p.pw_shift = 0;
  while ((1 << p.pw_shift) < pw) ++p.pw_shift;
  p.pmask = pw == 128 ? 7 : (pw == 64 ? 3 : (pw == 32 ? 1 : 0));
  p.panels = BN / pw;
  p.n_tiles = (d.K + BN - 1) / BN;
  p.k_pad = p.n_tiles * BN;
  if (p.a_mode == kAHalo) {
    p.tw = ht.tw; p.th = ht.th; p.twb = ht.twb; p.hb = ht.hb;
    p.q_tiles = (a.Q + ht.tw - 1) / ht.tw;
    p.p_tiles = (a.P + ht.th - 1) / ht.th;
    p.m_tiles = d.N * p.p_tiles * p.q_tiles;
  } else {
    p.m_tiles = (int)((a.M + kBM - 1) / kBM);
  }
  p.fd_ntiles = make_fastdiv(p.n_tiles);
  p.fd_perimg = make_fastdiv(p.a_mode == kAHalo ? p.p_tiles * p.q_tiles : 1);
  p.fd_qtiles = make_fastdiv(p.a_mode == kAHalo ? p.q_tiles : 1);
  p.fd_pq = make_fastdiv(p.PQ);
  p.fd_q = make_fastdiv(p.Q);
  p.tile8_bytes = (unsigned)(kBM * BN);  // a multiple of 2 KiB
  p.acc_stride = 32;
  while (p.acc_stride < BN) p.acc_stride *= 2;
  p.nacc = 512 / p.acc_stride < kMaxAcc ? 512 / p.acc_stride : kMaxAcc;
  p.tmem_cols = p.nacc * p.acc_stride;  // a power of two in [32, 512]
  // Three issuing warps where four accumulators allow it: 64-column tiles gain (3x3 64->64 at 300x300, batch 32: 130 ->
  // 106 us; at 56x56, batch 64: 13.4 -> 12.4 us), wider ones are within 4 % either way (64->128 at 150x150 43.6 -> 45.4 us).
  // With two accumulators a third lane could wait on an accumulator barrier two phases ahead (the release it waits
  // for may belong to a tile that another lane has not issued yet); with four, the tile that last used the
  // accumulator was issued before this lane's previous tile.
  p.mma_lanes = tune_env("Q8_LANES", p.nacc >= 4 ? 3 : 2, 2, 3);
  if (p.mma_lanes > 2 && p.nacc < 4) p.mma_lanes = 2;
  p.b_tile_bytes = (unsigned)(BN * BK);
  p.b_sub_bytes = round_up(p.b_tile_bytes, 1024u);

  // ---- shared memory plan: [resident weights] [A stages] [weight ring] [8-bit tile buffers] [bias, scale]
  // Launches with at most two work items per CTA cannot keep several groups busy on different tiles: there all
  // four groups share every tile, each taking a quarter of its columns (any tile width, both accumulators).
  {
    const long long items = (long long)p.m_tiles * p.n_tiles * splits;
    const long long ctas = items < sm_count() ? items : sm_count();
    const int may = (BN >= 64 && d.y_type != Q8_S32) ? 1 : 0;
    p.epi_split = tune_env("Q8_SPLIT", ((items + ctas - 1) / ctas <= 2 && may) ? 1 : 0, 0, may);
  }
  int G = tune_env("Q8_G", (BN > 128 && !p.epi_split) ? 2 : 4, 2, 4);
  if (G == 3) G = 4;
  if (G > p.nacc && !p.epi_split) G = 2;  // a group may run at most one accumulator phase ahead of the MMA warp
  const unsigned chan_bytes = round_up((unsigned)p.k_pad * 8u, 1024u);
  const unsigned budget = (unsigned)(kSmemLimit - kStaticSmemReserve) - 1024u /* alignment slack */ - chan_bytes;
  // Weights stay resident when the whole layer's B operand is small: no per-tile weight traffic at all.
  // A tile of bn*bk bytes keeps every tap tile aligned to the swizzle pattern.
  const unsigned b_all = (unsigned)(p.n_tiles * p.c_blocks * p.taps) * p.b_tile_bytes;
  // A launch of one item per CTA needs one tile of columns only, not the weights of all of them.
  const long long n_items = (long long)p.m_tiles * p.n_tiles * splits;
  const int can_reside = (b_all <= 80u * 1024u && (paired || p.n_tiles == 1 || n_items > sm_count()) && p.taps <= 256 && p.b_tile_bytes % (8u * BK) == 0) ? 1 : 0;
  const bool resident = tune_env("Q8_BRES", can_reside, 0, can_reside) != 0;
  p.b_mode = resident ? kBResident : (p.a_mode == kAHalo ? kBRing : kBStage);
  const unsigned bres_bytes = resident ? round_up(b_all, 1024u) : 0u;
  // CTA pairs for the large layers with 256-wide tiles and streamed weights.  There the shared-memory port is
  // the limit: every 128 x 256 x 128 block reads 48 KB of operands while TMA writes 32 KB of weights.  With
  // tcgen05.mma.cta_group::2 two CTAs work on two m tiles of the same n tile, each holds half of the weight
  // rows, and both the operand reads and the weight writes per SM drop by a third and a half.
  p.cta2 = 0;
  p.m_tiles_real = p.m_tiles;
  {
    // Long launches only, three items per pair of SMs and more: batch 32 at 150x150 128->128 97.0 -> 78.5 us, 75x75
    // 256->256 80.0 -> 68.0 us, batch 64 at 73x73 128->192 67.8 -> 60.1 us, at 35x35 96->96 16.5 -> 14.7 us.  At the lower
    // end they can lose (28x28 128->128, batch 64: 11.7 -> 12.7 us), and inside a network whose branches run on several
    // streams a cluster needs two free SMs of one pair at the same time.  Tile widths whose halves keep whole 16-row
    // groups.  Layers with resident weights stay single CTAs: 3x3 64->64 at 300x300, batch 32 takes 106 us with them, 199 us
    // with streamed weights, 167 us with those as pairs.
    const long long pair_items = (long long)((p.m_tiles + 1) / 2) * p.n_tiles;
    const bool can = p.a_mode == kAHalo && !paired && p.b_mode == kBRing && BN >= 96 && BN % 32 == 0 && out8 &&
                     !rows && splits == 1 && (BK == 128 || BK == 64) &&
                     !p.epi_split && pair_items >= tune_env("Q8_CTA2MIN", 2 * (sm_count() / 2), 1, 1 << 30);
    if (can && tune_env("Q8_CTA2", 1, 0, 1)) {
      p.cta2 = 1;
      p.m_tiles = (p.m_tiles + 1) / 2;              // work items are pairs of m tiles, more than two per pair of SMs
      // Teams: tiles above 128 columns leave two accumulators, hence two teams, and with two groups each an accumulator is
      // back in half the time (3x3 128->192 at 73x73, batch 64: 62.1 -> 57.3 us).  Four teams for narrower tiles (128->128
      // at 150x150 as teams of two: 74 -> 108 us, what a tile costs a group beside its columns is paid twice).
      p.pair_shift = BN > 128 ? 1 : 0;
      G = 4;
      p.b_tile_bytes = (unsigned)((BN / 2) * BK);   // this CTA's half of the weight rows
      p.b_sub_bytes = round_up(p.b_tile_bytes, 1024u);
    }
  }
  const bool use_bufs = allow_bufs && (out8 ? !rows : d.y_type == Q8_F32 && res_mode == kResVec) && tune_env("Q8_BUFS", buffered(a, p, true) || buffered(a, p, false), 0, 1);
  if (use_bufs && p.epi_split) {
    p.epi_split = 0;
    if (BN > 128 || G > p.nacc) G = 2;
  }
  const unsigned teams = (unsigned)(p.cta2 ? G >> p.pair_shift : G);
  const unsigned row_bytes = rows ? (unsigned)(p.epi_split ? 1 : G) * p.tile8_bytes : 0u;
  p.b_T = 1;
  p.b_chunks = p.taps;
  unsigned min_pipe;
  if (p.a_mode == kAHalo) {
    // the taps read up to (ext_h * twb + ext_w) pixels beyond accumulator row 127
    const unsigned reach = (unsigned)(kBM + (d.R - 1) * d.dil_h * ht.twb + (ht.s_eff - 1) * (paired ? 1 : d.dil_w)) * BK;
    p.a_sub_bytes = (unsigned)(BK * ht.twb * ht.hb);
    p.a_stage_bytes = round_up(reach > p.a_sub_bytes ? reach : p.a_sub_bytes, 1024u);
    p.kb = 1;
    // (measured: a gain with four accumulators, i.e. tiles up to 128 columns; a loss with two)
    if (p.b_mode == kBRing && p.b_tile_bytes % (8u * BK) == 0 && (p.nacc >= 4 || p.cta2)) {
      // Weight ring stages of several filter taps, one TMA operation each (the copy engine spends ~600 cycles
      // per operation whatever its size): as many taps as fit in about 48 KiB while two such stages fit beside
      // two activation stages and the tile buffers, spread evenly over a channel block.
      const unsigned fixed = bres_bytes + row_bytes + (use_bufs ? teams * p.tile8_bytes : 0u) + 2u * p.a_stage_bytes;
      const unsigned avail = budget > fixed ? budget - fixed : 0u;
      int T = (int)(48u * 1024u / p.b_tile_bytes);
      if (T > (int)(avail / (2u * p.b_tile_bytes))) T = (int)(avail / (2u * p.b_tile_bytes));
      T = tune_env("Q8_BT", T, 1, T > 1 ? T : 1);
      if (T > p.taps) T = p.taps;
      if (T < 1) T = 1;
      p.b_chunks = (p.taps + T - 1) / T;
      p.b_T = (p.taps + p.b_chunks - 1) / p.b_chunks;
      p.b_chunks = (p.taps + p.b_T - 1) / p.b_T;
      p.b_sub_bytes = round_up((unsigned)p.b_T * p.b_tile_bytes, 1024u);
    }
    min_pipe = 2u * p.a_stage_bytes + (p.b_mode == kBRing ? (p.b_T > 1 ? 2u : 3u) * p.b_sub_bytes : 0u);
  } else {
    p.a_sub_bytes = (unsigned)(kBM * BK);
    const unsigned unit = p.a_sub_bytes + (p.b_mode == kBStage ? p.b_sub_bytes : 0u);
    int kb = (int)(40u * 1024u / unit);
    if (kb < 1) kb = 1;
    if (kb > p.kps) kb = p.kps;
    p.kb = tune_env("Q8_KB", kb, 1, kb);
    p.a_stage_bytes = (unsigned)p.kb * unit;
    min_pipe = 2u * p.a_stage_bytes;
  }
  p.nbuf = 0;
  if (use_bufs) {
    // two buffers per group (team) when that still leaves a comfortable pipeline
    const bool fit = budget >= bres_bytes + teams * p.tile8_bytes + min_pipe;
    const bool two = budget >= bres_bytes + 2u * teams * p.tile8_bytes + 2u * min_pipe && 2 * teams <= (unsigned)kMaxSlots;
    if (!fit || !tune_env("Q8_BUFS", buffered(a, p, two), 0, 1)) return plan_tiles(a, splits, bk_cap, allow_halo, false, plan);
    p.nbuf = two ? 2 : 1;
  }
  const unsigned buf_bytes = row_bytes + teams * (unsigned)p.nbuf * p.tile8_bytes;
  if (budget < bres_bytes + buf_bytes + min_pipe) return false;
  unsigned rest = budget - bres_bytes - buf_bytes;
  p.b_stages = 0;
  if (p.b_mode == kBRing) {
    int bst = (int)((rest - 2u * p.a_stage_bytes) / p.b_sub_bytes);
    if (bst > kMaxBStages) bst = kMaxBStages;
    p.b_stages = tune_env("Q8_BSTAGES", bst, 2, bst > 2 ? bst : 2);
    rest -= (unsigned)p.b_stages * p.b_sub_bytes;
  }
  int stages = (int)(rest / p.a_stage_bytes);
  if (stages > kMaxStages) stages = kMaxStages;
  p.stages = tune_env("Q8_STAGES", stages, 2, stages > 2 ? stages : 2);
  p.off_a = bres_bytes;
  p.off_bring = p.off_a + (unsigned)p.stages * p.a_stage_bytes;
  p.off_bufs = p.off_bring + (unsigned)p.b_stages * p.b_sub_bytes;
  p.off_chan = p.off_bufs + buf_bytes;
  size_t dyn = 1024u + p.off_chan + chan_bytes;
  if (dyn > (size_t)(kSmemLimit - kStaticSmemReserve)) return false;
  // at least 120 KiB so that one CTA owns an SM and with it the whole TMEM
  plan->dyn = dyn < 120 * 1024 ? 120 * 1024 : dyn;
  plan->G = G; plan->res_mode = res_mode; plan->c_eff = c_eff;
  plan->rows = rows; plan->paired = paired; plan->resident = resident;
  return true;
}

int launch_planned(const ConvArgs& a, int splits) {
  const q8_conv_desc& d = a.d;
  UmmaPlan plan;
  if (!plan_conv(a, splits, &plan)) return kPlanNoFit;
  const DriverFns& fn = driver_fns();
  if (!fn.tiled || !fn.im2col) return fail(Q8_ERR_CUDA, "conv_umma: cuTensorMapEncode* entry points not available");
  unsigned int* status = status_word_device_ptr();
  if (!status) return fail(Q8_ERR_CUDA, "conv_umma: status word not available");
  UmmaParams& p = plan.p;
  const HaloTile& ht = plan.ht;
  const int BK = p.bk, BN = p.bn, G = plan.G, res_mode = plan.res_mode, c_eff = plan.c_eff;
  const bool rows = plan.rows, paired = plan.paired, resident = plan.resident;
  const bool out8 = d.y_type == Q8_U8 || d.y_type == Q8_S8;
  const size_t dyn = plan.dyn;
  const CUtensorMapSwizzle swz = swizzle_for_bytes(BK);

  // ---- tensor maps
  CUtensorMap tmA, tmB;
  CUresult cr;
  const cuuint32_t ones[4] = {1, 1, 1, 1};
  if (p.a_mode == kAPlain) {
    cuuint64_t dims[2] = {(cuuint64_t)d.C, (cuuint64_t)a.M};
    cuuint64_t strides[1] = {(cuuint64_t)d.C};
    cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)kBM};
    cr = fn.tiled(&tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(a.x), dims, strides, box, ones,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  } else {
    cuuint64_t dims[4] = {(cuuint64_t)d.C, (cuuint64_t)d.W, (cuuint64_t)d.H, (cuuint64_t)d.N};
    cuuint64_t strides[3] = {(cuuint64_t)d.C, (cuuint64_t)d.W * d.C, (cuuint64_t)d.H * d.W * d.C};
    if (p.a_mode == kAHalo) {
      if (paired) { dims[0] = (cuuint64_t)c_eff; dims[1] = (cuuint64_t)(d.W / 2); strides[0] = (cuuint64_t)c_eff; }
      cuuint32_t box[4] = {(cuuint32_t)BK, (cuuint32_t)ht.twb, (cuuint32_t)ht.hb, 1};
      cr = fn.tiled(&tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(a.x), dims, strides, box, ones,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    } else {
      int lower[2] = {-d.pad_w, -d.pad_h};
      int upper[2] = {d.pad_w - (d.S - 1) * d.dil_w, d.pad_h - (d.R - 1) * d.dil_h};
      cuuint32_t estr[4] = {1, (cuuint32_t)d.stride_w, (cuuint32_t)d.stride_h, 1};
      cr = fn.im2col(&tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(a.x), dims, strides, lower, upper,
                     (cuuint32_t)BK, (cuuint32_t)kBM, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    }
  }
  if (cr != CUDA_SUCCESS) return fail(Q8_ERR_CUDA, "conv_umma: activation tensor map rejected (CUresult %d)", (int)cr);
  if (resident && paired) {
    // (S*C, K, R) view of the KRSC weights: a box of 2C bytes along the (s, c) axis is one pixel-pair tap
    cuuint64_t dims[3] = {(cuuint64_t)d.S * d.C, (cuuint64_t)d.K, (cuuint64_t)d.R};
    cuuint64_t strides[2] = {(cuuint64_t)d.R * d.S * d.C, (cuuint64_t)d.S * d.C};
    cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)BN, (cuuint32_t)d.R};
    cr = fn.tiled(&tmB, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<int8_t*>(a.w), dims, strides, box, ones,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  } else if (resident) {
    // (C, K, taps) view of the KRSC weights: one box brings bn rows of every tap
    cuuint64_t dims[3] = {(cuuint64_t)d.C, (cuuint64_t)d.K, (cuuint64_t)p.taps};
    cuuint64_t strides[2] = {(cuuint64_t)p.taps * d.C, (cuuint64_t)d.C};
    cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)BN, (cuuint32_t)p.taps};
    cr = fn.tiled(&tmB, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<int8_t*>(a.w), dims, strides, box, ones,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  } else if (p.b_mode == kBRing) {
    // (C, K, taps) view: one box brings bn rows of b_T consecutive taps, one K-major tile per tap
    cuuint64_t dims[3] = {(cuuint64_t)d.C, (cuuint64_t)d.K, (cuuint64_t)p.taps};
    cuuint64_t strides[2] = {(cuuint64_t)p.taps * d.C, (cuuint64_t)d.C};
    cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)(p.cta2 ? BN / 2 : BN), (cuuint32_t)p.b_T};
    cr = fn.tiled(&tmB, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<int8_t*>(a.w), dims, strides, box, ones,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  } else {
    cuuint64_t dims[3] = {(cuuint64_t)d.C, (cuuint64_t)p.taps, (cuuint64_t)d.K};
    cuuint64_t strides[2] = {(cuuint64_t)d.C, (cuuint64_t)p.taps * d.C};
    cuuint32_t box[3] = {(cuuint32_t)BK, 1, (cuuint32_t)BN};
    cr = fn.tiled(&tmB, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<int8_t*>(a.w), dims, strides, box, ones,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  }
  if (cr != CUDA_SUCCESS) return fail(Q8_ERR_CUDA, "conv_umma: weight tensor map rejected (CUresult %d)", (int)cr);

  // 8-bit tiles through buffers: [M][channels] matrices, or for halo tiles (channels, Q, P, N) tensors whose TH x TW box
  // lands as TH*TW dense rows.  The output map ends at the last channel this layer owns, a multiple of 16 (stores are
  // clipped in units of 16 bytes), so the store clips ragged Cout tiles and never touches a neighbouring slice of a
  // concatenated tensor.
  RowMaps<true> maps;
  memset(&maps, 0, sizeof(maps));
  if (p.nbuf) {
    const int pw = 1 << p.pw_shift;
    auto encode_rows = [&](CUtensorMap* tm, void* ptr, int channels, int ld, CUtensorMapL2promotion promo) -> CUresult {
      if (p.a_mode == kAHalo) {
        cuuint64_t dims[4] = {(cuuint64_t)channels, (cuuint64_t)a.Q, (cuuint64_t)a.P, (cuuint64_t)d.N};
        cuuint64_t strides[3] = {(cuuint64_t)ld, (cuuint64_t)a.Q * ld, (cuuint64_t)a.P * a.Q * ld};
        cuuint32_t box[4] = {(cuuint32_t)pw, (cuuint32_t)ht.tw, (cuuint32_t)ht.th, 1};
        return fn.tiled(tm, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, ptr, dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        swizzle_for_bytes(pw), promo, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      }
      cuuint64_t dims[2] = {(cuuint64_t)channels, (cuuint64_t)a.M};
      cuuint64_t strides[1] = {(cuuint64_t)ld};
      cuuint32_t box[2] = {(cuuint32_t)pw, (cuuint32_t)kBM};
      return fn.tiled(tm, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, ptr, dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
                      swizzle_for_bytes(pw), promo, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    };
    if (a.residual) {
      cr = encode_rows(&maps.res, const_cast<void*>(a.residual), d.K, d.K, CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
      if (cr != CUDA_SUCCESS) return fail(Q8_ERR_CUDA, "conv_umma: residual tensor map rejected (CUresult %d)", (int)cr);
    }
    if (out8) {
      cr = encode_rows(&maps.y, a.y, a.c_off + d.K, a.ldc, CU_TENSOR_MAP_L2_PROMOTION_NONE);
      if (cr != CUDA_SUCCESS) return fail(Q8_ERR_CUDA, "conv_umma: output tensor map rejected (CUresult %d)", (int)cr);
    }
    p.res_tx_bytes = (unsigned)BN * (p.a_mode == kAHalo ? (unsigned)(ht.tw * ht.th) : (unsigned)kBM);
  }

  // instruction descriptor: D = s32 (2 << 4); A format at bit 7 (0 = u8, 1 = s8); B = s8 at bit 10;
  // both operands K-major; N/8 at bit 17; M/16 at bit 24.
  p.idesc = (2u << 4) | ((d.x_type == Q8_S8 ? 1u : 0u) << 7) | (1u << 10) | ((unsigned)(BN >> 3) << 17) |
            ((unsigned)((p.cta2 ? 2 * kBM : kBM) >> 4) << 24);
  // shared-memory matrix descriptor of a K-major operand tile whose rows are BK bytes (= one swizzle
  // span): 8-row groups are 8*BK bytes apart (stride byte offset, bits 32-45), the leading byte offset
  // (bits 16-29) is unused for swizzled K-major tiles and set to 1, descriptor version 1 (bit 46),
  // swizzle mode from BK (bits 61-63).  Only the high word is kept here; the low word is
  // (start address >> 4) | (1 << 16).
  {
    const unsigned layout = BK == 128 ? 2u : (BK == 64 ? 4u : 6u);
    p.desc_hi = (unsigned)((8 * BK) >> 4) | (1u << 14) | (layout << 29);
  }
  p.bias = a.bias; p.scale = a.scale; p.scale_count = d.scale_count;
  p.res = static_cast<const unsigned char*>(a.residual);
  p.res_mode = res_mode;
  p.res_signed = d.res_type == Q8_S8;
  p.res_scale = a.residual_scale;
  p.y = a.y; p.y_type = d.y_type; p.ldc = a.ldc; p.c_off = a.c_off; p.relu = d.relu;
  // an 8-bit row is stored and its residual loaded in whole 32-byte sectors where the pitch allows it
  p.y_wide = out8 && !rows && (reinterpret_cast<uintptr_t>(a.y) & 31u) == 0 && a.ldc % 32 == 0 && a.c_off % 32 == 0;
  p.res_wide = res_mode == kResVec && (reinterpret_cast<uintptr_t>(a.residual) & 31u) == 0 && d.K % 32 == 0;
  p.y_vec = out8 ? 1 : (aligned16(a.y) && a.ldc % 4 == 0 && a.c_off % 4 == 0);
  p.status = status;

  const long long tiles = (long long)p.m_tiles * p.n_tiles * splits;  // work items
  int grid = (int)(tiles < sm_count() ? tiles : sm_count());
  grid = tune_env("Q8_GRID", grid, 1, grid);
  if (p.cta2) {  // one cluster of two CTAs per work item in flight
    const long long pairs = sm_count() / 2;
    grid = 2 * (int)(tiles < pairs ? tiles : pairs);
  }
  if (p.cta2) {
    // planned only for 8-bit outputs on the 16-byte grid.  These are the large 3x3 layers, which seldom take a
    // residual: without tile buffers their kernels keep that choice at compile time.
#define Q8_PAIR_LAUNCH(GG, OUT, RES)                                                                                      \
  do {                                                                                                                   \
    if (p.scale_count == 1) return launch_variant<GG, OUT, RES, true, true>(tmA, tmB, maps, p, dyn, grid, a.stream); \
    return launch_variant<GG, OUT, RES, true, false>(tmA, tmB, maps, p, dyn, grid, a.stream);                      \
  } while (0)
#define Q8_PAIR(GG)                                                                                                      \
  do {                                                                                                                   \
    if (p.nbuf && d.y_type == Q8_U8) Q8_PAIR_LAUNCH(GG, Q8_U8, kResTma);                                                 \
    if (p.nbuf) Q8_PAIR_LAUNCH(GG, Q8_S8, kResTma);                                                                      \
    if (d.y_type == Q8_U8 && res_mode == kResVec) Q8_PAIR_LAUNCH(GG, Q8_U8, kResVec);                                    \
    if (d.y_type == Q8_U8) Q8_PAIR_LAUNCH(GG, Q8_U8, kResNone);                                                          \
    if (res_mode == kResVec) Q8_PAIR_LAUNCH(GG, Q8_S8, kResVec);                                                         \
    Q8_PAIR_LAUNCH(GG, Q8_S8, kResNone);                                                                                 \
  } while (0)
    Q8_PAIR(4);
#undef Q8_PAIR
#undef Q8_PAIR_LAUNCH
  }
  if (G == 2) return launch_groups<2>(tmA, tmB, maps, p, rows, dyn, grid, a.stream);
  return launch_groups<4>(tmA, tmB, maps, p, rows, dyn, grid, a.stream);
}
}  // namespace

}  // namespace q8

// Implicit-GEMM convolution on the sm_100a tensor cores (tcgen05.mma, accumulator in tensor memory),
// operands staged by TMA: the activation operand by im2col-mode loads straight from the NHWC tensor,
// the weight operand by tiled loads of a [C_n][taps * C_a] matrix.  One kernel serves
//   forward        Z  = omega' (*) X + b'      (Sec. 3.1 / 3.3): activation X,  weights omega'
//   backward data  dX = omega'_rot (*) dZ      (Sec. 3.2.1)    : activation dZ, weights omega' with
//                  taps flipped and channel roles swapped (stride-1 convolutions)
// GEMM view (Sec. 3.2.2): M = output pixels, N = output channels, K = taps x input channels.
//
// CTA = 11 warps: warp 0 loads the activation tiles by TMA, warp 10 the weight tiles, warp 1 owns tensor memory and issues the
// MMAs, warps 2-5 and 6-9 take the two 128 x BN fp32 accumulators in turn from tensor memory to registers, apply scale and
// bias, round to 16 bits and store.  A ring of `stages` shared-memory slots decouples loads from MMAs.  Every wait is
// bounded; a wait that gives up sets the device error word and the CTA drains and exits.
#include <mutex>

#include "kernels.h"
#include "mma_sync.cuh"
#include "packed_f32.cuh"
#include "sm100_ptx.cuh"

namespace convbn {

using namespace ptx;

constexpr int kBM = 128;       // output pixels per tile (UMMA M)
constexpr int kBK = 64;        // K elements per stage = one 128-byte swizzle row of bf16
constexpr int kUmmaK = 16;     // K per tcgen05.mma of kind::f16
constexpr int kMaxStages = 12;
constexpr int kConvThreads = 352;                             // activation TMA warp, MMA warp, 2 x 4 epilogue warps, weight TMA warp
constexpr int kWeightWarp = kConvThreads / 32 - 1;
constexpr uint32_t kStagingWarpBytes = 32 * 128;              // [32 rows][64 bf16]
constexpr uint32_t kStagingBytes = 8 * kStagingWarpBytes;     // one buffer per epilogue warp

struct ConvGemm {
    int ho, wo;              // output spatial extent
    int cn;                  // output channels (GEMM N)
    int ca;                  // activation channels (multiple of 64)
    int taps_h, taps_w;
    int nbuf;                // staging buffers per epilogue warp: 1 or 2
    int chunk_outer;         // order of K: 1: channel chunk by chunk, all taps of each; 0: tap by tap, all chunks of each
    int lower_h, lower_w;    // input coordinate read by output (0,0) at tap (0,0)
    int stride_h, stride_w, dil_h, dil_w;
    long long p;             // output pixels n * ho * wo
    int stages;
    int blockdiag;           // grouped conv as block-diagonal GEMM: tile n0 reads channels [n0, n0 + 64) only
    // Strided output (one parity class of a strided backward-data pass): pixel (img, i, j) of the
    // class goes to out_strided + img out_sn + i out_sh + j out_sw (elements).  NULL: dense TMA stores.
    __nv_bfloat16 *out_strided;
    long long out_sn;
    int out_sh, out_sw;
    // Small-C_in ("stem") mode: the activation map is a 5-D window view {64, wo, ho, r, n} of a packed,
    // zero-bordered copy of X (8 channels per pixel; 8 pixels x 8 channels = one 128-byte K row per tap
    // row r), tiles are stem_th x stem_tw output patches (stem_th * stem_tw = 128), the output map is 4-D.
    int stem, stem_tw, stem_th, stem_tiles_w, stem_tiles_h;
    int resident;            // 1: the CTA's whole weight slab [BN][K] stays in shared memory (loaded once)
    int f16;                 // 16-bit storage type: 0 bf16, 1 IEEE half
    BnFold fold;             // fold.gamma != NULL: scale and shift formed in the kernel from the BN parameters
    // Transposed convolution whose kernel is its stride (tap_c != 0): GEMM column tap tap_c + c of pixel (i, j) is channel
    // c of output pixel (i kh + r, j kw + q), tap = r kw + q, in out_strided; out_sh / out_sw are the steps of i and j,
    // tap_sh / tap_sw those of r and q.  The weight tensor is then read as it is, [ca][cn], as an MN-major operand.
    int tap_c, tap_kw, tap_sh, tap_sw;
    FastDiv by_n, by_wo, by_ho;                     // by the tiles of a row of tiles, wo, ho
    const __nv_bfloat16 *post_add, *post_mask;      // at the output's offsets
    int post_relu;
};

struct ConvSmemCtl {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    uint64_t tmem_full[2];     // MMA issuer -> epilogue, one per accumulator buffer
    uint64_t tmem_empty[2];    // epilogue -> MMA issuer (4 arrivals: one per epilogue warp)
    uint64_t bfull;            // resident weight slab has landed
    uint64_t post_full[8];     // kPost: an epilogue warp's boxes of the other tensors have landed
    uint32_t tmem_base;
    int abort_flag;
    float2 one;                // (1, 1) for mul_add2
};

// Persistent: CTA b works on tiles b, b + gridDim.x, ...; tile t covers output pixels
// [128 (t / n_tiles), +128) and output channels [BN (t % n_tiles), +BN).  The accumulator is
// double-buffered in tensor memory (2 x BN columns), so the MMAs of a tile overlap the epilogue of
// the tile before, and the TMA ring runs ahead across tile boundaries.
//
// MODE kDual (Eval mode, dense stores): Y = acc + fold.b goes to tm_out and Z = s Y + (beta - mean s), from the rounded
// Y, to tm_out2.  A pass of its own re-read Y: conv + pass took 37 us for the 64 -> 256 layer at 56 x 56, N = 32.  (An
// instantiation of its own: as a run-time branch it cost the plain kernel 40 registers, and with 168 of them no block
// of the kernels beside it fits next to a CTA: 3x3 512 -> 512 at 7 x 7, N = 64, forward + backward 85 -> 93 us.  The
// bound of 512 threads holds the plain kernel to 128 registers for the same reason.)
// MODE kTap: the transposed convolution of ConvGemm::tap_c.
// MODE kRelu: the plain kernel with max(., 0) at the end (by kPost, with its 168 registers, 64 -> 256 at 56 x 56, N = 32 took 20.4 us, now
// 16.7; 512 -> 128 at 28 x 28 9.3 and 8.2).
// MODE kPost: post_add, post_relu, post_mask follow.  A warp's [32 rows][64 columns] of the other tensors are brought into
// buffers of their own by TMA, the next one while this one is used (read from global memory beside the stores, the
// 64 -> 256 layer at 56 x 56, N = 32 took 90 us with an addend).  MODE kPostStrided: the same for strided outputs, whose
// rows are no box: read from global memory.
enum ConvMode { kPlain, kDual, kTap, kPost, kPostStrided, kRelu };
//
// PAIR: two CTAs of a cluster share a 256 x BN product (cta_group::2).  Each brings its own 128 pixels and HALF of the
// weight tile, and gets the accumulator of its own pixels; the first CTA issues the MMAs of both (see pick_tile for what that gains).
template <int BN, ConvMode MODE, bool PAIR>
__global__ void __launch_bounds__(MODE == kPlain || MODE == kRelu || MODE == kTap ? 512 : kConvThreads) umma_conv_kernel(const __grid_constant__ CUtensorMap tm_act,
                                                                const __grid_constant__ CUtensorMap tm_w,
                                                                const __grid_constant__ CUtensorMap tm_out,
                                                                const __grid_constant__ CUtensorMap tm_out2,
                                                                const __grid_constant__ CUtensorMap tm_mask,
                                                                const ConvGemm g, const float *__restrict__ bias,
                                                                int *err) {
    extern __shared__ uint8_t smem_raw[];
    constexpr bool DUAL = MODE == kDual, TAP = MODE == kTap, POST = MODE == kPost, POST_STRIDED = MODE == kPostStrided;
    constexpr uint32_t kABytes = kBM * kBK * 2, kBBytes = BN * kBK * 2 / (PAIR ? 2 : 1);
    constexpr int CTAS = PAIR ? 2 : 1;
    const uint32_t rank = PAIR ? cluster_rank() : 0u;
    const int cchunks = g.blockdiag ? 1 : g.ca / kBK;
    const int num_kb = g.taps_h * g.taps_w * cchunks;
    // Ring slots hold the activation tile and, unless the weights are resident, the weight tile.
    const uint32_t kStageBytes = g.resident ? kABytes : kABytes + kBBytes;
    uint8_t *tiles = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *slab = tiles + (size_t)g.stages * kStageBytes;            // resident weights: num_kb x [BN][64]
    uint8_t *staging = slab + (g.resident ? (size_t)num_kb * kBBytes : 0);   // 8 warps x nbuf x [32 rows][128 B]
    const int extra = POST ? (g.post_add != nullptr) + (g.post_mask != nullptr) : 0;     // staging areas of the other tensors
    ConvSmemCtl *ctl = (ConvSmemCtl *)(staging + (size_t)(g.nbuf + extra) * kStagingBytes);
    float *bias_s = (float *)(((uintptr_t)(ctl + 1) + 15) & ~(uintptr_t)15);   // cn floats
    float *scale_s = bias_s + g.cn;                                            // cn floats (fold mode)
    float *shift_s = scale_s + g.cn;                                           // cn floats (DUAL)
    const bool fold = g.fold.gamma != nullptr;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int stages = g.stages;
    const uint32_t n_tiles = g.by_n.d;
    const uint32_t m_tiles = (uint32_t)((g.p + kBM - 1) / kBM);
    const uint32_t total_tiles = (PAIR ? (m_tiles + 1) / 2 : m_tiles) * n_tiles;
    // Tile i of this CTA.  Resident weights: the CTA keeps one n-tile (blockIdx.x % n_tiles) and walks
    // m-tiles; otherwise tiles are dealt round-robin with the n-tiles of an m-tile on neighbouring CTAs.
    auto tile_of = [&](uint32_t i, uint32_t &mt, uint32_t &nt) -> bool {
        if (g.resident) {
            const uint32_t row = g.by_n.div(blockIdx.x);
            nt = blockIdx.x - row * n_tiles;
            mt = row + i * g.by_n.div(gridDim.x);
            return mt < m_tiles;
        }
        const uint32_t t = blockIdx.x / CTAS + i * (gridDim.x / CTAS);
        if (t >= total_tiles) return false;
        mt = g.by_n.div(t);
        nt = t - mt * n_tiles;
        if constexpr (PAIR) mt = 2 * mt + rank;         // (of an odd number of m-tiles the last has no partner: all out of range)
        return true;
    };
    volatile int *abort_flag = &ctl->abort_flag;
    // a pair's boxes all count on its first CTA's barriers
    const uint32_t full_of_first = PAIR ? cluster_addr(&ctl->full[0], 0) : smem_u32(&ctl->full[0]);

    // the tensor maps are kernel parameters, not data of an earlier kernel: their way to the copy engine starts at once
    if (threadIdx.x == 64) { prefetch_tensormap(&tm_act); prefetch_tensormap(&tm_w); prefetch_tensormap(&tm_out); }
    // What the first load of the activations needs is worked out beside the set-up (after it, with divisions, that load went out
    // 1100 clocks late: with the same in umma_wgrad.cu ResNet-50, N = 32 2463 -> 2426 us).
    auto pixel_of = [&](uint32_t mt, int &img, int &ho, int &wo) {
        if (g.stem) {           // m-tile -> (image, patch row, patch column)
            const uint32_t tq = mt / (uint32_t)g.stem_tiles_w;
            wo = (int)(mt - tq * (uint32_t)g.stem_tiles_w) * g.stem_tw;
            img = (int)(tq / (uint32_t)g.stem_tiles_h);
            ho = (int)(tq - (uint32_t)img * (uint32_t)g.stem_tiles_h) * g.stem_th;
        } else {
            const uint32_t m0 = (PAIR && mt >= m_tiles ? m_tiles - 1 : mt) * kBM, tq = g.by_wo.div(m0);
            wo = (int)(m0 - tq * (uint32_t)g.wo);
            img = (int)g.by_ho.div(tq);
            ho = (int)(tq - (uint32_t)img * (uint32_t)g.ho);
        }
    };
    uint32_t first_mt = 0, first_nt = 0;
    int first_img = 0, first_ho = 0, first_wo = 0;
    if (warp == 0) {
        tile_of(0, first_mt, first_nt);
        pixel_of(first_mt, first_img, first_ho, first_wo);
    }
    if (threadIdx.x == 96) {
        CONVBN_TRACE_POINT(0);
        for (int s = 0; s < stages; ++s) { mbar_init(&ctl->full[s], g.resident ? 1 : 2); mbar_init(&ctl->empty[s], 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(&ctl->tmem_full[a], 1); mbar_init(&ctl->tmem_empty[a], 4 * CTAS); }
        mbar_init(&ctl->bfull, 1);
        if constexpr (POST)
            for (int a = 0; a < 8; ++a) mbar_init(&ctl->post_full[a], 1);
        ctl->abort_flag = 0;
        ctl->one = make_float2(1.f, 1.f);
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc<CTAS>(&ctl->tmem_base, 2 * BN);
        tmem_relinquish<CTAS>();
    }
    tc_fence_before_sync();
    __syncthreads();
    if constexpr (PAIR) cluster_sync_all();                 // both CTAs' barriers and columns are there
    tc_fence_after_sync();
    // Everything above touched only this CTA's own shared / tensor memory.  Global memory (inputs that
    // an earlier kernel may still be writing, outputs it may still be reading) comes after this wait.
    pdl_wait();
    if (threadIdx.x == 0) CONVBN_TRACE_POINT(1);
    pdl_launch_dependents();       // not earlier than here: this CTA owns its tensor-memory columns
    const uint32_t tmem_base = ctl->tmem_base;
    if (threadIdx.x == 0) CONVBN_TRACE_POINT(2);

    // The first CTA's commits arrive in the second too: a loading thread sees the last of them before its CTA may exit.
    auto drain = [&](uint32_t it, bool &ok) {
        for (uint32_t j = it > (uint32_t)stages ? it - stages : 0; ok && j < it; ++j)
            ok = mbar_wait_bounded(&ctl->empty[j % stages], (j / stages) & 1u, abort_flag);
    };
    if (warp == 0) {
        // ---------------- TMA producer ----------------
        // One thread for the activations, one (of the last warp) for the weights, stepped addresses, the next slot's barrier
        // tested while this slot's load is issued, and loops unrolled by four: a taken branch back to a barrier wait costs
        // about 100 clocks, and a k-block of 128 x 64 x 64 is only 199 clocks of MMAs (267 at 128 columns).  Clocks per k-block
        // and forward time of 3x3 512 -> 512 at 7 x 7, N = 32: two lanes of one warp forming every address anew 515, 25.6 us;
        // one thread, stepped 430, 21.0; two threads 350, 18.0; tested ahead 310, 17.2; unrolled 247, 14.6.  (Before, neither
        // smaller loads nor half of them, by CTA pairs, changed the time: the chip was waiting for these loops.)
        if (elect_one()) {
            const uint32_t full0 = full_of_first, empty0 = smem_u32(&ctl->empty[0]), tiles0 = smem_u32(tiles);
            uint32_t it = 0;                         // k-blocks issued so far
            uint32_t sb = 0, slot = tiles0, ph = 1;  // ring slot: 8 x its number, its address; parity that says it is free
            const uint32_t sb_end = 8u * (uint32_t)stages;
            bool ok = true, free = false;
            uint32_t mt, nt;
            for (uint32_t i = 0; ok && tile_of(i, mt, nt); ++i) {
                const int n0 = (int)nt * BN;
                int img0 = first_img, ho0 = first_ho, wo0 = first_wo;
                if (i) pixel_of(mt, img0, ho0, wo0);
                const int base_w = g.lower_w + wo0 * g.stride_w, base_h = g.lower_h + ho0 * g.stride_h;
                // K: an inner run over the channels of a tap (or, chunk_outer, over a row of taps) with one addition a step
                const int c_first = g.blockdiag ? n0 : 0, w_end = g.taps_w * g.dil_w, h_end = g.taps_h * g.dil_h;
                const int inner = g.chunk_outer ? g.taps_w : cchunks, dc = g.chunk_outer ? 0 : kBK, dw = g.chunk_outer ? g.dil_w : 0;
                int c = c_first, off_w = 0, off_h = 0, left = inner;
#pragma unroll 4
                for (int kb = 0; kb < num_kb; ++kb) {
                    if (!free) ok = mbar_wait_bounded(empty0 + sb, ph, abort_flag);
                    if (!ok) break;
                    const uint32_t bar = full0 + sb, dst = slot;
                    ++it; sb += 8; slot += kStageBytes;
                    if (sb == sb_end) { sb = 0; slot = tiles0; ph ^= 1u; }
                    free = mbar_test_wait(empty0 + sb, ph);              // of the next slot, while this one's load is issued
                    if (rank == 0) mbar_arrive_expect_tx(bar, CTAS * kABytes);
                    if constexpr (PAIR)
                        tma_load_im2col_4d_pair(dst, &tm_act, bar, c, base_w, base_h, img0, (uint16_t)off_w, (uint16_t)off_h);
                    else if (g.stem)
                        tma_load_5d(dst, &tm_act, bar, 0, wo0, ho0, kb, img0);
                    else
                        tma_load_im2col_4d(dst, &tm_act, bar, c, base_w, base_h, img0, (uint16_t)off_w, (uint16_t)off_h);
                    c += dc; off_w += dw;
                    if (--left == 0) {
                        left = inner;
                        if (g.chunk_outer) {
                            off_w = 0;
                            if ((off_h += g.dil_h) == h_end) { off_h = 0; c += kBK; }
                        } else {
                            c = c_first;
                            if ((off_w += g.dil_w) == w_end) { off_w = 0; off_h += g.dil_h; }
                        }
                    }
                }
            }
            if constexpr (PAIR) drain(it, ok);
            if (!ok) {
                atomicOr(err, ERRW_TIMEOUT);
                ctl->abort_flag = 1;
                if constexpr (PAIR)       // counted in the first CTA as far as that has got: a millisecond is ample for any of them
                    for (const uint64_t t0 = globaltimer_ns(); globaltimer_ns() - t0 < 1000000ull;) {}
                // Let the copies already issued land (bounded) before the CTA may exit.
                const uint32_t first = it > (uint32_t)stages ? it - stages : 0;
                for (uint32_t j = first; !PAIR && j < it; ++j)
                    mbar_wait_bounded(&ctl->full[j % stages], (j / stages) & 1u, nullptr, 200000000ull);
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (rank == 0 && elect_one()) {
            // MN-major weights: 64-column blocks of [64 k][128 bytes], 8192 bytes apart; 16 k = 2048 bytes
            const uint32_t idesc = idesc_h16_f32(kBM * CTAS, BN, 0, TAP ? 1 : 0, g.f16);
            const uint32_t hi = smem_desc_hi_sw128(1024), b_lead = TAP ? 8192u : 16u;
            const uint32_t tiles_lo = smem_desc_lo(smem_u32(tiles), 16), slab_lo = smem_desc_lo(smem_u32(slab), b_lead);
            const uint32_t ring_b_lo = smem_desc_lo(smem_u32(tiles) + kABytes, b_lead);
            const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
            const bool resident = g.resident;
            auto commit = [](auto bar) {
                if constexpr (PAIR) umma_commit_pair(bar); else umma_commit(bar);
            };
            const uint32_t a_step = kStageBytes >> 4, b_step = resident ? kBBytes >> 4 : a_step, b_first = resident ? slab_lo : ring_b_lo;
            const uint32_t sb_end = 8u * (uint32_t)stages;
            uint32_t sb = 0, ph = 0, a_lo = tiles_lo, b_lo = b_first;
            bool ok = true, ready = false;
            if (resident) {
                ok = mbar_wait_bounded(&ctl->bfull, 0, abort_flag);
                tc_fence_after_sync();
            }
            uint32_t mt, nt;
            for (uint32_t i = 0; ok && tile_of(i, mt, nt); ++i) {
                const uint32_t acc = i & 1u;
                { CONVBN_TRACE_T0();
                if (!mbar_wait_bounded(&ctl->tmem_empty[acc], ((i >> 1) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
                CONVBN_TRACE_ACC(13); }
                tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + acc * BN;
                if (resident) b_lo = b_first;
#pragma unroll 4
                for (int kb = 0; kb < num_kb; ++kb) {
                    { CONVBN_TRACE_T0();
                    if (!ready && !mbar_wait_bounded(full0 + sb, ph, abort_flag)) { ok = false; break; }
                    CONVBN_TRACE_ACC(14); }
                    if (i == 0 && kb == 0) CONVBN_TRACE_POINT(4);
                    // descriptors as halves: only the start-address field (16-byte units) moves
                    const uint32_t a0 = a_lo, b0 = b_lo, done = empty0 + sb;
                    sb += 8; a_lo += a_step; b_lo += b_step;
                    if (sb == sb_end) {
                        sb = 0; ph ^= 1u; a_lo = tiles_lo;
                        if (!resident) b_lo = b_first;
                    }
                    ready = mbar_test_wait(full0 + sb, ph);              // of the next slot, while these MMAs are issued
                    umma_bf16_ss_sel<CTAS>(d_tmem, a0, hi, b0, hi, idesc, (uint32_t)kb);
#pragma unroll
                    for (int k = 1; k < kBK / kUmmaK; ++k)
                        umma_bf16_ss_halves<true, CTAS>(d_tmem, a0 + (uint32_t)k * 2u, hi, b0 + (uint32_t)k * (TAP ? 128u : 2u), hi, idesc);
                    commit(done);
                }
                if (ok) commit(&ctl->tmem_full[acc]);
                CONVBN_TRACE_POINT(6);
            }
            if (!ok) { atomicOr(err, ERRW_TIMEOUT); ctl->abort_flag = 1; }
        }
    } else if (warp == kWeightWarp) {
        // ---------------- weight loads: the CTA's resident slab once, or a tile per ring slot ----------------
        if (elect_one()) {
            const uint32_t full0 = full_of_first, empty0 = smem_u32(&ctl->empty[0]), tiles0 = smem_u32(tiles) + kABytes;
            const uint32_t sb_end = 8u * (uint32_t)stages;
            uint32_t it = 0, sb = 0, slot = tiles0, ph = 1, mt, nt;
            const int k_step = g.chunk_outer ? g.ca : kBK;
            bool ok = true, free = false;
            if (g.resident) {
                const int n0 = (int)(blockIdx.x - g.by_n.div(blockIdx.x) * n_tiles) * BN;
                mbar_arrive_expect_tx(&ctl->bfull, (uint32_t)num_kb * kBBytes);
                int k = 0;
                for (int kb = 0; kb < num_kb; ++kb) {
                    uint8_t *dst = slab + (size_t)kb * kBBytes;
                    if constexpr (TAP)
                        for (int c = 0; c < BN; c += 64) tma_load_2d(dst + c * 128, &tm_w, &ctl->bfull, n0 + c, k);
                    else
                        tma_load_2d(dst, &tm_w, &ctl->bfull, k, n0);
                    k += k_step;
                    if (k >= num_kb * kBK) k += kBK - num_kb * kBK;
                }
            } else {
                for (uint32_t i = 0; ok && tile_of(i, mt, nt); ++i) {
                    const int n0 = (int)nt * BN;
                    int k = 0;
#pragma unroll 4
                    for (int kb = 0; kb < num_kb; ++kb) {
                        if (!free) ok = mbar_wait_bounded(empty0 + sb, ph, abort_flag);
                        if (!ok) break;
                        const uint32_t bar = full0 + sb, dst = slot;
                        ++it; sb += 8; slot += kStageBytes;
                        if (sb == sb_end) { sb = 0; slot = tiles0; ph ^= 1u; }
                        free = mbar_test_wait(empty0 + sb, ph);
                        if (rank == 0) mbar_arrive_expect_tx(bar, CTAS * kBBytes);
                        if constexpr (PAIR)
                            tma_load_2d_pair(dst, &tm_w, bar, k, n0 + (int)rank * (BN / 2));
                        else if constexpr (TAP)
                            for (int cb = 0; cb < BN; cb += 64) tma_load_2d(dst + cb * 128, &tm_w, bar, n0 + cb, k);
                        else
                            tma_load_2d(dst, &tm_w, bar, k, n0);
                        k += k_step;
                        if (k >= num_kb * kBK) k += kBK - num_kb * kBK;      // (chunk_outer: the next chunk's first tap)
                    }
                }
            }
            if constexpr (PAIR) drain(it, ok);
            if (!ok) {
                atomicOr(err, ERRW_TIMEOUT);
                ctl->abort_flag = 1;
                if constexpr (PAIR)       // counted in the first CTA as far as that has got: a millisecond is ample for any of them
                    for (const uint64_t t0 = globaltimer_ns(); globaltimer_ns() - t0 < 1000000ull;) {}
                const uint32_t first = it > (uint32_t)stages ? it - stages : 0;
                for (uint32_t j = first; !PAIR && j < it; ++j)
                    mbar_wait_bounded(&ctl->full[j % stages], (j / stages) & 1u, nullptr, 200000000ull);
            }
        }
    } else {
        // ---------------- epilogue: tensor memory -> registers -> bf16 -> shared -> TMA store --------
        // Two groups of four warps; group e drains accumulator buffer e, i.e. every other tile of this
        // CTA, so two tiles are in their epilogue at once; the last tile is halved between them, from 128 columns on.  Each warp
        // owns 32 accumulator rows and one or two
        // private [32 rows][64 columns] staging buffers (128-byte swizzle): warp-level sync only.
        // First the per-channel parameters, by these warps alone: the loads and the first MMAs do not wait for them.
        const int pc = TAP ? g.tap_c : g.cn;               // channels the per-channel parameters belong to
        if constexpr (DUAL) {
            for (int c = (int)threadIdx.x - 64; c < g.cn; c += 256) {
                const float sc = g.fold.gamma[c] * (1.0f / sqrtf(g.fold.var[c] + g.fold.eps));
                bias_s[c] = g.fold.b ? g.fold.b[c] : 0.f;
                scale_s[c] = sc;
                shift_s[c] = g.fold.beta[c] - g.fold.mean[c] * sc;
            }
        } else if (fold) {
            // On-the-fly reparameterisation (Sec. 3.3 / 3.4): s = gamma / sqrt(var + eps), b' = (b - mu) s + beta.
            // s multiplies the fp32 accumulator (the associative law of Sec. 3.2.2), so omega is used unrounded.
            for (int c = (int)threadIdx.x - 64; c < pc; c += 256) {
                const float r = 1.0f / sqrtf(g.fold.var[c] + g.fold.eps);
                const float sc = g.fold.gamma[c] * r;
                const float bf = ((g.fold.b ? g.fold.b[c] : 0.f) - g.fold.mean[c]) * sc + g.fold.beta[c];
                scale_s[c] = sc;
                bias_s[c] = bf;
                if (blockIdx.x == 0 && g.fold.vec3) {
                    g.fold.vec3[c] = sc; g.fold.vec3[pc + c] = bf; g.fold.vec3[2 * pc + c] = r;
                }
            }
        } else {
            // (scale 1 and shift -0 leave every value as it is, so the epilogue has one form)
            for (int c = (int)threadIdx.x - 64; c < g.cn; c += 256) { scale_s[c] = 1.f; bias_s[c] = bias ? bias[c] : -0.f; }
        }
        named_bar_sync(1, 256);
        const int quarter = warp & 3;                      // tensor-memory lanes this warp may read
        const uint32_t egroup = (uint32_t)(warp - 2) >> 2; // 0: warps 2-5, 1: warps 6-9
        uint8_t *stage_buf = staging + (size_t)(warp - 2) * kStagingWarpBytes;
        // The accumulator is read as matrix fragments: this lane gets columns 8 i + 2 (lane % 4) and the next of rows lane / 4 and
        // lane / 4 + 8 of every 16, so the parameters of a 64-column chunk are 16 values of each kind, read while the accumulator
        // is on its way, and stmatrix writes the swizzled rows.  (A row per lane needs the parameters of all 64 columns in every
        // lane, 32 16-byte loads: a chunk took 1550 clocks instead of 1040; forward + backward of the transposed 2x2 256 -> 128 layer
        // at 56 x 56, N = 8 62.0 -> 57.7 us, Eval 64 -> 256 at 56 x 56, N = 32 94.4 -> 84.1, ResNet-50, N = 32 2586 -> 2512.)
        const uint32_t shift_at = smem_u32(bias_s) + (uint32_t)(lane & 3) * 8u, scale_at = shift_at + (uint32_t)g.cn * 4u;
        // stmatrix: lanes 8 m to 8 m + 7 name the rows of matrix m; matrices 0, 1: rows 0-7, 8-15, matrices 2, 3: the next 8 columns
        const uint32_t frag_row = (uint32_t)((lane & 7) + (lane & 8)) * 128u, frag_chunk = (uint32_t)(((lane >> 4) ^ (lane & 7)) << 4);
        // the buffer for the next box: the last store from it has been read, an earlier one (nbuf = 2) may still be under way
        uint32_t turn = 0;
        auto next_buf = [&]() -> uint8_t * {
            if (lane == 0) { if ((MODE == kPlain || MODE == kRelu) && g.nbuf == 2) tma_store_wait_read<1>(); else tma_store_wait_read<0>(); }
            __syncwarp();
            uint8_t *b = stage_buf + turn;
            if ((MODE == kPlain || MODE == kRelu) && g.nbuf == 2) turn ^= kStagingBytes;
            return b;
        };
        const f32x2 one = lds_f32x2(smem_u32(&ctl->one));
        uint32_t mt, nt;
        // kPost: tm_out2 is the addend's map.  One box of each tensor in flight per warp.
        uint8_t *add_buf = staging + (size_t)g.nbuf * kStagingBytes + (size_t)(warp - 2) * kStagingWarpBytes, *mask_buf = add_buf + (g.post_add ? kStagingBytes : 0);
        uint32_t post_ph = 0;
        bool post_pending = false;
        // Columns [lo, hi) of tile i are this group's: the groups take tiles in turn, and halve the last one, which nothing is
        // left to overlap with (forward + backward of 3x3 stride 2 128 -> 128 at 200 x 334, N = 2 58.9 -> 57.4 us,
        // ResNet-50, N = 32 2480 -> 2463).
        auto columns_of = [&](uint32_t i, uint32_t &m, uint32_t &n, int &lo, int &hi) -> bool {
            if (!tile_of(i, m, n)) return false;
            const bool own = (i & 1u) == egroup;
            uint32_t m2, n2;
            if (BN >= 128 && !tile_of(i + 1, m2, n2)) { lo = own ? 0 : BN / 2; hi = lo + BN / 2; }
            else { lo = 0; hi = own ? BN : 0; }
            const int valid = g.cn - (int)n * BN;
            if (hi > valid) hi = valid;
            return true;
        };
        auto fetch_post = [&](uint32_t m, uint32_t n, int c0) {
            post_pending = extra > 0;
            if (!post_pending || lane != 0) return;
            uint64_t *bar = &ctl->post_full[warp - 2];
            mbar_arrive_expect_tx(bar, (uint32_t)extra * kStagingWarpBytes);
            const int x = (int)n * BN + c0, y = (int)(m * kBM) + quarter * 32;
            if (g.post_add) tma_load_2d(add_buf, &tm_out2, bar, x, y);
            if (g.post_mask) tma_load_2d(mask_buf, &tm_mask, bar, x, y);
        };
        auto fetch_from = [&](uint32_t i) {                   // the first chunk of this group's next tile, from tile i on
            uint32_t m, n;
            int lo, hi;
            post_pending = false;
            for (; columns_of(i, m, n, lo, hi); ++i)
                if (lo < hi) { fetch_post(m, n, lo); return; }
        };
        if constexpr (POST) fetch_from(0);
        int c_lo, c_hi;
        for (uint32_t i = 0; columns_of(i, mt, nt, c_lo, c_hi); ++i) {
            if (c_lo >= c_hi) continue;
            const uint32_t acc = i & 1u;
            // (the other group's buffer, for the last tile: this group has drained tile i - 1, whose products were complete
            // after those of tile i - 2, so the barrier is past that earlier phase of the same parity)
            CONVBN_TRACE_T0();
            const bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(&ctl->tmem_full[acc], (i >> 1) & 1u, abort_flag));
            if (warp == 2 && lane == 0) CONVBN_TRACE_ACC(15);
            if (!ok) {
                if (lane == 0) { atomicOr(err, ERRW_TIMEOUT); ctl->abort_flag = 1; }
                break;
            }
            tc_fence_after_sync();
            const uint32_t m0 = mt * kBM;
            const int n0 = (int)nt * BN;
            const uint32_t t_row = tmem_base + acc * BN + ((uint32_t)(quarter * 32) << 16);
            __nv_bfloat16 *srow = nullptr;                  // strided mode: this thread's output pixel
            if (g.out_strided) {
                const uint32_t m = m0 + quarter * 32 + lane;
                if ((long long)m < g.p) {
                    const uint32_t tq = g.by_wo.div(m), img = g.by_ho.div(tq);
                    srow = g.out_strided + (size_t)img * g.out_sn + (size_t)(tq - img * (uint32_t)g.ho) * g.out_sh +
                           (size_t)(m - tq * (uint32_t)g.wo) * g.out_sw;
                    if constexpr (TAP) {                    // (a tile lies inside one tap: BN divides tap_c)
                        const int tap = n0 / g.tap_c, tr = tap / g.tap_kw;
                        srow += (size_t)tr * g.tap_sh + (size_t)(tap - tr * g.tap_kw) * g.tap_sw + (n0 - tap * g.tap_c);
                    } else {
                        srow += n0;
                    }
                }
            }
            const int p0 = TAP ? n0 % g.tap_c : n0;         // first per-channel parameter of this tile
#pragma unroll 1
            for (int c0 = c_lo; c0 < c_hi; c0 += 64) {
                uint32_t v[2][32];                          // rows 0-15 and 16-31 of this warp
                f32x2 sc[4], sh[4];                         // parameters of 32 columns
                auto params = [&](int i0, uint32_t sc_at, uint32_t sh_at) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        sh[i] = lds_f32x2(sh_at + (uint32_t)(p0 + c0 + 8 * (i0 + i)) * 4u);
                        if (sc_at) sc[i] = lds_f32x2(sc_at + (uint32_t)(p0 + c0 + 8 * (i0 + i)) * 4u);
                    }
                };
                tmem_ld_16x64(t_row + (uint32_t)c0, v[0]);
                tmem_ld_16x64(t_row + (16u << 16) + (uint32_t)c0, v[1]);
                params(0, DUAL ? 0u : scale_at, shift_at);
                tmem_ld_wait();
                if (c0 + 64 >= c_hi && acc == egroup) {
                    // every column of this accumulator has been read: hand the buffer back (nobody waits for the last one)
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) {
                        if constexpr (PAIR) mbar_arrive_cluster(cluster_addr(&ctl->tmem_empty[acc], 0));
                        else mbar_arrive(&ctl->tmem_empty[acc]);
                    }
                }
                {
                    uint8_t *buf = next_buf();
                    const uint32_t frag = smem_u32(buf) + frag_row;
                    if constexpr (POST) {
                        if (post_pending) {
                            const bool here = mbar_wait_bounded(&ctl->post_full[warp - 2], post_ph, abort_flag);
                            post_ph ^= 1u;
                            if (!here && lane == 0) { atomicOr(err, ERRW_TIMEOUT); ctl->abort_flag = 1; }
                            __syncwarp();
                        }
                    }
                    // (what follows the rounding is fixed outside the loop over the columns: one uniform branch per chunk)
                    auto pack_rows = [&](auto half_tag, auto add_tag, auto relu_tag, auto mask_tag) {
                        constexpr bool H = decltype(half_tag)::value, ADD = decltype(add_tag)::value;
                        constexpr bool RELU = decltype(relu_tag)::value, MASK = decltype(mask_tag)::value;
#pragma unroll
                        for (int i = 0; i < 8; i += 2) {
                            if (i == 4) params(4, DUAL ? 0u : scale_at, shift_at);
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                uint32_t o[4];                 // columns 8 i and 8 i + 8: rows 0-7, 8-15 of each
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    const uint32_t *q = &v[h][(i + (e >> 1)) * 4 + (e & 1) * 2];
                                    const f32x2 f = pair(__uint_as_float(q[0]), __uint_as_float(q[1]));
                                    const f32x2 shift = sh[(i & 3) + (e >> 1)];
                                    o[e] = narrow_t<H>(DUAL ? fma2(f, one, shift) : mul_add2(f, sc[(i & 3) + (e >> 1)], shift, one));
                                    if constexpr (MODE == kRelu) o[e] = post_pair<H>(o[e], false, 0u, true, false, 0u);
                                }
                                const uint32_t at16 = (uint32_t)h * 2048u + (((uint32_t)i << 4) ^ frag_chunk);
                                if constexpr (POST) {
                                    uint32_t a[4] = {0u, 0u, 0u, 0u}, m[4] = {0u, 0u, 0u, 0u};
                                    if constexpr (ADD) ldmatrix_x4(a[0], a[1], a[2], a[3], smem_u32(add_buf) + frag_row + at16);
                                    if constexpr (MASK) ldmatrix_x4(m[0], m[1], m[2], m[3], smem_u32(mask_buf) + frag_row + at16);
#pragma unroll
                                    for (int e = 0; e < 4; ++e) o[e] = post_pair<H>(o[e], ADD, a[e], RELU, MASK, m[e]);
                                }
                                stmatrix_x4(frag + at16, o[0], o[1], o[2], o[3]);
                                if constexpr (DUAL) {          // kept for the second output, in the accumulator's registers
#pragma unroll
                                    for (int e = 0; e < 4; ++e) v[h][i * 2 + e] = o[e];
                                }
                            }
                        }
                    };
                    auto pack = [&](auto add_tag, auto relu_tag, auto mask_tag) {
                        if (g.f16) pack_rows(std::true_type{}, add_tag, relu_tag, mask_tag);
                        else pack_rows(std::false_type{}, add_tag, relu_tag, mask_tag);
                    };
                    constexpr std::true_type yes{};
                    constexpr std::false_type no{};
                    if constexpr (!POST) pack(no, no, no);
                    else if (g.post_mask) { if (g.post_add) pack(yes, no, yes); else pack(no, no, yes); }
                    else if (g.post_relu) pack(yes, yes, no);
                    else pack(yes, no, no);
                    if constexpr (POST) {
                        __syncwarp();                          // every lane has read its rows of the boxes
                        if (c0 + 64 < c_hi) fetch_post(mt, nt, c0 + 64); else fetch_from(i + 1);
                    }
                    if constexpr (POST_STRIDED) {
                        // as below, with the other tensors' values of four pixels requested before the first is used
                        __syncwarp();
                        const int ch = lane & 7;
#pragma unroll 1
                        for (int i0 = 0; i0 < 8; i0 += 4) {
                            uint4 av[4], mv[4];
                            ptrdiff_t at8[4];
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const __nv_bfloat16 *dst = (const __nv_bfloat16 *)__shfl_sync(
                                    0xffffffffu, (unsigned long long)srow, (i0 + k) * 4 + (lane >> 3));
                                const bool on = dst && c0 + ch * 8 < c_hi;
                                at8[k] = on ? dst - g.out_strided + c0 + ch * 8 : -1;
                                av[k] = mv[k] = make_uint4(0u, 0u, 0u, 0u);
                                if (on && g.post_add) av[k] = *(const uint4 *)(g.post_add + at8[k]);
                                if (on && g.post_mask) mv[k] = *(const uint4 *)(g.post_mask + at8[k]);
                            }
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const int rr = (i0 + k) * 4 + (lane >> 3);
                                const uint4 q = *(const uint4 *)(buf + rr * 128 + (((ch ^ (rr & 7)) & 7) << 4));
                                const uint4 o = g.f16 ? post_chunk<true>(q, g.post_add, av[k], g.post_relu, g.post_mask, mv[k])
                                                      : post_chunk<false>(q, g.post_add, av[k], g.post_relu, g.post_mask, mv[k]);
                                if (at8[k] >= 0) *(uint4 *)(g.out_strided + at8[k]) = o;
                            }
                        }
                        __syncwarp();
                        continue;
                    }
                    if (TAP || g.out_strided) {
                        // eight lanes write the 128 bytes of a pixel, four pixels per instruction
                        __syncwarp();
#pragma unroll 2
                        for (int it = 0; it < 8; ++it) {
                            const int rr = it * 4 + (lane >> 3), ch = lane & 7;
                            __nv_bfloat16 *dst = (__nv_bfloat16 *)__shfl_sync(0xffffffffu, (unsigned long long)srow, rr);
                            const uint4 q = *(const uint4 *)(buf + rr * 128 + (((ch ^ (rr & 7)) & 7) << 4));
                            if (dst && c0 + ch * 8 < c_hi) *(uint4 *)(dst + c0 + ch * 8) = q;
                        }
                        __syncwarp();
                        continue;
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        if (g.stem) {
                            // this warp's 32 accumulator rows are (32 / stem_tw) patch rows of stem_tw pixels
                            const uint32_t tq2 = mt / (uint32_t)g.stem_tiles_w, im2 = tq2 / (uint32_t)g.stem_tiles_h;
                            tma_store_4d(&tm_out, buf, n0 + c0, (int)(mt - tq2 * (uint32_t)g.stem_tiles_w) * g.stem_tw,
                                         (int)(tq2 - im2 * (uint32_t)g.stem_tiles_h) * g.stem_th + quarter * (32 / g.stem_tw),
                                         (int)im2);
                        } else {
                            tma_store_2d(&tm_out, buf, n0 + c0, (int)(m0 + quarter * 32));
                        }
                        tma_store_commit();
                    }
                    if constexpr (DUAL) {
                        buf = next_buf();
                        const uint32_t frag2 = smem_u32(buf) + frag_row;
                        auto normalise = [&](auto half_tag) {
                            constexpr bool H = decltype(half_tag)::value;
#pragma unroll
                            for (int i = 0; i < 8; i += 2) {
                                if ((i & 3) == 0) params(i, scale_at, scale_at + (uint32_t)g.cn * 4u);
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    uint32_t o[4];
#pragma unroll
                                    for (int e = 0; e < 4; ++e)
                                        o[e] = narrow_t<H>(fma2(widen_t<H>(v[h][i * 2 + e]), sc[(i & 3) + (e >> 1)], sh[(i & 3) + (e >> 1)]));
                                    stmatrix_x4(frag2 + (uint32_t)h * 2048u + (((uint32_t)i << 4) ^ frag_chunk), o[0], o[1], o[2], o[3]);
                                }
                            }
                        };
                        if (g.f16) normalise(std::true_type{}); else normalise(std::false_type{});
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            tma_store_2d(&tm_out2, buf, n0 + c0, (int)(m0 + quarter * 32));
                            tma_store_commit();
                        }
                    }
                }
            }
        }
        if (warp == 2 && lane == 0) CONVBN_TRACE_POINT(9);
        if constexpr (POST)                                 // (after a give-up: let the boxes in flight land)
            if (post_pending) mbar_wait_bounded(&ctl->post_full[warp - 2], post_ph, nullptr, 200000000ull);
        if (lane == 0) tma_store_wait_all<0>();             // global writes done before the CTA exits
        if (warp == 2 && lane == 0) CONVBN_TRACE_POINT(10);
    }
    tc_fence_before_sync();
    __syncthreads();
    if constexpr (PAIR) cluster_sync_all();                 // neither CTA's barriers, tiles or columns are in use any more
    if (threadIdx.x == 0) CONVBN_TRACE_POINT(11);
    if (warp == 1) tmem_dealloc<CTAS>(tmem_base, 2 * BN);
}

// ---- failure-path self-test: the bounded wait of the kernels above, on a barrier nobody completes --------
__global__ void selftest_wait_timeout_kernel(unsigned long long limit_ns, int *err) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_barrier_init();
        if (!mbar_wait_bounded(&bar, 0, nullptr, limit_ns)) atomicOr(err, ERRW_TIMEOUT);
    }
}

cudaError_t launch_selftest_wait_timeout(unsigned long long limit_ns, cudaStream_t st) {
    int *err = nullptr;
    cudaError_t e = error_word_address(&err);
    if (e != cudaSuccess) return e;
    selftest_wait_timeout_kernel<<<1, 32, 0, st>>>(limit_ns, err);
    return cudaGetLastError();
}

// ---- host side: tensor maps and launch ---------------------------------------------------------
namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
typedef CUresult (*EncodeIm2colFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const int *, const int *, cuuint32_t, cuuint32_t,
                                   const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode_tiled = nullptr;
EncodeIm2colFn g_encode_im2col = nullptr;
std::once_flag g_encode_once;

bool load_encoders() {
    std::call_once(g_encode_once, [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode_tiled = (EncodeTiledFn)f;
        f = nullptr;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeIm2col", &f, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode_im2col = (EncodeIm2colFn)f;
    });
    return g_encode_tiled && g_encode_im2col;
}

}  // namespace

// bf16 row-major matrix [rows][cols] -> box of box_rows x 64 columns, 128-byte swizzle.
bool make_tmap_matrix_bf16(CUtensorMap *tm, const void *base, long long rows, long long cols, int box_rows,
                           int box_cols) {
    if (!load_encoders()) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return g_encode_tiled(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box,
                          estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// NHWC bf16 tensor [n][h][w][c] -> im2col-mode map: `pixels` consecutive output positions x 64 channels
// per load, 128-byte swizzle, zero fill outside the image.
bool make_tmap_im2col_bf16(CUtensorMap *tm, const void *base, int n, int h, int w, int c, int lower_h,
                           int lower_w, int upper_h, int upper_w, int stride_h, int stride_w, int pixels,
                           int channels) {
    if (!load_encoders()) return false;
    cuuint64_t dims[4] = {(cuuint64_t)c, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)n};
    cuuint64_t strides[3] = {(cuuint64_t)c * 2, (cuuint64_t)w * c * 2, (cuuint64_t)h * w * c * 2};
    int lower[2] = {lower_w, lower_h};
    int upper[2] = {upper_w, upper_h};
    cuuint32_t estr[4] = {1, (cuuint32_t)stride_w, (cuuint32_t)stride_h, 1};
    return g_encode_im2col(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides, lower,
                           upper, (cuuint32_t)channels, (cuuint32_t)pixels, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static bool encode_tiled_bf16(CUtensorMap *tm, const void *base, int rank, const unsigned long long *dims,
                              const unsigned long long *strides_bytes, const unsigned int *box, CUtensorMapSwizzle sw) {
    if (!load_encoders() || rank < 1 || rank > 5) return false;
    cuuint64_t d[5], st[4];
    cuuint32_t bx[5], es[5];
    for (int i = 0; i < rank; ++i) { d[i] = dims[i]; bx[i] = box[i]; es[i] = 1; }
    for (int i = 1; i < rank; ++i) st[i - 1] = strides_bytes[i];
    return g_encode_tiled(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void *>(base), d, st, bx,
                          es, CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_tmap_tiled_bf16(CUtensorMap *tm, const void *base, int rank, const unsigned long long *dims,
                          const unsigned long long *strides_bytes, const unsigned int *box) {
    return encode_tiled_bf16(tm, base, rank, dims, strides_bytes, box, CU_TENSOR_MAP_SWIZZLE_128B);
}

bool make_tmap_tiled_bf16_linear(CUtensorMap *tm, const void *base, int rank, const unsigned long long *dims,
                                 const unsigned long long *strides_bytes, const unsigned int *box) {
    return encode_tiled_bf16(tm, base, rank, dims, strides_bytes, box, CU_TENSOR_MAP_SWIZZLE_NONE);
}

bool umma_conv_eligible(const UmmaConvShape &s) {
    if (s.ca % kBK || s.cn % 8 || s.cn < 64 || s.cn > 4096) return false;
    if (s.blockdiag && (s.ca != s.cn)) return false;
    if (s.lower_h < -128 || s.lower_h > 127 || s.lower_w < -128 || s.lower_w > 127) return false;
    if ((s.taps_h - 1) * s.dil_h > 255 || (s.taps_w - 1) * s.dil_w > 255) return false;
    if (s.stride_h > 8 || s.stride_w > 8) return false;
    if ((long long)s.taps_h * s.taps_w * s.ca > (1 << 24)) return false;
    if ((long long)s.n * s.ho * s.wo >= (1LL << 31) - 256) return false;
    return true;
}

static int sm_count() { return device_sm_count(); }

template <int BN, ConvMode MODE = kPlain, bool PAIR = false>
static cudaError_t launch_bn(const CUtensorMap &ta, const CUtensorMap &tw, const CUtensorMap &tout,
                             const CUtensorMap &tout2, const CUtensorMap &tmask, ConvGemm g, const float *bias, int *err,
                             cudaStream_t st) {
    const size_t a_bytes = (size_t)kBM * kBK * 2, b_bytes = (size_t)BN * kBK * 2 / (PAIR ? 2 : 1);
    const int extra = MODE == kPost ? (g.post_add != nullptr) + (g.post_mask != nullptr) : 0;
    const int num_kb = g.taps_h * g.taps_w * (g.blockdiag ? 1 : g.ca / kBK);
    // Short K: the epilogues bound the kernel, and the second buffer is worth more than the ring slots it takes (1x1 256 -> 64
    // at 56 x 56, N = 256, forward 86.4 -> 82.6 us; the other modes, with staging areas of their own, gain nothing).
    g.nbuf = (MODE == kPlain || MODE == kRelu) && num_kb <= 8 ? 2 : 1;
    // (256: the epilogue reads the per-channel parameters of whole 64-column chunks)
    size_t fixed = 1024 + 256 + (size_t)(g.nbuf + extra) * kStagingBytes + sizeof(ConvSmemCtl) + (MODE == kDual ? 3 : 2) * (size_t)g.cn * sizeof(float) + 16;
    const long long m_tiles = (g.p + kBM - 1) / kBM, n_tiles = (g.cn + BN - 1) / BN;
    g.by_n = FastDiv((uint32_t)n_tiles); g.by_wo = FastDiv((uint32_t)g.wo); g.by_ho = FastDiv((uint32_t)g.ho);
    long long grid_l = m_tiles * n_tiles < sm_count() ? m_tiles * n_tiles : sm_count();
    if (PAIR) {
        const long long pairs = (m_tiles + 1) / 2 * n_tiles;
        grid_l = 2 * (pairs < sm_count() / 2 ? pairs : sm_count() / 2);
    }
    // Weights stay resident when the CTA's slab fits beside at least four activation slots and the
    // grid can give every CTA one fixed n-tile.
    const size_t slab = (size_t)num_kb * b_bytes;
    g.resident = 0;
    if (!PAIR && slab <= 104 * 1024 && fixed + slab + 4 * a_bytes <= 220 * 1024 && m_tiles * n_tiles >= sm_count() &&
        n_tiles <= sm_count()) {
        g.resident = 1;
        grid_l = sm_count() - sm_count() % n_tiles;
        fixed += slab;
    }
    const size_t stage = g.resident ? a_bytes : a_bytes + b_bytes;
    int stages = (int)((220 * 1024 - fixed) / stage);  // one CTA per SM owns the shared memory
    if (stages > kMaxStages) stages = kMaxStages;
    g.stages = stages;
    const size_t smem = stages * stage + fixed;
    static PerDevice attr_done;
    if (cudaError_t e = max_dynamic_smem_once(umma_conv_kernel<BN, MODE, PAIR>, 224 * 1024, &attr_done); e != cudaSuccess) return e;
    static PerDevice carve;
    prefer_max_shared_once(umma_conv_kernel<BN, MODE, PAIR>, &carve);
    const unsigned grid = (unsigned)grid_l;
    return launch_pdl<PAIR ? 2 : 1>(umma_conv_kernel<BN, MODE, PAIR>, dim3(grid), dim3(kConvThreads), smem, st, ta, tw, tout, tout2, tmask, g, bias, err);
}

template <ConvMode MODE>
static cudaError_t launch_mode(int bn, bool pair, const CUtensorMap &ta, const CUtensorMap &tw, const CUtensorMap &tout,
                               const CUtensorMap &tout2, const CUtensorMap &tmask, const ConvGemm &g, const float *bias,
                               int *err, cudaStream_t st) {
    if constexpr (MODE == kPlain || MODE == kRelu || MODE == kPost) {
        if (pair && bn == 64) return launch_bn<64, MODE, true>(ta, tw, tout, tout2, tmask, g, bias, err, st);
        if (pair && bn == 128) return launch_bn<128, MODE, true>(ta, tw, tout, tout2, tmask, g, bias, err, st);
        if (pair) return launch_bn<256, MODE, true>(ta, tw, tout, tout2, tmask, g, bias, err, st);
    }
    if (bn == 64) return launch_bn<64, MODE>(ta, tw, tout, tout2, tmask, g, bias, err, st);
    if (bn == 128) return launch_bn<128, MODE>(ta, tw, tout, tout2, tmask, g, bias, err, st);
    return launch_bn<256, MODE>(ta, tw, tout, tout2, tmask, g, bias, err, st);
}

// Tile width, and whether CTAs work in pairs: the least time by a model of clocks fitted to 24 layers (3x3 and 1x1, 64 to 2048
// channels, N = 8 to 256, both directions) at all six choices.  A round of tiles takes the larger of its k-blocks and its
// epilogue (1x1 64 -> 256 at 56 x 56, N = 256: 83.7 us with 128 columns, 96.5 with 256); the last tile's epilogue and a pair's
// start-up (a cluster launch, two CTAs meeting twice) come on top.  A k-block costs a CTA of a pair 20 to 90 clocks less, being
// half a weight tile to write to and read from shared memory, so pairs pay for long K or many rounds (1x1 512 -> 1024 at 28 x
// 28, N = 32 28.6 us alone with 128 columns, 22.7 in pairs with 256; 64 -> 64 at 56 x 56, N = 8 3.7 alone, 4.6 in pairs).  The
// terms of the epilogue date from one that took 1.5 times as long: over 112 passes (the layers above, also at N = 64) the
// choice is now 3 % from the best on average, and furthest where wide pairs win (1x1 512 -> 256 at 14 x 14, N = 256 18.1 us and
// 13.4).
struct TilePick { int bn; bool pair; };
static TilePick pick_tile(long long tiles_m, int cn, int num_kb, bool pairs, int max_bn) {
    static const double clk[2][3] = {{645, 300, 260}, {555, 280, 205}};
    TilePick best{64, false};
    double best_cost = 1e30;
    for (int pr = 0; pr <= (pairs ? 1 : 0); ++pr)
        for (int c = 0; c < 3; ++c) {
            const int bn = 256 >> c;
            if (bn > max_bn || (bn > 64 && cn <= bn / 2)) continue;
            const long long n_tiles = (cn + bn - 1) / bn, slots = pr ? sm_count() / 2 : sm_count();
            const long long rounds = ((pr ? (tiles_m + 1) / 2 : tiles_m) * n_tiles + slots - 1) / slots;
            const double mma = num_kb * clk[pr][c], epi = bn * (bn == 64 ? 17.0 : (bn == 128 ? 14.7 : 16.0));
            const double cost = (double)rounds * ((mma > epi ? mma : epi) + 220.0) + 6.0 * bn + (pr ? 1900.0 : 0.0);
            if (cost < best_cost) { best_cost = cost; best = TilePick{bn, pr != 0}; }
        }
    return best;
}

cudaError_t launch_umma_conv(const UmmaConvShape &s, const void *act, const void *wmat, const float *bias,
                             void *out, cudaStream_t st, const BnFold *fold, void *out2, const PostOp *post) {
    ConvGemm g;
    g.ho = s.ho; g.wo = s.wo; g.cn = s.cn; g.ca = s.ca; g.taps_h = s.taps_h; g.taps_w = s.taps_w;
    g.lower_h = s.lower_h; g.lower_w = s.lower_w; g.stride_h = s.stride_h; g.stride_w = s.stride_w;
    g.dil_h = s.dil_h; g.dil_w = s.dil_w; g.p = (long long)s.n * s.ho * s.wo; g.stages = 1;
    g.blockdiag = s.blockdiag;
    g.chunk_outer = umma_strip_possible(s);              // the strip kernel's order, so that results do not depend on the choice
    g.f16 = call_f16();
    g.stem = 0; g.stem_tw = g.stem_th = g.stem_tiles_w = g.stem_tiles_h = 1;
    g.fold = fold ? *fold : BnFold{nullptr, nullptr, nullptr, nullptr, nullptr, 0.f, nullptr};
    g.out_strided = s.out_sw ? (__nv_bfloat16 *)out : nullptr;
    g.out_sn = s.out_sn; g.out_sh = s.out_sh; g.out_sw = s.out_sw;
    const bool with_post = post && post->any();
    g.post_add = with_post ? (const __nv_bfloat16 *)post->add : nullptr;
    g.post_mask = with_post ? (const __nv_bfloat16 *)post->mask : nullptr;
    g.post_relu = with_post ? post->relu : 0;
    g.tap_c = s.tap_c; g.tap_kw = s.tap_kw; g.tap_sh = s.tap_sh; g.tap_sw = s.tap_sw;
    // The bounding box of base pixels has ho x wo positions: upper = lower + (out-1) stride - (in-1).
    const int upper_h = s.lower_h + (s.ho - 1) * s.stride_h - (s.ha - 1);
    const int upper_w = s.lower_w + (s.wo - 1) * s.stride_w - (s.wa - 1);
    const long long tiles_m = (g.p + kBM - 1) / kBM;
    int max_bn = s.blockdiag ? 64 : 256;
    while (s.tap_c && s.tap_c % max_bn) max_bn /= 2;     // a tile lies inside one tap
    if (!s.out_sw && (g.post_add || g.post_mask) && max_bn > 128) max_bn = 128;       // room for the other tensors' staging areas
    const bool pairs = !s.blockdiag && !s.tap_c && !out2 && !(with_post && s.out_sw);
    const TilePick pick = pick_tile(tiles_m, s.cn, s.taps_h * s.taps_w * (s.blockdiag ? 1 : s.ca / kBK), pairs, max_bn);
    const int bn = pick.bn;
    const bool pair = pick.pair;
    CUtensorMap ta, tw, tout;
    // (in strided mode the output map is encoded but never used: every row is stored by its thread)
    if (!make_tmap_matrix_bf16(&tout, out, s.out_sw ? 32 : g.p, s.cn, 32, 64)) return cudaErrorInvalidValue;
    if (!make_tmap_im2col_bf16(&ta, act, s.n, s.ha, s.wa, s.ca, s.lower_h, s.lower_w, upper_h, upper_w, s.stride_h,
                               s.stride_w, kBM, kBK))
        return cudaErrorInvalidValue;
    if (s.tap_c ? !make_tmap_matrix_bf16(&tw, wmat, s.ca, s.cn, kBK, 64)
                : !make_tmap_matrix_bf16(&tw, wmat, s.cn, (long long)s.taps_h * s.taps_w * (s.blockdiag ? 64 : s.ca), pair ? bn / 2 : bn, kBK))
        return cudaErrorInvalidValue;
    int *err = nullptr;
    cudaError_t e = error_word_address(&err);
    if (e != cudaSuccess) return e;
    CUtensorMap tout2 = tout;
    if (out2 && !make_tmap_matrix_bf16(&tout2, out2, g.p, s.cn, 32, 64)) return cudaErrorInvalidValue;
    CUtensorMap tmask = tout;
    if (with_post && !s.out_sw) {
        if (g.post_add && !make_tmap_matrix_bf16(&tout2, post->add, g.p, s.cn, 32, 64)) return cudaErrorInvalidValue;
        if (g.post_mask && !make_tmap_matrix_bf16(&tmask, post->mask, g.p, s.cn, 32, 64)) return cudaErrorInvalidValue;
        if (!g.post_add && !g.post_mask) return launch_mode<kRelu>(bn, pair, ta, tw, tout, tout2, tmask, g, bias, err, st);
        return launch_mode<kPost>(bn, pair, ta, tw, tout, tout2, tmask, g, bias, err, st);
    }
    if (with_post) return launch_mode<kPostStrided>(bn, pair, ta, tw, tout, tout2, tmask, g, bias, err, st);
    if (out2) return launch_mode<kDual>(bn, pair, ta, tw, tout, tout2, tmask, g, bias, err, st);
    if (g.tap_c) return launch_mode<kTap>(bn, pair, ta, tw, tout, tout2, tmask, g, bias, err, st);
    return launch_mode<kPlain>(bn, pair, ta, tw, tout, tout2, tmask, g, bias, err, st);
}

// Forward pass of a small-C_in layer on the packed input (see stem_kernels.cu): tiles of 8 x 16 output
// pixels, K = stem_krows rows of 64, weights resident.
cudaError_t launch_stem_fwd(const Problem &pb, const void *x_packed, const void *wst, const float *bias, void *out,
                            cudaStream_t st, const BnFold *fold) {
    const int krows = stem_krows(pb);
    ConvGemm g;
    g.chunk_outer = 0;
    g.tap_c = 0; g.post_add = g.post_mask = nullptr; g.post_relu = 0;
    g.ho = pb.h_out; g.wo = pb.w_out; g.cn = pb.c_out; g.ca = 64; g.taps_h = krows; g.taps_w = 1;
    g.lower_h = g.lower_w = 0; g.stride_h = g.stride_w = g.dil_h = g.dil_w = 1;
    g.stem = 1; g.stem_tw = 16; g.stem_th = 8;
    g.stem_tiles_w = (pb.w_out + 15) / 16; g.stem_tiles_h = (pb.h_out + 7) / 8;
    g.p = (long long)pb.n * g.stem_tiles_h * g.stem_tiles_w * kBM;      // m-tiles x 128 (patches, ragged edges clipped)
    g.stages = 1; g.blockdiag = 0; g.out_strided = nullptr; g.out_sn = 0; g.out_sh = g.out_sw = 0;
    g.f16 = call_f16();
    g.fold = fold ? *fold : BnFold{nullptr, nullptr, nullptr, nullptr, nullptr, 0.f, nullptr};
    CUtensorMap ta, tw, tout;
    {   // overlapping windows: 64 elements (8 pixels x 8 channels) starting at every output column
        const unsigned long long dims[5] = {64, (unsigned long long)pb.w_out, (unsigned long long)pb.h_out,
                                            (unsigned long long)krows, (unsigned long long)pb.n};
        unsigned long long str[5];
        stem_window_strides(pb, str);
        const unsigned int box[5] = {64, 16, 8, 1, 1};
        if (!make_tmap_tiled_bf16(&ta, x_packed, 5, dims, str, box)) return cudaErrorInvalidValue;
    }
    {
        const unsigned long long dims[4] = {(unsigned long long)pb.c_out, (unsigned long long)pb.w_out,
                                            (unsigned long long)pb.h_out, (unsigned long long)pb.n};
        const unsigned long long str[4] = {0, (unsigned long long)pb.c_out * 2,
                                           (unsigned long long)pb.w_out * pb.c_out * 2,
                                           (unsigned long long)pb.h_out * pb.w_out * pb.c_out * 2};
        const unsigned int box[4] = {64, 16, 2, 1};
        if (!make_tmap_tiled_bf16(&tout, out, 4, dims, str, box)) return cudaErrorInvalidValue;
    }
    if (!make_tmap_matrix_bf16(&tw, wst, pb.c_out, (long long)krows * 64, 64, kBK)) return cudaErrorInvalidValue;
    int *err = nullptr;
    cudaError_t e = error_word_address(&err);
    if (e != cudaSuccess) return e;
    return launch_bn<64>(ta, tw, tout, tout, tout, g, bias, err, st);
}

}  // namespace convbn

// Weight-gradient implicit GEMM on the sm_100a tensor cores:  domega' = dZ (.) X  (Sec. 3.2.1; Table 2,
// Tune row), the reduction over all N H_out W_out output pixels.
//
// GEMM view: D[k][co] = sum_p Xcol[p][k] dZ[p][co] with k = (tap, ci).  Both operands have the
// reduction index p as their slow axis in NHWC memory, so both are fed to tcgen05.mma as MN-major
// tiles: the A tile is two [64 pixels][64 channels] im2col loads of X (two consecutive 64-wide slices
// of k), the B tile is BN/64 plain [64 pixels][64 channels] boxes of dZ.  The pixel range is cut into
// `splits` slices (grid.z); every CTA accumulates its slice in tensor memory in fp32 and writes one
// fp32 partial tile, in the weights' layout part[split][co][k].  A second kernel adds the slices in fixed order and forms
// domega, dgamma, ... from the fp32 sums (never from rounded values).
#include "kernels.h"
#include "sm100_ptx.cuh"

namespace convbn {

using namespace ptx;

constexpr int kWM = 128;          // k rows per tile (two 64-channel slices)
constexpr int kWP = 64;           // pixels per stage (reduction depth per stage)
constexpr int kWUmmaK = 16;
constexpr int kWMaxStages = 8;
constexpr int kWThreads = 224;    // X loads, MMA, 4 epilogue warps, dZ loads
constexpr int kWDzWarp = kWThreads / 32 - 1;
constexpr uint32_t kChunkBytes = kWP * 64 * 2;   // one [64 pixels][64 channels] bf16 box

struct WgradGemm {
    int ho, wo, c_in, c_out, taps_w;
    int lower_h, lower_w, stride_h, stride_w, dil_h, dil_w;
    int kdim;               // taps * c_in
    long long p;            // output pixels
    long long per_split;    // pixels per slice (multiple of 64)
    FastDiv by_wo, by_ho, by_ci, by_tw;      // by wo, ho, c_in, taps_w
    int stages;
    int blockdiag;          // grouped conv: c_in = 64 here, k rows are (tap, channel of block blockIdx.y)
    // Small-C_in ("stem") mode: tm_x is the 5-D window view of the packed input (one 64-wide slice per
    // filter row), tm_dz a 4-D map of dZ; a "pixel block" is a 4 x 16 patch of output pixels.
    int stem, stem_tiles_w, stem_tiles_h;
    // Where the per-channel sums come from.  kSumNone: nowhere (the packed stem input carries a constant-1 slot instead).
    // kSumSlice: a slice of ones behind the last slice of k; its accumulator rows are sum_p dZ[p][co].  kSumX: the rows of the X
    // tiles, added in fp32 by the epilogue warps while the tiles are multiplied (the sums of a transposed layer's dZ, which is
    // the windowed operand there; by products of ones in a second accumulator they were 1.2e-6 off instead of 1e-7).  Ones times
    // the dZ tile in an accumulator of its own, instead of the slice, were measured where the number of slices is even and the
    // slice costs another row of tiles: 2 to 6 % slower for most layers (3x3 256 at 23 x 21, N = 8 34.9 -> 36.7 us, ResNet-50,
    // N = 32 2464 -> 2500), the products being a second full MMA per step.
    int sums;
    int f16;                // 16-bit storage type: 0 bf16, 1 IEEE half
    int rows;               // 1: partials are [split][C_out][kdim], 0: [split][k][C_out]
};

enum { kSumNone, kSumSlice, kSumX };
struct WgradSmemCtl {
    uint64_t full[kWMaxStages];
    uint64_t empty[kWMaxStages];
    uint64_t tmem_full;
    uint32_t tmem_base;
    int abort_flag;
};

// X_SUMS: g.sums is kSumX.
template <int BN, bool X_SUMS>
__global__ void __launch_bounds__(kWThreads) umma_wgrad_kernel(const __grid_constant__ CUtensorMap tm_x,
                                                              const __grid_constant__ CUtensorMap tm_dz,
                                                              const WgradGemm g, float *__restrict__ partials,
                                                              float *__restrict__ bsum,
                                                              unsigned int *__restrict__ counters, int ncounters,
                                                              int *err) {
    extern __shared__ uint8_t smem_raw[];
    constexpr uint32_t kABytes = 2 * kChunkBytes, kBBytes = (BN / 64) * kChunkBytes, kStageBytes = kABytes + kBBytes;
    uint8_t *tiles = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    WgradSmemCtl *ctl = (WgradSmemCtl *)(tiles + (size_t)g.stages * kStageBytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int stages = g.stages;
    const int k0 = blockIdx.x * kWM;                    // first k row of this tile
    const int n0 = blockIdx.y * BN;                     // first output channel
    const long long p0 = (long long)blockIdx.z * g.per_split;
    const long long p1 = p0 + g.per_split < g.p ? p0 + g.per_split : g.p;
    const int num_kb = (int)((p1 - p0 + kWP - 1) / kWP);
    const int nch = g.kdim / 64, c_first = k0 / 64;
    const int a_chunks = nch - c_first >= 2 ? 2 : (nch - c_first >= 1 ? 1 : 0);   // slices loaded by TMA
    const int ones_slot = g.sums != kSumSlice ? -1 : ((c_first == nch) ? 0 : (c_first + 1 == nch ? 1 : -1));
    const bool adds = X_SUMS && blockIdx.y == 0;         // (kSumX: the first tile of channels)
    int b_chunks = (g.c_out - n0) / 64;
    if (b_chunks > BN / 64) b_chunks = BN / 64;
    volatile int *abort_flag = &ctl->abort_flag;

    // the tensor maps are kernel parameters, not data of an earlier kernel: fetch them before the wait
    if (threadIdx.x == 96) { prefetch_tensormap(&tm_x); prefetch_tensormap(&tm_dz); }
    // The X loads' coordinates, worked out beside the set-up: the slices' k = tap * c_in + ci is fixed for the whole CTA, the pixel
    // is that of the slice's start.
    int ci[2] = {0, 0}, wo0 = 0, ho0 = 0;
    uint16_t off_w[2] = {0, 0}, off_h[2] = {0, 0};
    uint32_t img = 0;
    if (warp == 0) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int kk = k0 + j * 64, tap = (int)g.by_ci.div((uint32_t)kk), tr = (int)g.by_tw.div((uint32_t)tap);
            ci[j] = kk - tap * g.c_in + (g.blockdiag ? n0 : 0);
            off_w[j] = (uint16_t)((tap - tr * g.taps_w) * g.dil_w);
            off_h[j] = (uint16_t)(tr * g.dil_h);
        }
        const uint32_t pp = (uint32_t)p0, t0 = g.by_wo.div(pp);
        wo0 = (int)(pp - t0 * (uint32_t)g.wo);
        img = g.by_ho.div(t0);
        ho0 = (int)(t0 - img * (uint32_t)g.ho);
    }
    if (threadIdx.x == 64) {
        for (int s = 0; s < stages; ++s) { mbar_init(&ctl->full[s], 2); mbar_init(&ctl->empty[s], adds ? 5 : 1); }
        mbar_init(&ctl->tmem_full, 1);
        ctl->abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc(&ctl->tmem_base, BN);
        tmem_relinquish();
    }
    pdl_wait();                 // global memory only after every earlier kernel has finished
    // counters of the epilogue kernel that runs after this one start from zero
    if (counters && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0)
        for (int i = threadIdx.x; i < ncounters; i += kWThreads) counters[i] = 0u;
    if (ones_slot >= 0) {
        // 1.0 everywhere (invariant under the swizzle); TMA never writes this slice
        const uint32_t one2 = one_h16(g.f16) * 0x10001u;
        const uint4 ones = make_uint4(one2, one2, one2, one2);
        for (int s = 0; s < stages; ++s) {
            uint4 *dst = (uint4 *)(tiles + (size_t)s * kStageBytes + (size_t)ones_slot * kChunkBytes);
            for (int i = threadIdx.x; i < (int)(kChunkBytes / 16); i += kWThreads) dst[i] = ones;
        }
        fence_proxy_async_smem();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = ctl->tmem_base;

    // the two loading threads' walk through the ring
    const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]), tiles0 = smem_u32(tiles), sb_end = 8u * (uint32_t)stages;
    uint32_t sb = 0, slot = tiles0, ph = 1;
    int issued = 0;
    bool ok = true, free = false;
    auto give_up = [&]() {
        if (ok) return;
        atomicOr(err, ERRW_TIMEOUT);
        ctl->abort_flag = 1;
        for (int kb = issued > stages ? issued - stages : 0; kb < issued; ++kb)     // let the copies in flight land
            mbar_wait_bounded(&ctl->full[kb % stages], (uint32_t)(kb / stages) & 1u, nullptr, 200000000ull);
    };
    // stem: pixel block -> (image, patch row, patch column) of 4 x 16 output pixels
    auto patch = [&](uint32_t blk, int &pw, int &phh, int &im) {
        const uint32_t t1 = blk / (uint32_t)g.stem_tiles_w, i1 = t1 / (uint32_t)g.stem_tiles_h;
        pw = (int)(blk - t1 * (uint32_t)g.stem_tiles_w) * 16;
        phh = (int)(t1 - i1 * (uint32_t)g.stem_tiles_h) * 4;
        im = (int)i1;
    };

    if (warp == 0) {
        // One thread for the X slices, one (of the last warp) for dZ; stepped addresses, the next slot's barrier tested ahead,
        // loops unrolled: what one thread has to do per stage bounded this kernel (see umma_conv.cu).
        // Weight phase with its second kernel, graph replay: 3x3 512 at 7 x 7, N = 64 29.5 -> 25.5 us, N = 32 22.6 -> 20.6,
        // 3x3 64 at 56 x 56, N = 32 21.9 -> 19.4.
        if (elect_one()) {
            const uint32_t tx_bytes = (uint32_t)a_chunks * kChunkBytes;
            const uint32_t blk0 = (uint32_t)(p0 / kWP);
#pragma unroll 4
            for (int kb = 0; kb < num_kb; ++kb) {
                if (!free) ok = mbar_wait_bounded(empty0 + sb, ph, abort_flag);
                if (!ok) break;
                const uint32_t bar = full0 + sb, dst = slot;
                ++issued; sb += 8; slot += kStageBytes;
                if (sb == sb_end) { sb = 0; slot = tiles0; ph ^= 1u; }
                free = mbar_test_wait(empty0 + sb, ph);
                mbar_arrive_expect_tx(bar, tx_bytes);
                if (g.stem) {
                    int pw, phh, im;
                    patch(blk0 + (uint32_t)kb, pw, phh, im);
                    if (a_chunks > 0) tma_load_5d(dst, &tm_x, bar, 0, pw, phh, c_first, im);
                    if (a_chunks > 1) tma_load_5d(dst + kChunkBytes, &tm_x, bar, 0, pw, phh, c_first + 1, im);
                } else {
                    const int base_w = g.lower_w + wo0 * g.stride_w, base_h = g.lower_h + ho0 * g.stride_h;
                    if (a_chunks > 0) tma_load_im2col_4d(dst, &tm_x, bar, ci[0], base_w, base_h, (int)img, off_w[0], off_h[0]);
                    if (a_chunks > 1) tma_load_im2col_4d(dst + kChunkBytes, &tm_x, bar, ci[1], base_w, base_h, (int)img, off_w[1], off_h[1]);
                    wo0 += kWP;
                    while (wo0 >= g.wo) { wo0 -= g.wo; if (++ho0 == g.ho) { ho0 = 0; ++img; } }
                }
            }
            give_up();
        }
    } else if (warp == kWDzWarp) {
        if (elect_one()) {
            const uint32_t blk0 = (uint32_t)(p0 / kWP);
            slot += kABytes;
#pragma unroll 4
            for (int kb = 0; kb < num_kb; ++kb) {
                if (!free) ok = mbar_wait_bounded(empty0 + sb, ph, abort_flag);
                if (!ok) break;
                const uint32_t bar = full0 + sb, dst = slot;
                ++issued; sb += 8; slot += kStageBytes;
                if (sb == sb_end) { sb = 0; slot = tiles0 + kABytes; ph ^= 1u; }
                free = mbar_test_wait(empty0 + sb, ph);
                if (g.stem) {
                    int pw, phh, im;
                    patch(blk0 + (uint32_t)kb, pw, phh, im);
                    mbar_arrive_expect_tx(bar, (uint32_t)b_chunks * kChunkBytes);
                    for (int j = 0; j < b_chunks; ++j) tma_load_4d(dst + j * kChunkBytes, &tm_dz, bar, n0 + j * 64, pw, phh, im);
                } else {
                    mbar_arrive_expect_tx(bar, kBBytes);             // (slices past C_out arrive as zeros)
                    tma_load_3d(dst, &tm_dz, bar, 0, (int)p0 + kb * kWP, n0 / 64);
                }
            }
            give_up();
        }
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc = idesc_h16_f32(kWM, BN, 1, 1, g.f16);   // both operands MN-major
            const uint32_t hi = smem_desc_hi_sw128(1024);
            const uint32_t tiles_lo = smem_desc_lo(smem_u32(tiles), kChunkBytes);
            uint32_t a_lo = tiles_lo;
            ph = 0;
#pragma unroll 4
            for (int kb = 0; kb < num_kb; ++kb) {
                if (!free && !mbar_wait_bounded(full0 + sb, ph, abort_flag)) {
                    atomicOr(err, ERRW_TIMEOUT);
                    ctl->abort_flag = 1;
                    ok = false;
                    break;
                }
                // 16 pixels = two groups of 8 rows (1024 B apart); 64-channel slices 8192 B apart; descriptors as
                // halves, only the start-address field (16-byte units) moves
                const uint32_t a0 = a_lo, b0 = a_lo + (kABytes >> 4), done = empty0 + sb;
                sb += 8; a_lo += kStageBytes >> 4;
                if (sb == sb_end) { sb = 0; a_lo = tiles_lo; ph ^= 1u; }
                free = mbar_test_wait(full0 + sb, ph);
                umma_bf16_ss_sel(tmem_base, a0, hi, b0, hi, idesc, (uint32_t)kb);
#pragma unroll
                for (int k = 1; k < kWP / kWUmmaK; ++k)
                    umma_bf16_ss_halves<true>(tmem_base, a0 + (uint32_t)k * (kWUmmaK * 128 >> 4), hi,
                                              b0 + (uint32_t)k * (kWUmmaK * 128 >> 4), hi, idesc);
                umma_commit(done);
            }
            if (ok) umma_commit(&ctl->tmem_full);
        }
    } else {
        const int quarter = warp & 3;
        if (adds) {
            // two warps per 64-channel slice, half of the pixels each; a lane has two channels, a row is 128 bytes
            const int slice = quarter >> 1, half = quarter & 1;
            float lo = 0.f, hi = 0.f;
            auto add_rows = [&](auto half_tag, uint32_t tile) {
                constexpr bool H = decltype(half_tag)::value;
#pragma unroll 8
                for (int r = 0; r < 32; ++r) {
                    uint32_t u;
                    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(u) : "r"(tile + (uint32_t)r * 128u + (((uint32_t)(lane >> 2) ^ (r & 7)) << 4)));
                    float a, b;
                    unpack2_t<H>(u, a, b);
                    lo += a;
                    hi += b;
                }
            };
            const uint32_t first = tiles0 + (uint32_t)slice * kChunkBytes + (uint32_t)half * 32u * 128u + (uint32_t)(lane & 3) * 4u;
            uint32_t at = first, sb2 = 0, ph2 = 0;
            bool fine = true;
            for (int kb = 0; kb < num_kb && fine; ++kb) {
                fine = __all_sync(0xffffffffu, mbar_wait_bounded(full0 + sb2, ph2, abort_flag));
                if (!fine) break;
                if (slice < a_chunks) { if (g.f16) add_rows(std::true_type{}, at); else add_rows(std::false_type{}, at); }
                __syncwarp();
                if (lane == 0) mbar_arrive(empty0 + sb2);
                sb2 += 8; at += kStageBytes;
                if (sb2 == sb_end) { sb2 = 0; at = first; ph2 ^= 1u; }
            }
            const int k = k0 + slice * 64 + 2 * lane;
            if (slice < a_chunks) *(float2 *)(bsum + ((size_t)blockIdx.z * 2 + half) * g.kdim + k) = make_float2(lo, hi);
        }
        const bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(&ctl->tmem_full, 0, abort_flag));
        if (!ok && lane == 0) { atomicOr(err, ERRW_TIMEOUT); ctl->abort_flag = 1; }
        // The adding kernel is let go only here: its blocks, waiting for this grid, would take the shared memory that the
        // 220 KB CTAs of the data pass beside it need (forward + backward of 3x3 64 -> 64 at 56 x 56, N = 32 49.8 -> 47.4 us,
        // 3x3 stride 2 128 -> 128 at 200 x 334, N = 2 62.1 -> 59.9, 3x3 128 at 52 x 85, N = 9 55.1 -> 50.2).
        pdl_launch_dependents();
        if (ok) {
            tc_fence_after_sync();
            const int k = k0 + quarter * 32 + lane;
            const bool row_ok = k < g.kdim;
            const bool sum_row = g.sums == kSumSlice && k == g.kdim;      // first row of the ones slice
            float *brow = bsum + (size_t)blockIdx.z * g.c_out + n0;
            float *orow = g.blockdiag
                              ? partials + (((size_t)blockIdx.z * gridDim.y + blockIdx.y) * g.kdim + (row_ok ? k : 0)) * 64
                              : partials + ((size_t)blockIdx.z * g.kdim + (row_ok ? k : 0)) * g.c_out + n0;
#pragma unroll 1
            for (int c0 = 0; c0 < BN; c0 += 32) {
                if (n0 + c0 >= g.c_out) break;
                uint32_t v[32];
                tmem_ld_32x32(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0, v);
                tmem_ld_wait();
                if (row_ok && g.rows) {
                    // lanes are consecutive k: each store is 128 contiguous bytes of a weight row
                    float *wrow = partials + ((size_t)blockIdx.z * g.c_out + n0 + c0) * g.kdim + k;
#pragma unroll
                    for (int j = 0; j < 32; ++j) wrow[(size_t)j * g.kdim] = __uint_as_float(v[j]);
                } else if (row_ok) {
#pragma unroll
                    for (int j = 0; j < 32; j += 4)
                        *(uint4 *)(orow + c0 + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                } else if (sum_row) {
#pragma unroll
                    for (int j = 0; j < 32; j += 4)
                        *(uint4 *)(brow + c0 + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                }
            }
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, BN);
}

bool grouped_bd_eligible(const Problem &pb) {
    if (pb.groups <= 1 || pb.cg != pb.cog || pb.cg < 2 || 64 % pb.cg || pb.c_in % 64) return false;
    if (pb.pad_h > 128 || pb.pad_w > 128) return false;
    if ((pb.kh - 1) * pb.dil_h > 255 || (pb.kw - 1) * pb.dil_w > 255) return false;
    if (pb.stride_h > 8 || pb.stride_w > 8) return false;
    if (pb.p >= (1LL << 31) - 256 || pb.pin >= (1LL << 31) - 256) return false;
    return true;
}

bool umma_wgrad_eligible(const Problem &pb) {
    if (pb.groups != 1 || pb.c_in % 64 || pb.c_out % 64) return false;
    if (pb.pad_h > 128 || pb.pad_w > 128) return false;
    if ((pb.kh - 1) * pb.dil_h > 255 || (pb.kw - 1) * pb.dil_w > 255) return false;
    if (pb.stride_h > 8 || pb.stride_w > 8) return false;
    if (pb.p >= (1LL << 31)) return false;
    return true;
}

// (256-wide tiles, one CTA per SM, measured 0 to 5 % slower than two 128-wide ones; the packed stem still uses them)
static int wgrad_bn(const Problem &pb) { return pb.c_out >= 128 ? 128 : 64; }
static int stem_wgrad_bn(const Problem &pb) { return pb.c_out >= 256 ? 256 : wgrad_bn(pb); }

// Output tiles of bn columns.
static long long wgrad_k_slices(const Problem &pb) { return (pb.groups > 1 ? (long long)pb.kh * pb.kw * 64 : pb.kdim) / 64; }
static long long wgrad_tiles(const Problem &pb, int bn, bool ones_slice) {
    return (wgrad_k_slices(pb) + (ones_slice ? 2 : 1)) / 2 * ((pb.c_out + bn - 1) / bn);
}

// The slice count minimises  rounds over the resident slots x (pixels per slice + a fixed cost per
// CTA, in pixels) + a small cost per slice for the epilogue that adds the slices up (four pixels, set when a block added a whole
// channel); a grid a few CTAs larger than the slots would otherwise run a second, nearly empty round.
static UmmaWgradPlan wgrad_slices(const Problem &pb, long long tiles, long long slots) {
    UmmaWgradPlan pl;
    const long long max_splits = (pb.p + 4 * kWP - 1) / (4 * kWP);     // at least 256 pixels per slice
    long long splits = 1;
    double best_cost = -1.0;
    for (long long sp = 1; sp <= max_splits; ++sp) {
        const long long rounds = (tiles * sp + slots - 1) / slots;
        const double cost = (double)rounds * ((double)pb.p / (double)sp + 384.0) + 4.0 * (double)sp;
        if (best_cost < 0 || cost < best_cost) { best_cost = cost; splits = sp; }
        if (tiles * sp > 4 * slots) break;
    }
    long long per = (pb.p + splits - 1) / splits;
    per = (per + kWP - 1) / kWP * kWP;
    pl.per_split = per;
    pl.splits = (int)((pb.p + per - 1) / per);
    return pl;
}

UmmaWgradPlan umma_wgrad_plan(const Problem &pb, WgradSums sums) {
    // Resident CTAs: two per SM (the stage rings are sized for it, launch_w): one's partial tile leaves while the other
    // multiplies.  A deeper ring for one CTA gains nothing.
    // Few tiles mean many slices, and where those are short the partial tensors weigh more than what a second CTA hides: up to
    // 24 tiles with slices of up to 2048 pixels get one CTA per SM (N = 32: 1x1 128 -> 512 at 28 x 28 15.3 -> 13.4 us, 1024 ->
    // 256 at 14 x 14 13.3 -> 11.4, 3x3 128 at 28 x 28 17.6 -> 15.5; but 3x3 256 at 14 x 14, 38 tiles, 15.8 -> 18.1, and 1x1
    // 128 -> 512 at 28 x 28, N = 256 58.3 -> 73.6).  Not where output rows are shorter than four pixels: the boxes of X then
    // arrive pixel by pixel and a second CTA hides that (29173 rows, 1024 -> 64: 44.5 and 27.4 us; 2 x 2 about even; from
    // 4 x 4 on one CTA is the faster).
    const long long tiles = wgrad_tiles(pb, pb.groups > 1 ? 64 : wgrad_bn(pb), sums == WgradSums::kDz), sms = device_sm_count();
    return wgrad_slices(pb, tiles, sms * (tiles <= 24 && pb.p * tiles <= 2048 * sms && pb.w_out >= 4 ? 1 : 2));
}

// The slices of a call whose scratch is bounded, where the plan above wants more than there is: 256 columns count as one tile
// with an SM of its own, which makes fewer slices of wide layers (3x3 768 -> 384 at 13 x 13, N = 12: 10 MiB, above 30).
UmmaWgradPlan umma_wgrad_plan_bounded(const Problem &pb) {
    const int bn = pb.groups > 1 ? 64 : (pb.c_out >= 256 ? 256 : wgrad_bn(pb));
    return wgrad_slices(pb, wgrad_tiles(pb, bn, true), (long long)device_sm_count() * (bn == 256 ? 1 : 2));
}

int wgrad_kmajor_rows(const Problem &pb) { return (pb.kdim + 1) / 2; }

template <int BN, bool X_SUMS = false>
static cudaError_t launch_w(const CUtensorMap &tx, const CUtensorMap &tdz, WgradGemm g, const UmmaWgradPlan &pl,
                            const Problem &pb, float *partials, float *bsum, int *err, cudaStream_t st,
                            unsigned int *counters = nullptr, int ncounters = 0) {
    g.by_wo = FastDiv((uint32_t)g.wo); g.by_ho = FastDiv((uint32_t)g.ho); g.by_ci = FastDiv((uint32_t)g.c_in); g.by_tw = FastDiv((uint32_t)g.taps_w);
    constexpr size_t stage = 2 * kChunkBytes + (BN / 64) * kChunkBytes;
    int stages = BN == 128 ? 3 : 4;                    // 128-wide: 3 x 32 KB, so that two CTAs share an SM
    const long long max_kb = (pl.per_split + kWP - 1) / kWP;
    if (stages > max_kb) stages = (int)max_kb;
    g.stages = stages;
    size_t smem = stages * stage + 1024 + sizeof(WgradSmemCtl);
    const size_t floor_smem = (size_t)(228 * 1024) / (512 / BN + 1) + 1024;
    if (smem < floor_smem) smem = floor_smem;
    static PerDevice attr_done;
    if (cudaError_t e = max_dynamic_smem_once(umma_wgrad_kernel<BN, X_SUMS>, 210 * 1024, &attr_done); e != cudaSuccess) return e;
    static PerDevice carve;
    prefer_max_shared_once(umma_wgrad_kernel<BN, X_SUMS>, &carve);
    dim3 grid((unsigned)((g.kdim / 64 + (g.sums == kSumSlice ? 2 : 1)) / 2), (unsigned)((pb.c_out + BN - 1) / BN),
              (unsigned)pl.splits);
    return launch_pdl(umma_wgrad_kernel<BN, X_SUMS>, grid, dim3(kWThreads), smem, st, tx, tdz, g, partials, bsum, counters,
                      ncounters, err);
}

cudaError_t launch_umma_wgrad(const Problem &pb, const UmmaWgradPlan &pl, const void *dz, const void *x,
                              float *partials, float *bsum, cudaStream_t st, unsigned int *counters, int ncounters, WgradSums sums) {
    WgradGemm g;
    g.ho = pb.h_out; g.wo = pb.w_out; g.c_in = pb.c_in; g.c_out = pb.c_out; g.taps_w = pb.kw;
    g.lower_h = -pb.pad_h; g.lower_w = -pb.pad_w; g.stride_h = pb.stride_h; g.stride_w = pb.stride_w;
    g.dil_h = pb.dil_h; g.dil_w = pb.dil_w; g.kdim = pb.kdim; g.p = pb.p; g.per_split = pl.per_split; g.stages = 1;
    g.blockdiag = pb.groups > 1 ? 1 : 0;
    g.rows = g.blockdiag ? 0 : 1;
    g.stem = 0; g.stem_tiles_w = g.stem_tiles_h = 1; g.f16 = call_f16();
    g.sums = sums == WgradSums::kX ? kSumX : (sums == WgradSums::kNone ? kSumNone : kSumSlice);
    if (g.blockdiag) { g.c_in = 64; g.kdim = pb.kh * pb.kw * 64; }
    const int upper_h = g.lower_h + (pb.h_out - 1) * pb.stride_h - (pb.h_in - 1);
    const int upper_w = g.lower_w + (pb.w_out - 1) * pb.stride_w - (pb.w_in - 1);
    CUtensorMap tx, tdz;
    if (!make_tmap_im2col_bf16(&tx, x, pb.n, pb.h_in, pb.w_in, pb.c_in, g.lower_h, g.lower_w, upper_h, upper_w,
                               pb.stride_h, pb.stride_w, kWP, 64))
        return cudaErrorInvalidValue;
    const int bn = g.blockdiag ? 64 : wgrad_bn(pb);
    {   // a stage's [64 pixels][64 channels] slices of dZ, side by side in shared memory, are one box
        const unsigned long long dims[3] = {64, (unsigned long long)pb.p, (unsigned long long)pb.c_out / 64};
        const unsigned long long str[3] = {0, (unsigned long long)pb.c_out * 2, 128};
        const unsigned int box[3] = {64, (unsigned int)kWP, (unsigned int)(bn / 64)};
        if (!make_tmap_tiled_bf16(&tdz, dz, 3, dims, str, box)) return cudaErrorInvalidValue;
    }
    int *err = nullptr;
    cudaError_t e = error_word_address(&err);
    if (e != cudaSuccess) return e;
    if (g.sums == kSumX)
        return bn == 64 ? launch_w<64, true>(tx, tdz, g, pl, pb, partials, bsum, err, st, counters, ncounters)
                        : launch_w<128, true>(tx, tdz, g, pl, pb, partials, bsum, err, st, counters, ncounters);
    if (bn == 64) return launch_w<64>(tx, tdz, g, pl, pb, partials, bsum, err, st, counters, ncounters);
    return launch_w<128>(tx, tdz, g, pl, pb, partials, bsum, err, st, counters, ncounters);
}

// ---- epilogue over partial weight tensors -----------------------------------------------------------
// part[split][C_out][kdim] fp32, the layout of the weights.  One block per output channel finishes everything that
// belongs to it (Table 2, Tune row):
//     acc[k] = sum_split part[split][co][k]
//     domega = s acc,   dbeta = sum_split bsum,   db = s dbeta,   dgamma = r (sum_k acc omega + dbeta (b - mu_hat)).
// Plain mode (vec3 == NULL): domega = acc, db = sum dZ if requested; need_sums = 0: domega alone.
// CL blocks (a cluster) share a channel, a span of k each; their parts of the dot product meet in the first one.
// Threads of a block: VL along k (a float4 each, so that reads and stores are whole lines) x SL groups of slices, added in
// order through shared memory; a thread requests up to eight slices before it uses the first.  Bound by the latency of those
// reads (9 to 19 MB, most of them from L2): few channels of long rows would leave most SMs idle with a block each (how many: see
// the launch).
// With k-major partial tiles the GEMM's stores were 16 bytes per lane in 32 lines, this kernel had to transpose,
// and the per-channel sums needed a counter or a second kernel.  Weight phase (GEMM + this), graph replay, N = 32: 1x1
// 512 -> 128 at 28 x 28 20.3 -> 12.0 us, 3x3 256 at 14 x 14 22.8 -> 17.2, 3x3 512 at 7 x 7 30.0 -> 22.8.
constexpr int kRowsMaxThreads = 512, kRowsMaxCluster = 4;
template <int CL>
__global__ void __launch_bounds__(kRowsMaxThreads) wgrad_rows_kernel(int c_out, int kdim, int span, int VL, int SL,
                                                                     const float *__restrict__ part, int splits,
                                                                     const float *__restrict__ bsum,
                                                                     const __nv_bfloat16 *__restrict__ w,
                                                                     const float *__restrict__ vec3, const float *__restrict__ b,
                                                                     const float *__restrict__ mean, float *__restrict__ dw,
                                                                     float *__restrict__ db, float *__restrict__ dgamma,
                                                                     float *__restrict__ dbeta, int need_sums, int f16) {
    __shared__ float4 red[kRowsMaxThreads];
    __shared__ float fin[2][kRowsMaxThreads / 32], dots[kRowsMaxCluster];
    const int rank = CL > 1 ? (int)cluster_rank() : 0, co = blockIdx.x / CL;
    const int z = threadIdx.x / VL, l = threadIdx.x - z * VL;        // (z >= SL: threads that fill up the last warp)
    const size_t slice = (size_t)c_out * kdim, row = (size_t)co * kdim;
    if (CL > 1 && need_sums) cluster_arrive_started();
    pdl_wait();
    pdl_launch_dependents();
    const float s = vec3 ? vec3[co] : 1.f;
    float dot = 0.f, ds = 0.f;
    if (need_sums && rank == 0)
        for (int sp = threadIdx.x; sp < splits; sp += blockDim.x) ds += __ldcg(bsum + (size_t)sp * c_out + co);
    const int k_end = min(kdim, (rank + 1) * span);
    for (int k0 = rank * span; k0 < k_end; k0 += 4 * VL) {
        const int k = k0 + 4 * l;
        const bool on = k < k_end;
        uint2 wq = make_uint2(0u, 0u);
        if (vec3 && need_sums && z == 0 && on) wq = *(const uint2 *)(w + row + k);
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        if (on && z < SL) {
            const float *src = part + row + k;
            const size_t step = (size_t)SL * slice;
            int sp = z;
            src += (size_t)z * slice;
            for (; sp + 7 * SL < splits; sp += 8 * SL, src += 8 * step) {
                float4 v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = __ldcg((const float4 *)(src + u * step));
#pragma unroll
                for (int u = 0; u < 8; ++u) { a.x += v[u].x; a.y += v[u].y; a.z += v[u].z; a.w += v[u].w; }
            }
            if (sp < splits) {
                float4 v[7];
#pragma unroll
                for (int u = 0; u < 7; ++u)
                    v[u] = sp + u * SL < splits ? __ldcg((const float4 *)(src + u * step)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int u = 0; u < 7; ++u) { a.x += v[u].x; a.y += v[u].y; a.z += v[u].z; a.w += v[u].w; }
            }
        }
        if (SL > 1) {
            if (k0 != rank * span) __syncthreads();
            red[threadIdx.x] = a;
            // groups z and z + h in halves: log2(SL) short steps
            for (int h = SL / 2; h > 0; h /= 2) {
                __syncthreads();
                if (z < h) {
                    const float4 o = red[threadIdx.x + h * VL];
                    a.x += o.x; a.y += o.y; a.z += o.z; a.w += o.w;
                    red[threadIdx.x] = a;
                }
            }
        }
        if (z == 0 && on) {
            *(float4 *)(dw + row + k) = make_float4(s * a.x, s * a.y, s * a.z, s * a.w);
            dot = fmaf(a.x, unpack_h16((uint16_t)(wq.x & 0xFFFFu), f16), dot);
            dot = fmaf(a.y, unpack_h16((uint16_t)(wq.x >> 16), f16), dot);
            dot = fmaf(a.z, unpack_h16((uint16_t)(wq.y & 0xFFFFu), f16), dot);
            dot = fmaf(a.w, unpack_h16((uint16_t)(wq.y >> 16), f16), dot);
        }
    }
    if (!need_sums) return;
    const int lane = threadIdx.x & 31, warps = blockDim.x / 32;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) { dot += __shfl_xor_sync(0xffffffffu, dot, o); ds += __shfl_xor_sync(0xffffffffu, ds, o); }
    if (lane == 0) { fin[0][threadIdx.x / 32] = dot; fin[1][threadIdx.x / 32] = ds; }
    __syncthreads();
    if (threadIdx.x < 32) {
        dot = lane < warps ? fin[0][lane] : 0.f;
        ds = lane < warps ? fin[1][lane] : 0.f;
#pragma unroll
        for (int o = kRowsMaxThreads / 64; o > 0; o >>= 1) { dot += __shfl_xor_sync(0xffffffffu, dot, o); ds += __shfl_xor_sync(0xffffffffu, ds, o); }
    }
    if constexpr (CL > 1) {
        // the first block has started (a block whose span lies past the row's end comes here at once); then its `dots` may be
        // written, and the second meeting says that all are there
        cluster_wait_started();
        if (threadIdx.x == 0) st_cluster_f32(cluster_addr(&dots[rank], 0), dot);
        __syncwarp();
        cluster_sync_all();
    }
    if (threadIdx.x || rank) return;
    if constexpr (CL > 1) {
        dot = 0.f;
#pragma unroll
        for (int i = 0; i < CL; ++i) dot += dots[i];
    }
    if (!vec3) {
        if (db) db[co] = ds;
        return;
    }
    dbeta[co] = ds;
    if (db) db[co] = s * ds;
    dgamma[co] = vec3[2 * c_out + co] * (dot + ds * ((b ? b[co] : 0.f) - mean[co]));
}

// kdim: a multiple of 4 (rows of the weight tensor start on 16-byte boundaries)
cudaError_t launch_wgrad_rows(const Problem &pb, int splits, const float *partials, const float *bsum, const void *w,
                              const float *vec3, const float *b, const float *mean, float *dw, float *db, float *dgamma,
                              float *dbeta, bool need_sums, cudaStream_t st) {
    // Slice groups so that a thread adds at most eight slices, threads along the span in equal turns.  Blocks per channel: up
    // to two per SM for rows with 1600 vectors (of all slices) or more to read, one otherwise: below that and with more
    // channels the blocks' meeting and their number cost more than they share.  Weight phase with 1, 2, 4, 8 blocks per
    // channel: 1x1 256 -> 64, 1000 rows, 256 vectors 9.4 9.7 10.0 9.8 us; 3x3 256 -> 128, 26 x 26, 1728 vectors 7.8 7.2 7.4
    // 7.4; 3x3 64 -> 64, 56 x 56, N = 32, 8496 vectors 21.1 18.2 16.2 16.3; 3x3 512 -> 512, 7 x 7, N = 64 21.0 22.5 25.3 26.0;
    // 5x5 640 -> 384, 13 x 13, N = 9 40.4 44.7 49.8 60.2; whole backward calls at 192 and 256 channels, 4000 to 4400 vectors:
    // 3x3 256 -> 256, 14 x 14, N = 32 27.0 27.4 27.1 29.0, 1x1 832 -> 256 57.0 58.8 57.9 59.2, 3x3 192 -> 192, 28 x 28, N = 16
    // 32.8 34.1 33.4 34.6.
    int SL = 1, CL = 1;
    while (SL < 32 && SL * 8 < splits) SL *= 2;
    auto vectors = [&](int cl) { return ((pb.kdim / 4 + cl - 1) / cl + 7) / 8 * 8; };
    const long long work = (long long)(pb.kdim / 4) * splits;
    while (work >= 1600 && CL < kRowsMaxCluster && pb.kdim / 4 >= 16 * CL && (long long)pb.c_out * CL <= device_sm_count()) CL *= 2;
    const int span = 4 * vectors(CL);
    int VL = vectors(CL);
    if (VL * SL > kRowsMaxThreads) {
        const int turns = (VL * SL + kRowsMaxThreads - 1) / kRowsMaxThreads;
        VL = ((VL + turns - 1) / turns + 7) / 8 * 8;
        if (VL * SL > kRowsMaxThreads) VL = kRowsMaxThreads / SL;
    }
    const int threads = (VL * SL + 31) / 32 * 32;
    if ((long long)pb.c_out * CL > 0x7fffffffLL) return cudaErrorInvalidValue;
    auto go = [&](auto cl) {
        constexpr int N = decltype(cl)::value;
        static PerDevice carve;
        prefer_max_shared_once(wgrad_rows_kernel<N>, &carve);
        return launch_pdl<N>(wgrad_rows_kernel<N>, dim3(pb.c_out * N), dim3(threads), 0, st, pb.c_out, pb.kdim, span, VL, SL,
                             partials, splits, bsum, (const __nv_bfloat16 *)w, vec3, b, mean, dw, db, dgamma, dbeta,
                             need_sums ? 1 : 0, call_f16());
    };
    if (CL == 1) return go(std::integral_constant<int, 1>());
    if (CL == 2) return go(std::integral_constant<int, 2>());
    return go(std::integral_constant<int, 4>());
}

// ---- epilogue over k-major partials (the stem's weight gradient) --------------------------------------
// part[split][k][C_out]: the stem's accumulators hold an output channel per lane.  Two kernels:
//
// wgrad_add_kernel: block = 64 output channels x KR weight rows k.  Thread (float4 of channels, k, slice group z < SL)
// adds slices z, z + SL, ..., eight loads in flight, then the groups are added in order through shared memory and
//     dw[co][k] = s[co] acc,    dotpart[k block][co] = sum over the block's k of acc w[co][k].
// wgrad_finish_kernel: dbeta = sum dZ,  db = s dbeta,  dgamma = r (sum_k domega' omega + dbeta (b - mu_hat)).
// Plain mode (vec3 == NULL): dw = acc, db = sum dZ if requested.  Bound by the latency of the L2 reads (5.5 MB).
template <int KR, int SL>
__global__ void __launch_bounds__(KR * 16 * SL) wgrad_add_kernel(int c_out, int kdim, const float *__restrict__ part, int splits,
                                                                const __nv_bfloat16 *__restrict__ w,
                                                                const float *__restrict__ scale, float *__restrict__ dw,
                                                                float *__restrict__ dotpart, int f16) {
    constexpr int T = KR * 16 * SL, E = KR * 64;                    // threads, elements
    constexpr int SUB = T > E ? T / E : 1, PER = T > E ? 1 : E / T; // threads per element, elements per thread
    __shared__ float tile[SL][KR][65];
    pdl_wait();
    pdl_launch_dependents();
    const int co0 = blockIdx.x * 64, k0 = blockIdx.y * KR;
    // the element(s) this thread finishes: k runs fastest, over neighbouring groups of SUB lanes
    const int sub = threadIdx.x % SUB;
    float wv[PER], sv[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int e = threadIdx.x / SUB + i * (T / SUB), k = k0 + e % KR, co = co0 + e / KR;
        wv[i] = dotpart && sub == 0 && k < kdim ? load_h16(w + (size_t)co * kdim + k, f16) : 0.f;
        sv[i] = scale ? scale[co] : 1.f;
    }
    {
        const int l = threadIdx.x & 15, ky = (threadIdx.x >> 4) % KR, z = threadIdx.x / (16 * KR), k = k0 + ky;
        const size_t slice = (size_t)kdim * c_out;
        const float *src = part + (size_t)k * c_out + co0 + l * 4;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k < kdim)
            for (int sp = z; sp < splits; sp += 8 * SL) {
                float4 v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    v[u] = sp + u * SL < splits ? __ldcg((const float4 *)(src + (size_t)(sp + u * SL) * slice))
                                                : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int u = 0; u < 8; ++u) { a.x += v[u].x; a.y += v[u].y; a.z += v[u].z; a.w += v[u].w; }
            }
        float *t = &tile[z][ky][l * 4];
        t[0] = a.x; t[1] = a.y; t[2] = a.z; t[3] = a.w;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int e = threadIdx.x / SUB + i * (T / SUB), k = k0 + e % KR, cl = e / KR;
        float v = 0.f;
#pragma unroll
        for (int z = sub; z < SL; z += SUB) v += tile[z][e % KR][cl];
#pragma unroll
        for (int o = 1; o < SUB; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (sub == 0 && k < kdim) dw[(size_t)(co0 + cl) * kdim + k] = sv[i] * v;
        if (dotpart) {
            float d = v * wv[i];
#pragma unroll
            for (int o = SUB; o < SUB * KR; o <<= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            if (sub == 0 && e % KR == 0) dotpart[(size_t)blockIdx.y * c_out + co0 + cl] = d;
        }
    }
}

// dotpart [rows][C_out], bsum [bsplits][C_out]: one block per 32 channels, 32 groups of rows added in order.
__global__ void __launch_bounds__(1024) wgrad_finish_kernel(int c_out, int rows, const float *__restrict__ dotpart, int bsplits,
                                                            const float *__restrict__ bsum, const float *__restrict__ vec3,
                                                            const float *__restrict__ b, const float *__restrict__ mean,
                                                            float *__restrict__ db, float *__restrict__ dgamma,
                                                            float *__restrict__ dbeta) {
    __shared__ float red[2][32][33];
    pdl_wait();
    pdl_launch_dependents();
    const int ch = threadIdx.x & 31, grp = threadIdx.x >> 5, co = blockIdx.x * 32 + ch;
    auto column = [&](const float *v, int n) {
        float acc = 0.f;
        for (int r = grp; r < n; r += 128) {
            float q[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) q[u] = r + 32 * u < n ? __ldcg(v + (size_t)(r + 32 * u) * c_out + co) : 0.f;
            acc += (q[0] + q[1]) + (q[2] + q[3]);
        }
        return acc;
    };
    red[0][grp][ch] = column(bsum, bsplits);
    red[1][grp][ch] = vec3 ? column(dotpart, rows) : 0.f;
    __syncthreads();
    if (grp) return;
    float dsum = 0.f, d = 0.f;
#pragma unroll
    for (int i = 0; i < 32; ++i) { dsum += red[0][i][ch]; d += red[1][i][ch]; }
    if (!vec3) {
        if (db) db[co] = dsum;
        return;
    }
    dbeta[co] = dsum;
    if (db) db[co] = vec3[co] * dsum;
    dgamma[co] = vec3[2 * c_out + co] * (d + dsum * ((b ? b[co] : 0.f) - mean[co]));
}

cudaError_t launch_wgrad_epilogue_kmajor(const Problem &pb, int splits, const float *partials, const float *bsum,
                                         const void *w, const float *vec3, const float *b, const float *mean, float *dw,
                                         float *dotpart, float *db, float *dgamma, float *dbeta, bool need_sums,
                                         cudaStream_t st) {
    const int rows = wgrad_kmajor_rows(pb);
    static PerDevice carve_a, carve_f;
    prefer_max_shared_once(wgrad_add_kernel<2, 32>, &carve_a);
    cudaError_t e = launch_pdl(wgrad_add_kernel<2, 32>, dim3(pb.c_out / 64, rows), dim3(1024), 0, st, pb.c_out, pb.kdim, partials,
                               splits, (const __nv_bfloat16 *)w, vec3, dw, vec3 && need_sums ? dotpart : nullptr, call_f16());
    if (e != cudaSuccess || !need_sums) return e;
    prefer_max_shared_once(wgrad_finish_kernel, &carve_f);
    return launch_pdl(wgrad_finish_kernel, dim3(pb.c_out / 32), dim3(1024), 0, st, pb.c_out, rows, dotpart, splits, bsum, vec3, b,
                      mean, db, dgamma, dbeta);
}

// ---- small-C_in ("stem") layers -------------------------------------------------------------------
UmmaWgradPlan stem_wgrad_plan(const Problem &pb) {
    UmmaWgradPlan pl;
    const int bn = stem_wgrad_bn(pb);
    const long long patches = (long long)pb.n * ((pb.h_out + 3) / 4) * ((pb.w_out + 15) / 16);
    const long long m_tiles = (stem_krows(pb) + (stem_ones_in_pack(pb) ? 1 : 2)) / 2, n_tiles = (pb.c_out + bn - 1) / bn;
    long long splits = (device_sm_count() + m_tiles * n_tiles - 1) / (m_tiles * n_tiles);
    if (splits > (patches + 3) / 4) splits = (patches + 3) / 4;
    if (splits < 1) splits = 1;
    const long long per = (patches + splits - 1) / splits;
    pl.per_split = per * kWP;                       // in pixels of 4 x 16 patches
    pl.splits = (int)((patches + per - 1) / per);
    return pl;
}

// partials: [splits][krows * 64][C_out]; bsum: [splits][C_out]
cudaError_t launch_stem_wgrad(const Problem &pb, const UmmaWgradPlan &pl, const void *dz, const void *x_packed,
                              float *partials, float *bsum, cudaStream_t st) {
    const int krows = stem_krows(pb);
    WgradGemm g;
    g.ho = pb.h_out; g.wo = pb.w_out; g.c_in = 64; g.c_out = pb.c_out; g.taps_w = 1;
    g.lower_h = g.lower_w = 0; g.stride_h = g.stride_w = g.dil_h = g.dil_w = 1;
    g.kdim = krows * 64;
    g.rows = 0;
    g.stem = 1; g.stem_tiles_w = (pb.w_out + 15) / 16; g.stem_tiles_h = (pb.h_out + 3) / 4;
    g.sums = stem_ones_in_pack(pb) ? kSumNone : kSumSlice;
    g.f16 = call_f16();
    g.p = (long long)pb.n * g.stem_tiles_h * g.stem_tiles_w * kWP;
    g.per_split = pl.per_split; g.stages = 1; g.blockdiag = 0;
    CUtensorMap tx, tdz;
    {
        const unsigned long long dims[5] = {64, (unsigned long long)pb.w_out, (unsigned long long)pb.h_out,
                                            (unsigned long long)krows, (unsigned long long)pb.n};
        unsigned long long str[5];
        stem_window_strides(pb, str);
        const unsigned int box[5] = {64, 16, 4, 1, 1};
        if (!make_tmap_tiled_bf16(&tx, x_packed, 5, dims, str, box)) return cudaErrorInvalidValue;
    }
    {
        const unsigned long long dims[4] = {(unsigned long long)pb.c_out, (unsigned long long)pb.w_out,
                                            (unsigned long long)pb.h_out, (unsigned long long)pb.n};
        const unsigned long long str[4] = {0, (unsigned long long)pb.c_out * 2,
                                           (unsigned long long)pb.w_out * pb.c_out * 2,
                                           (unsigned long long)pb.h_out * pb.w_out * pb.c_out * 2};
        const unsigned int box[4] = {64, 16, 4, 1};
        if (!make_tmap_tiled_bf16(&tdz, dz, 4, dims, str, box)) return cudaErrorInvalidValue;
    }
    int *err = nullptr;
    cudaError_t e = error_word_address(&err);
    if (e != cudaSuccess) return e;
    Problem q = pb;
    q.kdim = g.kdim;                                   // grid: (kh + 2) / 2 row tiles
    const int bn = stem_wgrad_bn(pb);
    if (bn == 64) return launch_w<64>(tx, tdz, g, pl, q, partials, bsum, err, st);
    if (bn == 128) return launch_w<128>(tx, tdz, g, pl, q, partials, bsum, err, st);
    return launch_w<256>(tx, tdz, g, pl, q, partials, bsum, err, st);
}

// One block per output channel: gathers the kh x kw x C_in real entries out of the krows x 64 padded rows,
// adds the slices in order and finishes domega, db, dgamma, dbeta (Table 2, Tune row) or the plain sums.
__global__ void __launch_bounds__(256) wgrad_epilogue_stem_kernel(int c_out, int kh, int kw, int c_in, int krows, int s2d,
                                                                 int sum_row,
                                                                 const float *__restrict__ part, int splits,
                                                                 const float *__restrict__ bsum,
                                                                 const __nv_bfloat16 *__restrict__ w,
                                                                 const float *__restrict__ vec3,
                                                                 const float *__restrict__ b,
                                                                 const float *__restrict__ mean,
                                                                 float *__restrict__ dw, float *__restrict__ db,
                                                                 float *__restrict__ dgamma,
                                                                 float *__restrict__ dbeta, int need_sums, int f16) {
    __shared__ float red[256];
    const int co = blockIdx.x, kdim = kh * kw * c_in;
    const size_t slice = (size_t)krows * 64 * c_out;
    const float s = vec3 ? vec3[co] : 1.f;
    float dot = 0.f;
    for (int k = threadIdx.x; k < kdim; k += blockDim.x) {
        const int c = k % c_in, t = k / c_in, q = t % kw, r = t / kw;
        const size_t o = (s2d ? (size_t)(r >> 1) * 64 + (q >> 1) * 16 + (r & 1) * 8 + (q & 1) * 4 + c
                              : (size_t)r * 64 + q * 8 + c) * c_out + co;
        float acc = 0.f;
        for (int sp = 0; sp < splits; ++sp) acc += part[(size_t)sp * slice + o];
        dw[(size_t)co * kdim + k] = s * acc;
        if (vec3) dot = fmaf(acc, load_h16(w + (size_t)co * kdim + k, f16), dot);
    }
    float bs = 0.f;
    if (need_sums)
        for (int sp = threadIdx.x; sp < splits; sp += blockDim.x)   // sum dZ: its own array, or k row `sum_row`
            bs += sum_row >= 0 ? part[(size_t)sp * slice + (size_t)sum_row * c_out + co] : bsum[(size_t)sp * c_out + co];
    red[threadIdx.x] = dot;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) { if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o]; __syncthreads(); }
    const float dot_all = red[0];
    __syncthreads();
    red[threadIdx.x] = bs;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) { if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o]; __syncthreads(); }
    if (threadIdx.x == 0 && need_sums) {
        const float dsum = red[0];
        if (vec3) {
            const float r = vec3[2 * c_out + co];
            dbeta[co] = dsum;
            if (db) db[co] = s * dsum;
            dgamma[co] = r * (dot_all + dsum * ((b ? b[co] : 0.f) - mean[co]));
        } else if (db) {
            db[co] = dsum;
        }
    }
}

cudaError_t launch_wgrad_epilogue_stem(const Problem &pb, const UmmaWgradPlan &pl, const float *partials,
                                       const float *bsum, const void *w, const float *vec3, const float *b,
                                       const float *mean, float *dw, float *db, float *dgamma, float *dbeta,
                                       bool need_sums, cudaStream_t st) {
    wgrad_epilogue_stem_kernel<<<pb.c_out, 256, 0, st>>>(pb.c_out, pb.kh, pb.kw, pb.c_in, stem_krows(pb), stem_s2d(pb) ? 1 : 0,
                                                         stem_ones_in_pack(pb) ? 3 : -1, partials, pl.splits, bsum,
                                                         (const __nv_bfloat16 *)w, vec3, b, mean, dw, db, dgamma, dbeta,
                                                         need_sums ? 1 : 0, call_f16());
    return cudaGetLastError();
}

}  // namespace convbn

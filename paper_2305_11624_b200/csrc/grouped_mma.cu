// Grouped convolution with 8 channels per group (C_in/G = C_out/G = 8), bf16 NHWC, unit stride and dilation:
//   Z[p, 8g + o] = b'[8g + o] + sum_{tap, ci} omega'[8g + o][tap][ci] X[p + tap, 8g + ci]     (Sec. 3.1 / 3.3)
// and, with rotated and transposed weights, the backward-data pass (Sec. 3.2.1).
// One group is a GEMM with N = 8 and K = 8 per tap (about 36 FLOP per byte moved): far too narrow for a
// 128-row tcgen05 tile, whose block-diagonal emulation spends 8x the MMA work and was bound by it, but an
// exact fit for the warp-level m16n8k16 MMA: 16 pixels x (2 taps x 8 input channels) x 8 output channels.
// The kernel is organised around the memory stream.  Work item = (image, band of R output rows (of a column strip),
// 64-channel chunk); a producer warp brings the item's input patch ((R + kh - 1) rows x (W + kw - 1) columns x 64
// channels, zero fill outside the image) into a ring of shared-memory stages with one TMA box (128-byte
// swizzle).  Compute warp w owns group w of the chunk: its A fragments are ldmatrix loads of [pixel][8
// channels] rows at the tap's shifted start address (virtual pixels, row pitch W + kw - 1: the outputs of
// the halo columns are computed and dropped), which the swizzle makes bank-conflict free; its B fragments
// (the group's 8 x 8 weights per tap) sit in registers.  The warps' results (16 bytes per pixel and group) meet in
// a shared-memory image of the band, which leaves as one TMA box: stored by the lanes themselves they were half
// sectors, 8 lines per instruction, and the load/store unit (77 % busy with them and the ldmatrix reads) was the bound.
// The per-channel transform costs no launch of its own: the forward pass forms s and b'
// per lane and applies them to the fp32 accumulators (omega is not rounded), the backward-data pass builds
// s omega, rotated and transposed, while it loads its B fragments (reparam + flip kernels: 6 us of a 76 us
// step at C = 256, 28 x 28, N = 64).
#include "kernels.h"
#include "mma_sync.cuh"
#include "sm100_ptx.cuh"

namespace convbn {

namespace {

using namespace ptx;

constexpr int kGMaxStages = 8;
constexpr int kGMaxKSteps = 5;       // up to 10 taps (3 x 3), two per k-step; the loops over them are unrolled
constexpr int kGThreads = 288;       // 8 compute warps + the producer warp
constexpr int kGTiles = 4;           // 16-pixel MMA tiles a warp works on at a time

struct GroupedCtl {
    uint64_t full[kGMaxStages], empty[kGMaxStages];
    int abort_flag;
};

struct GroupedGeom {
    int n, ho, wo, c, kh, kw, lower_h, lower_w;
    int R, Wt, rows_in, tiles_h;
    int cols, tiles_w;         // output columns of a band (convolution only: wide images are cut into column strips)
    int stages;
    uint32_t patch_bytes;      // bytes one TMA box writes
    uint32_t stage_stride;     // allocation per stage (multiple of 1024, includes the read-ahead tail)
    uint32_t out_bytes;        // output image of a band, R x W x 128, and one row for what is dropped (multiple of 1024)
};

// DGRAD: w is the layer's own [C][taps][8] weight tensor, read rotated and with the channel roles exchanged,
// times scale[output channel of the layer] (NULL = 1).  Otherwise out = w (*) act + bias, or with
// fold.gamma != NULL out = s (w (*) act) + b' from the BatchNorm parameters.
template <bool H, bool DGRAD>            // H: IEEE-half storage, else bf16
__global__ void __launch_bounds__(kGThreads, 3) grouped8_conv_kernel(const __grid_constant__ CUtensorMap tm_act,
                                                                 const __grid_constant__ CUtensorMap tm_out,
                                                                 const GroupedGeom g,
                                                                 const __nv_bfloat16 *__restrict__ w,
                                                                 const float *__restrict__ bias,
                                                                 const float *__restrict__ scale, const BnFold fold, int *err) {
    extern __shared__ uint8_t grouped_smem_raw[];
    uint8_t *ring = (uint8_t *)(((uintptr_t)grouped_smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *image = ring + (size_t)g.stages * g.stage_stride;
    GroupedCtl *ctl = (GroupedCtl *)(image + g.out_bytes);
    volatile int *abort_flag = &ctl->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int taps = g.kh * g.kw, ksteps = (taps + 1) / 2, chunks = g.c / 64;
    if (threadIdx.x == 0) {
        for (int s = 0; s < g.stages; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 8); }
        ctl->abort_flag = 0;
        fence_barrier_init();
    }
    if (threadIdx.x == 256) { prefetch_tensormap(&tm_act); prefetch_tensormap(&tm_out); }
    __syncthreads();
    pdl_wait();
    pdl_launch_dependents();
    if (threadIdx.x == 0) { CONVBN_TRACE_POINT(0); }
    const uint32_t items = (uint32_t)g.n * g.tiles_h * g.tiles_w * chunks;   // chunk fastest: a patch's chunks run together
    if (warp == 8) {
        if (lane == 0) {
            uint32_t s = 0, ph = 0;
            bool ok = true;
            for (uint32_t it = blockIdx.x; it < items; it += gridDim.x) {
                const int cc = (int)(it % (uint32_t)chunks);
                const uint32_t t1 = it / (uint32_t)chunks;
                const uint32_t t2 = t1 / (uint32_t)g.tiles_w;
                const int w0 = (int)(t1 - t2 * (uint32_t)g.tiles_w) * g.cols;
                const int h0 = (int)(t2 % (uint32_t)g.tiles_h) * g.R, img = (int)(t2 / (uint32_t)g.tiles_h);
                if (!mbar_wait_bounded(&ctl->empty[s], ph ^ 1u, abort_flag)) { ok = false; break; }
                mbar_arrive_expect_tx(&ctl->full[s], g.patch_bytes);
                tma_load_4d(ring + (size_t)s * g.stage_stride, &tm_act, &ctl->full[s], cc * 64, w0 + g.lower_w,
                            h0 + g.lower_h, img);
                if (++s == (uint32_t)g.stages) { s = 0; ph ^= 1u; }
            }
            if (!ok) { atomicOr(err, ERRW_TIMEOUT); ctl->abort_flag = 1; }
        }
        return;
    }
    // ---- compute warps: warp = group inside the 64-channel chunk ----
    const int gr = lane >> 2, t = lane & 3;
    // ldmatrix.x4: lanes 0-7 address the rows of matrix 0 (pixels 0-7, first tap), 8-15 matrix 1 (pixels
    // 8-15, first tap), 16-23 matrix 2 (pixels 0-7, second tap), 24-31 matrix 3 (pixels 8-15, second tap)
    const int lm_pix = (lane & 7) + ((lane >> 3) & 1) * 8, lm_tap = lane >> 4;
    // the grid is a multiple of the chunk count: a block keeps one chunk, so its weights are loaded once
    const int cc = (int)(blockIdx.x % (uint32_t)chunks);
    const int ch0 = cc * 64 + warp * 8;                    // first channel of this warp's group
    // B fragments: k = 8 (tap in the step) + ci, n = output channel gr; lane holds ci = 2t, 2t + 1
    uint32_t bf[kGMaxKSteps][2];
    float sc0 = 1.f, sc1 = 1.f, b0 = 0.f, b1 = 0.f;
    if constexpr (DGRAD) {
        // row gr of this pass is the layer's input channel, k its output channel: s[o] w[o][taps - 1 - tap][gr]
        const __nv_bfloat16 *w0 = w + ((size_t)(ch0 + 2 * t) * taps + taps - 1) * 8 + gr, *w1 = w0 + (size_t)taps * 8;
        if (scale) { sc0 = scale[ch0 + 2 * t]; sc1 = scale[ch0 + 2 * t + 1]; }
#pragma unroll
        for (int i = 0; i < 2 * kGMaxKSteps; ++i)
            bf[i / 2][i % 2] = i < taps ? pack2_t<H>(sc0 * load_h16(w0 - (ptrdiff_t)i * 8, H), sc1 * load_h16(w1 - (ptrdiff_t)i * 8, H)) : 0u;
    } else {
        const __nv_bfloat16 *wrow = w + ((size_t)(ch0 + gr) * taps) * 8 + 2 * t;
#pragma unroll
        for (int i = 0; i < 2 * kGMaxKSteps; ++i)
            bf[i / 2][i % 2] = i < taps ? *reinterpret_cast<const uint32_t *>(wrow + (size_t)i * 8) : 0u;
        if (fold.gamma) {
            float r[2], sc[2], sh[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int c = ch0 + 2 * t + e;
                r[e] = 1.0f / sqrtf(fold.var[c] + fold.eps);
                sc[e] = fold.gamma[c] * r[e];
                sh[e] = ((fold.b ? fold.b[c] : 0.f) - fold.mean[c]) * sc[e] + fold.beta[c];
                if (blockIdx.x < (uint32_t)chunks && gr == 0 && fold.vec3) {     // blocks 0 .. chunks - 1: one per chunk of channels
                    fold.vec3[c] = sc[e]; fold.vec3[g.c + c] = sh[e]; fold.vec3[2 * g.c + c] = r[e];
                }
            }
            sc0 = sc[0]; sc1 = sc[1]; b0 = sh[0]; b1 = sh[1];
        } else if (bias) {
            b0 = bias[ch0 + 2 * t]; b1 = bias[ch0 + 2 * t + 1];
        }
    }
    // this lane's ldmatrix row of k-step ks, relative to the tile start: its pixel plus the shift of its tap
    int vrow[kGMaxKSteps];
    {
        int r = 0, q = 0;                                  // tap 2 ks
#pragma unroll
        for (int ks = 0; ks < kGMaxKSteps; ++ks) {
            int r1 = r, q1 = q + 1;                        // tap 2 ks + 1
            if (q1 == g.kw) { q1 = 0; ++r1; }
            const bool second = lm_tap && 2 * ks + 1 < taps;   // an absent second tap re-reads the first (weights 0)
            vrow[ks] = lm_pix + (second ? r1 * g.Wt + q1 : r * g.Wt + q);
            r = r1; q = q1 + 1;
            if (q >= g.kw) { q -= g.kw; ++r; }
        }
    }
    const int npix = g.R * g.Wt;                               // virtual pixels of a full band
    const uint32_t image_s = smem_u32(image);
    uint32_t s = 0, ph = 0;
    bool ok = true;
    for (uint32_t it = blockIdx.x; it < items && ok; it += gridDim.x) {
        const uint32_t t1 = it / (uint32_t)chunks, t2 = t1 / (uint32_t)g.tiles_w;
        const int w0 = (int)(t1 - t2 * (uint32_t)g.tiles_w) * g.cols;
        const int h0 = (int)(t2 % (uint32_t)g.tiles_h) * g.R, img = (int)(t2 / (uint32_t)g.tiles_h);
        ok = mbar_wait_bounded(&ctl->full[s], ph, abort_flag);
        // the image buffer is free once the box of the item before has been read out of it; the warps leave together
        if (threadIdx.x == 0) tma_store_wait_read<0>();
        ok = named_bar_all(1, 256, ok);
        if (!ok) break;
        if (threadIdx.x == 0) { if (it == blockIdx.x) CONVBN_TRACE_POINT(1); CONVBN_TRACE_POINT(3); }
        const uint32_t patch = smem_u32(ring + (size_t)s * g.stage_stride);
        // four 16-pixel tiles at a time: their MMA chains are independent, so the loads of one overlap
        // the arithmetic of the others
        for (int v0 = 0; v0 < npix; v0 += 16 * kGTiles) {
            float acc[kGTiles][4];
#pragma unroll
            for (int u = 0; u < kGTiles; ++u) acc[u][0] = acc[u][1] = acc[u][2] = acc[u][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < kGMaxKSteps; ++ks) {
                if (ks >= ksteps) break;                       // the same for every lane
                const int v = v0 + vrow[ks];
                // tiles are 16 rows = 2048 bytes apart, which leaves the swizzle term unchanged
                const uint32_t addr = patch + (uint32_t)v * 128u + (uint32_t)((warp ^ (v & 7)) << 4);
                uint32_t a[kGTiles][4];
#pragma unroll
                for (int u = 0; u < kGTiles; ++u) ldmatrix_x4(a[u][0], a[u][1], a[u][2], a[u][3], addr + (uint32_t)u * 2048u);
#pragma unroll
                for (int u = 0; u < kGTiles; ++u) mma_16x8x16_t<H>(acc[u], a[u][0], a[u][1], a[u][2], a[u][3], bf[ks][0], bf[ks][1]);
            }
            // rows 0-7 / 8-15 of tile u are matrices 2 u / 2 u + 1 of the stores: this lane addresses virtual pixel
            // v0 + lane of the first two tiles, v0 + 32 + lane of the last two; halo columns go to the spare row
            uint32_t o[2 * kGTiles];
#pragma unroll
            for (int u = 0; u < kGTiles; ++u)
#pragma unroll
                for (int half = 0; half < 2; ++half)
                    o[2 * u + half] = DGRAD ? pack2_t<H>(acc[u][2 * half], acc[u][2 * half + 1])
                                            : pack2_t<H>(fmaf(acc[u][2 * half], sc0, b0), fmaf(acc[u][2 * half + 1], sc1, b1));
#pragma unroll
            for (int u = 0; u < kGTiles; u += 2) {
                const int v = v0 + 16 * u + lane, ti = v / g.Wt, tj = v - ti * g.Wt;
                const int row = (ti < g.R && tj < g.cols) ? ti * g.cols + tj : g.R * g.cols;
                stmatrix_x4(image_s + (uint32_t)row * 128u + (uint32_t)((warp ^ (row & 7)) << 4), o[2 * u], o[2 * u + 1],
                            o[2 * u + 2], o[2 * u + 3]);
            }
        }
        fence_proxy_async_smem();
        named_bar_sync(1, 256);
        if (threadIdx.x == 0) {                    // rows and columns outside the image are clipped by the map
            tma_store_4d(&tm_out, image, cc * 64, w0, h0, img);
            tma_store_commit();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl->empty[s]);
        if (threadIdx.x == 0) { if (it == blockIdx.x) CONVBN_TRACE_POINT(2); CONVBN_TRACE_POINT(4); }
        if (++s == (uint32_t)g.stages) { s = 0; ph ^= 1u; }
    }
    if (threadIdx.x == 0) tma_store_wait_all<0>();
    if (!ok && lane == 0) { atomicOr(err, ERRW_TIMEOUT); ctl->abort_flag = 1; }
}

// ---- backward weight -----------------------------------------------------------------------------------
//   domega'[8g + o][tap][ci] = sum_p dZ[p][8g + o] X[p + tap][8g + ci],   sum_p dZ[p][8g + o]      (Sec. 3.2.1)
// The same patch stream with two boxes per stage: the X patch and the dZ band, the latter on the same
// virtual-pixel grid (row pitch W + kw - 1, its extra columns lie outside the tensor and arrive as zeros,
// so the products of the halo positions vanish).  Per group and 16 virtual pixels: K = the pixels,
// M = (2 taps x 8 input channels), N = 8 output channels; both operands come out of shared memory with
// transposing ldmatrix loads.  sum dZ is a row of ones: it takes the place of the tap that an odd tap count leaves
// empty in the last step (a further MMA when there is none).  A block keeps one
// 64-channel chunk for its whole life, so the sums stay in registers across its bands; at the end every
// warp writes its group's partial block: part[slot][C][taps 8], bsum[slot][C].
template <bool H>
__global__ void __launch_bounds__(kGThreads) grouped8_wgrad_kernel(const __grid_constant__ CUtensorMap tm_x,
                                                                  const __grid_constant__ CUtensorMap tm_dz,
                                                                  const GroupedGeom g, uint32_t dz_off, int slots,
                                                                  float *__restrict__ part, float *__restrict__ bsum,
                                                                  int *err) {
    extern __shared__ uint8_t grouped_smem_raw[];
    uint8_t *ring = (uint8_t *)(((uintptr_t)grouped_smem_raw + 1023) & ~(uintptr_t)1023);
    GroupedCtl *ctl = (GroupedCtl *)(ring + (size_t)g.stages * g.stage_stride);
    volatile int *abort_flag = &ctl->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int taps = g.kh * g.kw, ksteps = (taps + 1) / 2, chunks = g.c / 64;
    // the regions TMA never writes (read-ahead tails, the gap between the two boxes) are read as operands:
    // they have to hold zeros, not whatever the last kernel left there
    for (uint32_t i = threadIdx.x; i < (uint32_t)g.stages * g.stage_stride / 16; i += kGThreads)
        reinterpret_cast<uint4 *>(ring)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (threadIdx.x == 0) {
        for (int s = 0; s < g.stages; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 8); }
        ctl->abort_flag = 0;
        fence_barrier_init();
    }
    fence_proxy_async_smem();
    if (threadIdx.x == 256) { prefetch_tensormap(&tm_x); prefetch_tensormap(&tm_dz); }
    __syncthreads();
    pdl_wait();
    const int cc = (int)(blockIdx.x % (uint32_t)chunks), slot = (int)(blockIdx.x / (uint32_t)chunks);
    const uint32_t items = (uint32_t)g.n * g.tiles_h;          // bands of this chunk
    const uint32_t x_bytes = g.patch_bytes, dz_bytes = (uint32_t)g.R * g.Wt * 128u;
    float acc[kGMaxKSteps][4], accs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int ks = 0; ks < kGMaxKSteps; ++ks) acc[ks][0] = acc[ks][1] = acc[ks][2] = acc[ks][3] = 0.f;
    if (warp == 8) {
        if (lane == 0) {
            uint32_t s = 0, ph = 0;
            bool ok = true;
            for (uint32_t it = (uint32_t)slot; it < items; it += (uint32_t)slots) {
                const int h0 = (int)(it % (uint32_t)g.tiles_h) * g.R, img = (int)(it / (uint32_t)g.tiles_h);
                if (!mbar_wait_bounded(&ctl->empty[s], ph ^ 1u, abort_flag)) { ok = false; break; }
                uint8_t *dst = ring + (size_t)s * g.stage_stride;
                mbar_arrive_expect_tx(&ctl->full[s], x_bytes + dz_bytes);
                tma_load_4d(dst, &tm_x, &ctl->full[s], cc * 64, g.lower_w, h0 + g.lower_h, img);
                tma_load_4d(dst + dz_off, &tm_dz, &ctl->full[s], cc * 64, 0, h0, img);
                if (++s == (uint32_t)g.stages) { s = 0; ph ^= 1u; }
            }
            if (!ok) { atomicOr(err, ERRW_TIMEOUT); ctl->abort_flag = 1; }
        }
        return;
    }
    const int gr = lane >> 2, t = lane & 3;
    // A: matrix 0 = pixels 0-7 of the first tap, 1 = pixels 0-7 of the second, 2 / 3 = pixels 8-15
    const int lm_pix = (lane & 7) + (lane >> 4) * 8, lm_tap = (lane >> 3) & 1;
    int vrow[kGMaxKSteps];
    {
        int r = 0, q = 0;
#pragma unroll
        for (int ks = 0; ks < kGMaxKSteps; ++ks) {
            int r1 = r, q1 = q + 1;
            if (q1 == g.kw) { q1 = 0; ++r1; }
            const bool second = lm_tap && 2 * ks + 1 < taps;   // an absent second tap re-reads the first (its rows are dropped)
            vrow[ks] = lm_pix + (second ? r1 * g.Wt + q1 : r * g.Wt + q);
            r = r1; q = q1 + 1;
            if (q >= g.kw) { q -= g.kw; ++r; }
        }
    }
    const int npix = g.R * g.Wt;
    const uint32_t ones = one_h16(H ? 1 : 0) * 0x10001u;       // 1.0 twice
    uint32_t s = 0, ph = 0;
    bool ok = true;
    for (uint32_t it = (uint32_t)slot; it < items && ok; it += (uint32_t)slots) {
        if (!mbar_wait_bounded(&ctl->full[s], ph, abort_flag)) { ok = false; break; }
        const uint32_t xpatch = smem_u32(ring + (size_t)s * g.stage_stride), dzpatch = xpatch + dz_off;
#pragma unroll 2
        for (int v0 = 0; v0 < npix; v0 += 16) {
            uint32_t b0, b1;
            {
                const int v = v0 + (lane & 15);
                ldmatrix_x2_trans(b0, b1, dzpatch + (uint32_t)v * 128u + (uint32_t)((warp ^ (v & 7)) << 4));
            }
            if (!(taps & 1)) mma_16x8x16_t<H>(accs, ones, ones, ones, ones, b0, b1);
#pragma unroll
            for (int ks = 0; ks < kGMaxKSteps; ++ks) {
                if (ks >= ksteps) break;
                const int v = v0 + vrow[ks];
                uint32_t a0, a1, a2, a3;
                ldmatrix_x4_trans(a0, a1, a2, a3, xpatch + (uint32_t)v * 128u + (uint32_t)((warp ^ (v & 7)) << 4));
                if (2 * ks + 1 >= taps) a1 = a3 = ones;
                mma_16x8x16_t<H>(acc[ks], a0, a1, a2, a3, b0, b1);
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl->empty[s]);
        if (++s == (uint32_t)g.stages) { s = 0; ph ^= 1u; }
    }
    if (!ok && lane == 0) { atomicOr(err, ERRW_TIMEOUT); ctl->abort_flag = 1; }
    pdl_launch_dependents();       // (earlier, the adding kernel's blocks would wait here and take the data pass's room:
                                   // forward + backward of 256 channels at 28 x 28, N = 64 57.9 -> 53.9 us)
    // accumulator registers: (row gr = input channel of the first tap, columns 2t, 2t + 1 = output channels),
    // (row gr + 8 = the same input channel of the second tap)
    const int ch0 = cc * 64 + warp * 8, kdim = taps * 8;
    float *prow0 = part + ((size_t)slot * g.c + ch0 + 2 * t) * kdim, *prow1 = prow0 + kdim;
#pragma unroll
    for (int ks = 0; ks < kGMaxKSteps; ++ks) {
        if (2 * ks < taps) {
            prow0[(2 * ks) * 8 + gr] = acc[ks][0];
            prow1[(2 * ks) * 8 + gr] = acc[ks][1];
        }
        if (2 * ks + 1 < taps) {
            prow0[(2 * ks + 1) * 8 + gr] = acc[ks][2];
            prow1[(2 * ks + 1) * 8 + gr] = acc[ks][3];
        } else if (2 * ks < taps) {
            accs[0] = acc[ks][2]; accs[1] = acc[ks][3];
        }
    }
    if (gr == 0) {
        bsum[(size_t)slot * g.c + ch0 + 2 * t] = accs[0];
        bsum[(size_t)slot * g.c + ch0 + 2 * t + 1] = accs[1];
    }
}

// Adds the block partials and forms the parameter gradients (Table 2, Tune row):
//   domega = s domega', dbeta = sum dZ, db = s dbeta, dgamma = r (sum_k domega' omega + dbeta (b - mu_hat)).
// vec3 == NULL: domega = domega', db = sum dZ.  One block per output channel: thread (k, j) adds slots
// j, j + ng, ... of entry k (a slot's kdim <= 80 entries are contiguous, so the loads coalesce), the ng
// slot groups are then added in order, and the last group column does the same for sum dZ.
// Bound by the latency of the slot reads (the partials are in L2): a thread requests four slots before it adds the first.
constexpr int kGFinThreads = 512;            // at most
__global__ void __launch_bounds__(kGFinThreads) grouped8_wgrad_finish_kernel(int c, int kdim, int slots,
                                                                            const float *__restrict__ part,
                                                                            const float *__restrict__ bsum,
                                                                            const __nv_bfloat16 *__restrict__ w,
                                                                            const float *__restrict__ vec3,
                                                                            const float *__restrict__ b,
                                                                            const float *__restrict__ mean,
                                                                            float *__restrict__ dw, float *__restrict__ db,
                                                                            float *__restrict__ dgamma,
                                                                            float *__restrict__ dbeta, int f16) {
    __shared__ float red[kGFinThreads];
    __shared__ float dots[96];
    pdl_wait();
    pdl_launch_dependents();
    const int co = blockIdx.x;
    const int ng = (int)blockDim.x / (kdim + 1);     // slot groups; column kdim of each group sums dZ
    const int k = threadIdx.x % (kdim + 1), j = threadIdx.x / (kdim + 1);
    float sum = 0.f;
    if (j < ng) {
        const float *src = k < kdim ? part + (size_t)co * kdim + k : bsum + co;
        const size_t pitch = k < kdim ? (size_t)c * kdim : (size_t)c;
        for (int sl = j; sl < slots; sl += 4 * ng) {
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = sl + u * ng < slots ? __ldcg(src + (size_t)(sl + u * ng) * pitch) : 0.f;
            sum += (v[0] + v[1]) + (v[2] + v[3]);
        }
    }
    red[threadIdx.x] = sum;
    __syncthreads();
    const float s = vec3 ? vec3[co] : 1.f;
    if (threadIdx.x <= kdim) {
        float tot = 0.f;
        for (int jj = 0; jj < ng; ++jj) tot += red[jj * (kdim + 1) + threadIdx.x];
        if (threadIdx.x < kdim) {
            dw[(size_t)co * kdim + threadIdx.x] = s * tot;
            dots[threadIdx.x] = vec3 ? tot * load_h16(w + (size_t)co * kdim + threadIdx.x, f16) : 0.f;
        } else {
            dots[kdim] = tot;                        // sum dZ
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        float d = 0.f;
        for (int i = threadIdx.x; i < kdim; i += 32) d += dots[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        if (threadIdx.x == 0) {
            const float dsum = dots[kdim];
            if (vec3) {
                dbeta[co] = dsum;
                if (db) db[co] = s * dsum;
                dgamma[co] = vec3[2 * c + co] * (d + dsum * ((b ? b[co] : 0.f) - mean[co]));
            } else if (db) {
                db[co] = dsum;
            }
        }
    }
}

struct GroupedPlan { bool ok = false; GroupedGeom g; size_t smem = 0; unsigned grid = 0; uint32_t dz_off = 0; int bps = 1; };

GroupedPlan plan_grouped8(int n, int h_in, int w_in, int c, int ho, int wo, int kh, int kw, int lower_h, int lower_w,
                          bool with_dz = false) {
    GroupedPlan pl;
    (void)h_in; (void)w_in;
    if (kh * kw > 2 * kGMaxKSteps || c % 64) return pl;
    const int sms = device_sm_count();
    // The compute warps of one block (8, two per scheduler) cannot hide the ldmatrix -> MMA latency on their own, so
    // the bands are kept small enough for two or three blocks per SM, two stages each (a third stage costs blocks:
    // 19.2 -> 21.5 us at R = 4).  Estimated time: bands of an SM, and one more for the tail, x input pixels of a band
    // and its fixed cost, derated for how many blocks share the SM.  C = 256, 28 x 28, N = 64, forward: R = 2 20.9 us,
    // 3 23.6, 4 19.2, 5 23.8, 7 23.6, 10 27.4.
    double best = -1.0;
    // Column strips of at most 64 keep several rows in a band of a wide image (a band is one TMA box of at most 256
    // columns, and two stages of it have to fit).  The weight gradient takes none: its dZ band relies on zeros to the
    // right of the image.  Narrow images are not cut: at 28 x 28, N = 64 two strips of 14 cost 64.7 us per forward +
    // backward, none 61.6.
    const int tiles_w = with_dz ? 1 : (wo + 63) / 64;
    const int cols = (wo + tiles_w - 1) / tiles_w, wt = cols + kw - 1;
    if (wt > 256 || wt < 8) return pl;
    for (int r = 1; r <= ho && r + kh - 1 <= 256; ++r) {
        const int rows_in = r + kh - 1;
        // stage = the box, plus what the last group of tiles reads past it
        const size_t px = (size_t)((r * wt + 16 * kGTiles - 1) / (16 * kGTiles) * (16 * kGTiles)) + (size_t)(kh - 1) * wt + kw;
        const size_t need = px > (size_t)rows_in * wt ? px : (size_t)rows_in * wt;
        size_t stride = (need * 128 + 1023) / 1024 * 1024;
        const size_t dz_off = stride;                          // the dZ band sits behind the X patch
        if (with_dz) stride += ((size_t)((r * wt + 15) / 16 * 16) * 128 + 1023) / 1024 * 1024;
        const size_t out_bytes = with_dz ? 0 : ((size_t)(r * cols + 1) * 128 + 1023) / 1024 * 1024;
        const int tiles_h = (ho + r - 1) / r;
        const long long items = (long long)n * tiles_h * tiles_w * (c / 64);
        for (int stages = 2; stages <= 4; ++stages) {
            const size_t smem = 1024 + (size_t)stages * stride + out_bytes + sizeof(GroupedCtl);
            if (smem > 220 * 1024) break;
            int bps = (int)((226 * 1024) / (smem + 1024));
            if (bps > 3) bps = 3;
            if (bps < 1) break;
            const long long slots = (long long)sms * bps;
            const double share = bps == 1 ? 1.9 : (bps == 2 ? 1.25 : 1.0);     // time per item relative to 3 blocks per SM
            const double cost = ((double)items / sms + 1.0) * (rows_in * (double)wt + 40.0) * share;
            if (best < 0 || cost < best) {
                best = cost;
                pl.ok = true;
                pl.g.R = r; pl.g.Wt = wt; pl.g.rows_in = rows_in; pl.g.tiles_h = tiles_h;
                pl.g.cols = cols; pl.g.tiles_w = tiles_w; pl.g.stages = stages;
                pl.g.patch_bytes = (uint32_t)((size_t)rows_in * wt * 128);
                pl.g.stage_stride = (uint32_t)stride;
                pl.g.out_bytes = (uint32_t)out_bytes;
                pl.dz_off = (uint32_t)dz_off;
                pl.bps = bps;
                pl.smem = smem;
                // a multiple of the chunk count (the items are one already): a block then keeps one chunk of channels
                pl.grid = (unsigned)(items < slots ? items : (slots >= c / 64 ? slots - slots % (c / 64) : c / 64));
            }
        }
    }
    pl.g.n = n; pl.g.ho = ho; pl.g.wo = wo; pl.g.c = c; pl.g.kh = kh; pl.g.kw = kw;
    pl.g.lower_h = lower_h; pl.g.lower_w = lower_w;
    return pl;
}

}  // namespace

bool grouped8_eligible(const Problem &pb) {
    return pb.groups > 1 && pb.cg == 8 && pb.cog == 8 && pb.c_in % 64 == 0 && pb.stride_h == 1 && pb.stride_w == 1 &&
           pb.dil_h == 1 && pb.dil_w == 1 && pb.kh * pb.kw <= 2 * kGMaxKSteps && pb.w_out + pb.kw - 1 <= 256 &&
           pb.w_in + pb.kw - 1 <= 256 && pb.pad_h <= 128 && pb.pad_w <= 128 && pb.p < (1LL << 30) &&
           pb.pin < (1LL << 30);
}

// act: [n][ha][wa][c]; out: [n][ho][wo][c]; w: [c][kh kw][8], the layer's weights in either direction
template <bool DGRAD>
static cudaError_t launch_grouped8(int n, int ha, int wa, int c, int ho, int wo, int kh, int kw, int lower_h,
                                   int lower_w, const void *act, const void *w, const float *bias, const float *scale,
                                   const BnFold *fold, void *out, cudaStream_t st) {
    const GroupedPlan pl = plan_grouped8(n, ha, wa, c, ho, wo, kh, kw, lower_h, lower_w);
    if (!pl.ok) return cudaErrorInvalidValue;
    CUtensorMap ta;
    const unsigned long long dims[4] = {(unsigned long long)c, (unsigned long long)wa, (unsigned long long)ha,
                                        (unsigned long long)n};
    const unsigned long long str[4] = {0, (unsigned long long)c * 2, (unsigned long long)wa * c * 2,
                                       (unsigned long long)ha * wa * c * 2};
    const unsigned int box[4] = {64, (unsigned)pl.g.Wt, (unsigned)pl.g.rows_in, 1};
    if (!make_tmap_tiled_bf16(&ta, act, 4, dims, str, box)) return cudaErrorInvalidValue;
    CUtensorMap tout;
    {
        const unsigned long long odims[4] = {(unsigned long long)c, (unsigned long long)wo, (unsigned long long)ho,
                                             (unsigned long long)n};
        const unsigned long long ostr[4] = {0, (unsigned long long)c * 2, (unsigned long long)wo * c * 2,
                                            (unsigned long long)ho * wo * c * 2};
        const unsigned int obox[4] = {64, (unsigned)pl.g.cols, (unsigned)pl.g.R, 1};
        if (!make_tmap_tiled_bf16(&tout, out, 4, odims, ostr, obox)) return cudaErrorInvalidValue;
    }
    int *err = nullptr;
    cudaError_t e = error_word_address(&err);
    if (e != cudaSuccess) return e;
    const BnFold fd = fold ? *fold : BnFold{nullptr, nullptr, nullptr, nullptr, nullptr, 0.f, nullptr};
    static PerDevice attr, attr_h;        // (one flag per instantiation)
    if (call_f16()) {
        if ((e = max_dynamic_smem_once(grouped8_conv_kernel<true, DGRAD>, 220 * 1024, &attr_h)) != cudaSuccess) return e;
        return launch_pdl(grouped8_conv_kernel<true, DGRAD>, dim3(pl.grid), dim3(kGThreads), pl.smem, st, ta, tout,
                          pl.g, (const __nv_bfloat16 *)w, bias, scale, fd, err);
    }
    if ((e = max_dynamic_smem_once(grouped8_conv_kernel<false, DGRAD>, 220 * 1024, &attr)) != cudaSuccess) return e;
    return launch_pdl(grouped8_conv_kernel<false, DGRAD>, dim3(pl.grid), dim3(kGThreads), pl.smem, st, ta, tout,
                      pl.g, (const __nv_bfloat16 *)w, bias, scale, fd, err);
}

cudaError_t launch_grouped8_fwd(const Problem &pb, const void *x, const void *w, const float *bias, void *z,
                                cudaStream_t st, const BnFold *fold) {
    return launch_grouped8<false>(pb.n, pb.h_in, pb.w_in, pb.c_in, pb.h_out, pb.w_out, pb.kh, pb.kw, -pb.pad_h, -pb.pad_w,
                                  x, w, bias, nullptr, fold, z, st);
}

// dX = omega'_rot (*) dZ: the same kernel on the mirrored problem
cudaError_t launch_grouped8_dgrad(const Problem &pb, const void *dz, const void *w, const float *s_vec, void *dx,
                                  cudaStream_t st) {
    return launch_grouped8<true>(pb.n, pb.h_out, pb.w_out, pb.c_out, pb.h_in, pb.w_in, pb.kh, pb.kw, pb.pad_h - (pb.kh - 1),
                                 pb.pad_w - (pb.kw - 1), dz, w, nullptr, s_vec, nullptr, dx, st);
}

// Blocks per 64-channel chunk of the backward-weight kernel = partial rows it writes.
static GroupedPlan plan_grouped8_wgrad(const Problem &pb, int *slots) {
    GroupedPlan pl = plan_grouped8(pb.n, pb.h_in, pb.w_in, pb.c_in, pb.h_out, pb.w_out, pb.kh, pb.kw, -pb.pad_h, -pb.pad_w,
                                   true);
    if (!pl.ok) return pl;
    const int sms = device_sm_count();
    const int chunks = pb.c_in / 64;
    long long per_chunk = (long long)sms * pl.bps / chunks;
    const long long bands = (long long)pb.n * pl.g.tiles_h;
    if (per_chunk > bands) per_chunk = bands;
    if (per_chunk < 1) per_chunk = 1;
    *slots = (int)per_chunk;
    pl.grid = (unsigned)(per_chunk * chunks);
    return pl;
}

int grouped8_wgrad_slots(const Problem &pb) {
    int slots = 0;
    return plan_grouped8_wgrad(pb, &slots).ok ? slots : 0;
}

// part: [slots][C][taps 8] floats, bsum: [slots][C] floats (slots = grouped8_wgrad_slots)
cudaError_t launch_grouped8_wgrad(const Problem &pb, const void *dz, const void *x, float *part, float *bsum,
                                  cudaStream_t st) {
    int slots = 0;
    const GroupedPlan pl = plan_grouped8_wgrad(pb, &slots);
    if (!pl.ok) return cudaErrorInvalidValue;
    CUtensorMap tx, tdz;
    {
        const unsigned long long dims[4] = {(unsigned long long)pb.c_in, (unsigned long long)pb.w_in,
                                            (unsigned long long)pb.h_in, (unsigned long long)pb.n};
        const unsigned long long str[4] = {0, (unsigned long long)pb.c_in * 2, (unsigned long long)pb.w_in * pb.c_in * 2,
                                           (unsigned long long)pb.h_in * pb.w_in * pb.c_in * 2};
        const unsigned int box[4] = {64, (unsigned)pl.g.Wt, (unsigned)pl.g.rows_in, 1};
        if (!make_tmap_tiled_bf16(&tx, x, 4, dims, str, box)) return cudaErrorInvalidValue;
    }
    {
        const unsigned long long dims[4] = {(unsigned long long)pb.c_out, (unsigned long long)pb.w_out,
                                            (unsigned long long)pb.h_out, (unsigned long long)pb.n};
        const unsigned long long str[4] = {0, (unsigned long long)pb.c_out * 2, (unsigned long long)pb.w_out * pb.c_out * 2,
                                           (unsigned long long)pb.h_out * pb.w_out * pb.c_out * 2};
        const unsigned int box[4] = {64, (unsigned)pl.g.Wt, (unsigned)pl.g.R, 1};
        if (!make_tmap_tiled_bf16(&tdz, dz, 4, dims, str, box)) return cudaErrorInvalidValue;
    }
    int *err = nullptr;
    cudaError_t e = error_word_address(&err);
    if (e != cudaSuccess) return e;
    static PerDevice attr, attr_h;
    if (call_f16()) {
        if ((e = max_dynamic_smem_once(grouped8_wgrad_kernel<true>, 220 * 1024, &attr_h)) != cudaSuccess) return e;
        return launch_pdl(grouped8_wgrad_kernel<true>, dim3(pl.grid), dim3(kGThreads), pl.smem, st, tx, tdz, pl.g, pl.dz_off,
                          slots, part, bsum, err);
    }
    if ((e = max_dynamic_smem_once(grouped8_wgrad_kernel<false>, 220 * 1024, &attr)) != cudaSuccess) return e;
    return launch_pdl(grouped8_wgrad_kernel<false>, dim3(pl.grid), dim3(kGThreads), pl.smem, st, tx, tdz, pl.g, pl.dz_off,
                      slots, part, bsum, err);
}

cudaError_t launch_grouped8_wgrad_finish(const Problem &pb, const float *part, const float *bsum, const void *w,
                                         const float *vec3, const float *b, const float *mean, float *dw, float *db,
                                         float *dgamma, float *dbeta, cudaStream_t st) {
    const int slots = grouped8_wgrad_slots(pb);
    if (slots <= 0) return cudaErrorInvalidValue;
    // With 256 threads five blocks share an SM.  512 where a thread would go through more than six batches of slots (C = 256,
    // 56 x 16, N = 31, 111 slots: 19.5 and 17.2 us with the GEMM); 1024, which many slots want alone, cost 1.3 to 3.8 times the
    // whole phase from 640 channels on (C = 768, 34 x 12, N = 29: 19.9 and 28.7).
    const int threads = slots > 24 * (256 / (pb.kh * pb.kw * 8 + 1)) ? kGFinThreads : 256;
    return launch_pdl(grouped8_wgrad_finish_kernel, dim3(pb.c_out), dim3(threads), 0, st, pb.c_out, pb.kh * pb.kw * 8,
                      slots, part, bsum, (const __nv_bfloat16 *)w, vec3, b, mean, dw, db, dgamma, dbeta, call_f16());
}

}  // namespace convbn

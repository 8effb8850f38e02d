// fp32 NCHW convolutions with unit stride and dilation, groups = 1 and a 1x1 or 3x3 kernel, up to 128 channels.  (Other fp32
// shapes: direct_kernels.cu.)
//
// At the sizes of unit tests, gradient checks and small networks a pass is bound by its launches and by the length of each
// thread's chain of loads (a 3x3 block of 16 -> 32 channels at 16 x 16, N = 2 is 14 MFLOP; one thread per output took 12 to
// 33 us a kernel in seven launches), so each direction is ONE launch there:
//   forward   Z = s (omega (*) X) + b', s and b' formed in the kernel;
//   backward  blocks of two kinds: domega', sum dZ and all parameter gradients in clusters of eight blocks that add up
//             through distributed shared memory, and dX = (s omega)_rot (*) dZ.
// With more pixels several clusters share the output channels and a second launch adds their sums (f32_wgrad_groups).
#include <cooperative_groups.h>

#include "kernels.h"

namespace cg = cooperative_groups;

namespace convbn {
namespace {

constexpr int kFThreads = 256;
constexpr int kFPix = 64;           // output pixels of a convolution block (of any images)
constexpr int kFChunk = 16;         // input channels whose weights are staged at a time
constexpr int kFCluster = 8;        // blocks of a weight-gradient cluster
constexpr int kFCo = 4;             // output channels of a cluster
constexpr int kFRun = 8;            // consecutive pixels a thread slides its window over

// Outside the image there is nothing to multiply: an infinite weight or dZ beside it must not become 0 x inf = NaN.  The
// loops multiply by staged zeros there; a thread with a sum that is not finite at the end forms its sums again, from global
// memory, without them.  (Looking at every value while it is staged cost the weight gradient 20 %.)
template <int N>
__device__ __forceinline__ bool all_finite(const float (&v)[N]) {
    bool yes = true;
#pragma unroll
    for (int i = 0; i < N; ++i) yes = yes && fabsf(v[i]) < INFINITY;
    return yes;
}

// out[n][oc][p] = scale[oc] sum_{ic, tap} act[n][ic][p + tap - pad] wt(oc, ic, tap) + shift[oc]
struct F32Conv {
    const float *act, *w;
    float *out;
    int n, ic, h, wd, oc, ho, wo, pad;     // pad: of this pass
    const float *k_scale;                  // DGRAD: s of the layer's output channel, here the input channel (NULL = 1)
    const float *bias;                     // without fold (NULL = 0)
    int tiles;                             // tiles of the n ho wo output pixels
};

// Block (oc tile, pixel tile).  256 threads = 64 pixels x 4 groups.  S == 1: the groups are R output channels each,
// the input channels go by in chunks of 16.  S == 4: the groups split the input channels and are added up at the end, R
// output channels per block, which keeps the chain of a thread short when there are too few blocks to hide it.
// Weights are staged as [ic][tap][oc]; a thread's value of the activation meets R of them in one or two broadcasts.
template <int K, int R, int S, bool DGRAD>
__device__ __forceinline__ void conv_tile(const F32Conv &c, int oc0, int tile, const float *scale_s, const float *shift_s,
                                          float *smem) {
    constexpr int KK = K * K, OCT = S == 1 ? 4 * R : R;
    const int lane = threadIdx.x % kFPix, grp = threadIdx.x / kFPix;
    const int hw = c.ho * c.wo, pg = tile * kFPix + lane, img = pg / hw, p = pg - img * hw;
    const bool valid = img < c.n;
    const int y = valid ? p / c.wo : 0, x = valid ? p - y * c.wo : 0;
    bool ok[KK];
#pragma unroll
    for (int r = 0; r < K; ++r)
#pragma unroll
        for (int q = 0; q < K; ++q) {
            const int yy = y - c.pad + r, xx = x - c.pad + q;
            ok[r * K + q] = valid && yy >= 0 && yy < c.h && xx >= 0 && xx < c.wd;
        }
    // (offsets fit an int: fewer than 2^30 elements)
    const int a0 = img * c.ic * c.h * c.wd + (y - c.pad) * c.wd + (x - c.pad), out0 = valid ? (img * c.oc + oc0) * hw + p : -1;
    float acc[R];
#pragma unroll
    for (int j = 0; j < R; ++j) acc[j] = 0.f;
    const int chunk = S == 1 ? kFChunk : c.ic;
    for (int ic0 = 0; ic0 < c.ic; ic0 += chunk) {
        const int nic = c.ic - ic0 < chunk ? c.ic - ic0 : chunk;
        if (ic0) __syncthreads();
        // consecutive threads read consecutive weights: the source rows are [ic][tap] (forward) or [oc][tap] (DGRAD)
        if constexpr (DGRAD) {
            for (int i = threadIdx.x; i < nic * OCT * KK; i += kFThreads) {
                const int t = i % KK, o = (i / KK) % OCT, ci = i / (KK * OCT);
                float v = 0.f;
                if (oc0 + o < c.oc) {
                    v = c.w[((size_t)(ic0 + ci) * c.oc + oc0 + o) * KK + t];
                    if (c.k_scale) v *= c.k_scale[ic0 + ci];
                }
                smem[(ci * KK + KK - 1 - t) * OCT + o] = v;
            }
        } else {
            for (int i = threadIdx.x; i < nic * OCT * KK; i += kFThreads) {
                const int t = i % KK, ci = (i / KK) % nic, o = i / (KK * nic);
                smem[(ci * KK + t) * OCT + o] = oc0 + o < c.oc ? c.w[((size_t)(oc0 + o) * c.ic + ic0 + ci) * KK + t] : 0.f;
            }
        }
        __syncthreads();
        const int per = S == 1 ? nic : (nic + 3) / 4, lo = S == 1 ? 0 : grp * per, hi = S == 1 ? nic : min(nic, lo + per);
#pragma unroll 2
        for (int ci = lo; ci < hi; ++ci) {
            const float *a = c.act + (ptrdiff_t)(a0 + (ic0 + ci) * c.h * c.wd);
            float v[KK];
#pragma unroll
            for (int t = 0; t < KK; ++t) v[t] = ok[t] ? __ldg(a + (t / K) * c.wd + t % K) : 0.f;
            const float *ws = smem + ci * KK * OCT + (S == 1 ? grp * R : 0);
#pragma unroll
            for (int t = 0; t < KK; ++t)
#pragma unroll
                for (int j = 0; j < R; j += 4) {
                    const float4 q = *(const float4 *)(ws + t * OCT + j);
                    acc[j] = fmaf(v[t], q.x, acc[j]); acc[j + 1] = fmaf(v[t], q.y, acc[j + 1]);
                    acc[j + 2] = fmaf(v[t], q.z, acc[j + 2]); acc[j + 3] = fmaf(v[t], q.w, acc[j + 3]);
                }
        }
    }
    if (!all_finite(acc)) {
        const int per = S == 1 ? c.ic : (c.ic + 3) / 4, lo = S == 1 ? 0 : grp * per, hi = min(c.ic, lo + per), o0 = oc0 + (S == 1 ? grp * R : 0);
#pragma unroll
        for (int j = 0; j < R; ++j) acc[j] = 0.f;
#pragma unroll 1
        for (int i = lo * KK; i < hi * KK; ++i) {
            const int ci = i / KK, t = i - ci * KK, yy = y - c.pad + t / K, xx = x - c.pad + t % K;
            if (!valid || yy < 0 || yy >= c.h || xx < 0 || xx >= c.wd) continue;
            const float v = __ldg(c.act + (((size_t)img * c.ic + ci) * c.h + yy) * c.wd + xx);
#pragma unroll
            for (int j = 0; j < R; ++j) {
                if (o0 + j >= c.oc) break;
                const float w = DGRAD ? c.w[((size_t)ci * c.oc + o0 + j) * KK + KK - 1 - t] * (c.k_scale ? c.k_scale[ci] : 1.f)
                                      : c.w[((size_t)(o0 + j) * c.ic + ci) * KK + t];
                acc[j] = fmaf(v, w, acc[j]);
            }
        }
    }
    if constexpr (S == 4) {
        __syncthreads();
#pragma unroll
        for (int j = 0; j < R; ++j) smem[(grp * R + j) * kFPix + lane] = acc[j];
        __syncthreads();
        static_assert(R == 4, "one output channel per group at the end");
        acc[0] = (smem[(0 * R + grp) * kFPix + lane] + smem[(1 * R + grp) * kFPix + lane]) +
                 (smem[(2 * R + grp) * kFPix + lane] + smem[(3 * R + grp) * kFPix + lane]);
    }
    constexpr int NO = S == 1 ? R : 1;
#pragma unroll
    for (int j = 0; j < NO; ++j) {
        const int o = S == 1 ? grp * R + j : grp;
        if (out0 >= 0 && oc0 + o < c.oc)
            c.out[(size_t)(out0 + o * hw)] = DGRAD ? acc[j] : fmaf(acc[j], scale_s[o], shift_s[o]);
    }
}

constexpr int conv_smem_floats(int kk, int r, int s, int ic) {
    const int w = s == 1 ? kFChunk * kk * 4 * r : ic * kk * r;
    return s == 4 && w < kFThreads * r ? kFThreads * r : w;
}

template <int K, int R, int S>
__global__ void __launch_bounds__(kFThreads, K == 1 ? 8 : (S == 1 ? 5 : 4)) f32_fwd_kernel(const F32Conv c, const BnFold fold) {
    extern __shared__ __align__(16) float f32_smem[];
    constexpr int OCT = S == 1 ? 4 * R : R;
    __shared__ float scale_s[OCT], shift_s[OCT];
    // (the kernel behind it starts when this one ends: with an early launch its waiting blocks held the places of blocks still to
    // run.  Forward + backward of 3x3 16 -> 32 at 16 x 16, N = 2 11.7 -> 10.8 us, of 1x1 layers at 56 x 56 36.9 -> 22.5)
    pdl_wait();
    const int oc0 = blockIdx.y * OCT;
    if (threadIdx.x < OCT) {
        const int o = oc0 + threadIdx.x;
        float sc = 1.f, sh = 0.f;
        if (o < c.oc) {
            if (fold.gamma) {
                const float r = 1.0f / sqrtf(fold.var[o] + fold.eps);
                sc = fold.gamma[o] * r;
                sh = ((fold.b ? fold.b[o] : 0.f) - fold.mean[o]) * sc + fold.beta[o];
                if (blockIdx.x == 0 && fold.vec3) {
                    fold.vec3[o] = sc; fold.vec3[c.oc + o] = sh; fold.vec3[2 * c.oc + o] = r;
                }
            } else if (c.bias) {
                sh = c.bias[o];
            }
        }
        scale_s[threadIdx.x] = sc;
        shift_s[threadIdx.x] = sh;
    }
    conv_tile<K, R, S, false>(c, oc0, blockIdx.x, scale_s, shift_s, f32_smem);
}

struct F32Wgrad {
    const float *x, *dz, *w;
    const float *vec3, *b, *mean;          // vec3 NULL: dw = domega', db = sum dZ
    float *dw, *db, *dgamma, *dbeta;
    int groups;                            // clusters that share kFCo output channels
    float *partials, *bsum;                // groups > 1: sums of a cluster, [groups][c_out][c_in K K] and [groups][c_out]
    int n, c_in, h, wd, c_out, ho, wo, pad;
    int cip;                               // power of two >= c_in, 4 .. 128: threads along the input channels
    int rows, bands;                       // output rows of a band, bands of an image
    int xp, zp;                            // pitches of a staged row of X / dZ
    int x_ci;                              // floats between the channels of the staged X (odd)
};

// Cluster = kFCo output channels and one of `groups` shares of the row bands: the 8 groups blocks that have the same channels
// take turns.  A band of X (all channels,
// its halo rows, zeros outside) and of dZ is staged; thread (ci, channel pair, pixel group) slides a K x K window of X
// along runs of eight pixels: K new values and two of dZ per 2 K K multiply-adds.  The pixel groups are added in the block,
// the blocks through distributed shared memory, in rank order; rank j < 4 then finishes output channel j:
//   domega = s domega', dbeta = sum dZ, db = s dbeta, dgamma = r (sum domega' omega + dbeta (b - mu_hat))   (Table 2)
template <int K>
__device__ __forceinline__ void wgrad_cluster(const F32Wgrad &g, int co0, int group, float *smem) {
    constexpr int KK = K * K;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int ci = threadIdx.x % g.cip, rest = threadIdx.x / g.cip;
    const int pair = rest & 1, pg = rest >> 1, npg = kFThreads / (2 * g.cip);
    float *xs = smem, *zs = smem + (size_t)g.c_in * g.x_ci + 1;
    float acc[2][KK], sum[kFCo] = {0.f, 0.f, 0.f, 0.f};      // sum: of the dZ values this thread stages
#pragma unroll
    for (int t = 0; t < KK; ++t) acc[0][t] = acc[1][t] = 0.f;
    const int xrows = g.rows + K - 1, runs = g.zp / kFRun, items = g.n * g.bands;
    for (int it = group * kFCluster + rank; it < items; it += g.groups * kFCluster) {
        const int img = it / g.bands, y0 = (it - img * g.bands) * g.rows;
        __syncthreads();
        for (int i = threadIdx.x; i < g.c_in * xrows * g.xp; i += kFThreads) {
            const int x = i % g.xp, t = i / g.xp, r = t % xrows, c = t / xrows;
            const int yy = y0 - g.pad + r, xx = x - g.pad;
            xs[(size_t)c * g.x_ci + r * g.xp + x] = (yy >= 0 && yy < g.h && xx >= 0 && xx < g.wd)
                                                        ? __ldg(g.x + (((size_t)img * g.c_in + c) * g.h + yy) * g.wd + xx) : 0.f;
        }
        for (int i = threadIdx.x; i < kFCo * g.rows * g.zp; i += kFThreads) {
            const int x = i % g.zp, t = i / g.zp, r = t % g.rows, o = t / g.rows;
            const float v = (co0 + o < g.c_out && y0 + r < g.ho && x < g.wo)
                                ? __ldg(g.dz + (((size_t)img * g.c_out + co0 + o) * g.ho + y0 + r) * g.wo + x) : 0.f;
            zs[i] = v;
#pragma unroll
            for (int q = 0; q < kFCo; ++q) sum[q] += q == o ? v : 0.f;
        }
        __syncthreads();
        const int nruns = min(g.rows, g.ho - y0) * runs;
        if (ci < g.c_in)
            for (int j = pg; j < nruns; j += npg) {
                const int r = j / runs, x = (j - r * runs) * kFRun;
                const float *xr = xs + (size_t)ci * g.x_ci + r * g.xp + x;
                const float *z0 = zs + ((2 * pair) * g.rows + r) * g.zp + x, *z1 = z0 + g.rows * g.zp;
                float win[K][K];
#pragma unroll
                for (int a = 0; a < K; ++a)
#pragma unroll
                    for (int q = 0; q < K - 1; ++q) win[a][q] = xr[a * g.xp + q];
#pragma unroll
                for (int i = 0; i < kFRun; ++i) {
                    const float d0 = z0[i], d1 = z1[i];
#pragma unroll
                    for (int a = 0; a < K; ++a) win[a][(i + K - 1) % K] = xr[a * g.xp + i + K - 1];
#pragma unroll
                    for (int a = 0; a < K; ++a)
#pragma unroll
                        for (int q = 0; q < K; ++q) {
                            const float v = win[a][(i + q) % K];
                            acc[0][a * K + q] = fmaf(d0, v, acc[0][a * K + q]);
                            acc[1][a * K + q] = fmaf(d1, v, acc[1][a * K + q]);
                        }
                }
            }
    }
    if (ci < g.c_in && !(all_finite(acc[0]) && all_finite(acc[1]))) {
#pragma unroll
        for (int t = 0; t < KK; ++t) acc[0][t] = acc[1][t] = 0.f;
#pragma unroll 1
        for (int it = group * kFCluster + rank; it < items; it += g.groups * kFCluster) {
            const int img = it / g.bands, y0 = (it - img * g.bands) * g.rows, nruns = min(g.rows, g.ho - y0) * runs;
#pragma unroll 1
            for (int i = pg * kFRun; i < nruns * kFRun; i += i % kFRun == kFRun - 1 ? (npg - 1) * kFRun + 1 : 1) {      // the same runs
                const int r = i / g.zp, x = i - r * g.zp, y = y0 + r;
                if (x >= g.wo) continue;
                float d[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int o = co0 + 2 * pair + h;
                    d[h] = o < g.c_out ? __ldg(g.dz + (((size_t)img * g.c_out + o) * g.ho + y) * g.wo + x) : 0.f;
                }
#pragma unroll
                for (int t = 0; t < KK; ++t) {
                    const int yy = y + t / K - g.pad, xx = x + t % K - g.pad;
                    if (yy < 0 || yy >= g.h || xx < 0 || xx >= g.wd) continue;
                    const float v = __ldg(g.x + (((size_t)img * g.c_in + ci) * g.h + yy) * g.wd + xx);
                    acc[0][t] = fmaf(d[0], v, acc[0][t]);
                    acc[1][t] = fmaf(d[1], v, acc[1][t]);
                }
            }
        }
    }
    // pixel groups -> block: [thread][K K], then part[co][c_in K K + 1] (the last entry is sum dZ)
    __shared__ float sums[kFCo][kFThreads];
#pragma unroll
    for (int q = 0; q < kFCo; ++q) sums[q][threadIdx.x] = sum[q];
    __syncthreads();
    const int kd = g.c_in * KK, row = kd + 1;
    float *part = smem, *red = smem + kFCo * row;
    for (int h = 0; h < 2; ++h) {
        float *mine = red + ((size_t)((pg * g.cip + ci) * 2 + pair)) * (KK + 1);
#pragma unroll
        for (int t = 0; t < KK; ++t) mine[t] = acc[h][t];
        __syncthreads();
        for (int i = threadIdx.x; i < 2 * kd; i += kFThreads) {
            const int pr = i / kd, e = i - pr * kd, c = e / KK, t = e % KK;
            float v = 0.f;
            for (int q = 0; q < npg; ++q) v += red[((size_t)((q * g.cip + c) * 2 + pr)) * (KK + 1) + t];
            part[(2 * pr + h) * row + e] = v;
        }
        __syncthreads();
    }
    if (threadIdx.x < 32 * kFCo) {        // one warp per output channel
        const int o = threadIdx.x / 32;
        float v = 0.f;
        for (int i = threadIdx.x % 32; i < kFThreads; i += 32) v += sums[o][i];
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
        if (threadIdx.x % 32 == 0) part[o * row + kd] = v;
    }
    cluster.sync();
    const int co = co0 + rank;
    if (rank < kFCo && co < g.c_out) {
        const float s = g.vec3 ? g.vec3[co] : 1.f;
        float dot = 0.f, dsum = 0.f;
        for (int e = threadIdx.x; e < row; e += kFThreads) {
            float v[kFCluster];
#pragma unroll
            for (int b = 0; b < kFCluster; ++b) v[b] = cluster.map_shared_rank(part, b)[rank * row + e];
            float tot = 0.f;
#pragma unroll
            for (int b = 0; b < kFCluster; ++b) tot += v[b];
            if (g.groups > 1) {
                if (e < kd) g.partials[((size_t)group * g.c_out + co) * kd + e] = tot;
                else g.bsum[(size_t)group * g.c_out + co] = tot;
            } else if (e < kd) {
                const size_t o = (size_t)co * kd + e;
                g.dw[o] = s * tot;
                if (g.vec3) dot = fmaf(tot, g.w[o], dot);
            } else {
                dsum = tot;
            }
        }
        __shared__ float fin[2][kFThreads / 32];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { dot += __shfl_xor_sync(0xffffffffu, dot, o); dsum += __shfl_xor_sync(0xffffffffu, dsum, o); }
        if (threadIdx.x % 32 == 0) { fin[0][threadIdx.x / 32] = dot; fin[1][threadIdx.x / 32] = dsum; }
        __syncthreads();
        if (threadIdx.x == 0 && g.groups == 1) {
            dot = dsum = 0.f;
            for (int i = 0; i < kFThreads / 32; ++i) { dot += fin[0][i]; dsum += fin[1][i]; }
            if (g.vec3) {
                g.dbeta[co] = dsum;
                if (g.db) g.db[co] = s * dsum;
                g.dgamma[co] = g.vec3[2 * g.c_out + co] * (dot + dsum * ((g.b ? g.b[co] : 0.f) - g.mean[co]));
            } else if (g.db) {
                g.db[co] = dsum;
            }
        }
    }
    cluster.sync();          // a block's shared memory stays until its neighbours have read it
}

// blocks [0, nw): weight-gradient clusters; [nw, nw + nd): dX tiles (rounded up to whole clusters)
template <int K, int R, int S>
__global__ void __cluster_dims__(kFCluster, 1, 1) __launch_bounds__(kFThreads, 4) f32_bwd_kernel(const F32Wgrad g, int nw, const F32Conv c,
                                                                                          int oc_tiles) {
    extern __shared__ __align__(16) float f32_smem[];
    pdl_wait();
    const int b = (int)blockIdx.x;
    if (b < nw) {
        const int cl = b / kFCluster / g.groups;
        wgrad_cluster<K>(g, cl * kFCo, b / kFCluster - cl * g.groups, f32_smem);
        return;
    }
    constexpr int OCT = S == 1 ? 4 * R : R;
    const int i = b - nw, t = i / oc_tiles;
    if (t < c.tiles) conv_tile<K, R, S, true>(c, (i - t * oc_tiles) * OCT, t, nullptr, nullptr, f32_smem);
}

// S = 4 while the 32-channel blocks of S = 1 would not give every SM two (16 -> 32 channels at 16 x 16, N = 2: 8 of them), and
// where it has less to do: a block's fixed cost and, per input channel and tap of a thread, a load and R multiply-adds, padded
// channels included (93 -> 1 at 96 x 96, N = 22: 119.9 us by 32 channels, 24 by 4; 3 -> 9 at 117 x 27, N = 37: 7.5 and 13.5).
bool split_channels(int tiles, int ic, int oc, int kk) {
    if ((long long)tiles * ((oc + 31) / 32) < 2LL * device_sm_count()) return true;
    return (oc + 3) / 4 * (100 + (ic + 3) / 4 * kk * 6) < (oc + 31) / 32 * (100 + ic * kk * 10);
}
int pixel_tiles(long long pixels) { return (int)((pixels + kFPix - 1) / kFPix); }

bool wgrad_geometry(const Problem &pb, F32Wgrad *g, size_t *bytes) {
    g->n = pb.n; g->c_in = pb.c_in; g->h = pb.h_in; g->wd = pb.w_in; g->c_out = pb.c_out; g->ho = pb.h_out; g->wo = pb.w_out;
    g->pad = pb.pad_h;
    g->cip = 4;
    while (g->cip < pb.c_in) g->cip *= 2;
    g->zp = (pb.w_out + kFRun - 1) / kFRun * kFRun;
    g->xp = g->zp + pb.kw - 1;
    const size_t kk = (size_t)pb.kh * pb.kw, red = kFCo * (pb.c_in * kk + 1) + kFThreads * (kk + 1);
    // the largest band of at most eight rows that leaves every block of a cluster one, within 96 KB (two blocks per SM)
    for (int rows = pb.h_out < 8 ? pb.h_out : 8; rows >= 1; --rows) {
        const int bands = (pb.h_out + rows - 1) / rows, x_ci = ((rows + pb.kh - 1) * g->xp) | 1;
        size_t stage = (size_t)pb.c_in * x_ci + 1 + (size_t)kFCo * rows * g->zp;
        if (stage < red) stage = red;
        if (stage * sizeof(float) > 96 * 1024 && rows > 1) continue;
        if ((long long)pb.n * bands < kFCluster && rows > 1) continue;
        g->rows = rows; g->bands = bands; g->x_ci = x_ci;
        *bytes = stage * sizeof(float);
        return *bytes <= 200 * 1024;
    }
    return false;
}

template <class F>
cudaError_t by_shape(int k, bool split, F f) {
    using I1 = std::integral_constant<int, 1>;
    using I3 = std::integral_constant<int, 3>;
    using I4 = std::integral_constant<int, 4>;
    using I8 = std::integral_constant<int, 8>;
    if (k == 1) return split ? f(I1(), I4(), I4()) : f(I1(), I8(), I1());
    return split ? f(I3(), I4(), I4()) : f(I3(), I8(), I1());
}

}  // namespace

bool f32_conv_eligible(const Problem &pb) {
    if (pb.groups != 1 || pb.kh != pb.kw || (pb.kh != 1 && pb.kh != 3) || pb.stride_h != 1 || pb.stride_w != 1 ||
        pb.dil_h != 1 || pb.dil_w != 1 || pb.pad_h != pb.pad_w || pb.pad_h >= pb.kh || pb.c_in > 128 || pb.c_out > 128)
        return false;
    if (pb.n > 65535 || pb.pin * pb.c_in >= (1LL << 30) || pb.p * pb.c_out >= (1LL << 30)) return false;
    F32Wgrad g;
    size_t bytes;
    return wgrad_geometry(pb, &g, &bytes);
}

// How many clusters share four output channels (their sums then go through launch_wgrad_epilogue), or 0: the direct kernels
// take the parameter gradients.  The least time by a model of microseconds, fitted to 400 layers (1 to 128 channels, planes of
// 1 x 1 to 200 x 200, N = 1 to 20000) at up to 13 counts each: on average 2 % above the best of them.  A block's row bands go by one after the other, each a staging pass and its multiply-adds;
// the direct kernels' threads go through the pixels of a slice.  One cluster whatever the pixels left few output channels to few
// blocks: 1x1 64 -> 8 at 56 x 56, N = 16 340 us, now 51, direct 145.  Planes narrower than a run of pixels in many images stay
// with the direct kernels: 1x1 1 -> 89 on 6876 rows 991 us with one cluster, direct 46.
int f32_wgrad_groups(const Problem &pb, bool need_sums) {
    F32Wgrad g;
    size_t bytes;
    if (!wgrad_geometry(pb, &g, &bytes)) return 0;
    const int kk = pb.kh * pb.kw, items = g.n * g.bands, npg = kFThreads / (2 * g.cip), lines = (pb.kdim + 255) / 256;
    const int blocks = (pb.c_out + kFCo - 1) / kFCo * kFCluster, inner = (g.rows * (g.zp / kFRun) + npg - 1) / npg * kFRun;
    const int steps = (g.c_in * (g.rows + pb.kh - 1) * g.xp + kFThreads - 1) / kFThreads + (kFCo * g.rows * g.zp + kFThreads - 1) / kFThreads;
    // (what the fit leaves out: the bands of one- and two-pixel rows take about half as long again)
    const double item = (0.72 + 0.0041 * inner * kk + 0.195 * steps) * (pb.w_out <= 2 ? 1.5 : 1.0);
    const int per_sm = 227 * 1024 / ((int)bytes + 5 * 1024), slots = device_sm_count() * (per_sm < 1 ? 1 : (per_sm > 4 ? 4 : per_sm));
    // The partial sums live in the direct kernels' workspace; no thread adds up more pixels than one of those would, or 512;
    // and thousands of clusters take longer to launch than they save (16292 rows, 1 -> 1, by 512 groups: 73 us, direct 30).
    const int slices = direct_wgrad_splits(pb), sums = channel_sum_splits(pb), most = slices < sums ? slices : sums, limit = most < 64 ? most : 64;
    const double chain = (double)pb.p / slices > 512.0 ? (double)pb.p / slices : 512.0;
    const double waves = (double)pb.c_out * pb.kdim * slices / (2048.0 * device_sm_count());
    // (sum dZ is a kernel of its own there; without it, in Eval mode, the direct kernels beside f32_bwd_kernel's dX were measured
    // to take 10 us more than the two alone; times 1.1: with that least is lost where the two are close)
    double best_cost = 1.1 * ((need_sums ? 6.0 + 0.166 * pb.p / sums : 14.0) +
                              (0.25 + (waves > 1.0 ? 1.57 * (waves - 1.0) : 0.0)) * pb.p / slices + 0.034 * slices * lines);
    int best = 0;
    for (int groups = 1; groups <= limit; groups += 1 + groups / 4) {
        const int per_block = (items + kFCluster * groups - 1) / (kFCluster * groups);
        if (per_block > 1 && (double)per_block * inner > chain && groups + 1 + groups / 4 <= limit) continue;
        const long long rounds = ((long long)blocks * groups + slots - 1) / slots;
        const double cost = 3.8 + (groups > 1 ? 2.6 + 0.02 * groups * lines : 0.0) + 2.2 * (rounds - 1) + per_block * item * rounds;
        if (cost < best_cost) { best_cost = cost; best = groups; }
    }
    return best;
}

cudaError_t launch_f32_fwd(const Problem &pb, const float *x, const float *w, const float *bias, float *z, cudaStream_t st,
                           const BnFold *fold) {
    F32Conv c{x, w, z, pb.n, pb.c_in, pb.h_in, pb.w_in, pb.c_out, pb.h_out, pb.w_out, pb.pad_h, nullptr, bias, 0};
    c.tiles = pixel_tiles(pb.p);
    const BnFold fd = fold ? *fold : BnFold{nullptr, nullptr, nullptr, nullptr, nullptr, 0.f, nullptr};
    return by_shape(pb.kh, split_channels(c.tiles, c.ic, c.oc, pb.kh * pb.kw), [&](auto k, auto r, auto s) {
        constexpr int K = decltype(k)::value, R = decltype(r)::value, S = decltype(s)::value, OCT = S == 1 ? 4 * R : R;
        const size_t smem = conv_smem_floats(K * K, R, S, pb.c_in) * sizeof(float);
        return launch_pdl(f32_fwd_kernel<K, R, S>, dim3(c.tiles, (c.oc + OCT - 1) / OCT), dim3(kFThreads), smem, st, c, fd);
    });
}

cudaError_t launch_f32_bwd(const Problem &pb, const float *dz, const float *x, const float *w, const float *scale, float *dx,
                           const float *vec3, const float *b, const float *mean, float *dw, float *db, float *dgamma,
                           float *dbeta, int groups, float *partials, float *bsum, cudaStream_t st) {
    F32Wgrad g{};
    size_t wbytes = 0;
    if (!wgrad_geometry(pb, &g, &wbytes)) return cudaErrorInvalidValue;
    g.x = x; g.dz = dz; g.w = w; g.vec3 = vec3; g.b = b; g.mean = mean; g.dw = dw; g.db = db; g.dgamma = dgamma; g.dbeta = dbeta;
    g.groups = groups; g.partials = partials; g.bsum = bsum;
    // dX is a convolution of dZ with the rotated weights: padding k - 1 - pad
    F32Conv c{dz, w, dx, pb.n, pb.c_out, pb.h_out, pb.w_out, pb.c_in, pb.h_in, pb.w_in, pb.kh - 1 - pb.pad_h, scale, nullptr, 0};
    c.tiles = pixel_tiles(pb.pin);
    const int nw = dw ? (pb.c_out + kFCo - 1) / kFCo * kFCluster * groups : 0;
    return by_shape(pb.kh, split_channels(c.tiles, c.ic, c.oc, pb.kh * pb.kw), [&](auto k, auto r, auto s) {
        constexpr int K = decltype(k)::value, R = decltype(r)::value, S = decltype(s)::value, OCT = S == 1 ? 4 * R : R;
        const int oc_tiles = (c.oc + OCT - 1) / OCT;
        const long long nd = dx ? ((long long)oc_tiles * c.tiles + kFCluster - 1) / kFCluster * kFCluster : 0;
        size_t smem = nw ? wbytes : 0;
        const size_t cbytes = conv_smem_floats(K * K, R, S, c.ic) * sizeof(float);
        if (nd && cbytes > smem) smem = cbytes;
        static PerDevice attr;
        if (cudaError_t e = max_dynamic_smem_once(f32_bwd_kernel<K, R, S>, 200 * 1024, &attr); e != cudaSuccess) return e;
        return launch_pdl(f32_bwd_kernel<K, R, S>, dim3((unsigned)(nw + nd)), dim3(kFThreads), smem, st, g, nw, c, oc_tiles);
    });
}

}  // namespace convbn

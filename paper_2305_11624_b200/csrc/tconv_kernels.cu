// Pointwise kernels of the Tune-mode TransposedConv-BN block.  The transposed convolution itself runs on the
// convolution kernels of the layer it transposes (its forward pass is that layer's backward data and vice versa);
// what differs is the axis the per-channel scale lives on: the weights are [C_in][taps][C_out/G] (NHWC) or
// [C_in][C_out/G][taps] (NCHW) and s belongs to the OUTPUT channel, the inner axis.
#include "kernels.h"

namespace convbn {
namespace {

// output channel of weight element idx
__device__ __forceinline__ int tconv_channel(long long idx, int taps, int cig, int cog, bool nhwc) {
    int j, ci;
    if (nhwc) {
        j = (int)(idx % cog);
        ci = (int)(idx / ((long long)cog * taps));
    } else {
        j = (int)((idx / taps) % cog);
        ci = (int)(idx / ((long long)cog * taps));
    }
    return (ci / cig) * cog + j;
}

// vec3 = [s | b' | r]  (Sec. 3.3 definitions; beta may be NULL where b' is not used)
__global__ void bn_vec3_kernel(int c_out, float eps, const float *__restrict__ b, const float *__restrict__ gamma,
                                  const float *__restrict__ beta, const float *__restrict__ mean,
                                  const float *__restrict__ var, float *__restrict__ vec3) {
    pdl_wait();
    pdl_launch_dependents();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= c_out) return;
    const float r = 1.0f / sqrtf(var[c] + eps), s = gamma[c] * r;
    vec3[c] = s;
    vec3[c_out + c] = ((b ? b[c] : 0.0f) - mean[c]) * s + (beta ? beta[c] : 0.0f);
    vec3[2 * c_out + c] = r;
}

template <class T>
__global__ void __launch_bounds__(256) tconv_rescale_kernel(long long count, int taps, int cig, int cog, bool nhwc,
                                                            const T *__restrict__ w, const float *__restrict__ s,
                                                            T *__restrict__ w_out) {
    pdl_wait();
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x)
        w_out[i] = from_f32<T>(to_f32(w[i]) * s[tconv_channel(i, taps, cig, cog, nhwc)]);
}

// NHWC with C_out/G a multiple of 8, 16-bit elements: eight consecutive channels a thread, 32-bit index arithmetic (the general
// kernel divides 64-bit numbers twice per weight).
template <bool H>
__global__ void __launch_bounds__(256) tconv_rescale8_kernel(uint32_t vecs, uint32_t row, uint32_t cig, uint32_t cog,
                                                             const uint4 *__restrict__ w, const float *__restrict__ s,
                                                             uint4 *__restrict__ w_out) {
    pdl_wait();
    pdl_launch_dependents();
    const uint32_t i = blockIdx.x * 256 + threadIdx.x;
    if (i >= vecs) return;
    const uint32_t j = i * 8 % cog, ci = i * 8 / row;                // row = taps C_out/G
    const float *sp = s + ci / cig * cog + j;
    const uint4 q = w[i];
    const float4 s0 = *(const float4 *)sp, s1 = *(const float4 *)(sp + 4);
    float f[8];
    unpack2_t<H>(q.x, f[0], f[1]); unpack2_t<H>(q.y, f[2], f[3]); unpack2_t<H>(q.z, f[4], f[5]); unpack2_t<H>(q.w, f[6], f[7]);
    w_out[i] = make_uint4(pack2_t<H>(f[0] * s0.x, f[1] * s0.y), pack2_t<H>(f[2] * s0.z, f[3] * s0.w),
                          pack2_t<H>(f[4] * s1.x, f[5] * s1.y), pack2_t<H>(f[6] * s1.z, f[7] * s1.w));
}

// z += b' per channel, in place
template <class T>
__global__ void __launch_bounds__(256) tconv_bias_kernel(long long count, int c, long long hw, bool nhwc,
                                                         const float *__restrict__ bias, T *__restrict__ z) {
    pdl_wait();
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
        const int ch = nhwc ? (int)(i % c) : (int)((i / hw) % c);
        z[i] = from_f32<T>(to_f32(z[i]) + bias[ch]);
    }
}

// One block per 32 output channels, 8 row slices per channel.  domega = s domega', dbeta = sum dZ, db = s dbeta,
// dgamma = r (sum over C_in/G and taps of domega' omega + dbeta (b - mu_hat))          (Table 2, Tune row)
template <class T>
__global__ void __launch_bounds__(256) tconv_param_epilogue_kernel(int c_out, int taps, int cig, int cog, bool nhwc,
                                                                   const float *__restrict__ dwp, const T *__restrict__ w,
                                                                   const float *__restrict__ vec3, const float *__restrict__ b,
                                                                   const float *__restrict__ mean,
                                                                   const float *__restrict__ bsum, int bsplits,
                                                                   float *__restrict__ dw, float *__restrict__ db,
                                                                   float *__restrict__ dgamma, float *__restrict__ dbeta) {
    pdl_wait();
    __shared__ float part[8][33];
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
    const int co = blockIdx.x * 32 + lane;
    float dot = 0.0f;
    if (co < c_out) {
        const int g = co / cog, j = co - g * cog;
        const float s = vec3[co];
        const int rows = cig * taps;                   // (ci, tap) pairs of this channel's group
        for (int rr = slice; rr < rows; rr += 8) {
            const int ci = g * cig + rr / taps, tap = rr - (rr / taps) * taps;
            const long long idx = nhwc ? ((long long)ci * taps + tap) * cog + j : ((long long)ci * cog + j) * taps + tap;
            const float v = dwp[idx];
            dot = fmaf(v, to_f32(w[idx]), dot);
            dw[idx] = s * v;
        }
    }
    part[slice][lane] = dot;
    __syncthreads();
    if (slice == 0 && co < c_out) {
        float d = 0.0f, sum = 0.0f;
        for (int q = 0; q < 8; ++q) d += part[q][lane];
        for (int q = 0; q < bsplits; ++q) sum += bsum[(long long)q * c_out + co];
        const float s = vec3[co], r = vec3[2 * c_out + co];
        dbeta[co] = sum;
        if (db) db[co] = s * sum;
        dgamma[co] = r * (d + sum * ((b ? b[co] : 0.0f) - mean[co]));
    }
}

// Block (bx, by): weight columns k = (tap, co) [32 bx, +32) x input channels [64 / Z by, + 64 / Z), one output channel group
// since 32 divides C_out.  Thread (l = four columns, ci, z = slice group) adds slices z, z + Z, ... of part[split][C_in][k], four
// loads in flight; the Z groups are added in halves through shared memory.  The last block of a group of 32
// output channels (a counter) adds the dot products and the sums of dZ in fixed order.  Bound by the latency of the reads of
// the partials (L2): 256 -> 128 channels, 2 x 2, 29 slices: 15 MB.  A thread per weight and all its slices (128 blocks of
// 1024 threads, four bytes a load) took 15 us; with the sum, the scale and the per-channel sums in kernels of their own the
// same work took 87 us.  Z follows the slices (see the launch).
constexpr int kTeThreads = 512;
template <int Z>
__global__ void __launch_bounds__(kTeThreads) tconv_wgrad_epilogue_kernel(int c_in, int c_out, int kdim, const float *__restrict__ part,
                                                                          int splits, const __nv_bfloat16 *__restrict__ w,
                                                                          const float *__restrict__ vec3, const float *__restrict__ b,
                                                                          const float *__restrict__ mean, const float *__restrict__ bsum,
                                                                          int bsplits, float *__restrict__ dotpart,
                                                                          unsigned int *__restrict__ counters, float *__restrict__ dw,
                                                                          float *__restrict__ db, float *__restrict__ dgamma,
                                                                          float *__restrict__ dbeta, int f16) {
    constexpr int CI = 64 / Z;
    __shared__ float4 red[Z > 1 ? kTeThreads : 1];
    __shared__ float tile[kTeThreads / 32][33], sums[kTeThreads / 32][33];
    __shared__ int is_last;
    pdl_wait();
    pdl_launch_dependents();
    const int tid = threadIdx.x, l = tid & 7, ci = (tid >> 3) & (CI - 1), z = tid / (8 * CI);
    const int k0 = blockIdx.x * 32, ci0 = blockIdx.y * CI, co0 = k0 % c_out;    // (the longer dimension is the unbounded one)
    const size_t slice = (size_t)kdim * c_in, at = (size_t)(ci0 + ci) * kdim + k0 + 4 * l;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int sp = z; sp < splits; sp += 4 * Z) {
        float4 q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            q[u] = sp + u * Z < splits ? __ldcg((const float4 *)(part + (size_t)(sp + u * Z) * slice + at))
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 4; ++u) { a.x += q[u].x; a.y += q[u].y; a.z += q[u].z; a.w += q[u].w; }
    }
    if constexpr (Z > 1) {
        red[tid] = a;
#pragma unroll
        for (int h = Z / 2; h > 0; h /= 2) {
            __syncthreads();
            if (z < h) {
                const float4 o = red[tid + h * 8 * CI];
                a.x += o.x; a.y += o.y; a.z += o.z; a.w += o.w;
                red[tid] = a;
            }
        }
    }
    if (z == 0) {                                       // CI / 4 warps: four input channels each
        const uint2 wq = *(const uint2 *)(w + at);
        const float4 s = *(const float4 *)(vec3 + co0 + 4 * l);
        *(float4 *)(dw + at) = make_float4(s.x * a.x, s.y * a.y, s.z * a.z, s.w * a.w);
        float d[4] = {a.x * unpack_h16((uint16_t)(wq.x & 0xFFFFu), f16), a.y * unpack_h16((uint16_t)(wq.x >> 16), f16),
                      a.z * unpack_h16((uint16_t)(wq.y & 0xFFFFu), f16), a.w * unpack_h16((uint16_t)(wq.y >> 16), f16)};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            d[e] += __shfl_xor_sync(0xffffffffu, d[e], 8);
            d[e] += __shfl_xor_sync(0xffffffffu, d[e], 16);
            if ((tid & 31) < 8) tile[tid / 32][4 * l + e] = d[e];
        }
    }
    __syncthreads();
    if (tid < 32) {
        float d = tile[0][tid];
#pragma unroll
        for (int i = 1; i < CI / 4; ++i) d += tile[i][tid];
        dotpart[(size_t)blockIdx.y * kdim + k0 + tid] = d;
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        const unsigned int per_group = gridDim.y * (unsigned)(kdim / c_out);
        is_last = atomicAdd(&counters[co0 / 32], 1u) == per_group - 1;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    // thread (tx = channel, ty = row group): rows of dotpart are (input-channel block, tap), then the slices of sum dZ
    constexpr int kTy = kTeThreads / 32;
    const int tx = tid & 31, ty = tid >> 5;
    const int taps = kdim / c_out, rows = (int)gridDim.y * taps;
    float d = 0.f, sum = 0.f;
    for (int r0 = ty; r0 < rows; r0 += 4 * kTy) {
        float q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = r0 + u * kTy;
            q[u] = r < rows ? __ldcg(dotpart + (size_t)(r / taps) * kdim + (r % taps) * c_out + co0 + tx) : 0.f;
        }
        d += (q[0] + q[1]) + (q[2] + q[3]);
    }
    for (int sp = ty; sp < bsplits; sp += 8 * kTy) {
        float q[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) q[u] = sp + kTy * u < bsplits ? __ldcg(bsum + (size_t)(sp + kTy * u) * c_out + co0 + tx) : 0.f;
        sum += ((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7]));
    }
    tile[ty][tx] = d;
    sums[ty][tx] = sum;
    __syncthreads();
    if (ty == 0) {
        const int co = co0 + tx;
        d = sum = 0.f;
#pragma unroll
        for (int i = 0; i < kTy; ++i) { d += tile[i][tx]; sum += sums[i][tx]; }
        dbeta[co] = sum;
        if (db) db[co] = vec3[co] * sum;
        dgamma[co] = vec3[2 * c_out + co] * (d + sum * ((b ? b[co] : 0.0f) - mean[co]));
    }
}

int grid_for(long long count) {
    long long blocks = (count + 255) / 256;
    const long long cap = (long long)device_sm_count() * 16;
    if (blocks > cap) blocks = cap;
    return (int)(blocks < 1 ? 1 : blocks);
}

}  // namespace

cudaError_t launch_bn_vec3(int c_out, float eps, const float *b, const float *gamma, const float *beta,
                              const float *mean, const float *var, float *vec3, cudaStream_t st) {
    return launch_pdl(bn_vec3_kernel, dim3((c_out + 127) / 128), dim3(128), 0, st, c_out, eps, b, gamma, beta, mean, var, vec3);
}

cudaError_t launch_tconv_wgrad_epilogue(int c_in, int c_out, int taps, const float *part, int splits, const void *w,
                                        const float *vec3, const float *b, const float *mean, const float *bsum,
                                        int bsplits, float *dotpart, unsigned int *counters, float *dw, float *db,
                                        float *dgamma, float *dbeta, cudaStream_t st) {
    // One batch of loads per thread: four slices a group, up to eight groups.  More groups than that leave threads idle, and what a
    // block does beside its loads (sums, counter, the last block's walk over a row of dot products per block) is then paid for
    // fewer weights: with eight groups always, forward + backward of 1024 -> 512, 14 x 14, N = 2 (three slices) took 86.9 us at
    // 2 x 2 and 431 at 4 x 4, with this rule 33.5 and 195.  Few weights spread over more blocks while there are slices to share.
    int z = 1;
    while (z < 8 && z * 4 < splits) z *= 2;
    while (z < 8 && z < splits && (long long)(taps * (long long)c_out / 32) * (c_in / 64) * z < 2LL * device_sm_count()) z *= 2;
    while (z > 1 && c_in / 64 * (long long)z > 65535) z /= 2;
    auto go = [&](auto groups) {
        constexpr int Z = decltype(groups)::value;
        static PerDevice carve;
        prefer_max_shared_once(tconv_wgrad_epilogue_kernel<Z>, &carve);
        return launch_pdl(tconv_wgrad_epilogue_kernel<Z>, dim3(taps * c_out / 32, c_in / 64 * Z), dim3(kTeThreads), 0, st, c_in,
                          c_out, taps * c_out, part, splits, (const __nv_bfloat16 *)w, vec3, b, mean, bsum, bsplits, dotpart,
                          counters, dw, db, dgamma, dbeta, call_f16());
    };
    if (z == 1) return go(std::integral_constant<int, 1>());
    if (z == 2) return go(std::integral_constant<int, 2>());
    if (z == 4) return go(std::integral_constant<int, 4>());
    return go(std::integral_constant<int, 8>());
}

cudaError_t launch_tconv_rescale(int dtype, bool nhwc, long long count, int taps, int cig, int cog, const void *w,
                                 const float *s, void *w_out, cudaStream_t st) {
    if (dtype == CONVBN_BF16 && nhwc && cog % 8 == 0 && count < (1LL << 31)) {
        const uint32_t vecs = (uint32_t)(count / 8);
        auto go = [&](auto kernel) {
            return launch_pdl(kernel, dim3((vecs + 255) / 256), dim3(256), 0, st, vecs, (uint32_t)(taps * cog), (uint32_t)cig,
                              (uint32_t)cog, (const uint4 *)w, s, (uint4 *)w_out);
        };
        return call_f16() ? go(tconv_rescale8_kernel<true>) : go(tconv_rescale8_kernel<false>);
    }
    if (dtype == CONVBN_BF16 && call_f16())     // a half call runs as its bf16 twin
        return launch_pdl(tconv_rescale_kernel<__half>, dim3(grid_for(count)), dim3(256), 0, st, count, taps, cig, cog, nhwc,
                          (const __half *)w, s, (__half *)w_out);
    if (dtype == CONVBN_BF16)
        return launch_pdl(tconv_rescale_kernel<__nv_bfloat16>, dim3(grid_for(count)), dim3(256), 0, st, count, taps, cig, cog,
                          nhwc, (const __nv_bfloat16 *)w, s, (__nv_bfloat16 *)w_out);
    return launch_pdl(tconv_rescale_kernel<float>, dim3(grid_for(count)), dim3(256), 0, st, count, taps, cig, cog, nhwc,
                      (const float *)w, s, (float *)w_out);
}

cudaError_t launch_tconv_bias(int dtype, bool nhwc, long long count, int c, long long hw, const float *bias, void *z,
                              cudaStream_t st) {
    if (dtype == CONVBN_BF16 && call_f16())
        return launch_pdl(tconv_bias_kernel<__half>, dim3(grid_for(count)), dim3(256), 0, st, count, c, hw, nhwc, bias, (__half *)z);
    if (dtype == CONVBN_BF16)
        return launch_pdl(tconv_bias_kernel<__nv_bfloat16>, dim3(grid_for(count)), dim3(256), 0, st, count, c, hw, nhwc, bias,
                          (__nv_bfloat16 *)z);
    return launch_pdl(tconv_bias_kernel<float>, dim3(grid_for(count)), dim3(256), 0, st, count, c, hw, nhwc, bias, (float *)z);
}

cudaError_t launch_tconv_param_epilogue(int dtype, bool nhwc, int c_out, int taps, int cig, int cog, const float *dwp,
                                        const void *w, const float *vec3, const float *b, const float *mean,
                                        const float *bsum, int bsplits, float *dw, float *db, float *dgamma,
                                        float *dbeta, cudaStream_t st) {
    const dim3 grid((c_out + 31) / 32);
    if (dtype == CONVBN_BF16 && call_f16())
        return launch_pdl(tconv_param_epilogue_kernel<__half>, grid, dim3(256), 0, st, c_out, taps, cig, cog, nhwc, dwp,
                          (const __half *)w, vec3, b, mean, bsum, bsplits, dw, db, dgamma, dbeta);
    if (dtype == CONVBN_BF16)
        return launch_pdl(tconv_param_epilogue_kernel<__nv_bfloat16>, grid, dim3(256), 0, st, c_out, taps, cig, cog, nhwc, dwp,
                          (const __nv_bfloat16 *)w, vec3, b, mean, bsum, bsplits, dw, db, dgamma, dbeta);
    return launch_pdl(tconv_param_epilogue_kernel<float>, grid, dim3(256), 0, st, c_out, taps, cig, cog, nhwc, dwp,
                      (const float *)w, vec3, b, mean, bsum, bsplits, dw, db, dgamma, dbeta);
}

}  // namespace convbn

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

// Block (bx, by): weight columns k = (tap, co) [32 bx, +32) x input channels [32 by, +32), one output channel group since
// 32 divides C_out.  Thread (tx = k, ty = ci) adds its element of part[split][C_in][k] over the slices, eight loads in
// flight, in slice order, scales it by s[co] and stores it.  The last block of a group of 32
// output channels (a counter) adds the dot products and the sums of dZ in fixed order.  Bound by the read of the
// partials (L2): 256 -> 128 channels, 2 x 2, 29 slices: 15 MB; with the sum, the scale and the per-channel
// sums in kernels of their own the same work took 87 us.
__global__ void __launch_bounds__(1024) tconv_wgrad_epilogue_kernel(int c_in, int c_out, int kdim, const float *__restrict__ part,
                                                                    int splits, const __nv_bfloat16 *__restrict__ w,
                                                                    const float *__restrict__ vec3, const float *__restrict__ b,
                                                                    const float *__restrict__ mean, const float *__restrict__ bsum,
                                                                    int bsplits, float *__restrict__ dotpart,
                                                                    unsigned int *__restrict__ counters, float *__restrict__ dw,
                                                                    float *__restrict__ db, float *__restrict__ dgamma,
                                                                    float *__restrict__ dbeta, int f16) {
    __shared__ float tile[32][33], prod[32][33];
    __shared__ int is_last;
    pdl_wait();
    pdl_launch_dependents();
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int k0 = blockIdx.x * 32, ci0 = blockIdx.y * 32, co0 = k0 % c_out;       // (the longer dimension is the unbounded one)
    const float wv = load_h16(w + (size_t)(ci0 + ty) * kdim + k0 + tx, f16);
    const float *src = part + (size_t)(ci0 + ty) * kdim + k0 + tx;
    const size_t slice = (size_t)kdim * c_in;
    float v = 0.f;
    for (int sp = 0; sp < splits; sp += 8) {
        float q[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) q[u] = sp + u < splits ? __ldcg(src + (size_t)(sp + u) * slice) : 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) v += q[u];
    }
    dw[(size_t)(ci0 + ty) * kdim + k0 + tx] = vec3[co0 + tx] * v;
    prod[ty][tx] = v * wv;
    __syncthreads();
    {
        float d = prod[tx][ty];                         // warp ty adds the 32 input channels of row k0 + ty
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        if (tx == 0) dotpart[(size_t)blockIdx.y * kdim + k0 + ty] = d;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned int per_group = gridDim.y * (unsigned)(kdim / c_out);
        is_last = atomicAdd(&counters[co0 / 32], 1u) == per_group - 1;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    // thread (tx = channel, ty = row group): rows of dotpart are (input-channel block, tap), then the slices of sum dZ
    float d = 0.f, sum = 0.f;
    const int taps = kdim / c_out, rows = (int)gridDim.y * taps;
    for (int r = ty; r < rows; r += 32) d += __ldcg(dotpart + (size_t)(r / taps) * kdim + (r % taps) * c_out + co0 + tx);
    for (int sp = ty; sp < bsplits; sp += 128) {
        float q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) q[u] = sp + 32 * u < bsplits ? __ldcg(bsum + (size_t)(sp + 32 * u) * c_out + co0 + tx) : 0.f;
        sum += (q[0] + q[1]) + (q[2] + q[3]);
    }
    tile[ty][tx] = d;
    prod[ty][tx] = sum;
    __syncthreads();
    if (ty == 0) {
        const int co = co0 + tx;
        d = sum = 0.f;
        for (int i = 0; i < 32; ++i) { d += tile[i][tx]; sum += prod[i][tx]; }
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
    static PerDevice carve;
    prefer_max_shared_once(tconv_wgrad_epilogue_kernel, &carve);
    return launch_pdl(tconv_wgrad_epilogue_kernel, dim3(taps * c_out / 32, c_in / 32), dim3(1024), 0, st, c_in, c_out,
                      taps * c_out, part, splits, (const __nv_bfloat16 *)w, vec3, b, mean, bsum, bsplits, dotpart, counters,
                      dw, db, dgamma, dbeta, call_f16());
}

cudaError_t launch_tconv_rescale(int dtype, bool nhwc, long long count, int taps, int cig, int cog, const void *w,
                                 const float *s, void *w_out, cudaStream_t st) {
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

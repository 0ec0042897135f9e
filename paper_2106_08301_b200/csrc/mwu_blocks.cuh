// fp64 statistics of one micro-block held in registers (Section 3.1): fixed pairwise tree, every
// operation rounded alone, so that the keys are the same bits whoever evaluates them.
#pragma once

#include "mwu_common.cuh"

namespace mwu {
namespace proj {

__device__ __forceinline__ unsigned long long key_bits(double x) { return (unsigned long long)__double_as_longlong(x); }

template <int B>
__device__ __forceinline__ double tree_sum(const double (&x)[B]) {
    double t[B];
#pragma unroll
    for (int l = 0; l < B; ++l) t[l] = x[l];
#pragma unroll
    for (int w = 1; w < B; w <<= 1)
#pragma unroll
        for (int i = 0; i < B; i += 2 * w) t[i] = __dadd_rn(t[i], t[i + w]);
    return t[0];
}

// v: the block's B values.  S = sum|v|, Lu = sum(|v| - S/B)^2, Kp = sum v^2 (or S for the L1 key)
template <int B>
__device__ __forceinline__ void block_keys(const float *v, int use_l1, double *S_out, double *Lu_out,
                                           double *Kp_out) {
    double a[B], t[B];
#pragma unroll
    for (int l = 0; l < B; ++l) a[l] = (double)fabsf(v[l]);
    const double S = tree_sum<B>(a);
    const double q = __dmul_rn(S, 1.0 / (double)B);
#pragma unroll
    for (int l = 0; l < B; ++l) {
        const double d = __dsub_rn(a[l], q);
        t[l] = __dmul_rn(d, d);
    }
    *Lu_out = tree_sum<B>(t);
    *S_out = S;
    if (use_l1) {
        *Kp_out = S;
    } else {
        // a*a is exact in fp64 for fp32-valued a, so fma(a,a,c) == round(a*a + c): the same
        // bits as a separately rounded multiply and add.
        double h[B / 2];
#pragma unroll
        for (int l = 0; l < B / 2; ++l) h[l] = __fma_rn(a[2 * l], a[2 * l], __dmul_rn(a[2 * l + 1], a[2 * l + 1]));
        *Kp_out = tree_sum<B / 2>(h);
    }
}

// sum v^2 of a block with the same pairing as the prune key of block_keys
template <int B>
__device__ __forceinline__ double block_sumsq(const float *v) {
    double h[B / 2];
#pragma unroll
    for (int l = 0; l < B / 2; ++l) {
        const double a0 = (double)v[2 * l], a1 = (double)v[2 * l + 1];
        h[l] = __fma_rn(a0, a0, __dmul_rn(a1, a1));
    }
    return tree_sum<B / 2>(h);
}

// sum over the CTA of one double per thread, added to *dst by one thread
__device__ __forceinline__ void block_add_double(double x, double *dst) {
    __shared__ double s_part[32];
    for (int m = 16; m > 0; m >>= 1) x += __shfl_xor_sync(0xffffffffu, x, m);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) s_part[wid] = x;
    __syncthreads();
    if (wid == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        double t = lane < nw ? s_part[lane] : 0.0;
        for (int m = 16; m > 0; m >>= 1) t += __shfl_xor_sync(0xffffffffu, t, m);
        if (lane == 0 && t != 0.0) atomicAdd(dst, t);
    }
}

}  // namespace proj
}  // namespace mwu

// Block reductions with a per-RHS "last block finishes" step: every block of
// one right-hand side writes its partial sums, the last block to arrive sums
// them in tile order (deterministic) and runs a finishing step.
#pragma once

#include "helm_internal.cuh"

namespace helm {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Reduce `nv` double2 values (vals[i] valid for i < nv) over the block, store
// the block's partials to `dst[0..nv)`, and report whether this block is the
// last of `ntiles` blocks of its RHS to finish (the counter is reset then).
// `smem` must hold (blockDim/32) * NV double2.  All threads must call it.
__device__ __forceinline__ double2 to_d2(double2 v) { return v; }
__device__ __forceinline__ double2 to_d2(float2 v) { return make_double2(v.x, v.y); }

template <int NV, class T>
__device__ bool reduce_block_last(const T (&vals)[NV], int nv, double2* dst, unsigned* counter,
                                  int ntiles, double2* smem) {
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int lane = tid & 31, warp = tid >> 5;
    const int nwarps = (blockDim.x * blockDim.y) >> 5;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        if (i < nv) {
            double2 v = to_d2(vals[i]);
            double a = warp_sum(v.x);
            double b = warp_sum(v.y);
            if (lane == 0) smem[warp * NV + i] = make_double2(a, b);
        }
    }
    __syncthreads();
    if (tid < nv) {
        double2 acc = make_double2(0.0, 0.0);
        for (int w = 0; w < nwarps; ++w) acc = dadd(acc, smem[w * NV + tid]);
        dst[tid] = acc;
    }
    __threadfence();
    __syncthreads();
    __shared__ unsigned s_last;
    if (tid == 0) {
        unsigned t = atomicAdd(counter, 1u);
        s_last = (t == (unsigned)ntiles - 1u) ? 1u : 0u;
        if (s_last) *counter = 0u;
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last != 0u;
}

// Sum partials[t][i] over tiles t in order (t fastest stride `stride`).
__device__ __forceinline__ double2 sum_partials(const double2* p, int ntiles, int stride, int i) {
    double2 acc = make_double2(0.0, 0.0);
    for (int t = 0; t < ntiles; ++t) {
        double2 v = __ldcg(p + (size_t)t * stride + i);
        acc = dadd(acc, v);
    }
    return acc;
}

// Two-term numbers (h + l, |l| <= ulp(h) / 2; about 46 bits): FP64 instructions take some 64 cycles each
// on this GPU two of them per SM and cycle, so that a warp's sum of a dozen values in FP64
// shuffles costs more than the pass over the data it belongs to.
struct ff {
    float h, l;
};
__device__ __forceinline__ ff ff_quick(float h, float l) {
    ff r;
    r.h = h + l;
    r.l = l - (r.h - h);
    return r;
}
__device__ __forceinline__ ff ff_add(ff a, ff b) {
    const float s = a.h + b.h, bb = s - a.h;
    return ff_quick(s, (a.h - (s - bb)) + (b.h - bb) + (a.l + b.l));
}
__device__ __forceinline__ ff ff_neg(ff a) { return {-a.h, -a.l}; }
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
    const float p = a.h * b.h;
    return ff_quick(p, fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p))));
}
__device__ __forceinline__ ff ff_rcp(ff a) {
    const float y = 1.0f / a.h;
    return ff_quick(y, y * (fmaf(-y, a.h, 1.0f) - y * a.l));
}
// 1 / sqrt(a), a > 0: one Newton step on the FP32 value
__device__ __forceinline__ ff ff_rsqrt(ff a) {
    const float y = rsqrtf(a.h);
    const ff t = ff_mul(a, ff_mul({y, 0.f}, {y, 0.f}));
    return ff_quick(y, 0.5f * y * ((1.0f - t.h) - t.l));
}
__device__ __forceinline__ ff ff_shfl(ff a, int src) {
    return {__shfl_sync(0xffffffffu, a.h, src), __shfl_sync(0xffffffffu, a.l, src)};
}

// Three-term numbers (h + m + l, about 70 bits): sums of FP32 values as good as exact, so that a result
// differs from its FP64 sum only by that sum's own rounding.
struct tf {
    float h, m, l;
};
__device__ __forceinline__ tf tf_add(tf a, tf b) {
    float s = a.h + b.h, bb = s - a.h;
    const float e1 = (a.h - (s - bb)) + (b.h - bb);
    float t = a.m + b.m;
    bb = t - a.m;
    const float e2 = (a.m - (t - bb)) + (b.m - bb);
    float m = t + e1;
    bb = m - t;
    const float e3 = (t - (m - bb)) + (e1 - bb);
    const ff hm = ff_quick(s, m), ml = ff_quick(hm.l, a.l + b.l + e2 + e3);
    return {hm.h, ml.h, ml.l};
}
__device__ __forceinline__ tf tf_shfl_xor(tf a, int o) {
    return {__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.m, o), __shfl_xor_sync(0xffffffffu, a.l, o)};
}
__device__ __forceinline__ tf tf_pick(bool c, tf a, tf b) { return {c ? a.h : b.h, c ? a.m : b.m, c ? a.l : b.l}; }

// reduce_block_last for FP32 values: three-term sums across the lanes (two FP64 additions per SM and cycle
// make FP64 shuffles cost more than the pass over the data), FP64 across the warps.  Eight floats take
// about 20 shuffles: each halving step leaves a lane with half of them.  `smem` holds
// (blockDim / 32) * (NV rounded up to 4) double2.
template <int NV>
__device__ bool reduce_block_last_f32(const float2 (&vals)[NV], double2* dst, unsigned* counter, int ntiles,
                                      double2* smem) {
    constexpr int NP = (NV + 3) / 4 * 4;
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int lane = tid & 31, warp = tid >> 5;
    const int nwarps = (blockDim.x * blockDim.y) >> 5;
    double* out = reinterpret_cast<double*>(smem + warp * NP);
    if constexpr (NV == 1) {
        tf x = {vals[0].x, 0.f, 0.f}, y = {vals[0].y, 0.f, 0.f};
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            x = tf_add(x, tf_shfl_xor(x, o));
            y = tf_add(y, tf_shfl_xor(y, o));
        }
        if (lane == 0) {
            out[0] = ((double)x.l + (double)x.m) + (double)x.h;
            out[1] = ((double)y.l + (double)y.m) + (double)y.h;
        }
    } else {
#pragma unroll
        for (int i0 = 0; i0 < NV; i0 += 4) {
            float a[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                a[2 * q] = i0 + q < NV ? vals[i0 + q < NV ? i0 + q : 0].x : 0.f;
                a[2 * q + 1] = i0 + q < NV ? vals[i0 + q < NV ? i0 + q : 0].y : 0.f;
            }
            tf h4[4], h2[2], h;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float keep = lane & 16 ? a[k + 4] : a[k], give = lane & 16 ? a[k] : a[k + 4];
                h4[k] = tf_add({keep, 0.f, 0.f}, {__shfl_xor_sync(0xffffffffu, give, 16), 0.f, 0.f});
            }
#pragma unroll
            for (int k = 0; k < 2; ++k)
                h2[k] = tf_add(tf_pick(lane & 8, h4[k + 2], h4[k]), tf_shfl_xor(tf_pick(lane & 8, h4[k], h4[k + 2]), 8));
            h = tf_add(tf_pick(lane & 4, h2[1], h2[0]), tf_shfl_xor(tf_pick(lane & 4, h2[0], h2[1]), 4));
#pragma unroll
            for (int o = 2; o > 0; o >>= 1) h = tf_add(h, tf_shfl_xor(h, o));
            if ((lane & 3) == 0) out[2 * i0 + (lane >> 2)] = ((double)h.l + (double)h.m) + (double)h.h;
        }
    }
    __syncthreads();
    if (tid < 2 * NV) {
        double t = 0.0;
        for (int w = 0; w < nwarps; ++w) t += reinterpret_cast<const double*>(smem + w * NP)[tid];
        reinterpret_cast<double*>(dst)[tid] = t;
    }
    __threadfence();
    __syncthreads();
    __shared__ unsigned s_last_f32;
    if (tid == 0) {
        const unsigned t = atomicAdd(counter, 1u);
        s_last_f32 = t == (unsigned)ntiles - 1u ? 1u : 0u;
        if (s_last_f32) *counter = 0u;
    }
    __syncthreads();
    if (s_last_f32) __threadfence();
    return s_last_f32 != 0u;
}

// The block sums entries 0 .. nv - 1 of all tiles' partials into out[0 .. nv) (shared memory): a warp per
// entry, lanes over the tiles, in a fixed order.  All threads must call it.
__device__ __forceinline__ void sum_tiles(const double2* part, int ntiles, int stride, int nv, double2* out) {
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    const int lane = tid & 31, nwarps = (blockDim.x * blockDim.y) >> 5;
    for (int i = tid >> 5; i < nv; i += nwarps) {
        double2 t = make_double2(0.0, 0.0);
        for (int k = lane; k < ntiles; k += 32) t = dadd(t, __ldcg(part + (size_t)k * stride + i));
        t = make_double2(warp_sum(t.x), warp_sum(t.y));
        if (lane == 0) out[i] = t;
    }
    __syncthreads();
}

}  // namespace helm

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

// float <-> double by integer operations: conversions run at the FP64 pipe's two lanes per SM and cycle,
// which would bound the FP64 residual.  Denormals, infinities and NaN take the instruction, narrow's zeros too.
__device__ __forceinline__ double widen(float f) {
    const unsigned u = __float_as_uint(f), e = (u >> 23) & 0xffu;
    if (e - 1u >= 254u) return (u << 1) == 0u ? __hiloint2double((int)u, 0) : (double)f;
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
}
// round to nearest even
__device__ __forceinline__ float narrow(double d) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(d);
    const unsigned e = (unsigned)(u >> 52) & 0x7ffu;
    if (e - 897u >= 253u) return (float)d;            // (the largest finite exponent too: it may round up to infinity)
    const unsigned long long v = u + 0x0fffffffull + ((u >> 29) & 1ull);
    return __uint_as_float(((unsigned)(u >> 32) & 0x80000000u) | ((unsigned)((v >> 29) & 0xffffffffull) - (896u << 23) & 0x7fffffffu));
}

// The FP64 pipe of this GPU takes two lanes per SM and cycle, half a lane per quarter of an SM: an FP64 instruction
// holds a warp's quarter for 64 cycles, and a warp's sums of a dozen values by FP64 shuffles cost
// more than the pass over the data they belong to.  Hence sums of several FP32 terms, by the error-free sum of two
// floats (Knuth; Moller 1965) and product by FMA (Dekker 1971).
//
// Two-term numbers (h + l, about 46 bits), for factors that are rounded to FP32 in the end.
struct ff {
    float h, l;
};
__device__ __forceinline__ ff ff_quick(float h, float l) {
    ff r;
    r.h = h + l;
    r.l = l - (r.h - h);
    return r;
}
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
    const float p = a.h * b.h;
    return ff_quick(p, fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p))));
}
__device__ __forceinline__ ff ff_rcp(ff a) {
    const float y = 1.0f / a.h;
    return ff_quick(y, y * (fmaf(-y, a.h, 1.0f) - y * a.l));
}

// Three-term numbers (h + m + l, about 70 bits of the largest value summed): sums of FP32 values as good as exact,
// so that a result differs from its FP64 sum only by that sum's own rounding.  The sums of the first and of the
// second terms are exact, their errors go one term down; the terms are not made to lie apart again (m may be above
// h where a sum cancels).
struct tf {
    float h, m, l;
};
__device__ __forceinline__ tf tf_add(tf a, tf b) {
    const float s = a.h + b.h;
    float bb = s - a.h;
    const float e1 = (a.h - (s - bb)) + (b.h - bb);
    const float t = a.m + b.m;
    bb = t - a.m;
    const float e2 = (a.m - (t - bb)) + (b.m - bb);
    const float m = t + e1;
    bb = m - t;
    const float e3 = (t - (m - bb)) + (e1 - bb);
    return {s, m, a.l + b.l + e2 + e3};
}
__device__ __forceinline__ tf tf_shfl_xor(tf a, int o) {
    return {__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.m, o), __shfl_xor_sync(0xffffffffu, a.l, o)};
}
__device__ __forceinline__ double tf_double(tf a) { return ((double)a.l + (double)a.m) + (double)a.h; }

__device__ __forceinline__ tf tf_pick(bool c, tf a, tf b) { return {c ? a.h : b.h, c ? a.m : b.m, c ? a.l : b.l}; }

// Pairs of FP32 additions and subtractions, an instruction each.
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    asm("{ .reg .b64 p, q;\n mov.b64 p, {%0, %1};\n mov.b64 q, {%2, %3};\n add.rn.f32x2 p, p, q;\n"
        " mov.b64 {%0, %1}, p; }"
        : "+f"(a.x), "+f"(a.y)
        : "f"(b.x), "f"(b.y));
    return a;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    asm("{ .reg .b64 p, q;\n mov.b64 p, {%0, %1};\n mov.b64 q, {%2, %3};\n sub.rn.f32x2 p, p, q;\n"
        " mov.b64 {%0, %1}, p; }"
        : "+f"(a.x), "+f"(a.y)
        : "f"(b.x), "f"(b.y));
    return a;
}
// Two three-term numbers, (first, second) per term.
struct tf2 {
    float2 h, m, l;
};
__device__ __forceinline__ tf first_of(const tf2& s) { return {s.h.x, s.m.x, s.l.x}; }
__device__ __forceinline__ tf second_of(const tf2& s) { return {s.h.y, s.m.y, s.l.y}; }
// a + b and its error
__device__ __forceinline__ float2 exact_sum2(float2 a, float2 b, float2* err) {
    const float2 s = add2(a, b), bb = sub2(s, a);
    *err = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
    return s;
}
__device__ __forceinline__ tf2 tf2_add(const tf2& a, const tf2& b) {
    float2 e1, e2, e3;
    const float2 s = exact_sum2(a.h, b.h, &e1), m = exact_sum2(exact_sum2(a.m, b.m, &e2), e1, &e3);
    return {s, m, add2(add2(add2(a.l, b.l), e2), e3)};
}
__device__ __forceinline__ float2 shfl_xor2(float2 a, int o) {
    return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
}
// The sum over groups of `wide` lanes (a power of two, the same in the whole warp), in every lane of a group.
__device__ __forceinline__ tf2 tf2_group_sum(tf2 a, int wide) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        if (wide > o) a = tf2_add(a, {shfl_xor2(a.h, o), shfl_xor2(a.m, o), shfl_xor2(a.l, o)});
    return a;
}
__device__ __forceinline__ float2 pick2(bool c, float2 a, float2 b) { return c ? a : b; }
// Sums of eight floats over the warp: value lane >> 2 in the lanes that are multiples of four.  Each halving step
// leaves a lane with half of the values, so that eight take about 20 shuffles.
__device__ __forceinline__ tf tf_warp_sum8(const float (&a)[8], int lane) {
    tf2 h[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float2 lo = make_float2(a[2 * k], a[2 * k + 1]), hi = make_float2(a[2 * k + 4], a[2 * k + 5]);
        h[k].h = exact_sum2(pick2(lane & 16, hi, lo), shfl_xor2(pick2(lane & 16, lo, hi), 16), &h[k].m);
        h[k].l = make_float2(0.f, 0.f);
    }
    const bool up = lane & 8;
    // (the third terms are zero here)
    const tf2 g = tf2_add({pick2(up, h[1].h, h[0].h), pick2(up, h[1].m, h[0].m), h[0].l},
                          {shfl_xor2(pick2(up, h[0].h, h[1].h), 8), shfl_xor2(pick2(up, h[0].m, h[1].m), 8), h[0].l});
    const tf x = first_of(g), y = second_of(g);
    tf s = tf_add(tf_pick(lane & 4, y, x), tf_shfl_xor(tf_pick(lane & 4, x, y), 4));
#pragma unroll
    for (int o = 2; o > 0; o >>= 1) s = tf_add(s, tf_shfl_xor(s, o));
    return s;
}

// reduce_block_last for FP32 values: three-term sums across the lanes (two FP64 additions per SM and cycle
// make FP64 shuffles cost more than the pass over the data), FP64 across the warps.  `smem` holds
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
            out[0] = tf_double(x);
            out[1] = tf_double(y);
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
            const tf h = tf_warp_sum8(a, lane);
            if ((lane & 3) == 0) out[2 * i0 + (lane >> 2)] = tf_double(h);
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

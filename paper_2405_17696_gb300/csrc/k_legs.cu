// The two legs of a V-cycle level with two damped-Jacobi sweeps each (Sec. 3.4), one
// pass over the fields per leg instead of one per sweep and transfer:
//   down: u1 = w D^-1 f, u2 = u1 + w D^-1 (f - A u1), rc = full weighting of f - A u2;
//         reads f, writes u2 and rc (18 bytes per node and right-hand side)
//   up:   v = u2 + bilinear interpolation of ec, then two sweeps;
//         reads u2, f, ec, writes u (26 bytes).
// The separate kernels move 58 and 66 bytes.  At 512 x 256, 192 right-hand sides, one GB300:
// fine 690 -> 296 us (1.1 GB: 3.7 TB/s), the level below 332 -> 275 us; about 100
// instructions per node and leg bound the fine ones, shared-memory reads of the nine
// coefficients and three operations per real product the coarse ones.
//
// A warp marches down a strip of 64 columns of one right-hand side.  A lane holds a pair
// of columns (2k, 2k + 1); its neighbours' values come by shuffles, and the last three rows
// of every intermediate field stay in registers: shared memory holds only the rows that are
// read, copied ahead.  The strip's outer columns and the first and last rows of a segment are
// computed twice, by the neighbours too: 29 (down) or 30 (up) of 32 lanes and all but 5 or
// 4 rows of a segment are written.  Values outside the grid are set to zero.  Every node is
// computed by the same operations in the same order as by the separate kernels.
//
// The warps of a block take different right-hand sides of the same tile.  On a coarse level
// they share the nine coefficients of its nodes (read per warp they are four times the
// traffic of the fields), at a barrier per row; right-hand sides of different frequencies in
// a block take turns.  On the fine grid the medium is an eighth of that and such a barrier
// costs more than it saves (139 -> 162 us at 512 x 256, 192 right-hand sides), so every warp
// reads its own and only the warp waits for its copies.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "helm_internal.cuh"

namespace helm {
namespace {

constexpr int LEG_WARPS = 4;        // warps (right-hand sides) per block
constexpr int LEG_CTAS = 4;         // blocks per SM (at most 128 registers per thread)

// two neighbouring complex values, their left and right neighbours
struct Row {
    float4 v;
    float2 l, r;
};

__device__ __forceinline__ Row make_row(float4 v) {
    Row o;
    o.v = v;
    o.l.x = __shfl_up_sync(0xffffffffu, v.z, 1);
    o.l.y = __shfl_up_sync(0xffffffffu, v.w, 1);
    o.r.x = __shfl_down_sync(0xffffffffu, v.x, 1);
    o.r.y = __shfl_down_sync(0xffffffffu, v.y, 1);
    return o;
}

__device__ __forceinline__ float4 sub4(float4 a, float4 b) {
    return make_float4(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y), __fsub_rn(a.z, b.z), __fsub_rn(a.w, b.w));
}
// The rounded operations below are spelled out: each node takes the ones the separate kernels take.
// a b + c d and a b - c d, the first product fused
__device__ __forceinline__ float mad2(float a, float b, float c, float d) { return __fmaf_rn(a, b, __fmul_rn(c, d)); }
__device__ __forceinline__ float msd2(float a, float b, float c, float d) { return __fmaf_rn(a, b, -__fmul_rn(c, d)); }
// u + w (r / d) for a pair, with i = 1 / |d|^2
__device__ __forceinline__ float4 relax2(float4 u, float w, float4 r, float4 d, float2 i) {
    return make_float4(__fmaf_rn(w, __fmul_rn(mad2(r.x, d.x, r.y, d.y), i.x), u.x),
                       __fmaf_rn(w, __fmul_rn(msd2(r.y, d.x, r.x, d.y), i.x), u.y),
                       __fmaf_rn(w, __fmul_rn(mad2(r.z, d.z, r.w, d.w), i.y), u.z),
                       __fmaf_rn(w, __fmul_rn(msd2(r.w, d.z, r.z, d.w), i.y), u.w));
}
__device__ __forceinline__ float2 inv_abs2(float4 d) {
    return make_float2(__frcp_rn(mad2(d.x, d.x, d.y, d.y)), __frcp_rn(mad2(d.z, d.z, d.w, d.w)));
}

// Operator of the fine grid as a leg uses it: per node pair the coefficient s (1 - i sigma)
// and 1 / |d|^2 of the diagonal d, from the {kappa, gamma} of the pair.
struct LegFine {
    OpFine5 op;
    static constexpr int NCO = 1;                      // float4 per pair and row
    static constexpr bool SHARED = false;              // every warp reads its own
    struct Co {
        float4 k;
        float2 i;
    };
    float w2;
    __device__ __forceinline__ void init(int f) {
        const float w = __ldg(op.omega + f);
        w2 = w * w;
    }
    __device__ __forceinline__ const void* src(int, int idx) const { return op.mg + idx; }
    __device__ __forceinline__ Co make(const float4 (*sh)[32], int lane) const {
        Co c;
        const float4 m = sh[0][lane];
        const float s0 = __fmul_rn(w2, __fmul_rn(m.x, m.x)), s1 = __fmul_rn(w2, __fmul_rn(m.z, m.z));
        const float g0 = op.sl ? (op.beta + (op.incg ? m.y : 0.0f)) : m.y;
        const float g1 = op.sl ? (op.beta + (op.incg ? m.w : 0.0f)) : m.w;
        c.k = make_float4(s0, -s0 * g0, s1, -s1 * g1);
        c.i = inv_abs2(diag(c));
        return c;
    }
    __device__ __forceinline__ float4 diag(const Co& c) const {
        return make_float4(2.0f * (op.ax + op.az) - c.k.x, -c.k.y, 2.0f * (op.ax + op.az) - c.k.z, -c.k.w);
    }
    __device__ __forceinline__ void clear(Co& c) const {
        c.k = make_float4(0.f, 0.f, 0.f, 0.f);
        c.i = make_float2(0.f, 0.f);
    }
    // A u at the pair of row b (rows a above, c below), in a sweep or for the residual that is restricted
    template <bool SWEEP>
    __device__ __forceinline__ float4 apply(const Co& k, const float4 (*)[32], int, const Row& a, const Row& b,
                                            const Row& c) const {
        // ax (2 m - l - r) + az (2 m - up - dn): the sweeps round the first product, the residual the second
        auto lap = [&](float m, float l, float r, float up, float dn) {
            const float tx = __fsub_rn(__fmaf_rn(2.f, m, -l), r), tz = __fsub_rn(__fmaf_rn(2.f, m, -up), dn);
            return SWEEP ? __fmaf_rn(op.az, tz, __fmul_rn(op.ax, tx)) : __fmaf_rn(op.ax, tx, __fmul_rn(op.az, tz));
        };
        float4 y;
        y.x = __fsub_rn(lap(b.v.x, b.l.x, b.v.z, a.v.x, c.v.x), msd2(k.k.x, b.v.x, k.k.y, b.v.y));
        y.y = __fsub_rn(lap(b.v.y, b.l.y, b.v.w, a.v.y, c.v.y), mad2(k.k.x, b.v.y, k.k.y, b.v.x));
        y.z = __fsub_rn(lap(b.v.z, b.v.x, b.r.x, a.v.z, c.v.z), msd2(k.k.z, b.v.z, k.k.w, b.v.w));
        y.w = __fsub_rn(lap(b.v.w, b.v.y, b.r.y, a.v.w, c.v.w), mad2(k.k.z, b.v.w, k.k.w, b.v.z));
        return y;
    }
};

// Galerkin level: the diagonal d and 1 / |d|^2 per pair, the nine coefficients shared per frequency.
struct LegC9 {
    OpC9 op;
    static constexpr int NCO = 9;
    static constexpr bool SHARED = true;               // by the block's warps of one frequency
    struct Co {
        float4 d;
        float2 i;
    };
    const float2* base;
    size_t plane;
    __device__ __forceinline__ void init(int f) {
        base = op.base(f);
        plane = (size_t)op.nx * op.nz;
    }
    __device__ __forceinline__ const void* src(int q, int idx) const { return base + q * plane + idx; }
    __device__ __forceinline__ Co make(const float4 (*sh)[32], int lane) const {
        Co c;
        c.d = sh[4][lane];
        c.i = inv_abs2(c.d);
        return c;
    }
    __device__ __forceinline__ float4 diag(const Co& c) const { return c.d; }
    __device__ __forceinline__ void clear(Co& c) const {
        c.d = make_float4(0.f, 0.f, 0.f, 0.f);
        c.i = make_float2(0.f, 0.f);
    }
    template <bool SWEEP>
    __device__ __forceinline__ float4 apply(const Co&, const float4 (*sh)[32], int lane, const Row& a, const Row& b,
                                            const Row& c) const {
        float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
        auto add = [&](float4 k, float4 v) {
            y.x = __fadd_rn(y.x, msd2(k.x, v.x, k.y, v.y));
            y.y = __fadd_rn(y.y, mad2(k.y, v.x, k.x, v.y));
            y.z = __fadd_rn(y.z, msd2(k.z, v.z, k.w, v.w));
            y.w = __fadd_rn(y.w, mad2(k.w, v.z, k.z, v.w));
        };
#pragma unroll
        for (int dz = 0; dz < 3; ++dz) {
            const Row& q = dz == 0 ? a : (dz == 1 ? b : c);
            add(sh[3 * dz][lane], make_float4(q.l.x, q.l.y, q.v.x, q.v.y));
            add(sh[3 * dz + 1][lane], q.v);
            add(sh[3 * dz + 2][lane], make_float4(q.v.z, q.v.w, q.r.x, q.r.y));
        }
        return y;
    }
};

// Row rings in shared memory, filled by asynchronous copies AHEAD rows ahead.  A lane copies and reads
// its own 16 bytes of a field's row; shared rows are copied by all warps and read after a barrier.
// A copy into a slot is issued after row z's barrier (of the warp or the block), when every lane is
// past row z - 1, so a ring holds rows z - 2 .. z + AHEAD.  Rows after a march's last one are not copied, only
// their empty groups are committed: the wait for the last row is then a wait for every copy of the march, and the
// next frequency's march may fill the same slots (asynchronous copies to one address have no order).
constexpr int AHEAD = 5, RING = 8;
struct Ring {
    float4 row[RING][32];
};
template <class L>
struct Coefs {
    float4 row[RING][L::NCO][32];
};
template <class L>
constexpr int COEF_RINGS = L::SHARED ? 1 : LEG_WARPS;
template <class L>
__device__ __forceinline__ void leg_sync() {
    if (L::SHARED) __syncthreads();
    else __syncwarp();
}
__device__ __forceinline__ void copy16(float4* dst, const void* src, bool in) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copy8(float2* dst, const void* src, bool in) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(in ? 8 : 0) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(AHEAD - 1) : "memory"); }

// Tile of a warp: right-hand side b, strip of column pairs, segment of rows.
struct LegTile {
    int strips, segs, rows;     // rows of a segment (even)
};

// The frequencies of a block's right-hand sides in turn: the smallest one above `last`, -1 when done.
__device__ __forceinline__ int next_freq(int mine, bool act, int last, int* sm) {
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = act && mine > last ? mine : 0x7fffffff;
    __syncthreads();
    int f = sm[0];
    for (int i = 1; i < LEG_WARPS; ++i) f = min(f, sm[i]);
    return f == 0x7fffffff ? -1 : f;
}

template <class L>
__global__ void __launch_bounds__(32 * LEG_WARPS, LEG_CTAS) leg_down_kernel(L lo, const float2* __restrict__ f,
                                                                            float2* __restrict__ u2out,
                                                                            float2* __restrict__ rc, float w, int nb,
                                                                            LegTile tl_, const int* mask, Tally tl) {
    extern __shared__ __align__(16) unsigned char leg_sm[];
    __shared__ int fsm[LEG_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Coefs<L>& rm = reinterpret_cast<Coefs<L>*>(leg_sm)[L::SHARED ? 0 : warp];
    unsigned char* rings = leg_sm + COEF_RINGS<L> * sizeof(Coefs<L>);
    Ring& rf = reinterpret_cast<Ring*>(rings)[warp];
    const int groups = (nb + LEG_WARPS - 1) / LEG_WARPS;
    const int tile = blockIdx.x / groups, b = (blockIdx.x - tile * groups) * LEG_WARPS + warp;
    const bool act = b < nb && mask[b] != 0;
    const int freq = act ? __ldg(lo.op.rhs_freq + b) : 0;
    if (act && tl.ctr && tile == 0 && lane == 0) atomicAdd(tl.ctr, tl.base);
    const int nx = lo.op.nx, nz = lo.op.nz, nxc = nx / 2;
    const int strip = tile % tl_.strips, seg = tile / tl_.strips;
    const int k = strip * 29 - 1 + lane;                  // this lane's column pair
    const bool col = k >= 0 && k < nxc;
    const bool wr = lane >= 1 && lane <= 29 && col;
    const int z0 = seg * tl_.rows, z1 = min(nz, z0 + tl_.rows);   // rows of u2 written here
    const size_t N = (size_t)nx * nz;
    const float2* fb = f + (size_t)b * N + 2 * k;
    float2* ub = u2out + (size_t)b * N + 2 * k;
    float2* rb = rc + (size_t)b * (N / 4) + k;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);

    for (int fq = -1;;) {
        if (L::SHARED) {
            fq = next_freq(freq, act, fq, fsm);
            if (fq < 0) break;
        } else if (!act) {
            break;
        }
        const bool mine = act && (!L::SHARED || freq == fq);
        lo.init(L::SHARED ? fq : freq);
        auto fetch = [&](int z) {
            if (z <= z1 + 2) {
                const bool in = col && z >= 0 && z < nz;
                if (mine) copy16(&rf.row[z & (RING - 1)][lane], in ? fb + (size_t)z * nx : f, in);
                for (int q = L::SHARED ? warp : 0; q < L::NCO; q += L::SHARED ? LEG_WARPS : 1)
                    copy16(&rm.row[z & (RING - 1)][q][lane], in ? lo.src(q, z * nx + 2 * k) : (const void*)f, in);
            }
            copy_commit();
        };
        for (int i = 0; i < AHEAD; ++i) fetch(z0 - 2 + i);
        Row U1[3], U2[3];
        typename L::Co C[3];
        float2 acc = make_float2(0.f, 0.f);                   // 16 rc of the coarse row under way
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            U1[i].v = U2[i].v = zero;
            U1[i].l = U1[i].r = U2[i].l = U2[i].r = make_float2(0.f, 0.f);
            lo.clear(C[i]);
        }
        // row z enters: u1[z], u2[z - 1], the residual of row z - 2 into the weighting (u2 is right from
        // row z0 - 1 on; the rows above it, made from rows that were not read, go nowhere)
        for (int zc = z0 - 2; zc <= z1 + 2; zc += 3) {
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int z = zc + i, s0 = i, s1 = (i + 2) % 3, s2 = (i + 1) % 3;   // slots of rows z, z - 1, z - 2
                if (z > z1 + 2) break;
                copy_wait();
                leg_sync<L>();
                fetch(z + AHEAD);
                if (!mine) continue;
                // slot s0 holds row z - 3 of u2 until u2[z] is due; the other arrays are free to take row z
                const Row u2m3 = U2[s0];
                C[s0] = lo.make(rm.row[z & (RING - 1)], lane);
                U1[s0] = make_row(col && z >= 0 && z < nz
                                      ? relax2(zero, w, rf.row[z & (RING - 1)][lane], lo.diag(C[s0]), C[s0].i)
                                      : zero);
                // u2[z - 1] from u1 rows z - 2, z - 1, z
                {
                    const float4 y = lo.template apply<true>(C[s1], rm.row[(z - 1) & (RING - 1)], lane, U1[s2], U1[s1], U1[s0]);
                    U2[s1] = make_row(col && z >= 1 && z <= nz
                                          ? relax2(U1[s1].v, w, sub4(rf.row[(z - 1) & (RING - 1)][lane], y),
                                                   lo.diag(C[s1]), C[s1].i)
                                          : zero);
                    if (wr && z - 1 >= z0 && z - 1 < z1)
                        *reinterpret_cast<float4*>(ub + (size_t)(z - 1) * nx) = U2[s1].v;
                }
                // residual of row y = z - 2 from u2 rows z - 3, z - 2, z - 1
                const int y = z - 2;
                if (y >= z0) {
                    const float4 t = lo.template apply<false>(C[s2], rm.row[y & (RING - 1)], lane, u2m3, U2[s2], U2[s1]);
                    const float4 r = col && y < nz ? sub4(rf.row[y & (RING - 1)][lane], t) : zero;
                    const float ex = __shfl_down_sync(0xffffffffu, r.x, 1), ey = __shfl_down_sync(0xffffffffu, r.y, 1);
                    // weights 1 2 1 along x, times 1 2 1 along z and 1 / 16 at the end (powers of two: exact)
                    const float wz = y & 1 ? 2.f : 1.f;
                    acc.x = __fmaf_rn(wz, ex, __fmaf_rn(2.f * wz, r.z, __fmaf_rn(wz, r.x, acc.x)));
                    acc.y = __fmaf_rn(wz, ey, __fmaf_rn(2.f * wz, r.w, __fmaf_rn(wz, r.y, acc.y)));
                    if (!(y & 1)) {
                        // the last row of coarse row y / 2 - 1, the first of y / 2
                        if (wr && y > z0)
                            rb[(size_t)(y / 2 - 1) * nxc] = make_float2(acc.x * (1.0f / 16.0f), acc.y * (1.0f / 16.0f));
                        acc = make_float2(__fadd_rn(__fmaf_rn(2.f, r.z, r.x), ex), __fadd_rn(__fmaf_rn(2.f, r.w, r.y), ey));
                    }
                }
            }
        }
        if (!L::SHARED) break;
    }
}

template <class L>
__global__ void __launch_bounds__(32 * LEG_WARPS, LEG_CTAS) leg_up_kernel(L lo, const float2* __restrict__ f,
                                                                          const float2* __restrict__ u2in,
                                                                          const float2* __restrict__ ec,
                                                                          float2* __restrict__ uout, float w, int nb,
                                                                          LegTile tl_, const int* mask, Tally tl) {
    extern __shared__ __align__(16) unsigned char leg_sm[];
    __shared__ int fsm[LEG_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Coefs<L>& rm = reinterpret_cast<Coefs<L>*>(leg_sm)[L::SHARED ? 0 : warp];
    unsigned char* rings = leg_sm + COEF_RINGS<L> * sizeof(Coefs<L>);
    Ring& rf = reinterpret_cast<Ring*>(rings)[2 * warp];
    Ring& rv = reinterpret_cast<Ring*>(rings)[2 * warp + 1];
    // coarse rows, entry lane + 1 the lane's column
    float2(*re)[33] =
        reinterpret_cast<float2(*)[33]>(rings + 2 * LEG_WARPS * sizeof(Ring)) + 4 * warp;
    const int groups = (nb + LEG_WARPS - 1) / LEG_WARPS;
    const int tile = blockIdx.x / groups, b = (blockIdx.x - tile * groups) * LEG_WARPS + warp;
    const bool act = b < nb && mask[b] != 0;
    const int freq = act ? __ldg(lo.op.rhs_freq + b) : 0;
    if (act && tl.ctr && tile == 0 && lane == 0) atomicAdd(tl.ctr, tl.base);
    const int nx = lo.op.nx, nz = lo.op.nz, nxc = nx / 2, nzc = nz / 2;
    const int strip = tile % tl_.strips, seg = tile / tl_.strips;
    const int k = strip * 30 - 1 + lane;
    const bool col = k >= 0 && k < nxc;
    const bool wr = lane >= 1 && lane <= 30 && col;
    const int z0 = seg * tl_.rows, z1 = min(nz, z0 + tl_.rows);
    const size_t N = (size_t)nx * nz;
    const float2* fb = f + (size_t)b * N + 2 * k;
    const float2* vb = u2in + (size_t)b * N + 2 * k;
    const float2* eb = ec + (size_t)b * (N / 4) + k;
    float2* ub = uout + (size_t)b * N + 2 * k;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);

    for (int fq = -1;;) {
        if (L::SHARED) {
            fq = next_freq(freq, act, fq, fsm);
            if (fq < 0) break;
        } else if (!act) {
            break;
        }
        const bool mine = act && (!L::SHARED || freq == fq);
        lo.init(L::SHARED ? fq : freq);
        auto fetch_e = [&](int J) {
            const bool in = J >= 0 && J < nzc;
            copy8(&re[J & 3][lane + 1], in && col ? eb + (size_t)J * nxc : ec, in && col);
            if (lane == 0) {
                const bool inl = in && k >= 1 && k <= nxc;
                copy8(&re[J & 3][0], inl ? eb + (size_t)J * nxc - 1 : ec, inl);
            }
        };
        // row z with, for an even z, the coarse row z / 2 (which it and the odd row after it need)
        auto fetch = [&](int z) {
            if (z <= z1 + 1) {
                const bool in = col && z >= 0 && z < nz;
                if (mine) {
                    copy16(&rf.row[z & (RING - 1)][lane], in ? fb + (size_t)z * nx : f, in);
                    copy16(&rv.row[z & (RING - 1)][lane], in ? vb + (size_t)z * nx : f, in);
                    if (!(z & 1)) fetch_e(z >> 1);
                }
                for (int q = L::SHARED ? warp : 0; q < L::NCO; q += L::SHARED ? LEG_WARPS : 1)
                    copy16(&rm.row[z & (RING - 1)][q][lane], in ? lo.src(q, z * nx + 2 * k) : (const void*)f, in);
            }
            copy_commit();
        };
        // coarse row J at columns k - 1 and k
        auto coarse = [&](int J) {
            const float2 l = re[J & 3][lane], e = re[J & 3][lane + 1];
            return make_float4(l.x, l.y, e.x, e.y);
        };
        if (mine) fetch_e((z0 - 2) / 2 - 1);                  // (joins the first row's group)
        for (int i = 0; i < AHEAD; ++i) fetch(z0 - 2 + i);
        Row V[3], S[3];
        typename L::Co C[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            V[i].v = S[i].v = zero;
            V[i].l = V[i].r = S[i].l = S[i].r = make_float2(0.f, 0.f);
            lo.clear(C[i]);
        }
        float4 e0 = zero, e1 = zero;                          // coarse rows z / 2 - 1 and z / 2
        for (int zc = z0 - 2; zc <= z1 + 1; zc += 3) {
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int z = zc + i, s0 = i, s1 = (i + 2) % 3, s2 = (i + 1) % 3;
                if (z > z1 + 1) break;
                copy_wait();
                leg_sync<L>();
                fetch(z + AHEAD);
                if (!mine) continue;
                const bool in = col && z >= 0 && z < nz;
                const Row sm3 = S[s0];
                C[s0] = lo.make(rm.row[z & (RING - 1)], lane);
                // v[z] = u2 + interpolation: an odd row takes coarse row (z - 1) / 2, an even one the mean of two
                float4 e;
                if (z & 1) {
                    e = e1;
                } else {
                    e0 = z == z0 - 2 ? coarse((z >> 1) - 1) : e1;
                    e1 = coarse(z >> 1);
                    e = make_float4(__fmaf_rn(0.5f, e0.x, 0.5f * e1.x), __fmaf_rn(0.5f, e0.y, 0.5f * e1.y),
                                    __fmaf_rn(0.5f, e0.z, 0.5f * e1.z), __fmaf_rn(0.5f, e0.w, 0.5f * e1.w));
                }
                const float4 vr = rv.row[z & (RING - 1)][lane];
                V[s0] = make_row(in ? make_float4(__fmaf_rn(0.5f, __fadd_rn(e.x, e.z), vr.x),
                                                  __fmaf_rn(0.5f, __fadd_rn(e.y, e.w), vr.y), __fadd_rn(vr.z, e.z),
                                                  __fadd_rn(vr.w, e.w))
                                    : zero);
                // first sweep, row z - 1
                {
                    const float4 y = lo.template apply<true>(C[s1], rm.row[(z - 1) & (RING - 1)], lane, V[s2], V[s1], V[s0]);
                    S[s1] = make_row(col && z >= 1 && z <= nz
                                         ? relax2(V[s1].v, w, sub4(rf.row[(z - 1) & (RING - 1)][lane], y),
                                                  lo.diag(C[s1]), C[s1].i)
                                         : zero);
                }
                // second sweep, row z - 2
                const int y2 = z - 2;
                if (y2 >= z0) {
                    const float4 y = lo.template apply<true>(C[s2], rm.row[y2 & (RING - 1)], lane, sm3, S[s2], S[s1]);
                    if (wr && y2 < z1)
                        *reinterpret_cast<float4*>(ub + (size_t)y2 * nx) =
                            relax2(S[s2].v, w, sub4(rf.row[y2 & (RING - 1)][lane], y), lo.diag(C[s2]), C[s2].i);
                }
            }
        }
        if (!L::SHARED) break;
    }
}

// Rows per segment: up to 64, of which 5 are computed twice; fewer while the warps do not fill the device
// (12 per SM), down to 2, since a small grid waits for the rows of one warp.
LegTile leg_tile(int nx, int nz, int nb, int useful) {
    LegTile t;
    t.strips = (nx / 2 + useful - 1) / useful;
    const long long want = 152 * 12;
    long long segs = std::max<long long>((nz + 63) / 64, (want + (long long)t.strips * nb - 1) / ((long long)t.strips * nb));
    segs = std::min<long long>(segs, std::max(1, nz / 2));
    t.rows = (int)((nz + segs - 1) / segs + 1) / 2 * 2;
    t.segs = (nz + t.rows - 1) / t.rows;
    return t;
}

template <class L>
constexpr size_t LEG_DOWN_SMEM = COEF_RINGS<L> * sizeof(Coefs<L>) + LEG_WARPS * sizeof(Ring);
template <class L>
constexpr size_t LEG_UP_SMEM = COEF_RINGS<L> * sizeof(Coefs<L>) + LEG_WARPS * (2 * sizeof(Ring) + 4 * 33 * sizeof(float2));

template <class L>
int leg_attributes() {
    static DeviceOnce once;
    HELM_CK(once_per_device(once, [] {
        const cudaError_t e = cudaFuncSetAttribute(leg_down_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LEG_DOWN_SMEM<L>);
        return e != cudaSuccess ? e : cudaFuncSetAttribute(leg_up_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                           (int)LEG_UP_SMEM<L>);
    }));
    return HELM_OK;
}

template <class Op>
auto leg_op(const Op& op) {
    if constexpr (std::is_same<Op, OpFine5>::value) {
        LegFine l{};
        l.op = op;
        return l;
    } else {
        LegC9 l{};
        l.op = op;
        return l;
    }
}

}  // namespace

template <class Op>
int launch_leg_down(const helm_ctx* c, const Op& op, const float2* f, float2* u2, float2* rc, int nb, const int* mask) {
    const int kid = std::is_same<Op, OpFine5>::value ? K_RESTRICT_FINE : K_RESTRICT_COARSE;
    LaunchScope scope(c, kid);
    const auto l = leg_op(op);
    const LegTile t = leg_tile(op.nx, op.nz, nb, 29);
    const unsigned blocks = (unsigned)((nb + LEG_WARPS - 1) / LEG_WARPS) * (unsigned)(t.strips * t.segs);
    HELM_TRY(leg_attributes<decltype(leg_op(op))>());
    { leg_down_kernel<<<blocks, 32 * LEG_WARPS, LEG_DOWN_SMEM<decltype(leg_op(op))>, c->stream>>>(
        l, f, u2, rc, c->opt.jacobi_w, nb, t, mask, tally(c, kid, 18ull * op.nx * op.nz)); count_launch(); }
    HELM_CK(cudaGetLastError());
    return HELM_OK;
}
template int launch_leg_down<OpFine5>(const helm_ctx*, const OpFine5&, const float2*, float2*, float2*, int, const int*);
template int launch_leg_down<OpC9>(const helm_ctx*, const OpC9&, const float2*, float2*, float2*, int, const int*);

template <class Op>
int launch_leg_up(const helm_ctx* c, const Op& op, const float2* f, const float2* u2, const float2* ec, float2* u, int nb,
                  const int* mask) {
    const int kid = std::is_same<Op, OpFine5>::value ? K_JACOBI_FINE : K_JACOBI_COARSE;
    LaunchScope scope(c, kid);
    const auto l = leg_op(op);
    const LegTile t = leg_tile(op.nx, op.nz, nb, 30);
    const unsigned blocks = (unsigned)((nb + LEG_WARPS - 1) / LEG_WARPS) * (unsigned)(t.strips * t.segs);
    HELM_TRY(leg_attributes<decltype(leg_op(op))>());
    { leg_up_kernel<<<blocks, 32 * LEG_WARPS, LEG_UP_SMEM<decltype(leg_op(op))>, c->stream>>>(
        l, f, u2, ec, u, c->opt.jacobi_w, nb, t, mask, tally(c, kid, 26ull * op.nx * op.nz)); count_launch(); }
    HELM_CK(cudaGetLastError());
    return HELM_OK;
}
template int launch_leg_up<OpFine5>(const helm_ctx*, const OpFine5&, const float2*, const float2*, const float2*, float2*,
                                    int, const int*);
template int launch_leg_up<OpC9>(const helm_ctx*, const OpC9&, const float2*, const float2*, const float2*, float2*, int,
                                 const int*);

}  // namespace helm

// Coarsest-level solve of the V-cycle with one thread-block cluster per right-hand
// side: k plain GMRES steps on the Galerkin shifted Laplacian from zero (Sec. 3.4),
// the Krylov basis and the nine stencil coefficients of every node on chip.
//
// A CTA owns a slab of grid rows.  A thread owns a strip of NPT rows of one column:
// its nodes of the current vector and (NPT <= 4) their coefficients stay in registers,
// the basis vectors lie in shared memory.  The rows next to a slab are pushed into the
// neighbour CTA's halo (distributed shared memory), the inner products into every CTA.
//
// The basis is kept unnormalised: A v_j = sum_i (d_ij / n_i^2) v_i + v_{j+1} / ie_j with
// d_ij = <v_i, A v_j> and n_i = ||v_i||, where the power of two ie_j near 1 / ||A v_j|| only sets
// the scale v_{j+1} is stored at (no drift from step to step, no rounding).  n_j^2 is reduced
// together with the inner products of step j, so a step takes one reduction: FP32 within a
// thread's strip, three-term sums, as good as FP64 ones (reduce.cuh), over lanes, warps and CTAs.
// The (k+1) x k least-squares problem is solved in FP64 at the end, by rotations without square
// roots (see there).
//
// Bound by latency: a step is two barriers, two sums and some 25 instructions per node and
// basis vector.  Ten steps on one GB300, against one 512-thread block per right-hand side
// with its vectors in L2 (k_coarse.cu, whose FP64 shuffle sums alone took about half):
// 40 x 40, 1 RHS 269 -> 45 us; 128 x 64, 192 RHS 734 -> 384 us (32 clusters of four CTAs at a
// time); 256 x 128, 16 RHS 1152 -> 213 us (sixteen CTAs); 340 x 172, 40 RHS 2636 -> 1408 us
// (spilled vectors, coefficients from L2).  With FP32 sums in a warp, two-term ones beyond and a two-term
// least-squares solve it was 41, 336, 187 and 1368 us.  Error of V-cycles against 64 bits, the
// mean over 24 grids for 4, 10 and 16 steps, as a multiple of that block's: 0.96, 0.96, 0.95 (0.99,
// 0.99, 1.00 with those sums).
#include <cooperative_groups.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "helm_internal.cuh"
#include "reduce.cuh"

namespace cg = cooperative_groups;

namespace helm {
namespace {

constexpr int CC_MAX = 16;          // CTAs per cluster at most (the non-portable limit)
constexpr int CC_WARPS = 24;        // warps per CTA at most
constexpr size_t CC_SMEM = 200 * 1024;   // dynamic shared memory at most

struct CoarsePlan {
    int npt = 0;        // rows of a thread's strip (0: the layer is not taken)
    int strips = 0;     // strips per CTA; its slab has npt * strips rows
    int ctas = 0;       // CTAs per cluster
    int nsm = 0;        // basis vectors in shared memory (the others in global memory)
    int threads = 0;
    size_t smem = 0;
};

// The power of two that takes a vector of squared norm x > 0 to a norm in [1, 2).
__device__ __forceinline__ float pow2_rsqrt(float x) {
    const int e = (int)(__float_as_uint(x) >> 23) - 127;
    return __uint_as_float((unsigned)(127 - (e >> 1)) << 23);
}

template <int NPT, bool SPILL>
__global__ void __launch_bounds__(SPILL ? 32 * CC_WARPS : 512)
coarse_cluster_kernel(OpC9 op, const float2* __restrict__ f, float2* __restrict__ u, float2* __restrict__ V,
                      size_t vstride, int kmax, int S, int C, int nsm, const int* mask, Tally tl) {
    extern __shared__ __align__(16) unsigned char dynsm[];
    // the warps' sums of a step and, once the steps are done, the least-squares columns
    __shared__ union Work {
        float2 redw[3][CC_WARPS][20];               // terms (re, im) of a value per warp
        struct {
            double2 D[KMAX + 1][KMAX + 1], T[KMAX + 1][KMAX];   // columns, the right-hand side last
            double2 a[KMAX];
            double n2[KMAX + 1], u[KMAX];
        } ls;
    } wk;
    __shared__ tf2 part[CC_MAX][KMAX + 2];
    __shared__ tf2 hist[KMAX][KMAX + 1];            // d_ij
    __shared__ tf n2h[KMAX + 1];                    // n_j^2
    __shared__ float2 qs[KMAX + 1];                 // 1 / n_j^2 (hi, lo)
    __shared__ float ieh[KMAX];
    __shared__ float2 cfs[KMAX + 1];
    __shared__ unsigned wmax[CC_WARPS], cmax[CC_MAX];
    __shared__ float ie_s;
    __shared__ int stop_s;

    const int b = blockIdx.x / C, rank = blockIdx.x - b * C;
    if (!mask[b]) return;                            // the whole cluster leaves together
    tally_once(tl, rank == 0);
    cg::cluster_group cl = cg::this_cluster();
    const int nx = op.nx, nz = op.nz, t = threadIdx.x, lane = t & 31, warp = t >> 5, nwarp = blockDim.x >> 5;
    const int R = S * NPT, slab = R * nx;
    float2* slots = reinterpret_cast<float2*>(dynsm);
    float2* htop = slots + (size_t)(nsm + (SPILL ? 1 : 0)) * slab;
    float2* hbot = htop + nx;
    const int s = t / nx, ix = t - s * nx;
    const bool own = s < S;
    const int z0 = rank * R + s * NPT;               // first row of this thread's strip
    const int loc = s * NPT * nx + ix;               // its node in a slot
    const int loc_r = own ? loc : 0, z0r = own ? z0 : 0, ixr = own ? ix : 0;
    const int n = nx * nz;
    const size_t plane = (size_t)n;
    const float2* coef = op.base(__ldg(op.rhs_freq + b));
    const int xl = ix > 0 ? -1 : 0, xr = ix < nx - 1 ? 1 : 0;   // (the coefficients beyond an edge are zero)
    auto sync_all = [&]() {
        __syncwarp();
        if (C > 1) cl.sync();
        else __syncthreads();
    };

    // coefficients of this thread's nodes; rows beyond the grid have none
    constexpr int NC = SPILL ? 1 : NPT;
    float2 cf[NC][9];
    if constexpr (!SPILL) {
#pragma unroll
        for (int m = 0; m < NPT; ++m)
#pragma unroll
            for (int q = 0; q < 9; ++q)
                cf[m][q] = own && z0 + m < nz ? __ldg(coef + q * plane + (size_t)(z0 + m) * nx + ix)
                                              : make_float2(0.f, 0.f);
    }
    float2 v[NPT], w[NPT];
#pragma unroll
    for (int m = 0; m < NPT; ++m)
        v[m] = own && z0 + m < nz ? f[(size_t)b * n + (size_t)(z0 + m) * nx + ix] : make_float2(0.f, 0.f);
    for (int i = t; i < 2 * nx; i += blockDim.x) htop[i] = make_float2(0.f, 0.f);

    // Sum nv complex values over the cluster, the caller having each warp's sums in redw: groups of `wide`
    // lanes (which cover the warps and, since lane c sends the sum to CTA c, the CTAs) take a value
    // each, sum it over the CTA's warps with a shuffle tree of three-term adds, send it to every CTA,
    // and after the cluster barrier sum the CTAs' values the same way.  use(k, value) runs in the first
    // lane of a value's group.  The values pass through entries at .. at + nv - 1 of `part`; a sum
    // whose entries may still be read takes others (the last one, which no halo barrier separates
    // from the one before).
    // (a spilling CTA has more than eight warps: fixed there, which keeps registers.)
    int wide = SPILL ? 32 : 1;
    while (!SPILL && (wide < C || wide < nwarp)) wide <<= 1;
    const int sub = lane & (wide - 1), k0 = (warp * 32 + lane) / wide, kstep = nwarp * 32 / wide;
    const tf2 none = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    auto cluster_sum = [&](int nv, int at, auto use) {
        __syncthreads();
        for (int kb = warp * 32 / wide, k = k0; kb < nv; kb += kstep, k += kstep) {
            tf2 x = none;
            if (sub < nwarp && k < nv) x = {wk.redw[0][sub][k], wk.redw[1][sub][k], wk.redw[2][sub][k]};
            x = tf2_group_sum(x, wide);
            if (k >= nv) continue;
            if (C == 1) {
                if (sub == 0) use(k, x);
            } else if (sub < C) {
                *cl.map_shared_rank(&part[rank][at + k], sub) = x;
            }
        }
        if (C == 1) return;
        sync_all();
        for (int kb = warp * 32 / wide, k = k0; kb < nv; kb += kstep, k += kstep) {
            const tf2 x = tf2_group_sum(sub < C && k < nv ? part[sub][at + k] : none, wide);
            if (sub == 0 && k < nv) use(k, x);
        }
    };

    // v_0 = f inv0 with a power of two that takes the largest component to about 1 / sqrt(n), so that ||v_0|| is at
    // most about 2 (n_0 below is the norm of what is stored).  Zero, infinite or NaN f: u = 0.
    float inv0;
    {
        unsigned a = 0u;
#pragma unroll
        for (int m = 0; m < NPT; ++m)
            a = max(a, max(__float_as_uint(v[m].x) & 0x7fffffffu, __float_as_uint(v[m].y) & 0x7fffffffu));
        a = __reduce_max_sync(0xffffffffu, a);
        if (lane == 0) wmax[warp] = a;
        sync_all();                                  // (every CTA of the cluster runs: remote stores may start)
        a = __reduce_max_sync(0xffffffffu, lane < nwarp ? wmax[lane] : 0u);
        if (C > 1) {
            if (warp == 0 && lane < C) *cl.map_shared_rank(&cmax[rank], lane) = a;
            sync_all();
            a = __reduce_max_sync(0xffffffffu, lane < C ? cmax[lane] : 0u);
        }
        if (a == 0u || a >= 0x7f800000u) {
#pragma unroll
            for (int m = 0; m < NPT; ++m)
                if (own && z0 + m < nz) u[(size_t)b * n + (size_t)(z0 + m) * nx + ix] = make_float2(0.f, 0.f);
            return;
        }
        const int e = 254 - (int)(a >> 23) - (31 - __clz(n)) / 2;
        inv0 = __uint_as_float((unsigned)min(max(e, 1), 253) << 23);
    }
#pragma unroll
    for (int m = 0; m < NPT; ++m) v[m] = cscale(inv0, v[m]);

    int steps = kmax;
    for (int j = 0;; ++j) {
        float2* cur = slots + (size_t)(SPILL ? (j < nsm ? j : nsm) : j) * slab;
        if (j < kmax) {
            // v_j into its slot and the neighbours' halos
            if (own) {
#pragma unroll
                for (int m = 0; m < NPT; ++m) cur[loc + m * nx] = v[m];
                if (SPILL && j >= nsm) {
#pragma unroll
                    for (int m = 0; m < NPT; ++m)
                        if (z0 + m < nz) V[(size_t)j * vstride + (size_t)b * n + (size_t)(z0 + m) * nx + ix] = v[m];
                }
                if (s == 0 && rank > 0) cl.map_shared_rank(hbot, rank - 1)[ix] = v[0];
                if (s == S - 1 && rank < C - 1) cl.map_shared_rank(htop, rank + 1)[ix] = v[NPT - 1];
            }
            sync_all();
            // w = A v_j
#pragma unroll
            for (int m = 0; m < NPT; ++m) w[m] = make_float2(0.f, 0.f);
            if (own) {
#pragma unroll
                for (int rr = -1; rr <= NPT; ++rr) {
                    const float2* row = rr < 0 ? (s == 0 ? htop + ix : cur + loc - nx)
                                               : (rr == NPT && s == S - 1 ? hbot + ix : cur + loc + rr * nx);
                    float2 e[3];
                    e[0] = row[xl];
                    e[1] = rr >= 0 && rr < NPT ? v[rr < 0 ? 0 : (rr < NPT ? rr : 0)] : row[0];
                    e[2] = row[xr];
#pragma unroll
                    for (int dz = 1; dz >= -1; --dz) {
                        const int m = rr - dz;       // row rr is neighbour dz of row m
                        if (m < 0 || m >= NPT) continue;
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx) {
                            const int q = (dz + 1) * 3 + dx;
                            const float2 c = SPILL ? (z0 + m < nz ? __ldg(coef + q * plane + (size_t)(z0 + m) * nx + ix)
                                                                  : make_float2(0.f, 0.f))
                                                   : cf[SPILL ? 0 : m][q];
                            w[m].x += c.x * e[dx].x - c.y * e[dx].y;
                            w[m].y += c.x * e[dx].y + c.y * e[dx].x;
                        }
                    }
                }
            }
        }
        // d_ij for i <= j, then (||w||^2, n_j^2); after the last step only n_k^2
        const int nv = j < kmax ? j + 2 : 1;
        for (int i0 = 0; i0 < nv; i0 += 4) {
            // (values past nv - 1 repeat an earlier vector and are not read; value nv - 1 is set below;
            // a thread without nodes reads node 0 and has w = 0)
            float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            if (j < kmax) {
                if constexpr (!SPILL) {
                    float2 x[4][NPT];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int m = 0; m < NPT; ++m) x[q][m] = slots[min(i0 + q, j) * slab + loc_r + m * nx];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int m = 0; m < NPT; ++m) {
                            a[2 * q] += x[q][m].x * w[m].x + x[q][m].y * w[m].y;
                            a[2 * q + 1] += x[q][m].x * w[m].y - x[q][m].y * w[m].x;
                        }
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int i = min(i0 + q, j);
                        const float2* vp = i < nsm ? slots + i * slab + loc_r
                                                   : V + (size_t)i * vstride + (size_t)b * n + z0r * nx + ixr;
#pragma unroll
                        for (int m = 0; m < NPT; ++m) {
                            const float2 x = i < nsm || z0r + m < nz ? vp[m * nx] : make_float2(0.f, 0.f);
                            a[2 * q] += x.x * w[m].x + x.y * w[m].y;
                            a[2 * q + 1] += x.x * w[m].y - x.y * w[m].x;
                        }
                    }
                }
            }
            if (i0 + 4 >= nv) {
                float ax = 0.f, ay = 0.f;
#pragma unroll
                for (int m = 0; m < NPT; ++m) {
                    ax += w[m].x * w[m].x + w[m].y * w[m].y;
                    ay += v[m].x * v[m].x + v[m].y * v[m].y;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (i0 + q == nv - 1) {
                        a[2 * q] = ax;
                        a[2 * q + 1] = ay;
                    }
            }
            const tf h = tf_warp_sum8(a, lane);
            if ((lane & 3) == 0) {                    // value lane >> 2 of the eight
                reinterpret_cast<float*>(&wk.redw[0][warp][i0])[lane >> 2] = h.h;
                reinterpret_cast<float*>(&wk.redw[1][warp][i0])[lane >> 2] = h.m;
                reinterpret_cast<float*>(&wk.redw[2][warp][i0])[lane >> 2] = h.l;
            }
        }
        // the last value carries n_j^2 and ||w||^2; c_i = d_ij / n_i^2 waits for 1 / n_j^2 only at i = j
        // (c_i is an FP32 factor: two-term numbers on the way to it)
        cluster_sum(nv, j < kmax ? 0 : KMAX + 1, [&](int k, const tf2& d) {
            if (k == nv - 1) {
                n2h[j] = second_of(d);
                stop_s = j == kmax || !(d.h.y > 0.f) || !isfinite(d.h.y) ? 1 : 0;
                if (j < kmax) {
                    const float ie = d.h.x > 0.f ? pow2_rsqrt(d.h.x) : 1.f;
                    ie_s = ie;
                    ieh[j] = ie;
                }
                const ff q = ff_rcp({d.h.y, d.m.y});
                qs[j] = make_float2(q.h, q.l);
            } else {
                hist[j][k] = d;
                if (k < j) {
                    const ff q = {qs[k].x, qs[k].y};
                    cfs[k] = make_float2(ff_mul({d.h.x, d.m.x}, q).h, ff_mul({d.h.y, d.m.y}, q).h);
                }
            }
        });
        __syncthreads();
        if (stop_s) {                                 // k steps done, or v_j is zero or not finite: j steps
            steps = j;
            break;
        }
        // v_{j+1} = (w - sum_i (d_ij / n_i^2) v_i) ie
        if (own) {
            for (int i = 0; i <= j; ++i) {
                float2 c;
                if (i < j) {
                    c = cfs[i];
                } else {
                    const tf2 d = hist[j][j];
                    const ff q = {qs[j].x, qs[j].y};
                    c = make_float2(ff_mul({d.h.x, d.m.x}, q).h, ff_mul({d.h.y, d.m.y}, q).h);
                }
                if (!SPILL || i < nsm) {
                    const float2* vp = slots + (size_t)i * slab + loc;
#pragma unroll
                    for (int m = 0; m < NPT; ++m) {
                        const float2 x = vp[m * nx];
                        w[m].x -= c.x * x.x - c.y * x.y;
                        w[m].y -= c.x * x.y + c.y * x.x;
                    }
                } else {
                    const float2* vp = V + (size_t)i * vstride + (size_t)b * n + (size_t)z0 * nx + ix;
#pragma unroll
                    for (int m = 0; m < NPT; ++m) {
                        if (z0 + m >= nz) continue;
                        const float2 x = vp[(size_t)m * nx];
                        w[m].x -= c.x * x.x - c.y * x.y;
                        w[m].y -= c.x * x.y + c.y * x.x;
                    }
                }
            }
        }
        const float ie = ie_s;
#pragma unroll
        for (int m = 0; m < NPT; ++m) v[m] = cscale(ie, w[m]);
    }

    // Least squares in FP64: min || f inv0 - sum_c y_c ie_c A v_c ||, of which row i of column c is D[c][i] =
    // <v_i, ie_c A v_c> with weight 1 / n_i^2; its subdiagonal entry is n_{c+1}^2, the right-hand side (n_0^2, 0, ..).
    // Rotation i takes the running row t (entries T[c][i], a = T[i][i], weight 1 / u_i) and row i + 1, q, with h =
    // n_{i+1}^2, to the pivot row b = h conj(a) t + u_i h q, whose own entry is u_{i+1} = h |a|^2 + h^2 u_i, and the next
    // running row a q - h t of weight 1 / u_{i+1}: Givens rotations without their roots and quotients (Gentleman 1973).
    // An FP64 instruction takes a warp 64 cycles, so those off the chain run on other warps or once for all rows
    // (by Givens rotations in one warp this took 18 us for ten steps).
    {
        const int m = steps;
        auto& ls = wk.ls;
        auto wide2 = [](const tf& s) { return (widen(s.l) + widen(s.m)) + widen(s.h); };
        for (int e = t, c = 0, c0 = 0; e < m * (m + 1) / 2; e += blockDim.x) {   // entries i <= c
            while (e > c0 + c) c0 += ++c;
            const tf2 d = hist[c][e - c0];
            const double s = ieh[c];
            ls.D[c][e - c0] = make_double2(wide2(first_of(d)) * s, wide2(second_of(d)) * s);
        }
        if (t <= m) {
            const double h = wide2(n2h[t]);
            ls.n2[t] = h;
            ls.D[m][t] = make_double2(t == 0 ? h : 0.0, 0.0);
        }
        __syncthreads();
        double piv = 0.0;                             // lane i of warp 0: u_{i+1}
        const int col = lane / 2 + 1;                 // lanes 2 c - 2 and 2 c - 1: the parts of column c
        const bool im = lane & 1;
        if (warp == 0) {
            double tc = 0.0, ax = 0.0, ay = 0.0;
            if (col <= m) tc = im ? ls.D[col][0].y : ls.D[col][0].x;
            for (int i = 0; i < m; ++i) {
                double px = __shfl_sync(0xffffffffu, tc, 2 * i - 2 & 31), py = __shfl_sync(0xffffffffu, tc, 2 * i - 1 & 31);
                if (i == 0) {
                    px = ls.D[0][0].x;
                    py = ls.D[0][0].y;
                }
                if (lane == i) {
                    ax = px;
                    ay = py;
                }
                if (col > i && col <= m) {
                    const double2 q = ls.D[col][i + 1];
                    reinterpret_cast<double*>(&ls.T[col][i])[im] = tc;
                    tc = fma(px, im ? q.y : q.x, fma(im ? py : -py, im ? q.x : q.y, -ls.n2[i + 1] * tc));
                }
            }
            const double h = lane < m ? ls.n2[lane + 1] : 0.0, hx = h * ax, hy = h * ay, w = fma(hx, ax, hy * ay), hh = h * h;
            double u = ls.n2[0], uo = 0.0;
            for (int i = 0; i < m; ++i) {
                if (lane == i) uo = u;
                u = fma(__shfl_sync(0xffffffffu, hh, i), u, __shfl_sync(0xffffffffu, w, i));
                if (lane == i) piv = u;
            }
            if (lane < m) {
                ls.a[lane] = make_double2(hx, hy);
                ls.u[lane] = uo * h;
            }
        }
        __syncthreads();
        // the pivot rows over T while warp 0 takes the reciprocals of their own entries
        if (warp == 0) {
            // (0: no component; not finite: it stays so)
            piv = piv > 0.0 ? 1.0 / piv : piv;
        } else {
            for (int e = t - 32, c = 1, c0 = 0; e < m * (m + 1) / 2; e += blockDim.x - 32) {   // entries i < c <= m
                while (e >= c0 + c) c0 += c++;
                const int i = e - c0;
                const double2 a = ls.a[i], b = ls.T[c][i], q = ls.D[c][i + 1];
                const double w = ls.u[i];
                ls.T[c][i] = make_double2(fma(a.x, b.x, fma(a.y, b.y, w * q.x)), fma(a.x, b.y, fma(-a.y, b.x, w * q.y)));
            }
        }
        __syncthreads();
        if (warp == 0) {
            // back substitution: lanes 2 i and 2 i + 1 have the parts of row i
            const int row = lane / 2;
            const double r = __shfl_sync(0xffffffffu, piv, row);
            double g = 0.0;
            if (row < m) g = im ? ls.T[m][row].y : ls.T[m][row].x;
            for (int c = m - 1; c >= 0; --c) {
                const double y = g * r, yx = __shfl_sync(0xffffffffu, y, 2 * c), yy = __shfl_sync(0xffffffffu, y, 2 * c + 1);
                if (row < c) {
                    const double2 b = ls.T[c][row];
                    g = fma(-b.x, im ? yy : yx, fma(im ? -b.y : b.y, im ? yx : yy, g));
                } else if (lane == 2 * c) {
                    const double s = (double)ieh[c] * (double)(1.0f / inv0);   // powers of two
                    cfs[c] = make_float2((float)(yx * s), (float)(yy * s));
                }
            }
        }
    }
    __syncthreads();
    // u = sum_i y_i v_i
#pragma unroll
    for (int m = 0; m < NPT; ++m) w[m] = make_float2(0.f, 0.f);
    if (own) {
        for (int i = 0; i < steps; ++i) {
            const float2 c = cfs[i];
            const bool in_sm = !SPILL || i < nsm;
            const float2* vp = in_sm ? slots + (size_t)i * slab + loc
                                     : V + (size_t)i * vstride + (size_t)b * n + (size_t)z0 * nx + ix;
#pragma unroll
            for (int m = 0; m < NPT; ++m) {
                if (!in_sm && z0 + m >= nz) continue;
                const float2 x = vp[m * nx];
                w[m].x += c.x * x.x - c.y * x.y;
                w[m].y += c.x * x.y + c.y * x.x;
            }
        }
#pragma unroll
        for (int m = 0; m < NPT; ++m)
            if (z0 + m < nz) u[(size_t)b * n + (size_t)(z0 + m) * nx + ix] = w[m];
    }
}

template <int NPT, bool SPILL>
bool cc_attributes() {
    static DeviceOnce once;
    const cudaError_t e = once_per_device(once, [] {
        const cudaError_t s = cudaFuncSetAttribute(coarse_cluster_kernel<NPT, SPILL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CC_SMEM);
        return s != cudaSuccess ? s : cudaFuncSetAttribute(coarse_cluster_kernel<NPT, SPILL>,
                                                           cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    });
    if (e != cudaSuccess) (void)cudaGetLastError();
    return e == cudaSuccess;
}

void cc_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at, const CoarsePlan& p, int nb, cudaStream_t st) {
    cfg->gridDim = dim3((unsigned)(nb * p.ctas));
    cfg->blockDim = dim3((unsigned)p.threads);
    cfg->dynamicSmemBytes = p.smem;
    cfg->stream = st;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)p.ctas;
    at->val.clusterDim.y = 1;
    at->val.clusterDim.z = 1;
    cfg->attrs = at;
    cfg->numAttrs = 1;
}

// Clusters of a plan that the device holds at once (0: it cannot run there).
template <int NPT, bool SPILL>
int cc_resident(const CoarsePlan& p) {
    if (!cc_attributes<NPT, SPILL>()) return 0;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at;
    cc_config(&cfg, &at, p, 1, nullptr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, coarse_cluster_kernel<NPT, SPILL>, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return n;
}
int cc_resident(const CoarsePlan& p) {
    switch (p.npt) {
        case 1: return cc_resident<1, false>(p);
        case 2: return cc_resident<2, false>(p);
        case 4: return cc_resident<4, false>(p);
        default: return cc_resident<8, true>(p);
    }
}

// The plan of a grid, step count and batch; .npt = 0 when no cluster holds the grid.  A solve is bound
// by the latency of its barriers and sums, about 35 us for ten steps, plus 12 us per 1000 nodes on an
// SM (three times that when coefficients and late basis vectors come from L2), so the plan takes the
// smallest waves x latency: a large batch the fewest CTAs per right-hand side, a small one more.
CoarsePlan coarse_plan(int nx, int nz, int k, int nb, int sms) {
    CoarsePlan best;
    double best_us = 1e30;
    for (int npt : {1, 2, 4, 8}) {
        const bool spill = npt == 8;
        const int tmax = spill ? 32 * CC_WARPS : 512;
        for (int S = 1; S * nx <= tmax; ++S) {
            CoarsePlan p;
            p.npt = npt;
            p.strips = S;
            p.ctas = (nz + npt * S - 1) / (npt * S);
            if (p.ctas > CC_MAX) continue;
            if (S > 1 && (nz + npt * (S - 1) - 1) / (npt * (S - 1)) == p.ctas) continue;   // the same with fewer strips
            p.threads = std::max((nx * S + 31) / 32 * 32, 128);
            const size_t slab = (size_t)npt * S * nx * sizeof(float2), halo = 2 * (size_t)nx * sizeof(float2);
            const size_t room = CC_SMEM - halo;
            if (spill) {
                if (room < 2 * slab) continue;
                p.nsm = std::min<int>(k, (int)(room / slab) - 1);
                p.smem = (p.nsm + 1) * slab + halo;
            } else {
                if ((size_t)k * slab > room) continue;
                p.nsm = k;
                p.smem = k * slab + halo;
            }
            const int res = cc_resident(p);
            if (res < 1) continue;
            const int held = std::min(nb, res);
            const int per_sm = std::max(1, (held * p.ctas + sms - 1) / sms);
            const double us = ((nb + res - 1) / res) *
                              (35.0 + 0.3 * p.ctas + 0.0125 * (spill ? 3 : 1) * npt * S * nx * per_sm);
            if (us < best_us) {
                best_us = us;
                best = p;
            }
        }
    }
    return best;
}

// Plans by shape (a first call of a batch size takes no longer than the second: 115 us at 160 x 160).
CoarsePlan coarse_plan_cached(int nx, int nz, int k, int nb) {
    static std::mutex mu;
    static std::map<std::tuple<int, int, int, int, int>, CoarsePlan> plans;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return CoarsePlan{};
    }
    const auto key = std::make_tuple(dev, nx, nz, k, nb);
    std::lock_guard<std::mutex> lk(mu);
    auto it = plans.find(key);
    if (it == plans.end()) {
        if (plans.size() >= 4096) plans.clear();
        it = plans.emplace(key, coarse_plan(nx, nz, k, nb, sms)).first;
    }
    return it->second;
}

template <int NPT, bool SPILL>
int launch_cc(const helm_ctx* c, const CoarsePlan& p, const OpC9& op, const float2* f, float2* u, size_t vstride, int k,
              int nb, const int* mask, const Tally& tl) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at;
    cc_config(&cfg, &at, p, nb, c->stream);
    HELM_CK(cudaLaunchKernelEx(&cfg, coarse_cluster_kernel<NPT, SPILL>, op, f, u, c->Vc, vstride, k, p.strips, p.ctas,
                               p.nsm, mask, tl));
    count_launch();
    return HELM_OK;
}
}  // namespace

// The coarsest-level solve by clusters: u = k GMRES steps for A u = f from zero.  HELM_EUNSUPPORTED (nothing
// launched) when no cluster holds the grid (more than 16 slabs of 8 rows, or rows wider than a CTA).
int launch_coarse_cluster(const helm_ctx* c, int level, const float2* f, float2* u, int nb, const int* mask) {
    const Level& L = c->lev[level];
    const size_t Nc = (size_t)L.nx * L.nz;
    const int k = c->opt.coarse_iters;
    const CoarsePlan p = coarse_plan_cached(L.nx, L.nz, k, nb);
    if (!p.npt) return HELM_EUNSUPPORTED;
    LaunchScope scope(c, K_COARSE_GMRES);
    // f in, u out; of n spilled vectors each is written once and read twice in its own step and every later one, and
    // once for the combination: n^2 + 3 n
    const unsigned long long n = (unsigned long long)(k - p.nsm);
    const Tally tl = tally(c, K_COARSE_GMRES, 8ull * Nc * (2 + n * n + 3 * n));
    const OpC9 op = coarse_op(c, level);
    const size_t vs = (size_t)c->cap * Nc;
    switch (p.npt) {
        case 1: return launch_cc<1, false>(c, p, op, f, u, vs, k, nb, mask, tl);
        case 2: return launch_cc<2, false>(c, p, op, f, u, vs, k, nb, mask, tl);
        case 4: return launch_cc<4, false>(c, p, op, f, u, vs, k, nb, mask, tl);
        default: return launch_cc<8, true>(c, p, op, f, u, vs, k, nb, mask, tl);
    }
}
}  // namespace helm

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
// d_ij = <v_i, A v_j> and n_i = ||v_i||, where ie_j = 1 / ||A v_j|| only sets the scale
// v_{j+1} is stored at (no drift from step to step).  n_j^2 is reduced together
// with the inner products of step j, so a step takes one reduction: FP32 within a
// thread's strip and its warp, then two-term (hi + lo) sums over warps and CTAs.  The
// (k+1) x k least-squares problem with columns d_ij / n_i, n_{j+1} / ie_j is solved in
// two-term arithmetic at the end, each rotation applied to all later columns at once.
//
// Bound by latency: a step is two barriers, two sums and some 25 instructions per node and
// basis vector.  Ten steps on one GB300, against one 512-thread block per right-hand side
// with its vectors in L2 (k_coarse.cu, whose FP64 shuffle sums alone took about half):
// 40 x 40, 1 RHS 269 -> 41 us; 128 x 64, 192 RHS 734 -> 334 us (32 clusters of four CTAs at a
// time); 256 x 128, 16 RHS 1152 -> 184 us (sixteen CTAs); 340 x 172, 40 RHS 2636 -> 1470 us
// (spilled vectors, coefficients from L2).
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

template <int NPT, bool SPILL>
__global__ void __launch_bounds__(SPILL ? 32 * CC_WARPS : 512)
coarse_cluster_kernel(OpC9 op, const float2* __restrict__ f, float2* __restrict__ u, float2* __restrict__ V,
                      size_t vstride, int kmax, int S, int C, int nsm, const int* mask, Tally tl) {
    extern __shared__ __align__(16) unsigned char dynsm[];
    __shared__ float2 redw[CC_WARPS][20];
    __shared__ float4 part[CC_MAX][KMAX + 2];
    __shared__ float4 hist[KMAX][KMAX + 1];         // d_ij as (re hi, re lo, im hi, im lo)
    __shared__ float2 n2h[KMAX + 1], qs[KMAX + 1];  // n_j^2 and 1 / n_j^2 (hi, lo)
    __shared__ float ieh[KMAX];
    __shared__ float4 Hs[KMAX + 1][KMAX + 3];       // least-squares columns, the right-hand side last
    __shared__ float2 nsh[KMAX + 1], rns[KMAX + 1]; // n_j and 1 / n_j
    __shared__ float2 cfs[KMAX + 1];
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

    // Sum nv complex values over the cluster, the caller having each warp's sums in redw: warp k sums
    // value k (k + nwarp, ...) over the CTA's warps with a shuffle tree of two-term adds, sends it to
    // every CTA, and after the cluster barrier sums the CTAs' values the same way.  use(k, value) runs
    // in every lane of that warp.  The values pass through entries at .. at + nv - 1 of `part`; a sum
    // whose entries may still be read takes others (the last one, which no halo barrier separates
    // from the one before).
    auto tree = [&](float4 r, int width) -> float4 {
        for (int o = width >> 1; o > 0; o >>= 1) {
            const ff x = ff_add({r.x, r.y}, {__shfl_xor_sync(0xffffffffu, r.x, o), __shfl_xor_sync(0xffffffffu, r.y, o)});
            const ff y = ff_add({r.z, r.w}, {__shfl_xor_sync(0xffffffffu, r.z, o), __shfl_xor_sync(0xffffffffu, r.w, o)});
            r = make_float4(x.h, x.l, y.h, y.l);
        }
        return r;
    };
    // tree widths: cwide covers the CTAs; wwide the warps and, since lane c sends the sum to CTA c, the CTAs
    int cwide = 1;
    while (cwide < C) cwide <<= 1;
    int wwide = cwide;
    while (wwide < nwarp) wwide <<= 1;
    auto cluster_sum = [&](int nv, int at, auto use) {
        __syncthreads();
        for (int k = warp; k < nv; k += nwarp) {
            const float2 x = lane < nwarp ? redw[lane][k] : make_float2(0.f, 0.f);
            const float4 r = tree(make_float4(x.x, 0.f, x.y, 0.f), wwide);
            if (C == 1) use(k, r);
            else if (lane < C) *cl.map_shared_rank(&part[rank][at + k], lane) = r;
        }
        if (C == 1) return;
        sync_all();
        for (int k = warp; k < nv; k += nwarp)
            use(k, tree(lane < C ? part[lane][at + k] : make_float4(0.f, 0.f, 0.f, 0.f), cwide));
    };

    // beta = ||f||: v_0 = f / beta (in FP32; n_0 below is the exact norm of what is stored)
    {
        float a = 0.f;
#pragma unroll
        for (int m = 0; m < NPT; ++m) a += v[m].x * v[m].x + v[m].y * v[m].y;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) redw[warp][0] = make_float2(a, 0.f);
        if (C > 1) sync_all();                       // every CTA of the cluster runs: remote stores may start
        cluster_sum(1, 0, [&](int, const float4& r) {
            if (lane == 0) ie_s = r.x > 0.f && isfinite(r.x) ? rsqrtf(r.x) : 0.f;
        });
        __syncthreads();
    }
    const float inv0 = ie_s;
    if (!(inv0 > 0.f)) {
#pragma unroll
        for (int m = 0; m < NPT; ++m)
            if (own && z0 + m < nz) u[(size_t)b * n + (size_t)(z0 + m) * nx + ix] = make_float2(0.f, 0.f);
        return;
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
            // eight warp sums in nine shuffles: each halving step leaves a lane with half the values
            float h4[4], h2[2], h1;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float keep = lane & 16 ? a[k + 4] : a[k], give = lane & 16 ? a[k] : a[k + 4];
                h4[k] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const float keep = lane & 8 ? h4[k + 2] : h4[k], give = lane & 8 ? h4[k] : h4[k + 2];
                h2[k] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
            }
            {
                const float keep = lane & 4 ? h2[1] : h2[0], give = lane & 4 ? h2[0] : h2[1];
                h1 = keep + __shfl_xor_sync(0xffffffffu, give, 4);
            }
            h1 += __shfl_xor_sync(0xffffffffu, h1, 2);
            h1 += __shfl_xor_sync(0xffffffffu, h1, 1);
            if ((lane & 3) == 0)                      // value 4 bit4 + 2 bit3 + bit2 of the eight
                reinterpret_cast<float*>(&redw[warp][i0])[lane >> 2] = h1;
        }
        // the last value carries n_j^2 and ||w||^2; c_i = d_ij / n_i^2 waits for 1 / n_j^2 only at i = j
        cluster_sum(nv, j < kmax ? 0 : KMAX + 1, [&](int k, const float4& d) {
            if (lane != 0) return;
            if (k == nv - 1) {
                n2h[j] = make_float2(d.z, d.w);
                stop_s = j == kmax || !(d.z > 0.f) || !isfinite(d.z) ? 1 : 0;
                if (j < kmax) {
                    const float ie = d.x > 0.f ? rsqrtf(d.x) : 1.f;
                    ie_s = ie;
                    ieh[j] = ie;
                }
                const ff q = ff_rcp({d.z, d.w});
                qs[j] = make_float2(q.h, q.l);
            } else {
                hist[j][k] = d;
                if (k < j) {
                    const ff q = {qs[k].x, qs[k].y};
                    cfs[k] = make_float2(ff_mul({d.x, d.y}, q).h, ff_mul({d.z, d.w}, q).h);
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
                    const float4 d = hist[j][j];
                    const ff q = {qs[j].x, qs[j].y};
                    c = make_float2(ff_mul({d.x, d.y}, q).h, ff_mul({d.z, d.w}, q).h);
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

    // least squares min || beta e_1 - H y ||: lane c < steps has column c, lane `steps` the right-hand side
    if (warp == 0) {
        const int m = steps;
        if (lane <= m) {
            const ff n2 = {n2h[lane].x, n2h[lane].y};
            const ff r = n2.h > 0.f ? ff_rsqrt(n2) : ff{0.f, 0.f}, nn = ff_mul(n2, r);
            rns[lane] = make_float2(r.h, r.l);
            nsh[lane] = make_float2(nn.h, nn.l);
        }
        __syncwarp();
        if (lane < m) {
            for (int i = 0; i <= lane; ++i) {
                const float4 d = hist[lane][i];
                const ff rn = {rns[i].x, rns[i].y}, x = ff_mul(ff{d.x, d.y}, rn), y = ff_mul(ff{d.z, d.w}, rn);
                Hs[lane][i] = make_float4(x.h, x.l, y.h, y.l);
            }
            const ff x = ff_mul(ff{nsh[lane + 1].x, nsh[lane + 1].y}, ff_rcp(ff{ieh[lane], 0.f}));
            Hs[lane][lane + 1] = make_float4(x.h, x.l, 0.f, 0.f);
        } else if (lane == m) {
            const ff x = ff_mul(ff{nsh[0].x, nsh[0].y}, ff_rcp(ff{inv0, 0.f}));
            Hs[m][0] = make_float4(x.h, x.l, 0.f, 0.f);
            for (int i = 1; i <= m; ++i) Hs[m][i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncwarp();
        ff rinv = {0.f, 0.f};                         // lane i: 1 / R_ii
        float4 p = lane <= m ? Hs[lane][0] : make_float4(0.f, 0.f, 0.f, 0.f);   // row i of this lane's column
        for (int i = 0; i < m; ++i) {
            ff cx = {0.f, 0.f}, cy = {0.f, 0.f}, sn = {0.f, 0.f};
            if (lane == i) {
                const ff ax = {p.x, p.y}, ay = {p.z, p.w}, hb = {Hs[i][i + 1].x, Hs[i][i + 1].y};
                const ff x = ff_add(ff_add(ff_mul(ax, ax), ff_mul(ay, ay)), ff_mul(hb, hb));
                // (x = 0: no component; x not finite: it stays so)
                rinv = x.h > 0.f ? ff_rsqrt(x) : x;
                cx = ff_mul(ax, rinv);
                cy = ff_mul(ay, rinv);
                sn = ff_mul(hb, rinv);
            }
            cx = ff_shfl(cx, i);
            cy = ff_shfl(cy, i);
            sn = ff_shfl(sn, i);
            if (lane > i && lane <= m) {              // [conj(c) s; -s c] on rows i, i + 1
                const float4 q = Hs[lane][i + 1];
                const ff px = {p.x, p.y}, py = {p.z, p.w}, qx = {q.x, q.y}, qy = {q.z, q.w};
                const ff tx = ff_add(ff_add(ff_mul(cx, px), ff_mul(cy, py)), ff_mul(sn, qx));
                const ff ty = ff_add(ff_add(ff_mul(cx, py), ff_neg(ff_mul(cy, px))), ff_mul(sn, qy));
                const ff vx = ff_add(ff_add(ff_mul(cx, qx), ff_neg(ff_mul(cy, qy))), ff_neg(ff_mul(sn, px)));
                const ff vy = ff_add(ff_add(ff_mul(cx, qy), ff_mul(cy, qx)), ff_neg(ff_mul(sn, py)));
                Hs[lane][i] = make_float4(tx.h, tx.l, ty.h, ty.l);
                p = make_float4(vx.h, vx.l, vy.h, vy.l);
            }
        }
        __syncwarp();
        ff gx = {0.f, 0.f}, gy = {0.f, 0.f};
        if (lane < m) {
            const float4 g = Hs[m][lane];
            gx = {g.x, g.y};
            gy = {g.z, g.w};
        }
        for (int c = m - 1; c >= 0; --c) {
            const ff yx = ff_shfl(ff_mul(gx, rinv), c), yy = ff_shfl(ff_mul(gy, rinv), c);
            if (lane < c) {
                const float4 r = Hs[c][lane];
                const ff rx = ff_neg(ff{r.x, r.y}), ry = ff_neg(ff{r.z, r.w});
                gx = ff_add(ff_add(gx, ff_mul(rx, yx)), ff_neg(ff_mul(ry, yy)));
                gy = ff_add(ff_add(gy, ff_mul(rx, yy)), ff_mul(ry, yx));
            }
            if (lane == c) cfs[c] = make_float2(yx.h, yy.h);
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
    static std::once_flag once;
    static bool ok = false;
    std::call_once(once, [] {
        ok = cudaFuncSetAttribute(coarse_cluster_kernel<NPT, SPILL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)CC_SMEM) == cudaSuccess &&
             cudaFuncSetAttribute(coarse_cluster_kernel<NPT, SPILL>, cudaFuncAttributeNonPortableClusterSizeAllowed,
                                  1) == cudaSuccess;
        (void)cudaGetLastError();
    });
    return ok;
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

// Plans by shape: the occupancy queries of one cost some hundred microseconds.
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
    const unsigned long long kk = (unsigned long long)k;
    LaunchScope scope(c, K_COARSE_GMRES);
    // as the other coarsest solve counts: ||f||, per step 2 (j + 1) basis reads, v_j, w, v_{j+1}, the combination
    const Tally tl = tally(c, K_COARSE_GMRES, 8ull * Nc * (kk * kk + 5 * kk + 2));
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

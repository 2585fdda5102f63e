// Fine-grid Helmholtz kernels: the matrix-free five-point operator H(m, w)
// of Eq. 3.1-3.2 (and the shifted Laplacian of Eq. 3.12), the FP64 true
// residual used at every FGMRES restart, and the per-RHS restart logic.
#include <type_traits>

#include "helm_internal.cuh"
#include "reduce.cuh"

namespace helm {

namespace {

constexpr int NTHREADS = TILE_X * TILE_Y;
constexpr int NWARPS = NTHREADS / 32;

__global__ void apply_fine_kernel(OpFine5 op, const float2* __restrict__ x, float2* __restrict__ y,
                                  const int* mask, Tally tl) {
    const int b = blockIdx.z;
    if (!mask[b]) return;
    tally_once(tl, blockIdx.x == 0 && blockIdx.y == 0);
    const int ix = blockIdx.x * blockDim.x + threadIdx.x;
    const int iz = blockIdx.y * blockDim.y + threadIdx.y;
    if (ix >= op.nx || iz >= op.nz) return;
    const size_t N = (size_t)op.nx * op.nz;
    y[(size_t)b * N + (size_t)iz * op.nx + ix] = op.apply(x + (size_t)b * N, b, ix, iz);
}

// y = A x on node pairs (nx even): a thread carries three rows of its pair down `rows` rows, so that a
// field is read about once (the neighbours' columns come from L1) with 16-byte accesses.  The rounded
// operations are those of OpFine5::apply in apply_fine_kernel, spelled out: the training pairs made
// from H x do not depend on which kernel made it.  512 x 256, 192 fields, one GB300:
// 115 -> 68 us (403 MB: 5.9 TB/s), 135 -> 96 us with the call's host part.
__global__ void __launch_bounds__(NTHREADS) apply_fine2_kernel(OpFine5 op, const float2* __restrict__ x,
                                                               float2* __restrict__ y, int rows, const int* mask,
                                                               Tally tl) {
    const int b = blockIdx.z;
    if (!mask[b]) return;
    tally_once(tl, blockIdx.x == 0 && blockIdx.y == 0);
    const int nx = op.nx, nz = op.nz;
    const int ix = 2 * (blockIdx.x * TILE_X + threadIdx.x);
    const int iz0 = (blockIdx.y * TILE_Y + threadIdx.y) * rows;
    if (ix >= nx || iz0 >= nz) return;
    const size_t N = (size_t)nx * nz;
    const float2* xb = x + (size_t)b * N + ix;
    float2* yb = y + (size_t)b * N + ix;
    const float w = __ldg(op.omega + __ldg(op.rhs_freq + b)), w2 = __fmul_rn(w, w);
    const float ax = op.ax, az = op.az;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    auto row = [&](int iz) { return iz >= 0 && iz < nz ? __ldg(reinterpret_cast<const float4*>(xb + (size_t)iz * nx)) : zero; };
    // ax (2 c - l - r) + az (2 c - n - s)
    auto lap = [&](float c, float l, float r, float n, float s) {
        return __fmaf_rn(ax, __fsub_rn(__fmaf_rn(2.f, c, -l), r), __fmul_rn(az, __fsub_rn(__fmaf_rn(2.f, c, -n), s)));
    };
    float4 n = row(iz0 - 1), c = row(iz0);
#pragma unroll 4
    for (int rr = 0; rr < rows; ++rr) {
        const int iz = iz0 + rr;
        if (iz >= nz) break;
        const float4 s = row(iz + 1);
        const float2 l = ix > 0 ? __ldg(xb + (size_t)iz * nx - 1) : make_float2(0.f, 0.f);
        const float2 r = ix + 2 < nx ? __ldg(xb + (size_t)iz * nx + 2) : make_float2(0.f, 0.f);
        const float4 m = __ldg(reinterpret_cast<const float4*>(op.mg + (size_t)iz * nx + ix));
        const float s0 = __fmul_rn(w2, __fmul_rn(m.x, m.x)), s1 = __fmul_rn(w2, __fmul_rn(m.z, m.z));
        const float g0 = op.sl ? __fadd_rn(op.beta, op.incg ? m.y : 0.0f) : m.y;
        const float g1 = op.sl ? __fadd_rn(op.beta, op.incg ? m.w : 0.0f) : m.w;
        const float k0 = __fmul_rn(-s0, g0), k1 = __fmul_rn(-s1, g1);
        float4 o;
        o.x = __fsub_rn(lap(c.x, l.x, c.z, n.x, s.x), __fmaf_rn(s0, c.x, -__fmul_rn(k0, c.y)));
        o.y = __fsub_rn(lap(c.y, l.y, c.w, n.y, s.y), __fmaf_rn(s0, c.y, __fmul_rn(k0, c.x)));
        o.z = __fsub_rn(lap(c.z, c.x, r.x, n.z, s.z), __fmaf_rn(s1, c.z, -__fmul_rn(k1, c.w)));
        o.w = __fsub_rn(lap(c.w, c.y, r.y, n.w, s.w), __fmaf_rn(s1, c.w, __fmul_rn(k1, c.z)));
        *reinterpret_cast<float4*>(yb + (size_t)iz * nx) = o;
        n = c;
        c = s;
    }
}

// r = b - H x evaluated in FP64 from the complex128 iterate x (b conjugated
// when solving the adjoint system); r is stored in complex64 as the first
// (unscaled) Krylov vector.  ||r||^2 and, on the first call, ||b||^2 are
// reduced per RHS in FP64.
//
// Bound by the FP64 pipe (two operations per SM and cycle on this GPU): 20 per node and RHS as
//   r = b - ax (2 xc - xw - xe) + az ((xs - xc) - (xc - xn)) + w^2 m xc - i (w^2 m gamma) xc
// with w^2 m and its products shared by a thread's two right-hand sides of one frequency and xs - xc by
// the next row, against 34 in the order the operator is written, its conversions included.  512 x 256,
// 192 right-hand sides, one GB300: 1.93 -> 1.34 ms a call.
// The differences stay: with the five terms of xc in one product it takes 17 (1.32 ms a call), but the large
// terms cancel, and the error, over the norm of w^2 m x, at 10, 40 and 160 points per wavelength is
// 7e-16, 1e-14 and 2e-13 in place of 1e-16, 1e-15 and 8e-15 (2e-16, 2e-15 and 1e-14 in the written order).
template <bool FIRST>
__global__ void __launch_bounds__(NTHREADS) residual64_kernel(OpFine5 op, const double2* __restrict__ x,
                                                              const float2* __restrict__ bvec,
                                                              float2* __restrict__ r, int conj_b, int nb, int rows,
                                                              double ax, double az, OuterState os, Tally tl) {
    const int b0 = 2 * blockIdx.z;
    const bool act[2] = {os.outer_active[b0] != 0, b0 + 1 < nb && os.outer_active[b0 + 1] != 0};
    if (!act[0] && !act[1]) return;
    if (act[0]) tally_once(tl, blockIdx.x == 0 && blockIdx.y == 0);
    if (act[1]) tally_once(tl, blockIdx.x == 0 && blockIdx.y == 0);
    const int nx = op.nx, nz = op.nz;
    const size_t N = (size_t)nx * nz;
    const int ix = blockIdx.x * TILE_X + threadIdx.x;
    const int iz0 = (blockIdx.y * TILE_Y + threadIdx.y) * rows;
    const int f0 = op.rhs_freq[b0], f1 = b0 + 1 < nb ? op.rhs_freq[b0 + 1] : f0;
    double w2[2];
    {
        const double a = op.omega[f0], c = op.omega[f1];
        w2[0] = a * a;
        w2[1] = c * c;
    }
    double acc_r[2] = {0.0, 0.0}, acc_b[2] = {0.0, 0.0};
    if (ix < nx) {
        const double2 zero = make_double2(0.0, 0.0);
        double2 dn[2], xc[2];   // this row less the one above, this row
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const double2* xb = x + (size_t)(b0 + q) * N + ix;
            const double2 xn = act[q] && iz0 > 0 && iz0 < nz ? xb[(size_t)(iz0 - 1) * nx] : zero;
            xc[q] = act[q] && iz0 < nz ? xb[(size_t)iz0 * nx] : zero;
            dn[q] = make_double2(xc[q].x - xn.x, xc[q].y - xn.y);
        }
        for (int rr = 0; rr < rows; ++rr) {
            const int iz = iz0 + rr;
            if (iz >= nz) break;
            const size_t p = (size_t)iz * nx + ix;
            const float2 mg = op.mg[p];
            const double k = widen(mg.x), m = k * k, gam = widen(mg.y);
            double s = 0.0, ci = 0.0;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                if (!act[q]) continue;
                const double2* xb = x + (size_t)(b0 + q) * N + p;
                const double2 xs = iz < nz - 1 ? xb[nx] : zero;
                const double2 xw = ix > 0 ? xb[-1] : zero;
                const double2 xe = ix < nx - 1 ? xb[1] : zero;
                const float2 bv = bvec[(size_t)(b0 + q) * N + p];
                if (q == 0 || f1 != f0 || !act[0]) {
                    s = w2[q] * m;
                    ci = s * gam;                                  // coefficient s (1 - i gamma)
                }
                const double bx = widen(bv.x), by = widen(conj_b ? -bv.y : bv.y);
                const double2 ds = make_double2(xs.x - xc[q].x, xs.y - xc[q].y);
                const double lx = fma(2.0, xc[q].x, -xw.x) - xe.x, ly = fma(2.0, xc[q].y, -xw.y) - xe.y;
                const double rx = fma(ci, xc[q].y, fma(s, xc[q].x, fma(az, ds.x - dn[q].x, fma(-ax, lx, bx))));
                const double ry = fma(-ci, xc[q].x, fma(s, xc[q].y, fma(az, ds.y - dn[q].y, fma(-ax, ly, by))));
                r[(size_t)(b0 + q) * N + p] = make_float2(narrow(rx), narrow(ry));
                acc_r[q] = fma(rx, rx, fma(ry, ry, acc_r[q]));
                if (FIRST) acc_b[q] = fma(bx, bx, fma(by, by, acc_b[q]));
                dn[q] = ds;
                xc[q] = xs;
            }
        }
    }
    __shared__ double2 sm[2][NWARPS];
    __shared__ unsigned s_last[2];
    const int tid = threadIdx.x + threadIdx.y * TILE_X, lane = tid & 31, warp = tid >> 5;
    const int ntiles = gridDim.x * gridDim.y, tile = blockIdx.y * gridDim.x + blockIdx.x;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        if (!act[q]) continue;
        const double a = warp_sum(acc_r[q]), c = FIRST ? warp_sum(acc_b[q]) : 0.0;
        if (lane == 0) sm[q][warp] = make_double2(a, c);
    }
    __syncthreads();
    if (tid < 2 && act[tid]) {
        double2 t = make_double2(0.0, 0.0);
        for (int w = 0; w < NWARPS; ++w) t = dadd(t, sm[tid][w]);
        os.partials[(size_t)(b0 + tid) * ntiles + tile] = t;
        __threadfence();
        const unsigned n = atomicAdd(os.counters + b0 + tid, 1u);
        s_last[tid] = n == (unsigned)ntiles - 1u ? 1u : 0u;
        if (s_last[tid]) os.counters[b0 + tid] = 0u;
    }
    __syncthreads();
    // the last block of an RHS sums the tiles (warp q for RHS b0 + q, lanes over the tiles in a fixed order)
    if (warp < 2 && act[warp] && s_last[warp]) {
        __threadfence();
        double2 t = make_double2(0.0, 0.0);
        for (int i = lane; i < ntiles; i += 32) t = dadd(t, __ldcg(os.partials + (size_t)(b0 + warp) * ntiles + i));
        const double a = warp_sum(t.x), c = FIRST ? warp_sum(t.y) : 0.0;
        if (lane == 0) {
            os.rnorm2[b0 + warp] = a;
            if (FIRST) os.bnorm2[b0 + warp] = c;
        }
    }
}

__global__ void conj64_kernel(double2* x, size_t n) {
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < n; p += (size_t)gridDim.x * blockDim.x)
        x[p].y = -x[p].y;
}

// Decide per RHS after the restart residual: converged, out of steps,
// broken down, or start another cycle (g_0 = ||r||, s_0 = 1/||r||).
__global__ void restart_check_kernel(OuterState os, KState st, int nb, double tol, int max_iter, double inner,
                                     int* n_active) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    int act = os.outer_active[b];
    if (act) {
        os.iters[b] += st.steps[b];
        double rn = sqrt(os.rnorm2[b]);
        double bn = sqrt(os.bnorm2[b]);
        if (!isfinite(rn) || os.status[b] == HELM_EBREAKDOWN) {
            os.status[b] = HELM_EBREAKDOWN;
            act = 0;
        } else if (bn == 0.0 || rn <= tol * bn) {
            os.status[b] = HELM_OK;
            act = 0;
        } else if (os.iters[b] >= max_iter) {
            os.status[b] = HELM_ENOCONV;
            act = 0;
        } else {
            // a restart cycle that lowered the residual by less than 10 % marks the RHS:
            // its network composition is guarded from now on
            if (os.rprev[b] > 0.0 && rn > 0.9 * os.rprev[b]) os.guard[b] = 1;
            os.rprev[b] = rn;
            st.g[(size_t)b * (st.k + 1)] = make_double2(rn, 0.0);
            st.s[(size_t)b * (st.k + 1)] = 1.0 / rn;
            st.inv_est[b] = 1.0 / rn;
            st.tol_abs[b] = inner * tol * bn;
            atomicAdd(n_active, 1);
        }
        os.outer_active[b] = act;
    }
    st.steps[b] = 0;
    st.active[b] = act;
}

__global__ void outer_init_kernel(OuterState os, KState st, int nb) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    os.iters[b] = 0;
    os.status[b] = HELM_OK;
    os.outer_active[b] = 1;
    os.rnorm2[b] = 0.0;
    os.bnorm2[b] = 0.0;
    os.rprev[b] = 0.0;
    os.guard[b] = 0;
    st.steps[b] = 0;
    st.active[b] = 0;
}

// x = 0 for right-hand sides that are identically zero
__global__ void zero_x_kernel(OuterState os, double2* x, size_t n) {
    const int b = blockIdx.y;
    if (os.bnorm2[b] != 0.0) return;
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < n; p += (size_t)gridDim.x * blockDim.x)
        x[(size_t)b * n + p] = make_double2(0.0, 0.0);
}

}  // namespace

int launch_apply_fine(const helm_ctx* c, const OpFine5& op, const float2* x, float2* y, int nb, const int* mask) {
    LaunchScope scope(c, K_APPLY);
    // Node pairs when the rows and the fields start on 16 bytes, from 1.5 million nodes on: a pair's thread walks
    // its rows one after another, which a launch that does not fill the SMs has to wait for.  A call on one
    // GB300, a node and a pair per thread: 160 x 160 22.1 and 23.0 us, 512 x 256, 8 fields, 25.7 and 26.5,
    // 16 fields 29.5 and 28.0, 32 fields 36.8 and 31.1.
    if (op.nx % 2 == 0 && (((uintptr_t)x | (uintptr_t)y) & 15) == 0 && (size_t)op.nx * op.nz * nb >= (3u << 19)) {
        const int xt = (op.nx / 2 + TILE_X - 1) / TILE_X, rows = arnoldi_rows(xt, op.nz, nb);
        { apply_fine2_kernel<<<dim3(xt, (op.nz + TILE_Y * rows - 1) / (TILE_Y * rows), nb), dim3(TILE_X, TILE_Y), 0, c->stream>>>(
            op, x, y, rows, mask, tally(c, K_APPLY, 16ull * op.nx * op.nz)); count_launch(); }
        HELM_CK(cudaGetLastError());
        return HELM_OK;
    }
    { apply_fine_kernel<<<dim3((op.nx + 31) / 32, (op.nz + 7) / 8, nb), dim3(32, 8), 0, c->stream>>>(op, x, y, mask,
                                                                                               tally(c, K_APPLY, 16ull * op.nx * op.nz)); count_launch(); }
    HELM_CK(cudaGetLastError());
    return HELM_OK;
}

int launch_residual64(helm_ctx* c, const double2* x, const float2* b, float2* r, int nb, int conj_b, int first) {
    const OpFine5 op = fine_op(c, 0);
    // rows per thread as the Arnoldi kernels choose them: fewer on a small batch
    const int xt = (c->nx + TILE_X - 1) / TILE_X, pairs = (nb + 1) / 2, rows = arnoldi_rows(xt, c->nz, pairs);
    const dim3 grid(xt, (c->nz + TILE_Y * rows - 1) / (TILE_Y * rows), pairs);
    const double ax = 1.0 / ((double)c->hx * c->hx), az = 1.0 / ((double)c->hz * c->hz);
    const Tally tl = tally(c, K_RESIDUAL64, 32ull * c->nx * c->nz);
    LaunchScope scope(c, K_RESIDUAL64);
    if (first)
        { residual64_kernel<true><<<grid, dim3(TILE_X, TILE_Y), 0, c->stream>>>(op, x, b, r, conj_b, nb, rows, ax, az, c->outer, tl); count_launch(); }
    else
        { residual64_kernel<false><<<grid, dim3(TILE_X, TILE_Y), 0, c->stream>>>(op, x, b, r, conj_b, nb, rows, ax, az, c->outer, tl); count_launch(); }
    HELM_CK(cudaGetLastError());
    return HELM_OK;
}

int launch_conj64(helm_ctx* c, double2* x, int nb) {
    size_t n = (size_t)nb * npts(c);
    LaunchScope scope(c, K_MISC);
    { conj64_kernel<<<1184, 256, 0, c->stream>>>(x, n); count_launch(); }
    HELM_CK(cudaGetLastError());
    return HELM_OK;
}

int launch_outer_init(helm_ctx* c, int nb) {
    LaunchScope scope(c, K_MISC);
    { outer_init_kernel<<<(nb + 127) / 128, 128, 0, c->stream>>>(c->outer, c->fine, nb); count_launch(); }
    HELM_CK(cudaGetLastError());
    return HELM_OK;
}

int launch_zero_x(helm_ctx* c, double2* x, int nb) {
    LaunchScope scope(c, K_MISC);
    { zero_x_kernel<<<dim3(64, nb), 256, 0, c->stream>>>(c->outer, x, npts(c)); count_launch(); }
    HELM_CK(cudaGetLastError());
    return HELM_OK;
}

int launch_restart_check_dev(helm_ctx* c, int nb, double tol, int* n_active_dev) {
    LaunchScope scope(c, K_RESTART);
    { restart_check_kernel<<<(nb + 127) / 128, 128, 0, c->stream>>>(c->outer, c->fine, nb, tol, c->opt.max_iter, 0.7,
                                                                  n_active_dev); count_launch(); }
    HELM_CK(cudaGetLastError());
    return HELM_OK;
}

}  // namespace helm

// 3x3 convolution layers of the encoder-solver network (Fig. 1 caption,
// Sec. 3.4) as implicit GEMMs on the tensor cores, with the input staged once
// per tile by TMA and the nine taps read as shifted shared-memory views.
//
// Staging.  For every group of 16 input channels TMA copies the tile's input
// into shared memory as 8-channel planes stored pixel-major, 16 bytes per
// pixel: exactly the K-major, no-swizzle core-matrix layout (8 pixels x 16
// bytes per core matrix) that tcgen05.mma reads.  The A operand of a tap for a
// block of 128 output pixels is then a plane seen from a start address shifted
// by the tap's offset in pixels; no gather.  Pixels outside the image are
// zero-filled by TMA.  The weights of the group (9 taps x 16 channels x N)
// arrive in the same layout, by one contiguous copy (staged_weight).
//
// Sampling modes (output node -> input nodes of its taps):
//  0 same grid   (y, x)           -> (y + dy, x + dx); one (rows+2) x (tw+2) halo plane per 8 channels.
//  1 stride-2    (Y, X)           -> (2Y + 1 + dy, 2X + 1 + dx); the input is staged as four
//                                    parity sub-planes (even/odd rows x even/odd columns, TMA
//                                    element strides of 2), so that every tap is again a shift.
//  2 nearest x2  (2Y+py, 2X+px)   -> coarse ((2Y+py+dy) >> 1, (2X+px+dx) >> 1); the coarse halo
//                                    tile is staged as in mode 0 and each of the four output
//                                    parities (py, px) is its own set of M blocks.  Per parity
//                                    the nine taps read only 2 x 2 coarse nodes, so the kernel
//                                    takes the phase-merged weights (ConvArgs::wup, the taps
//                                    that read the same node added up): four MMAs per M block
//                                    and group instead of nine.
//  3 transpose of mode 1 (the input gradient of a stride-2 layer): fine (2Y+py, 2X+px) takes
//                                    tap (dy, dx) from coarse (Y + (py-1-dy)/2, X + (px-1-dx)/2)
//                                    when both are integers; staged as mode 2.
//  4 (opt-in, cnn_set_conv_path(2)) same grid as mode 0, for 16 output channels, with the three
//    column taps in N: one MMA per
//    tap row dy computes D[s][(dx, o)] for N = 48, and the epilogue adds
//    D[q][(-1, o)] + D[q + 1][(0, o)] + D[q + 2][(1, o)].  The A operand of an M block
//    takes its 16 core-matrix groups of 8 pixels at a 6-pixel stride (SBO = 96 B), so that
//    the two neighbours of the first six rows of a group are rows of the same group (same
//    warp: two shuffles).  Each staged pixel is read by 3 MMAs instead of 9; the rows 6
//    and 7 of each group are computed and dropped.  Accumulators live in a ring of
//    per-M-block TMEM slots, so that a tile's size is not bounded by TMEM.
//  5 (same grid as mode 0, same sums in the same order) an M block is one staged row (pitch
//    tw + 2 <= 128, lanes >= tw dropped) and the accumulators of a tile's output rows lie side
//    by side in TMEM, the last row first.  Staged row b adds to output rows b - 2, b - 1 and b
//    with tap rows 2, 1 and 0: adjacent columns, so that one MMA with N = 3 npad per column shift
//    serves all three (N = npad or 2 npad at the tile's ends).  A pixel is read by 3 MMAs instead
//    of 9, and an output row still sums (group, dy, dx) in mode 0's order, bit for bit.  One MMA
//    of zeros clears the tile's columns, since every other one adds to rows in progress.  Mode 0
//    at 32 -> 16 channels spends 76 % of the cycles on operand reads.  1024 x 512, 32 images, one GB300:
//    the 29 layers of a network pass 5.79 ms with mode 0 and 5.02 with mode 5 where rowsum_pays says so.
//  6 (16 or 32 output channels, same grid as mode 0) the three tap rows in N: an M block is
//    one staged row (pitch tw + 2 <= 128, lanes >= tw dropped) and per 16-channel group takes
//    three MMAs, one per column shift dx, computing D[b][x][(dy, o)] for N = 3 npad.  Output
//    row m sums D[m][x][(-1, o)] + D[m + 1][x][(0, o)] + D[m + 2][x][(1, o)]: the same TMEM
//    lane of three consecutive staged-row slots, no shuffles.  An MMA with M = 128, K = 16
//    costs about as much for N = 16 as for N = 64 on this GPU, so three N = 48 MMAs per
//    staged row replace nine N = 16 ones per output row.  Staged-row accumulators live in a
//    ring of TMEM slots (3 npad columns each); every group of a tile is resident.  Opt-in
//    (cnn_set_conv_path(3)): on the 1024x512 network's layers it measured 2.3x slower than
//    mode 0, which stays the default.
// Staged rows (tile + halo) are packed end to end into M blocks of 128 pixels;
// the accumulator rows of the halo columns between rows are discarded (each
// accumulator row depends only on its own A row).  Activations are in the
// chunked layout [n][C/8][H][W][8] (nc8), so every staged row is one
// contiguous TMA box row.
//
// Persistent warp-specialised CTAs (two per SM, or one when a tile needs more
// than 128 TMEM columns): warp 8 lane 0 streams (tile, channel group) stages
// through a ring by TMA; warp 9 walks the MMA loop together (warp-uniform
// descriptor arithmetic, a 32-bit add per MMA) and its lane 0 issues
// tcgen05.mma into one of two TMEM accumulator buffers; warps 0-7 drain the other buffer (bias, residual, ReLU,
// BF16 or FP32 store, or FP32 accumulation).  Every wait is bounded and gives
// up when another role aborts; on expiry the kernel raises the error flag,
// waits (bounded) for its copies and MMAs in flight, frees its TMEM and returns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <cstdio>
#include <map>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "helm_internal.cuh"
#include "conv.cuh"
#include "tc_ptx.cuh"

namespace helm {

namespace {

// Epilogue warps: two warpgroups drain TMEM (alternate M blocks; mode 6, alternate output
// rows).  + a TMA-producer warp and an MMA-issuer warp.
__host__ __device__ constexpr int epi_warps(int) { return 8; }
__host__ __device__ constexpr int threads_of(int mode) { return 32 * epi_warps(mode) + 64; }
constexpr int MAX_NS = 6;                       // stages (one 16-channel group of one tile each)
constexpr int MAX_SLOTS = 10;                   // TMEM slot barriers: mode 4 uses 4, mode 6 up to 10
constexpr int NSLOT4 = 4;                       // TMEM accumulator slots of mode 4 (two buffers otherwise)
constexpr int N3_PX = 96;                       // mode 4: staged pixels per M block (16 groups x 6)
constexpr size_t RING_BUDGET_RT16 = 100 * 1024;  // mode 6, 16 channels: two CTAs per SM (256 TMEM columns each)
constexpr size_t RING_BUDGET_RT32 = 200 * 1024;  // mode 6, 32 channels: one CTA per SM (512 TMEM columns)
constexpr int ROWS_RT_MAX = 32;                 // mode 6: output rows per tile at most
constexpr int RT_CHUNK = 4;                     // mode 6: staged rows per commit at most (a commit
                                                // costs about as much as several MMAs)
constexpr int ZERO_BYTES = 256 * 32;            // mode 5: zero operands of the clearing MMA
constexpr long long WAIT_LIMIT = 1ll << 22;     // polls of try_wait before a wait gives up
// No padding after a plane: the last M block of a packed tile may read up to
// 2 pitches + 130 pixels past its plane's staged pixels, which lands in the next
// plane or in the stage's weights (>= 288 pixels' worth), inside the stage.
constexpr int SLACK_PX = 0;
constexpr size_t STAGE_BUDGET = 47 * 1024;      // default bytes of one stage at most (fewer rows otherwise)
constexpr size_t RING_BUDGET = 96 * 1024;       // default bytes of the stage ring (two CTAs fit an SM)
// Stride-2 layers stage four parity sub-planes per channel chunk; within 47 KB a
// tile would hold a single output row (twice the input rows it needs, and the
// weights once per row), so they take one CTA per SM with larger stages.
constexpr size_t STAGE_BUDGET_S2 = 100 * 1024;
constexpr size_t RING_BUDGET_S2 = 200 * 1024;

struct Geometry {
    int tw, rows, pw;        // tile on the staged grid (output grid in mode 1); staged row pitch
    int mb;                  // 128-pixel M blocks per output parity
    int nph;                 // output parities per tile: 1 (modes 0, 1) or 4 (modes 2, 3)
    int tiles_x, tiles_y, tiles;
    int plane;               // bytes of one staged 8-channel plane (its two halves are this far apart)
    int pstride;             // bytes between parity sub-planes (two planes, rounded up to 128 B)
    int nplanes;             // parity sub-planes: 1, or 4 in mode 1
    int wbytes;              // bytes of one group's weights (9 taps x 2 chunks x npad rows x 16 B)
    int nslot, slot_cols;    // modes 4 and 6: TMEM slots (an M block / a staged row each) and their columns
    int nbuf;                // modes 0-3: TMEM accumulator buffers (2: the epilogue drains one while
                             // the MMAs fill the other; 1: twice the M blocks per tile)
    int nzero;               // mode 5: columns that the clearing MMA writes (rows * npad)
    int nwg;                 // mode 6: epilogue warpgroups that take output rows
    int chunk;               // mode 6: staged rows per commit
    int psplit;              // mode 2: a tile computes one output row parity py (nph = 2: px), the
                             // tiles of the two parities alternate; 0: all four parities per tile
    int stage;               // bytes of one stage
    int groups, groups0;     // 16-channel groups in total / taken from x0
    int ns;                  // stages in the ring
    uint32_t tx;             // bytes TMA delivers per stage
    uint32_t acc_cols;       // TMEM columns of one accumulator buffer (nph * mb * npad)
    uint32_t tmem_cols;      // allocated: two accumulator buffers, power of two
};

// Bounded wait that also gives up once another role has raised the abort flag.
// A thread that polls without useful work in between backs off for sleep_ns per
// failed poll, so that its instructions do not take issue slots from the warps
// that work (at most WAIT_LIMIT polls: under a second at 128 ns).
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, volatile int* abort_v,
                                         unsigned sleep_ns = 0) {
    long long it = 0;
    while (!tc::mbar_try_wait(bar, parity)) {
        ++it;
        if (it > WAIT_LIMIT) return false;
        if ((it & 255) == 0 && *abort_v) return false;
        if (sleep_ns) __nanosleep(sleep_ns);
    }
    return true;
}

// What the epilogue reads of one pixel's 16-channel segment, loaded ahead of its use.
struct Pre2 {
    uint4 a, b;
};

// The two halves of a packed BF16 pair, exactly.
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// (x, y) += (bx, by), two FP32 additions in one instruction.
__device__ __forceinline__ void add2(float& x, float& y, float bx, float by) {
    asm("{ .reg .b64 p, q;\n mov.b64 p, {%0, %1};\n mov.b64 q, {%2, %3};\n add.rn.f32x2 p, p, q;\n"
        " mov.b64 {%0, %1}, p; }"
        : "+f"(x), "+f"(y)
        : "f"(bx), "f"(by));
}

// Tap t = (dy + 1) * 3 + (dx + 1) of output parity (py, px): whether it
// contributes, and its A operand as (plane, offset in pixels from the tile's
// staged pixel q).
template <int MODE>
__device__ __forceinline__ bool tap_source(int t, int py, int px, int pw, int* plane, int* off) {
    const int dy = t / 3 - 1, dx = t % 3 - 1;
    if (MODE == 0) {
        *plane = 0;
        *off = (dy + 1) * pw + (dx + 1);
        return true;
    } else if (MODE == 1) {
        // row 2Y+1+dy: odd sub-plane row Y (dy = 0), even rows Y (dy = -1) or Y + 1 (dy = +1)
        *plane = (dy == 0 ? 2 : 0) + (dx == 0 ? 1 : 0);
        *off = (dy == 1 ? pw : 0) + (dx == 1 ? 1 : 0);
        return true;
    } else if (MODE == 2) {
        // merged tap t = 2 ey + ex of parity (py, px): coarse node (Y + py - 1 + ey, X + px - 1 + ex)
        (void)dy;
        (void)dx;
        *plane = 0;
        *off = (py + (t >> 1)) * pw + (px + (t & 1));
        return true;
    } else {
        const int uy = py - 1 - dy, ux = px - 1 - dx;
        if ((uy & 1) || (ux & 1)) return false;
        *plane = 0;
        *off = ((uy >> 1) + 1) * pw + ((ux >> 1) + 1);
        return true;
    }
}

template <int MODE, bool ACT>
__global__ void __launch_bounds__(threads_of(MODE), 2) conv3x3_tma_kernel(const __grid_constant__ CUtensorMap tm_x0,
                                                         const __grid_constant__ CUtensorMap tm_x1,
                                                         const __grid_constant__ CUtensorMap tm_w, ConvArgs a,
                                                         Geometry g) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ uint64_t full[MAX_NS], empty[MAX_NS], tfull[MAX_SLOTS], tempty[MAX_SLOTS], done;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag;
    __shared__ float bias_s[128];
    // mode 5: both operands of the clearing MMA (A 128 rows, B up to 256 rows of 16 zeros)
    __shared__ __align__(128) unsigned char zeros[MODE == 5 ? ZERO_BYTES : 16];

    constexpr int EPI_WARPS = epi_warps(MODE);
    constexpr int EPI = 32 * EPI_WARPS;             // epilogue threads
    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid < a.npad) bias_s[tid] = a.accum || !a.bias ? 0.0f : __ldg(a.bias + tid);
    if constexpr (MODE == 5) {
        for (int i = tid * 16; i < ZERO_BYTES; i += (int)blockDim.x * 16)
            *reinterpret_cast<uint4*>(zeros + i) = make_uint4(0u, 0u, 0u, 0u);
        tc::fence_proxy_async_smem();   // the MMAs read them through the async proxy
    }
    if (warp == 0) {
        tc::tmem_alloc(&tmem_base, g.tmem_cols);
        tc::tmem_relinquish();
    }
    if (tid == 0) {
        for (int s = 0; s < MAX_NS; ++s) {
            tc::mbar_init(&full[s], 1);     // the producer's expect_tx arrival + the TMA bytes
            tc::mbar_init(&empty[s], 1);    // one tcgen05.commit per use
        }
        for (int i = 0; i < MAX_SLOTS; ++i) {
            tc::mbar_init(&tfull[i], 1);    // tcgen05.commit after the last MMA of a tile (mode 4: M block)
            // every epilogue thread after its TMEM loads (mode 4: the warpgroup that drains the
            // slot; mode 6: the warpgroups of the three output rows that read the slot)
            tc::mbar_init(&tempty[i], MODE == 4 ? EPI / 2 : (MODE == 6 ? 3 * 128 : EPI));
        }
        tc::mbar_init(&done, 1);
        tc::fence_mbar_init();
        abort_flag = 0;
    }
    tc::tc_fence_before_sync();
    __syncthreads();
    tc::tc_fence_after_sync();
    const uint32_t tmem = tmem_base;
    volatile int* abort_v = &abort_flag;
    const int G = g.groups;
    const int ntiles = g.tiles > (int)blockIdx.x ? (g.tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int chunk_bytes = g.plane;                 // K-adjacent core matrices (LBO)
    const int wofs = g.nplanes * g.pstride;          // the group's weights within a stage

    // the output row parity of tile k when the parities are split (0 otherwise)
    auto tile_py = [&](int k) { return g.psplit ? (((int)blockIdx.x + k * (int)gridDim.x) & 1) : 0; };
    auto tile_coords = [&](int k, int& b, int& xs, int& ys) {
        int t = (int)blockIdx.x + k * (int)gridDim.x;
        if (g.psplit) t >>= 1;
        const int tx = t % g.tiles_x;
        t /= g.tiles_x;
        const int ty = t % g.tiles_y;
        b = t / g.tiles_y;
        xs = tx * g.tw;
        ys = ty * g.rows;
    };

    if (tid == EPI) {
        // ---------------- TMA producer ----------------
        long long j = 0;
        int s = 0, wraps = 0;   // j % ns and j / ns as counters
        bool ok = true;
        for (int k = 0; k < ntiles && ok; ++k) {
            int b, xs, ys;
            tile_coords(k, b, xs, ys);
            const int b1 = a.c1 ? (a.x1_map ? __ldg(a.x1_map + b) : (a.x1_bcast ? 0 : b)) : 0;
            for (int gi = 0; gi < G; ++gi, ++j) {
                if (gi > 0 || k > 0)
                    if (++s == g.ns) {
                        s = 0;
                        ++wraps;
                    }
                if (wraps > 0 && !wait_bar(&empty[s], (uint32_t)((wraps - 1) & 1), abort_v, 32)) { ok = false; break; }
                unsigned char* st = smem + (size_t)s * g.stage;
                tc::mbar_arrive_expect_tx(&full[s], g.tx);
                {
                    // both 8-channel halves of the group in one box (a group never straddles x0 and x1)
                    const int c = gi * 16;
                    const bool second = gi >= g.groups0;
                    const CUtensorMap* tm = second ? &tm_x1 : &tm_x0;
                    const int cc = second ? c - a.c0 : c;
                    const int bb = second ? b1 : b;
                    if (MODE == 1) {
                        // parity sub-planes: rows 2ys + rp + 2i, columns 2xs + cp + 2j
                        for (int rp = 0; rp < 2; ++rp)
                            for (int cp = 0; cp < 2; ++cp)
                                tc::tma_load_5d(st + (rp * 2 + cp) * g.pstride, tm, 0, 2 * xs + cp, 2 * ys + rp,
                                                cc >> 3, bb, &full[s]);
                    } else {
                        // 8-byte elements, two per pixel, the row (with halo) contiguous
                        tc::tma_load_4d(st, tm, 2 * (xs - 1), ys - 1, cc >> 3, bb, &full[s]);
                    }
                }
                unsigned char* ws = st + wofs;
                if (MODE == 4) {
                    // [dy][half][dx][npad][8]: the B operand of tap row dy is 3 npad rows (dx, o)
                    tc::tma_load_5d(ws, &tm_w, 0, 0, 0, 2 * gi, 0, &full[s]);
                } else if (MODE == 2) {
                    // the merged taps of all parities, or of the tile's row parity
                    const size_t gb = (size_t)512 * a.npad;   // bytes of a group: 16 taps x 16 channels
                    tc::bulk_load(ws, reinterpret_cast<const unsigned char*>(a.wup) + gi * gb + tile_py(k) * (gb / 2),
                                  (uint32_t)g.wbytes, &full[s]);
                } else {
                    // [dx][half][dy][npad][8]
                    tc::bulk_load(ws, reinterpret_cast<const unsigned char*>(a.wst) + (size_t)gi * g.wbytes,
                                  (uint32_t)g.wbytes, &full[s]);
                }
            }
        }
        if (!ok) {
            *abort_v = 1;
            // the copies of the last issued stages land before the CTA exits (bounded)
            for (long long jj = j - 1; jj >= 0 && jj >= j - g.ns; --jj) {
                long long it = 0;
                while (!tc::mbar_try_wait(&full[jj % g.ns], (uint32_t)((jj / g.ns) & 1)) && ++it < WAIT_LIMIT) {
                }
            }
        }
    } else if (warp == EPI_WARPS + 1) {
        // ---------------- MMA issuer ----------------
        // The whole warp walks the loop, so that the descriptor arithmetic is warp-uniform,
        // and lane 0 issues: one tcgen05.mma per (parity, M block, tap) with a 32-bit add
        // for its A start address; the B descriptors of the nine taps are set per stage.
        const bool leader = (tid & 31) == 0;
        const uint32_t idesc = tc::idesc_bf16_f32(128, a.npad);
        const uint32_t wplane = (uint32_t)a.npad * 16;
        // descriptors with a zero start address: the start (bits 0-13, 16-byte units) is added per MMA
        const uint64_t adesc0 = tc::smem_desc(0u, (uint32_t)chunk_bytes, 128);
        // (K halves of B: a merged tap's are npad rows apart, the others' 3 npad, see staged_weight)
        const uint64_t bdesc0 = tc::smem_desc(0u, MODE == 2 ? wplane : 3u * wplane, 128);
        const uint32_t a_lo0 = (uint32_t)adesc0, a_hi = (uint32_t)(adesc0 >> 32);
        const uint32_t b_lo0 = (uint32_t)bdesc0, b_hi = (uint32_t)(bdesc0 >> 32);
        long long j = 0;
        bool ok = true;
        if constexpr (MODE == 4) {
            // m outer: an M block takes every group of its tile (all G stages resident) and
            // three MMAs per group (tap rows dy), then commits its TMEM slot
            const uint32_t idesc4 = tc::idesc_bf16_f32(128, 3 * a.npad);
            const uint64_t adesc4 = tc::smem_desc(0u, (uint32_t)chunk_bytes, 16 * 6);   // 6-pixel group stride
            const uint64_t bdesc4 = tc::smem_desc(0u, 3u * wplane, 128);
            const uint32_t a4_lo = (uint32_t)adesc4, a4_hi = (uint32_t)(adesc4 >> 32);
            const uint32_t b4_lo = (uint32_t)bdesc4, b4_hi = (uint32_t)(bdesc4 >> 32);
            const uint32_t row_b16 = (6u * wplane) >> 4;   // B of one tap row (2 halves x 3 dx)
            int slot = 0, wraps = 0;                         // counters, no divisions per M block
            uint32_t a16s[MAX_NS];
            for (int k = 0; k < ntiles && ok; ++k) {
                for (int gi = 0; gi < G; ++gi) {
                    const long long js = j + gi;
                    const int s = (int)(js % g.ns);
                    const bool f_ok = wait_bar(&full[s], (uint32_t)((js / g.ns) & 1), abort_v, 32);
                    if (!__all_sync(0xffffffffu, f_ok)) { ok = false; break; }
                    a16s[gi] = (tc::smem_u32(smem + (size_t)s * g.stage) & 0x3FFFFu) >> 4;
                }
                if (!ok) break;
                tc::tc_fence_after_sync();
                for (int m = 0; m < g.mb; ++m) {
                    const bool t_ok = wraps == 0 || wait_bar(&tempty[slot], (uint32_t)((wraps - 1) & 1), abort_v, 32);
                    if (!__all_sync(0xffffffffu, t_ok)) { ok = false; break; }
                    tc::tc_fence_after_sync();
                    const uint32_t d = tmem + (uint32_t)(slot * g.slot_cols);
                    for (int gi = 0; gi < G; ++gi) {
                        const uint32_t a16 = a16s[gi];
                        const uint32_t a_m = a4_lo + a16 + (uint32_t)(m * N3_PX);
                        const uint32_t b_s = b4_lo + a16 + ((uint32_t)wofs >> 4);
#pragma unroll
                        for (int dy = 0; dy < 3; ++dy) {
                            if (leader) {
                                const uint64_t ad = ((uint64_t)a4_hi << 32) | (a_m + (uint32_t)(dy * g.pw));
                                const uint64_t bd = ((uint64_t)b4_hi << 32) | (b_s + (uint32_t)dy * row_b16);
                                tc::mma_bf16(d, ad, bd, idesc4, (gi | dy) ? 1u : 0u);
                            }
                        }
                    }
                    __syncwarp();
                    if (leader) tc::mma_commit(&tfull[slot]);
                    if (++slot == g.nslot) {
                        slot = 0;
                        ++wraps;
                    }
                }
                if (!ok) break;
                __syncwarp();
                if (leader)
                    for (int gi = 0; gi < G; ++gi) tc::mma_commit(&empty[(j + gi) % g.ns]);
                j += G;
            }
        } else if constexpr (MODE == 6) {
            // staged row b of every tile (global index jb) into TMEM slot jb % nslot: for each
            // group and column shift dx one MMA with N = 3 npad (B rows (dy, o)).  Rows are
            // committed in chunks of g.chunk (and at the tile's last row): commit id
            // k * ceil(mb / chunk) + b / chunk on tfull[id % MAX_SLOTS].  A slot is
            // refilled once the epilogue released it.  Slot, use and commit indices advance
            // as counters: a 64-bit division per row cost more than the row's MMAs.
            const uint32_t ncol = (uint32_t)g.slot_cols;
            const uint32_t idesc6 = tc::idesc_bf16_f32(128, 3 * a.npad);
            const uint64_t bdesc6 = tc::smem_desc(0u, 3u * wplane, 128);   // K halves 3 npad rows apart
            const uint32_t b6_lo = (uint32_t)bdesc6, b6_hi = (uint32_t)(bdesc6 >> 32);
            const uint32_t dx_b16 = (6u * wplane) >> 4;                    // B of one column shift
            int slot = 0, wraps = 0, cslot = 0;
            uint32_t a16s[MAX_NS];
            for (int k = 0; k < ntiles && ok; ++k) {
                for (int gi = 0; gi < G; ++gi) {
                    const long long js = j + gi;
                    const int s = (int)(js % g.ns);
                    const bool f_ok = wait_bar(&full[s], (uint32_t)((js / g.ns) & 1), abort_v, 32);
                    if (!__all_sync(0xffffffffu, f_ok)) { ok = false; break; }
                    a16s[gi] = (tc::smem_u32(smem + (size_t)s * g.stage) & 0x3FFFFu) >> 4;
                }
                if (!ok) break;
                tc::tc_fence_after_sync();
                int cb = 0;
                for (int b = 0; b < g.mb; ++b) {
                    const bool t_ok = wraps == 0 || wait_bar(&tempty[slot], (uint32_t)((wraps - 1) & 1), abort_v, 32);
                    if (!__all_sync(0xffffffffu, t_ok)) { ok = false; break; }
                    tc::tc_fence_after_sync();
                    const uint32_t d = tmem + (uint32_t)slot * ncol;
                    for (int gi = 0; gi < G; ++gi) {
                        const uint32_t a_b = a_lo0 + a16s[gi] + (uint32_t)(b * g.pw);
                        const uint32_t b_s = b6_lo + a16s[gi] + ((uint32_t)wofs >> 4);
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx) {
                            if (leader) {
                                const uint64_t ad = ((uint64_t)a_hi << 32) | (a_b + (uint32_t)dx);
                                const uint64_t bd = ((uint64_t)b6_hi << 32) | (b_s + (uint32_t)dx * dx_b16);
                                tc::mma_bf16(d, ad, bd, idesc6, (gi | dx) ? 1u : 0u);
                            }
                        }
                    }
                    if (++slot == g.nslot) {
                        slot = 0;
                        ++wraps;
                    }
                    if (++cb == g.chunk || b == g.mb - 1) {
                        __syncwarp();
                        if (leader) tc::mma_commit(&tfull[cslot]);
                        cb = 0;
                        if (++cslot == MAX_SLOTS) cslot = 0;
                    }
                }
                if (!ok) break;
                __syncwarp();
                if (leader)
                    for (int gi = 0; gi < G; ++gi) tc::mma_commit(&empty[(j + gi) % g.ns]);
                j += G;
            }
        } else if constexpr (MODE == 5) {
            // output row r of the tile accumulates in columns (rows - 1 - r) npad of the buffer;
            // staged row b and column shift dx: rows r = b - t for the tap rows t that exist
            const uint64_t bdesc5 = tc::smem_desc(0u, 3u * wplane, 128);   // K halves 3 npad rows apart
            const uint32_t b5_lo = (uint32_t)bdesc5, b5_hi = (uint32_t)(bdesc5 >> 32);
            const uint32_t dx_b16 = (6u * wplane) >> 4;                    // B of one column shift
            const uint32_t id1 = tc::idesc_bf16_f32(128, a.npad), id2 = tc::idesc_bf16_f32(128, 2 * a.npad),
                           id3 = tc::idesc_bf16_f32(128, 3 * a.npad), idz = tc::idesc_bf16_f32(128, g.nzero);
            const uint64_t az = tc::smem_desc(tc::smem_u32(zeros), 128 * 16, 128);
            const uint64_t bz = tc::smem_desc(tc::smem_u32(zeros), (uint32_t)g.nzero * 16, 128);
            const int R = g.rows;
            int s = 0, wraps = 0;   // j % ns and j / ns as counters
            for (int k = 0; k < ntiles && ok; ++k) {
                const int acc = g.nbuf == 2 ? (k & 1) : 0;
                const int ause = g.nbuf == 2 ? (k >> 1) : k;
                const bool t_ok = ause == 0 || wait_bar(&tempty[acc], (uint32_t)((ause - 1) & 1), abort_v, 32);
                if (!__all_sync(0xffffffffu, t_ok)) { ok = false; break; }
                tc::tc_fence_after_sync();
                const uint32_t dbase = tmem + (uint32_t)acc * g.acc_cols;
                if (leader) tc::mma_bf16(dbase, az, bz, idz, 0u);
                for (int gi = 0; gi < G; ++gi, ++j) {
                    if (gi > 0 || k > 0)
                        if (++s == g.ns) {
                            s = 0;
                            ++wraps;
                        }
                    const bool f_ok = wait_bar(&full[s], (uint32_t)(wraps & 1), abort_v, 32);
                    if (!__all_sync(0xffffffffu, f_ok)) { ok = false; break; }
                    tc::tc_fence_after_sync();
                    const uint32_t a16 = (tc::smem_u32(smem + (size_t)s * g.stage) & 0x3FFFFu) >> 4;
                    const uint32_t b_s = b5_lo + a16 + ((uint32_t)wofs >> 4);
                    uint32_t a_b = a_lo0 + a16;
                    for (int b = 0; b < R + 2; ++b, a_b += (uint32_t)g.pw) {
                        const int t0 = b < R ? 0 : b - R + 1;          // first and last tap row in use
                        const int t1 = b < 2 ? b : 2;
                        const uint32_t d = dbase + (uint32_t)((R - 1 - b + t0) * a.npad);
                        const uint32_t b_t = b_s + (uint32_t)(t0 * a.npad);   // 16 bytes per row of B
                        const uint32_t id = t1 - t0 == 2 ? id3 : (t1 - t0 == 1 ? id2 : id1);
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx) {
                            if (leader) {
                                const uint64_t ad = ((uint64_t)a_hi << 32) | (a_b + (uint32_t)dx);
                                const uint64_t bd = ((uint64_t)b5_hi << 32) | (b_t + (uint32_t)dx * dx_b16);
                                tc::mma_bf16(d, ad, bd, id, 1u);
                            }
                        }
                    }
                    __syncwarp();
                    if (leader) tc::mma_commit(&empty[s]);
                }
                __syncwarp();
                if (ok && leader) tc::mma_commit(&tfull[acc]);
            }
        } else {
            int s = 0, wraps = 0;   // j % ns and j / ns as counters
            for (int k = 0; k < ntiles && ok; ++k) {
                const int acc = g.nbuf == 2 ? (k & 1) : 0;
                const int ause = g.nbuf == 2 ? (k >> 1) : k;
                // (the lanes agree on every wait's outcome, so that they leave the loop together)
                const bool t_ok = ause == 0 || wait_bar(&tempty[acc], (uint32_t)((ause - 1) & 1), abort_v, 32);
                if (!__all_sync(0xffffffffu, t_ok)) { ok = false; break; }
                tc::tc_fence_after_sync();
                const uint32_t dbase = tmem + (uint32_t)acc * g.acc_cols;
                for (int gi = 0; gi < G; ++gi, ++j) {
                    if (gi > 0 || k > 0)
                        if (++s == g.ns) {
                            s = 0;
                            ++wraps;
                        }
                    const bool f_ok = wait_bar(&full[s], (uint32_t)(wraps & 1), abort_v, 32);
                    if (!__all_sync(0xffffffffu, f_ok)) { ok = false; break; }
                    tc::tc_fence_after_sync();
                    const uint32_t a16 = (tc::smem_u32(smem + (size_t)s * g.stage) & 0x3FFFFu) >> 4;
                    const uint32_t bw_lo = b_lo0 + a16 + ((uint32_t)wofs >> 4);
                    for (int ph = 0; ph < g.nph; ++ph) {
                        constexpr int NT = MODE == 2 ? 4 : 9;   // mode 2: the parity's merged taps
                        uint32_t ao[NT];   // A start of each tap for M block 0, descriptor low word
                        bool use[NT];
                        const int py = g.psplit ? tile_py(k) : ph >> 1, px = g.psplit ? ph : ph & 1;
#pragma unroll
                        for (int tap = 0; tap < NT; ++tap) {
                            int pl, off;   // A offset in 16-byte units from the stage
                            use[tap] = tap_source<MODE>(tap, py, px, g.pw, &pl, &off);
                            ao[tap] = a_lo0 + a16 + (uint32_t)(pl * (g.pstride >> 4) + off);
                        }
                        // B of the parity's first tap (mode 2: the merged weights are [parity][4 taps])
                        const uint32_t bph = MODE == 2 ? bw_lo + (uint32_t)(ph * 8 * a.npad) : bw_lo;
                        uint32_t d = dbase + (uint32_t)(ph * g.mb * a.npad);
                        for (int m = 0; m < g.mb; ++m, d += (uint32_t)a.npad) {
                            const uint32_t mo = (uint32_t)(m * 128);   // 128 pixels of 16 bytes
                            uint32_t accum = gi == 0 ? 0u : 1u;
#pragma unroll
                            for (int tap = 0; tap < NT; ++tap) {
                                if (!use[tap]) continue;
                                if (leader) {
                                    const uint64_t ad = ((uint64_t)a_hi << 32) | (ao[tap] + mo);
                                    const uint64_t bd = ((uint64_t)b_hi << 32) |
                                                        (bph + (uint32_t)((MODE == 2 ? 2 * tap : tap % 3 * 6 + tap / 3) * a.npad));
                                    tc::mma_bf16(d, ad, bd, idesc, accum);
                                }
                                accum = 1u;
                            }
                        }
                    }
                    __syncwarp();
                    if (leader) tc::mma_commit(&empty[s]);
                }
                __syncwarp();
                if (ok && leader) tc::mma_commit(&tfull[acc]);
            }
        }
        if (!ok) *abort_v = 1;
        __syncwarp();
        if (leader) {
            tc::mma_commit(&done);   // every MMA issued so far completes before `done`
            long long it = 0;
            while (!tc::mbar_try_wait(&done, 0u) && ++it < WAIT_LIMIT) {
            }
        }
        __syncwarp();
    } else if (warp < EPI_WARPS) {
        // ---------------- epilogue ----------------
        // warp w reads TMEM lanes 32 (w % 4) .. + 31 (accumulator row = M-block row);
        // warpgroup w / 4 drains every other M block (all npad columns of it)
        const int row = (warp & 3) * 32 + (tid & 31);
        const int wg = warp >> 2;
        const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const long long hw_out = (long long)a.hout * a.wout;
        const size_t plane_out = (size_t)hw_out * 8;   // elements between 8-channel planes
        const int nblk = g.nph * g.mb;
        // The epilogue's instructions bound the layers of 16 channels: some 260 per 32 pixels when each
        // value was rounded and packed by itself.  Pairs now: two additions, one conversion, one ReLU an
        // instruction.  1024 x 512, 32 images, one GB300, 29 layers of a network pass: 7.17 -> 6.93 ms, before the weights' contiguous copy.
        //
        // The operand that the epilogue reads besides the accumulators: the residual, or the activation
        // whose mask is applied.  It is loaded before the accumulators are waited for.
        const __nv_bfloat16* pre_src = ACT || a.res ? a.res : a.gmask;
        auto preload = [&](size_t ob, int n0, bool valid) {
            Pre2 r{make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
            if (pre_src && valid) {
                const __nv_bfloat16* q = pre_src + ob + (size_t)(n0 >> 3) * plane_out;
                r.a = __ldg(reinterpret_cast<const uint4*>(q));
                r.b = __ldg(reinterpret_cast<const uint4*>(q + plane_out));
            }
            return r;
        };
        // one 16-channel segment of pixel p = (image, pixel of it): bias, residual, ReLU, store
        auto segment = [&](float* vv, int n0, size_t ob, long long p, const Pre2& pre) {
#pragma unroll
            for (int i = 0; i < 16; i += 4) {
                const float4 bb = *reinterpret_cast<const float4*>(bias_s + n0 + i);
                add2(vv[i], vv[i + 1], bb.x, bb.y);
                add2(vv[i + 2], vv[i + 3], bb.z, bb.w);
            }
            const size_t o0 = ob + (size_t)(n0 >> 3) * plane_out;   // planes n0/8 and n0/8 + 1
            const uint32_t pw8[8] = {pre.a.x, pre.a.y, pre.a.z, pre.a.w, pre.b.x, pre.b.y, pre.b.z, pre.b.w};
            if (a.res) {
#pragma unroll
                for (int i = 0; i < 8; ++i) add2(vv[2 * i], vv[2 * i + 1], bf_lo(pw8[i]), bf_hi(pw8[i]));
            }
            const bool packed = ACT || (!a.gmask && !a.out_fp32);
            if (a.relu && !packed) {
#pragma unroll
                for (int i = 0; i < 16; ++i) vv[i] = fmaxf(vv[i], 0.0f);
            }
            if (!ACT && a.gmask) {
                // the gradient of an activation: what is there already, the ReLU mask, the skip's FP32 copy
                if (a.gprior) {
                    const float4* q4 = reinterpret_cast<const float4*>(a.gprior + (size_t)p * a.npad + n0);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 t = __ldg(q4 + q);
                        add2(vv[4 * q], vv[4 * q + 1], t.x, t.y);
                        add2(vv[4 * q + 2], vv[4 * q + 3], t.z, t.w);
                    }
                }
                uint32_t mw[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) mw[i] = pw8[i];
                if (a.res) {
                    *reinterpret_cast<uint4*>(mw) = __ldg(reinterpret_cast<const uint4*>(a.gmask + o0));
                    *reinterpret_cast<uint4*>(mw + 4) = __ldg(reinterpret_cast<const uint4*>(a.gmask + o0 + plane_out));
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (!(bf_lo(mw[i]) > 0.0f)) vv[2 * i] = 0.0f;
                    if (!(bf_hi(mw[i]) > 0.0f)) vv[2 * i + 1] = 0.0f;
                }
                if (a.gres) {
                    float4* r4 = reinterpret_cast<float4*>(a.gres + (size_t)p * a.npad + n0);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float4 t = a.gres_accum ? r4[q] : make_float4(0.f, 0.f, 0.f, 0.f);
                        t.x += vv[4 * q];
                        t.y += vv[4 * q + 1];
                        t.z += vv[4 * q + 2];
                        t.w += vv[4 * q + 3];
                        r4[q] = t;
                    }
                }
            }
            if (!ACT && a.out_fp32) {
                float* yo = reinterpret_cast<float*>(a.y) + (size_t)p * a.cstore;
                if ((a.cstore & 15) == 0) {
                    // whole 16-channel segments, 64-byte aligned: four 16-byte accesses
                    float4* y4 = reinterpret_cast<float4*>(yo + n0);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float4 t = a.accum ? y4[q] : make_float4(0.f, 0.f, 0.f, 0.f);
                        t.x += vv[4 * q];
                        t.y += vv[4 * q + 1];
                        t.z += vv[4 * q + 2];
                        t.w += vv[4 * q + 3];
                        y4[q] = t;
                    }
                } else if (a.accum) {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (n0 + i < a.cstore) yo[n0 + i] += vv[i];
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (n0 + i < a.cstore) yo[n0 + i] = vv[i];
                }
            } else {
                uint32_t w[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    __nv_bfloat162 h = __floats2bfloat162_rn(vv[2 * i], vv[2 * i + 1]);
                    // (rounding keeps the sign, so that ReLU may follow it)
                    if (a.relu && packed) h = __hmax2(h, __nv_bfloat162(__nv_bfloat16_raw{0}, __nv_bfloat16_raw{0}));
                    w[i] = *reinterpret_cast<const uint32_t*>(&h);
                }
                __nv_bfloat16* yq = reinterpret_cast<__nv_bfloat16*>(a.y) + o0;
                *reinterpret_cast<uint4*>(yq) = make_uint4(w[0], w[1], w[2], w[3]);
                *reinterpret_cast<uint4*>(yq + plane_out) = make_uint4(w[4], w[5], w[6], w[7]);
            }
        };
        if constexpr (MODE == 6) {
            // Output row m of a tile (warpgroup m % nwg) sums three staged-row slots in this
            // thread's lane (= column), all channels.  The commit that covers the newest of
            // the three rows implies the older two.  Every slot takes 3 x 128 arrivals per
            // fill: one from each output row that reads it, and for the tile's first and
            // last two staged rows (read by fewer rows) the extra arrivals come from the
            // tile's first and last output rows.  Indices are kept as 32-bit counters.
            const int nwg = g.nwg;
            const uint32_t ncol = (uint32_t)g.slot_cols;
            const int cpt = (g.mb + g.chunk - 1) / g.chunk;   // commits per tile
            int jslot = 0;                                    // slot of the tile's staged row 0
            bool ok = true;
            for (int k = 0; k < ntiles && ok; ++k) {
                int b, xs, ys;
                tile_coords(k, b, xs, ys);
                const size_t img_base = (size_t)b * (size_t)(a.npad >> 3) * (size_t)hw_out * 8;
                const int R = g.rows;
                for (int m = wg < nwg ? wg : R; m < R; m += nwg) {
                    const int cid = k * cpt + (m + 2) / g.chunk;
                    if (!wait_bar(&tfull[cid % MAX_SLOTS], (uint32_t)((cid / MAX_SLOTS) & 1), abort_v, 64)) {
                        *abort_v = 1;
                        ok = false;
                        break;
                    }
                    tc::tc_fence_after_sync();
                    int s0 = jslot + m;
                    while (s0 >= g.nslot) s0 -= g.nslot;
                    const int s1 = s0 + 1 == g.nslot ? 0 : s0 + 1;
                    const int s2 = s1 + 1 == g.nslot ? 0 : s1 + 1;
                    const int ox = xs + row, oy = ys + m;
                    const bool valid = row < g.tw && ox < a.wout && oy < a.hout;
                    const long long pix = (long long)oy * a.wout + ox;
                    const size_t ob = img_base + (size_t)pix * 8;
                    const long long p = (long long)b * hw_out + pix;
                    for (int c0 = 0; c0 < a.npad; c0 += 16) {
                        float v0[16], v1[16], v2[16];
                        tc::tmem_ld16x3(lane_base + (uint32_t)s0 * ncol + (uint32_t)c0,
                                        lane_base + (uint32_t)s1 * ncol + (uint32_t)(a.npad + c0),
                                        lane_base + (uint32_t)s2 * ncol + (uint32_t)(2 * a.npad + c0), v0, v1, v2);
                        if (c0 + 16 >= a.npad) {
                            // this thread's reads of the three slots are complete
                            tc::tc_fence_before_sync();
                            tc::mbar_arrive(&tempty[s0]);
                            tc::mbar_arrive(&tempty[s1]);
                            tc::mbar_arrive(&tempty[s2]);
                            if (m == 0) {
                                tc::mbar_arrive(&tempty[s0]);
                                tc::mbar_arrive(&tempty[s0]);
                                tc::mbar_arrive(&tempty[s1]);
                            }
                            if (m == R - 1) {
                                tc::mbar_arrive(&tempty[s1]);
                                tc::mbar_arrive(&tempty[s2]);
                                tc::mbar_arrive(&tempty[s2]);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 16; ++i) v0[i] += v1[i] + v2[i];
                        if (valid) segment(v0, c0, ob, p, preload(ob, c0, true));
                    }
                }
                jslot += g.mb;
                while (jslot >= g.nslot) jslot -= g.nslot;
            }
        } else if constexpr (MODE == 4) {
            // warpgroup wg drains the slots of parity wg (the slot count is even); row
            // (group gr, row i) of an M block is staged pixel 96 m + 6 gr + i
            const int gr = row >> 3, i8 = row & 7;
            int slot = 0, wraps = 0;
            bool ok = true;
            for (int k = 0; k < ntiles && ok; ++k) {
                int b, xs, ys;
                tile_coords(k, b, xs, ys);
                const size_t img_base = (size_t)b * (size_t)(a.npad >> 3) * (size_t)hw_out * 8;
                for (int m = 0; m < g.mb; ++m) {
                    const int sl = slot;
                    const uint32_t par = (uint32_t)(wraps & 1);
                    if (++slot == g.nslot) {
                        slot = 0;
                        ++wraps;
                    }
                    if ((sl & 1) != wg) continue;
                    if (!wait_bar(&tfull[sl], par, abort_v, 128)) {
                        *abort_v = 1;
                        ok = false;
                        break;
                    }
                    tc::tc_fence_after_sync();
                    const int q = m * N3_PX + 6 * gr + i8;
                    const int yy = q / g.pw, xx = q - yy * g.pw;
                    const int oy = ys + yy, ox = xs + xx;
                    const bool valid = i8 < 6 && xx < g.tw && yy < g.rows && oy < a.hout && ox < a.wout;
                    const long long pix = (long long)oy * a.wout + ox;
                    const size_t ob = img_base + (size_t)pix * 8;
                    const long long p = (long long)b * hw_out + pix;
                    const uint32_t tcol = lane_base + (uint32_t)(sl * g.slot_cols);
                    // columns 0-15: dx = -1 (this row); 16-31: dx = 0 (row + 1); 32-47: dx = +1 (row + 2)
                    float d[48];
                    tc::tmem_ld48(tcol, d);
                    tc::tc_fence_before_sync();
                    tc::mbar_arrive(&tempty[sl]);   // the slot's TMEM reads are done
                    float v[16];
#pragma unroll
                    for (int c = 0; c < 16; ++c)
                        v[c] = d[c] + __shfl_down_sync(0xffffffffu, d[16 + c], 1) +
                               __shfl_down_sync(0xffffffffu, d[32 + c], 2);
                    if (valid) segment(v, 0, ob, p, preload(ob, 0, true));
                }
            }
        } else {
            for (int k = 0; k < ntiles; ++k) {
                const int acc = g.nbuf == 2 ? (k & 1) : 0;
                const uint32_t par = (uint32_t)((g.nbuf == 2 ? (k >> 1) : k) & 1);
                int b, xs, ys;
                tile_coords(k, b, xs, ys);
                const uint32_t dbase = lane_base + (uint32_t)acc * g.acc_cols;
                const size_t img_base = (size_t)b * (size_t)(a.npad >> 3) * (size_t)hw_out * 8;
                // output pixel of this thread's row of block bi (-1: none); an up-sampled image may have more than 2^31
                // (see plan_launch)
                using Pixel = std::conditional_t<MODE == 2 || MODE == 3, long long, int>;
                auto pixel = [&](int bi) -> Pixel {
                    if (bi >= nblk) return -1;
                    const int ph = MODE == 5 ? 0 : bi / g.mb, m = bi - ph * g.mb;
                    int yy = m, xx = row;        // mode 5: a block is an output row
                    if (MODE != 5) {
                        const int q = m * 128 + row;
                        yy = q / g.pw;
                        xx = q - yy * g.pw;
                    }
                    int oy = ys + yy, ox = xs + xx;
                    if (MODE == 2 || MODE == 3) {
                        oy = 2 * oy + (g.psplit ? tile_py(k) : ph >> 1);
                        ox = 2 * ox + (g.psplit ? ph : ph & 1);
                    }
                    return xx < g.tw && yy < g.rows && oy < a.hout && ox < a.wout ? (Pixel)oy * a.wout + ox : (Pixel)-1;
                };
                // (16 channels: the next block's operand is under way while this one is finished)
                Pixel pix = pixel(wg);
                Pre2 pre{};
                if (ACT && a.npad == 16) pre = preload(img_base + (size_t)pix * 8, 0, pix >= 0);
                if (!wait_bar(&tfull[acc], par, abort_v, 128)) { *abort_v = 1; break; }
                tc::tc_fence_after_sync();
                for (int bi = wg; bi < nblk; bi += 2) {
                    const Pixel next = pixel(bi + 2);
                    const size_t ob = img_base + (size_t)pix * 8;   // channel 0 of this pixel
                    const long long p = (long long)b * hw_out + pix;
                    const uint32_t tcol = dbase + (uint32_t)((MODE == 5 ? g.rows - 1 - bi : bi) * a.npad);
                    if (a.npad == 16) {
                        Pre2 pn{};
                        if (ACT) pn = preload(img_base + (size_t)next * 8, 0, next >= 0);
                        else pre = preload(ob, 0, pix >= 0);
                        float v[16];
                        tc::tmem_ld16(tcol, v);
                        if (pix >= 0) segment(v, 0, ob, p, pre);
                        if (ACT) pre = pn;
                    } else {
                        for (int c0 = 0; c0 < a.npad; c0 += 32) {
                            const Pre2 p0 = preload(ob, c0, pix >= 0);
                            Pre2 p1{};
                            if (ACT) p1 = preload(ob, c0 + 16, pix >= 0);
                            float v[32];
                            tc::tmem_ld32(tcol + (uint32_t)c0, v);
                            if (pix < 0) continue;
                            segment(v, c0, ob, p, p0);
                            if (!ACT) p1 = preload(ob, c0 + 16, true);
                            segment(v + 16, c0 + 16, ob, p, p1);
                        }
                    }
                    pix = next;
                }
                // this thread's TMEM reads of the buffer are complete (tcgen05.ld waited)
                tc::tc_fence_before_sync();
                tc::mbar_arrive(&tempty[acc]);
            }
        }
    }

    tc::tc_fence_before_sync();
    __syncthreads();
    if (*abort_v && tid == 0) atomicExch(a.err, 1);
    if (warp == 0) tc::tmem_dealloc(tmem, g.tmem_cols);
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        else
            (void)cudaGetLastError();
    });
    return fn;
}

// Chunked BF16 activation [n][c/8][h][w][8] (see nc8).  Modes 0, 2, 3: viewed
// as 8-byte elements, a 4-D tensor (2w, h, c/8, n); box = 2 box_w elements (box_w
// pixels of one row, contiguous) x box_h rows x two 8-channel planes x one image.
// Mode 1: a 5-D tensor (2, w, h, c/8, n) traversed with element stride 2 in w and
// h (box_w / 2 x box_h / 2 pixels of each of the two planes land in shared memory).
bool encode_act(CUtensorMap* m, const void* base, int c, int w, int h, int n, int box_w, int box_h, int es) {
    const cuuint64_t plane = (cuuint64_t)w * h * 16;
    if (es == 1) {
        const cuuint64_t dims[4] = {(cuuint64_t)2 * w, (cuuint64_t)h, (cuuint64_t)(c / 8), (cuuint64_t)n};
        const cuuint64_t strides[3] = {(cuuint64_t)w * 16, plane, plane * (cuuint64_t)(c / 8)};
        const cuuint32_t box[4] = {(cuuint32_t)(2 * box_w), (cuuint32_t)box_h, 2u, 1u};
        const cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
        return encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_UINT64, 4, const_cast<void*>(base), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    const cuuint64_t dims[5] = {2u, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)(c / 8), (cuuint64_t)n};
    const cuuint64_t strides[4] = {16u, (cuuint64_t)w * 16, plane, plane * (cuuint64_t)(c / 8)};
    const cuuint32_t box[5] = {2u, (cuuint32_t)box_w, (cuuint32_t)box_h, 2u, 1u};
    const cuuint32_t estr[5] = {1u, (cuuint32_t)es, (cuuint32_t)es, 1u, 1u};
    return encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_UINT64, 5, const_cast<void*>(base), dims, strides, box, estr,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Chunked BF16 activation [n][c/8][h][w][8] as a TMA tensor map for other kernels
// (the weight gradient): es = 1, a 4-D view (2w, h, c/8, n) of 8-byte elements with
// box (2 box_w, box_h, box_chunks, 1); es = 2, a 5-D view (2, w, h, c/8, n) traversed
// with element stride 2 along w and h, box (2, box_w, box_h, box_chunks, 1), which
// lands box_w / 2 x box_h / 2 pixels per chunk.  Either way a box lands as
// [chunk][row][pixel][8 channels].
bool tma_map_act(CUtensorMap* m, const void* base, int c, int w, int h, int n, int box_w, int box_h, int box_chunks,
                 int es) {
    if (!encode_fn()) return false;
    const cuuint64_t plane = (cuuint64_t)w * h * 16;
    if (es == 1) {
        const cuuint64_t dims[4] = {(cuuint64_t)2 * w, (cuuint64_t)h, (cuuint64_t)(c / 8), (cuuint64_t)n};
        const cuuint64_t strides[3] = {(cuuint64_t)w * 16, plane, plane * (cuuint64_t)(c / 8)};
        const cuuint32_t box[4] = {(cuuint32_t)(2 * box_w), (cuuint32_t)box_h, (cuuint32_t)box_chunks, 1u};
        const cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
        return encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_UINT64, 4, const_cast<void*>(base), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    const cuuint64_t dims[5] = {2u, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)(c / 8), (cuuint64_t)n};
    const cuuint64_t strides[4] = {16u, (cuuint64_t)w * 16, plane, plane * (cuuint64_t)(c / 8)};
    const cuuint32_t box[5] = {2u, (cuuint32_t)box_w, (cuuint32_t)box_h, (cuuint32_t)box_chunks, 1u};
    const cuuint32_t estr[5] = {1u, 2u, 2u, 1u, 1u};
    return encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_UINT64, 5, const_cast<void*>(base), dims, strides, box, estr,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

namespace {

// Mode 4: weights [npad][9][cin] viewed as a 5-D tensor (8 channels, npad rows,
// 3 column taps, cin/8 chunks, 3 tap rows); box = (8, npad, 3, 2, 3) lands as
// [dy][half][dx][npad][8], so that the B operand of tap row dy is 3 npad rows.
bool encode_w5(CUtensorMap* m, const void* base, int cin, int npad) {
    const cuuint64_t dims[5] = {8u, (cuuint64_t)npad, 3u, (cuuint64_t)(cin / 8), 3u};
    const cuuint64_t strides[4] = {(cuuint64_t)9 * cin * 2, (cuuint64_t)cin * 2, 16u, (cuuint64_t)3 * cin * 2};
    const cuuint32_t box[5] = {8u, (cuuint32_t)npad, 3u, 2u, 3u};
    const cuuint32_t estr[5] = {1u, 1u, 1u, 1u, 1u};
    return encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims, strides, box, estr,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

std::atomic<int> g_rows_cap{0};   // tile-height limit set by cnn_set_conv_tiling (0 = automatic)

// Tiling of one launch: tile-height cap, stage and ring budgets (0 = default), and
// the variant of a narrow same-grid layer: narrow = 1, the column-taps-in-N kernel
// (mode 4, 16 output channels); narrow = 2, the row-taps-in-N kernel (mode 6, 16 or 32).
struct TileCfg {
    int rows_cap = 0, stage_kb = 0, ring_kb = 0, narrow = 0;
    int plain = 0;    // same-grid layers: mode 0 also where mode 5 takes fewer cycles (see rowsum_pays)
    int single = 0;   // modes 0-3: one accumulator buffer of up to 512 TMEM columns
    int upsplit = 0;  // mode 2: a tile per output row parity (half the weights per stage, twice the rows)
};
std::atomic<int> g_stage_kb{0}, g_ring_kb{0};
std::atomic<int> g_single{0};   // one accumulator buffer, set by cnn_set_conv_buffers
std::atomic<int> g_upsplit{0};  // up layers: a tile per output row parity, set by cnn_set_conv_upsplit
std::atomic<long long> g_launch_narrow{0};   // launches of mode 4
std::atomic<long long> g_launch_rowtaps{0};  // launches of mode 6   // stage / ring budgets set by cnn_set_conv_ring (0 = default)
int g_last_launch[6] = {0, 0, 0, 0, 0, 0};   // grid, CTAs per SM, CTAs registers/smem allow, shared memory,
                                             // registers per thread, static shared memory

// Tile plan; .tiles = 0 when the layer does not fit this kernel.
Geometry plan(const ConvArgs& a, const TileCfg& t) {
    Geometry g{};
    if (a.mode == 6) {
        // same grid, 16 or 32 output channels, tap rows in N (see the mode list above): an M
        // block is one staged row (pitch tw + 2 <= 128)
        if (a.npad != 16 && a.npad != 32) return Geometry{};
        const int H = a.hout, W = a.wout;
        g.groups = (a.c0 + a.c1) / 16;
        g.groups0 = a.c0 / 16;
        g.nph = 1;
        g.nplanes = 1;
        const int ntx = (W + 125) / 126;   // staged rows of at most 128 pixels: one 4-D TMA box row
        g.tw = (W + ntx - 1) / ntx;
        g.pw = g.tw + 2;
        g.wbytes = 9 * 2 * a.npad * 16;
        // 16 channels: 5 slots of 48 columns in 256 (two CTAs per SM, so that two MMA streams
        // overlap); 32 channels: 5 slots of 96 in 512 (one CTA per SM)
        g.slot_cols = 3 * a.npad;
        g.tmem_cols = a.npad == 16 ? 256 : 512;
        g.nslot = std::min(MAX_SLOTS, (int)g.tmem_cols / g.slot_cols);
        int rmax = std::min(H, ROWS_RT_MAX);
        if (t.rows_cap > 0 && rmax > t.rows_cap) rmax = t.rows_cap;
        const size_t ring_budget = t.ring_kb > 0 ? (size_t)t.ring_kb * 1024
                                   : (a.npad == 16 ? RING_BUDGET_RT16 : RING_BUDGET_RT32);
        // the tallest tile whose stages fit a ring holding every group of a tile and one more
        g.rows = 0;
        for (int rows = rmax; rows >= 1; --rows) {
            const int plane = (rows + 2) * g.pw * 16;
            const int pstride = (2 * plane + 127) / 128 * 128;
            const int stage = pstride + g.wbytes;
            if (t.stage_kb > 0 && (size_t)stage > (size_t)t.stage_kb * 1024) continue;
            int ns = (int)(ring_budget / (size_t)stage);
            if (ns > MAX_NS) ns = MAX_NS;
            if (ns < g.groups + 1) continue;
            g.rows = rows;
            g.plane = plane;
            g.pstride = pstride;
            g.stage = stage;
            g.ns = ns;
            break;
        }
        if (g.rows < 1) return Geometry{};
        g.mb = g.rows + 2;          // staged rows (TMEM slots) per tile
        // Warpgroup w takes output rows w, w + nwg, ...  Its parity wait on the commit that
        // covers its newest staged row is unambiguous when that barrier's previous commit is
        // known complete, which its own previous wait proves: consecutive waits of a
        // warpgroup are at most 2 nwg + 1 rows apart when every warpgroup has a row in every
        // tile, i.e. at most (2 nwg + 1) / chunk + 2 commits, fewer than MAX_SLOTS.  A chunk
        // of rows can complete only if its last row's slot is released by output rows that
        // wait on earlier commits: chunk <= nslot - 2.
        g.nwg = epi_warps(6) / 4;
        while (g.nwg > 1 && g.nwg > g.rows) g.nwg >>= 1;
        g.chunk = std::min(RT_CHUNK, g.nslot - 2);
        g.acc_cols = 0;
        g.tiles_x = (W + g.tw - 1) / g.tw;
        g.tiles_y = (H + g.rows - 1) / g.rows;
        g.tx = (uint32_t)(2 * (g.rows + 2) * g.pw * 16 + g.wbytes);
        g.tiles = g.tiles_x * g.tiles_y * a.nb;
        return g;
    }
    if (a.mode == 4) {
        // same grid, 16 output channels, column taps in N (see the mode list above)
        if (a.npad != 16) return Geometry{};
        const int H = a.hout, W = a.wout;
        g.groups = (a.c0 + a.c1) / 16;
        g.groups0 = a.c0 / 16;
        g.nph = 1;
        g.nplanes = 1;
        const int ntx = (W + 125) / 126;
        g.tw = (W + ntx - 1) / ntx;
        g.pw = g.tw + 2;
        g.wbytes = 9 * 2 * a.npad * 16;
        const size_t stage_budget = t.stage_kb > 0 ? (size_t)t.stage_kb * 1024 : STAGE_BUDGET;
        const size_t ring_budget = t.ring_kb > 0 ? (size_t)t.ring_kb * 1024 : RING_BUDGET;
        int rmax = std::min(H, 252);
        const int cap = t.rows_cap;
        if (cap > 0 && rmax > cap) rmax = cap;
        // the tallest tile whose stage fits, with a ring that holds every group of a tile
        // and one more stage (the MMA warp takes all groups of a tile at once)
        g.rows = 0;
        for (int rows = rmax; rows >= 1; --rows) {
            const int plane = (rows + 2) * g.pw * 16;
            const int pstride = (2 * plane + 127) / 128 * 128;
            const int stage = pstride + g.wbytes;
            if ((size_t)stage > stage_budget) continue;
            int ns = (int)(ring_budget / (size_t)stage);
            if (ns > MAX_NS) ns = MAX_NS;
            if (ns < g.groups + 1) continue;
            g.rows = rows;
            g.plane = plane;
            g.pstride = pstride;
            g.stage = stage;
            g.ns = ns;
            break;
        }
        if (g.rows < 1) return Geometry{};
        g.mb = (g.rows * g.pw + N3_PX - 1) / N3_PX;
        g.slot_cols = 64;            // 48 columns used: (dx, o) for dx = -1, 0, 1
        g.nslot = NSLOT4;
        g.tmem_cols = (uint32_t)(g.nslot * g.slot_cols);
        g.acc_cols = 0;
        g.tiles_x = (W + g.tw - 1) / g.tw;
        g.tiles_y = (H + g.rows - 1) / g.rows;
        g.tx = (uint32_t)(2 * (g.rows + 2) * g.pw * 16 + g.wbytes);
        g.tiles = g.tiles_x * g.tiles_y * a.nb;
        return g;
    }
    // the grid the tile lives on: output grid for modes 0, 1 and 5, coarse input grid for 2 and 3
    const bool rowsum = a.mode == 5;
    const int mode = rowsum ? 0 : a.mode;
    const int H = mode >= 2 ? a.hin : a.hout, W = mode >= 2 ? a.win : a.wout;
    g.groups = (a.c0 + a.c1) / 16;
    g.groups0 = a.c0 / 16;
    g.psplit = mode == 2 && t.upsplit ? 1 : 0;
    g.nph = mode >= 2 ? (g.psplit ? 2 : 4) : 1;
    g.nplanes = mode == 1 ? 4 : 1;
    if (mode == 1) {
        g.tw = W >= 127 ? 127 : W;   // 2 (tw + 1) traversed columns fit a 256-element box
        g.pw = g.tw + 1;
    } else {
        // a staged row (tile + halo) is one TMA box row of at most 256 8-byte
        // elements: tw <= 126; wide images are cut into equal tiles
        const int ntx = (W + 125) / 126;
        g.tw = (W + ntx - 1) / ntx;
        g.pw = g.tw + 2;
    }
    const int halo = mode == 1 ? 1 : 2;        // extra staged rows
    g.wbytes = (mode == 2 ? (g.psplit ? 8 : 16) : 9) * 2 * a.npad * 16;   // mode 2: parities x 4 merged taps
    // TMEM per accumulator buffer: 128 columns (two CTAs per SM), or 256 when one
    // block per parity already needs more (one CTA per SM)
    // (wide layers: 256, so that packed rows fill the 128-pixel M blocks)
    int acc_max = 128;
    if (g.nph * a.npad > acc_max || a.npad >= 64) acc_max = 256;
    // one buffer of up to 512 columns: twice the M blocks per stage (the weights of a
    // stage serve more pixels), but the MMAs of a tile wait for the previous epilogue
    g.nbuf = t.single ? 1 : 2;
    if (t.single) acc_max = rowsum ? 256 : 512;   // (mode 5: one MMA clears the buffer)
    const int maxmb = acc_max / (g.nph * a.npad);
    auto fill = [&](int rows) {
        g.rows = rows;
        g.mb = rowsum ? rows : (rows * g.pw + 127) / 128;
        g.plane = ((rows + halo) * g.pw + SLACK_PX) * 16;
        g.pstride = (2 * g.plane + 127) / 128 * 128;
        g.stage = g.nplanes * g.pstride + g.wbytes;
    };
    int rmax = rowsum ? maxmb : (maxmb * 128) / g.pw;
    const int cap = t.rows_cap;
    if (cap > 0 && rmax > cap) rmax = cap;
    if (rmax > H) rmax = H;
    const int box_rows_max = mode == 1 ? 127 : 254;   // staged rows fit a 256-element box
    if (rmax > box_rows_max) rmax = box_rows_max;
    if (rmax < 1) return Geometry{};   // tiles = 0: not this kernel
    int rows = rmax;
    fill(rows);
    const size_t stage_budget = t.stage_kb > 0 ? (size_t)t.stage_kb * 1024
                                : (mode == 1 ? STAGE_BUDGET_S2 : STAGE_BUDGET);
    const size_t ring_budget = t.ring_kb > 0 ? (size_t)t.ring_kb * 1024
                               : (mode == 1 ? RING_BUDGET_S2 : RING_BUDGET);
    while (rows > 1 && (size_t)g.stage > stage_budget) fill(--rows);
    if (g.mb < 1 || g.mb > maxmb) return Geometry{};
    g.ns = (int)(ring_budget / (size_t)g.stage);
    if (g.ns > MAX_NS) g.ns = MAX_NS;
    if (g.ns < 2) g.ns = 2;
    g.tiles_x = (W + g.tw - 1) / g.tw;
    g.tiles_y = (H + g.rows - 1) / g.rows;
    const int staged_px = mode == 1 ? (g.rows + 1) * g.pw : (g.rows + 2) * g.pw;
    g.tx = (uint32_t)(2 * g.nplanes * staged_px * 16 + g.wbytes);
    g.acc_cols = (uint32_t)(g.nph * g.mb * a.npad);
    g.nzero = rowsum ? g.mb * a.npad : 0;
    uint32_t cols = 32;
    while (cols < (uint32_t)g.nbuf * g.acc_cols) cols <<= 1;
    g.tmem_cols = cols;
    g.tiles = g.tiles_x * g.tiles_y * a.nb * (g.psplit ? 2 : 1);
    return g;
}

// Cycles that an M = 128, K = 16 MMA holds the tensor core: its product, or the shared-memory reads of
// its operands at 128 bytes per cycle (4 KB of A, 32 bytes of B per column).
int mma_cycles(int n) { return std::max(n / 2, 32 + n / 4); }

// Whether mode 5 (plan g5) takes fewer MMA cycles per output node and group than mode 0 (plan g0).  Mode
// 5 reads A a third as often, but gives the lanes beyond a row's tile away (mode 0 packs rows), and its
// tile ends carry fewer columns.  The line lies a little below equal counts, where the two tie.  One GB300,
// 32 images, mode 0 and mode 5 (modelled ratio): 16 channels, 1024 x 512, 220 and 163 us; 32 to 16 channels
// there, 406 and 260; 32 channels, 512 x 256, 134 and 108; 64 channels, 512 x 64, 16 images, 59 and 50; 64
// channels, 256 x 128, 199 and 198 (0.91); 32 channels, 128 x 64, 25 and 25 (1.00); 64 channels, 80 x 40, 28
// and 33 (1.06); but 64 channels, 64 x 32, 28 and 24, which the count does not see.
bool rowsum_pays(const ConvArgs& a, const Geometry& g0, const Geometry& g5) {
    if (g5.tiles <= 0 || 3 * a.npad > 256 || (size_t)g5.ns * g5.stage + ZERO_BYTES > 200 * 1024) return false;
    if (g0.tiles <= 0) return false;
    const double c0 = 9.0 * g0.mb * mma_cycles(a.npad) * g0.tiles;
    double c5 = mma_cycles(g5.nzero) / (double)g5.groups;
    for (int b = 0; b < g5.rows + 2; ++b) {
        const int nt = (b < 2 ? b : 2) - (b < g5.rows ? 0 : b - g5.rows + 1) + 1;
        c5 += 3.0 * mma_cycles(nt * a.npad);
    }
    c5 *= g5.tiles;
    return c5 < 0.9 * c0;
}

int smem_per_sm() {
    static int n = 0;
    static std::once_flag once;
    std::call_once(once, [] {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess)
            n = 0;
        (void)cudaGetLastError();
    });
    return n > 0 ? n : 228 * 1024;
}

int sm_count() {
    static int n = 0;
    static std::once_flag once;
    std::call_once(once, [] {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            n = 0;
        (void)cudaGetLastError();
    });
    return n > 0 ? n : 148;
}

template <int MODE, bool ACT>
int launch_kernel(const CUtensorMap& tm0, const CUtensorMap& tm1, const CUtensorMap& tmw, const ConvArgs& a,
                const Geometry& g, cudaStream_t st) {
    static DeviceOnce once;
    HELM_CK(once_per_device(once, [] {
        const cudaError_t e = cudaFuncSetAttribute(conv3x3_tma_kernel<MODE, ACT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        // all of the unified L1/shared storage as shared memory: two CTAs of ~100 KB per SM
        return e != cudaSuccess ? e : cudaFuncSetAttribute(conv3x3_tma_kernel<MODE, ACT>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    }));
    const size_t smem = (size_t)g.ns * g.stage;
    // two CTAs per SM when two fit the 512 TMEM columns, else one; a shared-memory
    // request above a third (half) of the SM keeps further CTAs off
    int per_sm = g.tmem_cols <= 256 ? 2 : 1;
    const size_t smem_req = std::max<size_t>(smem, per_sm == 2 ? 80 * 1024 : 120 * 1024);
    // resident CTAs per SM from this kernel's registers and shared memory (the
    // runtime's occupancy query assumes a smaller shared-memory carveout here)
    static int regs = 0, static_smem = 0;
    static std::once_flag attrs;
    std::call_once(attrs, [] {
        cudaFuncAttributes fa;
        if (cudaFuncGetAttributes(&fa, conv3x3_tma_kernel<MODE, ACT>) == cudaSuccess) {
            regs = fa.numRegs;
            static_smem = (int)fa.sharedSizeBytes;
        } else {
            (void)cudaGetLastError();
        }
    });
    const size_t per_cta_smem = smem_req + (size_t)static_smem + 1024;   // + the per-block shared memory the CUDA runtime reserves
    const int by_smem = (int)((size_t)smem_per_sm() / per_cta_smem);
    constexpr int NT = threads_of(MODE);
    const int by_regs = regs > 0 ? 65536 / (((regs * 32 + 255) / 256) * 256 * (NT / 32)) : 1;
    const int occ = std::min(by_smem, by_regs);
    per_sm = std::max(1, std::min(per_sm, occ));
    const long long grid = std::min<long long>(g.tiles, (long long)per_sm * sm_count());
    g_last_launch[0] = (int)grid;
    g_last_launch[1] = per_sm;
    g_last_launch[2] = occ;
    g_last_launch[3] = (int)smem_req;
    g_last_launch[4] = regs;
    g_last_launch[5] = static_smem;
    { conv3x3_tma_kernel<MODE, ACT><<<(unsigned)grid, NT, smem_req, st>>>(tm0, tm1, tmw, a, g); count_launch(); }
    return cudaGetLastError() == cudaSuccess ? HELM_OK : HELM_ECUDA;
}

// ACT: the instance for BF16 activations alone (no gradient output, no FP32 output), which holds no
// registers for the rest: two CTAs per SM with a block's operand loaded ahead.
template <int MODE>
int launch_mode(const CUtensorMap& tm0, const CUtensorMap& tm1, const CUtensorMap& tmw, const ConvArgs& a,
                const Geometry& g, cudaStream_t st) {
    if constexpr (MODE != 4 && MODE != 6)
        if (!a.gmask && !a.out_fp32) return launch_kernel<MODE, true>(tm0, tm1, tmw, a, g, st);
    return launch_kernel<MODE, false>(tm0, tm1, tmw, a, g, st);
}

}  // namespace

// Launches the TMA halo-tile kernel; returns HELM_EINVAL (nothing launched) when
// the layer does not fit it, so that the caller can use the gather kernel.
namespace {

// The launch decision of one layer, host code shared by the launcher and
// cnn_conv_plan: the shape checks of the kernel, the tile plan, and for a narrow
// same-grid layer the variant that t.narrow asks for: 1, the column-taps-in-N kernel
// (mode 4, 16 channels); 2, the row-taps-in-N kernel (mode 6, 16 or 32 channels).  Either
// falls back to mode 0 when its plan does not fit (mode 4 also when the caller says
// that its weight map could not be encoded: no_mode4).  *mode_out = the mode that
// runs.  HELM_EINVAL when the kernel does not take the layer (nothing launched);
// *g_out is the plan either way.
int plan_launch(const ConvArgs& a, const TileCfg& t, bool no_mode4, int* mode_out, Geometry* g_out) {
    *g_out = Geometry{};
    *mode_out = a.mode;
    if (a.mode < 0 || a.mode > 3) return HELM_EINVAL;
    if (a.npad != 16 && a.npad % 32) return HELM_EINVAL;   // the epilogue reads 16 or 32k columns
    if (a.npad > 128 || a.c0 % 8 || a.c1 % 8) return HELM_EINVAL;
    if (a.mode == 0 && (a.hin != a.hout || a.win != a.wout)) return HELM_EINVAL;
    if (a.mode == 1 && (a.hin != 2 * a.hout || a.win != 2 * a.wout)) return HELM_EINVAL;
    if (a.mode >= 2 && (a.hout != 2 * a.hin || a.wout != 2 * a.win)) return HELM_EINVAL;
    if ((long long)a.nb * (a.mode >= 2 ? (long long)a.hin * a.win : (long long)a.hout * a.wout) > 0x7fffffffLL)
        return HELM_EINVAL;
    ConvArgs b = a;
    Geometry g{};
    if (t.narrow == 1 && !no_mode4 && a.mode == 0 && a.npad == 16) {
        b.mode = 4;
        g = plan(b, t);
        if (g.tiles <= 0 || (size_t)g.ns * g.stage > 200 * 1024) b.mode = 0;
    } else if (t.narrow == 2 && !no_mode4 && a.mode == 0 && (a.npad == 16 || a.npad == 32)) {
        b.mode = 6;
        g = plan(b, t);
        if (g.tiles <= 0 || (size_t)g.ns * g.stage > 200 * 1024) b.mode = 0;
    }
    if (b.mode != 4 && b.mode != 6) {
        g = plan(b, t);
        if (a.mode == 0 && !t.plain && !no_mode4) {
            b.mode = 5;
            const Geometry g5 = plan(b, t);
            if (rowsum_pays(a, g, g5)) g = g5;
            else b.mode = 0;
        }
    }
    *g_out = g;
    *mode_out = b.mode;
    if (g.tiles <= 0) return HELM_EINVAL;
    if ((size_t)g.ns * g.stage > 200 * 1024 || g.tmem_cols > 512) return HELM_EINVAL;
    // box extents: modes 0/2/3 (tw + 2) pixels = 2 (tw + 2) elements x (rows + 2); mode 1
    // traverses 2 (tw + 1) x 2 (rows + 1) pixels with stride 2
    const int bw = b.mode == 1 ? 2 * g.pw : g.pw;
    const int bh = b.mode == 1 ? 2 * (g.rows + 1) : g.rows + 2;
    if ((b.mode == 1 ? bw : 2 * bw) > 256 || bh > 256) return HELM_EINVAL;
    return HELM_OK;
}

// One launch of the TMA kernel with tiling t; HELM_EINVAL when the layer does not fit it.
int launch_cfg(const ConvArgs& a_in, cudaStream_t st, const TileCfg& t) {
    ConvArgs a = a_in;
    if ((reinterpret_cast<uintptr_t>(a.x0) & 15) || (a.c1 && (reinterpret_cast<uintptr_t>(a.x1) & 15)) ||
        (reinterpret_cast<uintptr_t>(a.w) & 15))
        return HELM_EINVAL;
    const void* wst = a.mode == 2 ? a.wup : a.wst;   // (an up layer runs on its phase-merged weights)
    if (!wst || (reinterpret_cast<uintptr_t>(wst) & 15)) return HELM_EINVAL;
    Geometry g{};
    int mode = a.mode;
    if (plan_launch(a, t, false, &mode, &g) != HELM_OK) return HELM_EINVAL;
    alignas(64) CUtensorMap tmw;
    if (mode == 4 && !encode_w5(&tmw, a.w, a.c0 + a.c1, a.npad)) {
        // no weight map for the variant: the plain same-grid kernel
        if (plan_launch(a, t, true, &mode, &g) != HELM_OK) return HELM_EINVAL;
    }
    a.mode = mode;
    const int es = a.mode == 1 ? 2 : 1;
    const int bw = a.mode == 1 ? 2 * g.pw : g.pw;
    const int bh = a.mode == 1 ? 2 * (g.rows + 1) : g.rows + 2;
    alignas(64) CUtensorMap tm0, tm1;
    auto enc = [&](CUtensorMap* m, const void* base, int c, int n) {
        return encode_act(m, base, c, a.win, a.hin, n, bw, bh, es);
    };
    if (!enc(&tm0, a.x0, a.c0, a.nb)) return HELM_EINVAL;
    if (a.c1) {
        const int n1 = a.nb1 > 0 ? a.nb1 : (a.x1_bcast ? 1 : a.nb);
        if (!enc(&tm1, a.x1, a.c1, n1)) return HELM_EINVAL;
    } else {
        tm1 = tm0;
    }
    if (a.mode != 4) tmw = tm0;   // (unused)
    switch (a.mode) {
        case 4: ++g_launch_narrow; return launch_mode<4>(tm0, tm1, tmw, a, g, st);
        case 5: return launch_mode<5>(tm0, tm1, tmw, a, g, st);
        case 6: ++g_launch_rowtaps; return launch_mode<6>(tm0, tm1, tmw, a, g, st);
        case 0: return launch_mode<0>(tm0, tm1, tmw, a, g, st);
        case 1: return launch_mode<1>(tm0, tm1, tmw, a, g, st);
        case 2: return launch_mode<2>(tm0, tm1, tmw, a, g, st);
        default: return launch_mode<3>(tm0, tm1, tmw, a, g, st);
    }
}

// Autotuning: the tiling that ran a layer shape fastest, by shape (batch size left out,
// so that the active-RHS batches of a solve find the entry of the full batch).
std::mutex g_tune_mu;
std::map<std::string, TileCfg> g_tuned;
std::atomic<int> g_tuning{0};

std::string shape_key(const ConvArgs& a) {
    char buf[160];
    std::snprintf(buf, sizeof buf, "%d:%d:%d:%d:%d:%d:%d:%d:%d:%d:%d:%d:%d", a.mode, a.c0, a.c1, a.x1_bcast,
                  a.x1_map ? 1 : 0, a.hin, a.win, a.npad, a.res ? 1 : 0, a.out_fp32, a.accum, a.relu, a.bias ? 1 : 0);
    return buf;
}

// Runs the candidate tilings of a layer twice each (the second timed with CUDA events),
// keeps the fastest and launches it once more, so that y holds its result.  Only
// layers whose output aliases none of their inputs and that do not accumulate are
// re-run (the caller checks).
int tune_and_launch(const ConvArgs& a, cudaStream_t st, const std::string& key, const TileCfg& base) {
    std::vector<TileCfg> cands;
    cands.push_back(base);
    const int budgets[][2] = {{36, 110}, {56, 112}, {100, 200}, {47, 200}};
    for (const auto& b : budgets) {
        TileCfg c = base;
        c.stage_kb = b[0];
        c.ring_kb = b[1];
        c.narrow = 0;
        c.plain = 1;
        cands.push_back(c);
    }
    {
        TileCfg c = base;
        c.rows_cap = 4;
        c.narrow = 0;
        c.plain = 1;
        cands.push_back(c);
    }
    if (a.mode == 0) {
        TileCfg c = base;
        c.narrow = 0;
        c.plain = 1;
        cands.push_back(c);
    }
    if (a.mode == 0 && a.npad == 16 && base.narrow != 1) {
        TileCfg c = base;
        c.narrow = 1;
        cands.push_back(c);
    }
    if (base.narrow) {
        TileCfg c = base;
        c.narrow = 0;
        cands.push_back(c);
    }
    {
        TileCfg c = base;
        c.narrow = 0;
        c.single = 1;
        c.plain = 1;
        cands.push_back(c);
    }
    if (a.mode == 2) {
        // a tile per output row parity: with the default budgets, a larger ring, one buffer
        const int v[][3] = {{0, 0, 0}, {100, 200, 0}, {0, 0, 1}, {47, 200, 1}};
        for (const auto& x : v) {
            TileCfg c = base;
            c.narrow = 0;
            c.upsplit = 1;
            c.stage_kb = x[0];
            c.ring_kb = x[1];
            c.single = x[2];
            cands.push_back(c);
        }
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        if (e0) cudaEventDestroy(e0);
        (void)cudaGetLastError();
        return launch_cfg(a, st, base);
    }
    TileCfg best = base;
    float best_ms = 1e30f;
    int s = HELM_OK;
    for (const TileCfg& c : cands) {
        s = launch_cfg(a, st, c);
        if (s == HELM_EINVAL) { s = HELM_OK; continue; }   // this tiling does not fit the layer
        if (s != HELM_OK) break;
        cudaEventRecord(e0, st);
        s = launch_cfg(a, st, c);
        cudaEventRecord(e1, st);
        if (s != HELM_OK) break;
        float ms = 0.0f;
        if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
            s = HELM_ECUDA;
            break;
        }
        if (ms < best_ms) {
            best_ms = ms;
            best = c;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (s != HELM_OK) return s;
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        g_tuned[key] = best;
    }
    return launch_cfg(a, st, best);
}

}  // namespace

int launch_conv3x3_tma(const ConvArgs& a, cudaStream_t st, int narrow) {
    if (!encode_fn()) return HELM_EINVAL;
    if (a.mode < 0 || a.mode > 3) return HELM_EINVAL;
    TileCfg t;
    t.rows_cap = g_rows_cap.load();
    t.stage_kb = g_stage_kb.load();
    t.ring_kb = g_ring_kb.load();
    t.narrow = narrow;
    t.single = g_single.load();
    t.upsplit = g_upsplit.load();
    // explicit tiling knobs take precedence over the tuned table
    if (t.rows_cap || t.stage_kb || t.ring_kb || t.single || t.upsplit) {
        t.plain = 1;
        return launch_cfg(a, st, t);
    }
    const std::string key = shape_key(a);
    bool tune = false;
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tuned.find(key);
        if (it != g_tuned.end())
            t = it->second;
        else   // a layer is re-run while tuning only if that leaves its result unchanged
            tune = g_tuning.load() && !a.accum && !a.gres && a.y != a.x0 && a.y != a.x1 && a.y != a.res;
    }
    return tune ? tune_and_launch(a, st, key, t) : launch_cfg(a, st, t);
}

void conv_tuning(bool on) { g_tuning.store(on ? 1 : 0); }

int conv_tuned_count() {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    return (int)g_tuned.size();
}

void conv_tune_reset() {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tuned.clear();
}

}  // namespace helm

extern "C" int cnn_set_conv_buffers(int nbuf) {
    if (nbuf < 0 || nbuf > 2) {
        helm::set_error("cnn_set_conv_buffers: nbuf must be 0 (automatic), 1 or 2");
        return HELM_EINVAL;
    }
    helm::g_single.store(nbuf == 1 ? 1 : 0);
    return HELM_OK;
}

extern "C" int cnn_set_conv_upsplit(int on) {
    if (on < 0 || on > 1) {
        helm::set_error("cnn_set_conv_upsplit: on must be 0 (automatic) or 1");
        return HELM_EINVAL;
    }
    helm::g_upsplit.store(on);
    return HELM_OK;
}

extern "C" int cnn_set_conv_tiling(int max_rows) {
    if (max_rows < 0 || max_rows > 254) {
        helm::set_error("cnn_set_conv_tiling: max_rows must be in [0, 254]");
        return HELM_EINVAL;
    }
    helm::g_rows_cap.store(max_rows);
    return HELM_OK;
}

extern "C" int cnn_set_conv_ring(int stage_kb, int ring_kb) {
    if (stage_kb < 0 || stage_kb > 128 || ring_kb < 0 || ring_kb > 200 || (stage_kb && ring_kb && ring_kb < stage_kb)) {
        helm::set_error("cnn_set_conv_ring: stage_kb in [0, 128], ring_kb in [0, 200], ring_kb >= stage_kb");
        return HELM_EINVAL;
    }
    helm::g_stage_kb.store(stage_kb);
    helm::g_ring_kb.store(ring_kb);
    return HELM_OK;
}

extern "C" long long cnn_conv_narrow_launches(void) { return helm::g_launch_narrow.load(); }
extern "C" long long cnn_conv_rowtaps_launches(void) { return helm::g_launch_rowtaps.load(); }

// Tile plan of the TMA kernel for a layer shape (host only, no GPU needed): out19 =
// {tiles, tw, rows, pw, mb, nph, nplanes, plane, pstride, wbytes, stage, ns, tmem_cols,
// nslot, slot_cols, mode, nwg, chunk, nbuf}; narrow = 3 asks for the single-buffer tiling, 6 for the
// tiling that a default launch takes (mode 5 or 0).
// For checking the plan's bounds on the CPU.
extern "C" int cnn_conv_plan(int mode, int c0, int c1, int npad, int hin, int win, int nb, int stage_kb,
                             int ring_kb, int rows_cap, int narrow, int* out19) {
    if (!out19 || mode < 0 || mode > 3 || c0 < 16 || c0 % 16 || c1 < 0 || c1 % 16 || nb < 1 || hin < 1 ||
        win < 1 || (npad != 16 && npad % 32) || npad > 128 || narrow < 0 || narrow > 6) {
        helm::set_error("cnn_conv_plan: invalid layer shape");
        return HELM_EINVAL;
    }
    helm::ConvArgs a{};
    a.c0 = c0;
    a.c1 = c1;
    a.nb = nb;
    a.hin = hin;
    a.win = win;
    a.hout = mode == 1 ? hin / 2 : (mode >= 2 ? 2 * hin : hin);
    a.wout = mode == 1 ? win / 2 : (mode >= 2 ? 2 * win : win);
    a.npad = npad;
    a.mode = mode;
    helm::TileCfg t;
    t.rows_cap = rows_cap;
    t.stage_kb = stage_kb;
    t.ring_kb = ring_kb;
    t.narrow = narrow >= 3 ? 0 : narrow;
    t.single = narrow == 3 || narrow == 5 ? 1 : 0;
    t.upsplit = narrow == 4 || narrow == 5 ? 1 : 0;
    t.plain = narrow != 6;
    helm::Geometry g{};
    int used = mode;
    const int s = helm::plan_launch(a, t, false, &used, &g);
    const int v[19] = {g.tiles, g.tw, g.rows, g.pw, g.mb, g.nph, g.nplanes, g.plane, g.pstride, g.wbytes,
                       g.stage, g.ns, (int)g.tmem_cols, g.nslot, g.slot_cols, used, g.nwg, g.chunk, g.nbuf};
    for (int i = 0; i < 19; ++i) out19[i] = v[i];
    if (s != HELM_OK) {
        helm::set_error("cnn_conv_plan: the layer does not fit the TMA kernel");
        return HELM_EINVAL;
    }
    return HELM_OK;
}

// Launch shape of the last TMA convolution (diagnostics): grid, CTAs per SM,
// the CTAs per SM that registers and shared memory allow, dynamic
// shared memory per CTA, registers per thread, static shared memory.
extern "C" void cnn_conv_last_launch(int* out6) {
    if (!out6) return;
    for (int i = 0; i < 6; ++i) out6[i] = helm::g_last_launch[i];
}

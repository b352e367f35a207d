// Temporally blocked Taylor stages for two particles in complex FP32: D
// Horner stages per launch on shared-memory tiles with halos.
//
// The order-K polynomial of Algorithm 3 (Sec. 2.3) in Horner form,
//   w_K = psi + (A/K) psi,  w_j = psi + (A/j) w_{j+1},  psi(t+dt) = psi + A w_2,
// A = -i dt H, is split into launches of D consecutive stages.  A block owns
// a T x T tile of the N x N amplitude tile of one realization.  It loads the
// launch's input iterate and psi on the tile plus D rows and columns around
// it, applies the D stages in shared memory (stage d is exact on the tile
// grown by D - d, so the halo shrinks by one per stage), and writes the
// tile of the result.  Per launch HBM carries the input iterate, psi and the
// output once (the halo reloads are L2 hits): about 24/D bytes per
// site-update against 24 for one launch per stage.  The extra arithmetic is
// the halo, sum_d (T + 2(D - d))^2 / (D T^2) - 1 of the work (20% for T = 32,
// D = 4).
//
// Coordinates outside 0..N-1 wrap around: on a ring that is the lattice, on
// an open chain the wrap bond has J[N-1] = 0, so the wrapped halo holds valid
// values of real sites and nothing crosses the open boundary.  When the
// launch ends with the final stage, the increment A w_2 is added to psi with
// its rounding error carried in a second FP32 word (lo, in place: every
// element is read and written by its own tile only), and the new psi goes to
// a separate buffer because other tiles still read the old psi as halo.
#include <algorithm>
#include <type_traits>

#include "ctqw_internal.cuh"
#include "fused_common.cuh"

namespace {

using namespace fused;

// One launch for every size group (register tiles): the work items
// (realization, tile row, tile column) of all groups form one 1D grid,
// groups in descending N so that the block scheduler starts the largest
// items first and the small ones fill the tail.  Groups next to each other
// with the same number of tiles are one range of it (a block reads its own
// realization's N), so only batches of more than 32 tile counts take a second
// launch.  Where more than 32 sizes took one launch each, of a few
// realizations: 873 of sizes 192..512, 27 steps of K = 16, 344 -> 130 ms; 500 of
// 64..128, 20 of K = 8, 25.2 -> 3.0; 200 of 128..1024, 4 of K = 16, 30.8 -> 12.8.
constexpr int kMaxFlatGroups = 32;
struct FlatGroups {
    int n;                              // ranges in the launch (0: one launch per group)
    int64_t item_off[kMaxFlatGroups + 1];   // first item of each range
    int list_off[kMaxFlatGroups];       // its realizations in by_group (the launch's list)
    int tiles_y[kMaxFlatGroups], tiles_x[kMaxFlatGroups];
};

struct TiledArgs {
    RealTable tab;
    FlatGroups flat;
    const int32_t *list;     // realizations of this launch's size group (all groups when flat.n > 0)
    const float *eps, *J;    // float32 parameters (packed per realization)
    const float2 *w_in;      // input iterate (w_{j0+1}; psi itself when j0 = K)
    const float2 *psi;       // state of the step
    float2 *w_out;           // output iterate w_{j0-D+1}, or the new state when final
    float2 *lo;              // carried rounding error (final launches when compensated)
    float dt, dtU;
    int T;                   // tile side for this size group (<= the compiled maximum)
    int j0;                  // first stage of the launch (stage j maps w_{j+1} -> w_j)
    int n_stages;            // D, or fewer for the last launch of a step
    int final;               // the launch's last stage is j = 1 (state update)
    int compensated;
    int aligned16;           // every buffer starts on a 16-byte boundary
};


// The block's work item: its realization and tile (row, column).
struct TileItem {
    int r, ty, tx;
};

__device__ __forceinline__ TileItem tile_item(const TiledArgs &a) {
    TileItem t;
    if (a.flat.n == 0) {
        t.r = a.list[blockIdx.z];
        t.ty = blockIdx.y;
        t.tx = blockIdx.x;
        return t;
    }
    const int64_t it = blockIdx.x;
    int g = 0;
    while (g + 1 < a.flat.n && it >= a.flat.item_off[g + 1]) ++g;
    const int64_t local = it - a.flat.item_off[g];
    const int per_r = a.flat.tiles_y[g] * a.flat.tiles_x[g];
    const int q = (int)(local / per_r), rem = (int)(local - (int64_t)q * per_r);
    t.r = a.list[a.flat.list_off[g] + q];
    t.ty = rem / a.flat.tiles_x[g];
    t.tx = rem - t.ty * a.flat.tiles_x[g];
    return t;
}

// T x T output tile (T <= TMAX, chosen per size group so that the tiles
// cover N evenly), D halo, blockDim = 256 (warps over rows, lanes over
// columns).  Region rows are stored with the compiled stride RS.
template <int TMAX, int D>
__global__ void __launch_bounds__(256) taylor_tiled_kernel(const __grid_constant__ TiledArgs a) {
    constexpr int RS = TMAX + 2 * D;    // region row stride
    constexpr int RE = RS * RS;
    const int T = a.T;
    const int RC = T + 2 * D;           // region side
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *bufA = reinterpret_cast<float2 *>(smem_raw);   // [RE]
    float2 *bufB = bufA + RE;                              // [RE]
    float2 *Q = bufB + RE;                                 // [RE] psi on the region
    float *e_row = reinterpret_cast<float *>(Q + RE);      // [RS] dt eps of the region's rows
    float *e_col = e_row + RS;                             // [RS]
    float *j_row = e_col + RS;                             // [RS + 1] -dt J of the bond above row i
    float *j_col = j_row + RS + 1;                         // [RS + 1] -dt J of the bond left of column k
    int *x_row = reinterpret_cast<int *>(j_col + RS + 1);  // [RS] wrapped coordinates
    int *x_col = x_row + RS;                               // [RS]

    const int r = a.list[blockIdx.z];
    const int N = a.tab.N[r];
    const int tiles = (N + T - 1) / T;
    if ((int)blockIdx.x >= tiles || (int)blockIdx.y >= tiles) return;   // never: one grid per group
    const int x1_0 = blockIdx.y * T - D, x2_0 = blockIdx.x * T - D;
    const int64_t base = a.tab.st_off[r];
    const int64_t po = a.tab.par_off[r];
    const float dt = a.dt;

    for (int i = threadIdx.x; i < RC; i += blockDim.x) {
        const int X1 = ((x1_0 + i) % N + N) % N, X2 = ((x2_0 + i) % N + N) % N;
        x_row[i] = X1;
        x_col[i] = X2;
        e_row[i] = dt * a.eps[po + X1];
        e_col[i] = dt * a.eps[po + X2];
        j_row[i] = -dt * a.J[po + (X1 + N - 1) % N];
        j_col[i] = -dt * a.J[po + (X2 + N - 1) % N];
    }
    if (threadIdx.x == 0) {
        const int X1 = ((x1_0 + RC - 1) % N + N) % N, X2 = ((x2_0 + RC - 1) % N + N) % N;
        j_row[RC] = -dt * a.J[po + X1];
        j_col[RC] = -dt * a.J[po + X2];
    }
    __syncthreads();
    // the region of the input iterate and of psi (warps over rows, lanes over
    // columns), copied asynchronously so that every load of the block is in
    // flight at once
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, ny = blockDim.x >> 5;
    const float2 *win = a.w_in + base, *gpsi = a.psi + base;
    const uint32_t sA = smem_u32(bufA), sQ = smem_u32(Q);
    for (int i = ty; i < RC; i += ny) {
        const int64_t grow = (int64_t)x_row[i] * N;
        for (int k = tx; k < RC; k += 32) {
            const uint32_t o = (uint32_t)(i * RS + k) * 8u;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sA + o), "l"(win + grow + x_col[k])
                         : "memory");
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sQ + o), "l"(gpsi + grow + x_col[k])
                         : "memory");
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    // every warp owns RS/8 consecutive region rows for the whole launch and
    // keeps psi of its rows and its two column passes in registers
    constexpr int CH = RS / 8;           // rows a warp (8 warps)
    static_assert(RS % 8 == 0 && RS <= 64, "region rows split over 8 warps, two column passes");
    const int r0 = ty * CH;
    float2 qv[2][CH];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
#pragma unroll
        for (int t = 0; t < CH; ++t) qv[p][t] = Q[(r0 + t) * RS + tx + 32 * p];
    }

    float2 *src = bufA, *dst = bufB;
    const float dU = a.dtU;
#pragma unroll 1
    for (int d = 1; d <= a.n_stages; ++d) {
        const int j = a.j0 - d + 1;
        const bool last_final = a.final && d == a.n_stages;   // j == 1
        const float inv_j = 1.0f / (float)j;
        // stage d is exact on the region shrunk by d; the final stage is
        // needed on the tile only
        const int lo = last_final ? D : d, hi = last_final ? D + T : RC - d;
        const int i0 = max(lo, r0), i1 = min(hi, r0 + CH);   // this warp's rows of the stage
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int k = tx + 32 * p;
            if (k < lo || k >= hi || i0 >= i1) continue;
            const float ec = e_col[k], jl = j_col[k], jr = j_col[k + 1];
            const int X2w = x_col[k];
            const bool col_in = x2_0 + k < N;
            float2 wu = src[(i0 - 1) * RS + k], wc = src[i0 * RS + k];
            float ju = j_row[i0];
#pragma unroll
            for (int t = 0; t < CH; ++t) {
                const int i = r0 + t;
                if (i < i0 || i >= i1) continue;
                const int c = i * RS + k;
                const float2 wd = src[c + RS], wl = src[c - 1], wr = src[c + 1];
                const float jd = j_row[i + 1];
                float v = e_row[i] + ec;
                if (x_row[i] == X2w) v += dU;
                // y = dt H w
                float yx = v * wc.x, yy = v * wc.y;
                yx = fmaf(ju, wu.x, yx); yy = fmaf(ju, wu.y, yy);
                yx = fmaf(jd, wd.x, yx); yy = fmaf(jd, wd.y, yy);
                yx = fmaf(jl, wl.x, yx); yy = fmaf(jl, wl.y, yy);
                yx = fmaf(jr, wr.x, yx); yy = fmaf(jr, wr.y, yy);
                const float2 q = qv[p][t];
                if (!last_final) {
                    // w_j = psi + (-i/j) y
                    dst[c] = make_float2(fmaf(inv_j, yy, q.x), fmaf(-inv_j, yx, q.y));
                } else if (col_in && x1_0 + i < N) {
                    // psi(t+dt) = psi + (-i) y, rounding error carried in lo
                    const int64_t g = base + (int64_t)x_row[i] * N + X2w;
                    float2 h = q;
                    const float2 inc = make_float2(yy, -yx);
                    if (a.compensated) {
                        float2 l = a.lo[g];
                        compensated_add(h.x, l.x, inc.x);
                        compensated_add(h.y, l.y, inc.y);
                        a.lo[g] = l;
                    } else {
                        h.x += inc.x;
                        h.y += inc.y;
                    }
                    a.w_out[g] = h;
                }
                wu = wc;
                wc = wd;
                ju = jd;
            }
        }
        __syncthreads();
        float2 *tsw = src;
        src = dst;
        dst = tsw;
    }
    if (!a.final) {
        // the tile of the launch's last iterate (exact on the tile)
        for (int i = D + ty; i < D + T; i += ny) {
            const int X1 = x1_0 + i;
            if (X1 >= N) break;
            for (int k = D + tx; k < D + T; k += 32) {
                const int X2 = x2_0 + k;
                if (X2 < N) a.w_out[base + (int64_t)X1 * N + X2] = src[i * RS + k];
            }
        }
    }
}

// The same D stages with the iterate in registers: the region is 8W rows x
// 64 columns (tile (8W - 2D) x (64 - 2 DC), DC = D or D + 1), every warp holds 8 region rows
// and every lane the two adjacent columns 2l, 2l+1 of them.  Neighbours along x2 are in the lane or
// one 64-bit shuffle away; along x1 in registers except the warp's first
// and last rows, which pass through shared memory once per stage (one
// __syncthreads).  psi of the region stays in shared memory.  The shuffles
// wrap from column 63 to 0 and the outermost warps read zero rows: both
// only touch the halo's outer ring, which stage 1 already leaves inexact.
//
// Everything a block reads from HBM is requested before its first stage:
// psi of the region and, for a final launch, the carried error word of the
// tile, both by cp.async into shared memory (a lane reads back only slots it
// filled itself, so they need no barrier).  The row coefficients are 8-byte
// broadcasts: 16-byte ones cost twice the shared-memory wavefronts, and that
// pipe is the bound (78% busy; 8 warps x 3 blocks an SM; at their 80 registers a
// thread spills 44 bytes, loaded 88 to 128 bytes at a time and 324 for odd N,
// through the same pipe).  The ragged batch
// of 512 realizations, N = 128..1024, K = 8, 20 steps: 97.5 ms with the
// error words read in the final stage and psi read twice, 79.9 ms with both
// fetched at the start, 74.2 ms with the 8-byte coefficients and the regions
// that tiled_default_shape picks.
//
// The halo along x2 is D rounded up to a whole pair of columns, so a lane's
// pair starts on 16 bytes at odd depths too (even N): one 16-byte copy where
// there were two of 8.  10 steps: 64 x N = 512, K = 14 (D = 7) 5.97 -> 5.07 ms,
// K = 10 (D = 5) 4.44 -> 3.67; 16 x N = 1000, K = 7 2.80 -> 2.35.  FLUSH keeps a
// halo of D columns at odd depths (settle_columns).
template <int D, int W, bool FLUSH>
struct RegTile {
    static constexpr int RS = 8 * W, RL = 8;              // region rows, rows a warp
    static constexpr int DC = FLUSH ? D : (D + 1) & ~1;   // halo along x2: whole pairs of columns
    static constexpr int T = RS - 2 * D, T2 = 64 - 2 * DC;  // tile rows and columns
    static constexpr size_t q_bytes = sizeof(float4) * RS * 32;
    static constexpr size_t lo_bytes = (sizeof(float2) * T * T2 + 15) / 16 * 16;
    static constexpr size_t edge_bytes = sizeof(float4) * 2 * W * 2 * 32;
    static constexpr size_t smem = q_bytes + lo_bytes + edge_bytes + sizeof(float4) * 32 + sizeof(float2) * (RS + 1) + sizeof(int) * RS;
};

// One stencil stage of a warp's 8 x 64 block: y = dt H P, then
//   !FINAL: P <- psi + (-i / j) y;
//   FINAL: psi + (-i) y on the tile, with the rounding error carried in lo.
// u4, d4: the rows above and below; Q: this lane's psi (row stride 32
// float4); diag: bit (2 i + k) set where row i, column k is on x1 = x2
// (DIAG: some bit of the warp is set).
template <bool DIAG>
__device__ __forceinline__ void reg_stencil_row(const float2 (&P)[8][2], int i, const float2 (&prev)[2], float4 d4,
                                                float2 rc, float2 rn, const float2 (&ec)[2], const float2 (&nJc)[3],
                                                float2 dU, unsigned diag, int from_left, int from_right,
                                                float2 &y0, float2 &y1) {
    const float2 c0 = P[i][0], c1 = P[i][1];
    const float2 lft = shfl2(c1, from_left), rgt = shfl2(c0, from_right);
    const float2 n0 = i < 7 ? P[i < 7 ? i + 1 : 7][0] : make_float2(d4.x, d4.y);
    const float2 n1 = i < 7 ? P[i < 7 ? i + 1 : 7][1] : make_float2(d4.z, d4.w);
    const float2 er = make_float2(rc.x, rc.x), jup = make_float2(rc.y, rc.y), jdn = make_float2(rn.y, rn.y);
    y0 = __fmul2_rn(ec[0], c0);
    y1 = __fmul2_rn(ec[1], c1);
    y0 = __ffma2_rn(er, c0, y0);
    y1 = __ffma2_rn(er, c1, y1);
    y0 = __ffma2_rn(jup, prev[0], y0);
    y1 = __ffma2_rn(jup, prev[1], y1);
    y0 = __ffma2_rn(jdn, n0, y0);
    y1 = __ffma2_rn(jdn, n1, y1);
    y0 = __ffma2_rn(nJc[0], lft, y0);
    y1 = __ffma2_rn(nJc[1], c0, y1);
    y0 = __ffma2_rn(nJc[1], c1, y0);
    y1 = __ffma2_rn(nJc[2], rgt, y1);
    if (DIAG) {
        if (diag & (1u << (2 * i))) y0 = __ffma2_rn(dU, c0, y0);
        if (diag & (1u << (2 * i + 1))) y1 = __ffma2_rn(dU, c1, y1);
    }
}

template <int D, int W, bool FLUSH>
__global__ void __launch_bounds__(32 * W, W == 8 ? 3 : 2) taylor_tiled_reg_kernel(const __grid_constant__ TiledArgs a) {
    using Tile = RegTile<D, W, FLUSH>;
    constexpr int RS = Tile::RS, T = Tile::T, T2 = Tile::T2, RL = Tile::RL, DC = Tile::DC;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *Q = reinterpret_cast<float4 *>(smem_raw);                        // [RS][32] psi, (row, lane) -> 2 columns
    float2 *los = reinterpret_cast<float2 *>(smem_raw + Tile::q_bytes);      // [T][T2] carried error of the tile
    float4 *edge = reinterpret_cast<float4 *>(smem_raw + Tile::q_bytes + Tile::lo_bytes);   // [2 parity][W warps][2][32]
    float4 *zero = edge + 2 * W * 2 * 32;                         // [32] a row of zeros
    float2 *rowc = reinterpret_cast<float2 *>(zero + 32);         // [RS + 1] (dt eps, -dt J of the bond above)
    int *x_row = reinterpret_cast<int *>(rowc + RS + 1);          // [RS]

    const TileItem item = tile_item(a);
    const int r = item.r;
    const int N = a.tab.N[r];
    const int x1_0 = item.ty * T - D, x2_0 = item.tx * T2 - DC;
    const int64_t base = a.tab.st_off[r];
    const int64_t po = a.tab.par_off[r];
    const float dt = a.dt;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r0 = warp * RL;
    auto wrap = [N](int x) { return x < 0 || x >= N ? (x % N + N) % N : x; };

    // this warp's rows (a row index of its own: no barrier before the loads)
    if (lane < RL) x_row[r0 + lane] = wrap(x1_0 + r0 + lane);
    __syncwarp();
    int X2[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) X2[k] = wrap(x2_0 + 2 * lane + k);
    // pairs of columns are 16 bytes apart and never straddle the wrap
    const bool vec = a.aligned16 && DC % 2 == 0 && ((N | (int)(base & 1)) & 1) == 0;
    // the tile's part of this lane and warp
    bool col_in[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int ck = 2 * lane + k;
        col_in[k] = ck >= DC && ck < DC + T2 && x2_0 + ck < N;
    }
    auto row_in = [&](int ri) { return ri >= D && ri < D + T && x1_0 + ri < N; };

    const float2 *win = a.w_in + base, *gpsi = a.psi + base;
    const bool carried = a.final && a.compensated;
    const uint32_t sQ = smem_u32(Q) + (uint32_t)(r0 * 32 + lane) * 16u;
    // slot of (row, column) of the tile: negative rows and columns are never touched
    const int lo_at = (r0 - D) * T2 + 2 * lane - DC;
    const uint32_t sL = smem_u32(los);
    float2 P[RL][2];
    if (vec) {
#pragma unroll
        for (int i = 0; i < RL; ++i)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sQ + i * 512u),
                         "l"(gpsi + (int64_t)x_row[r0 + i] * N + X2[0])
                         : "memory");
    } else {
#pragma unroll
        for (int i = 0; i < RL; ++i) {
#pragma unroll
            for (int k = 0; k < 2; ++k)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sQ + i * 512u + 8u * k),
                             "l"(gpsi + (int64_t)x_row[r0 + i] * N + X2[k])
                             : "memory");
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (carried) {
        const float2 *glo = a.lo + base;
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            if (!row_in(r0 + i)) continue;
            const int64_t grow = (int64_t)x_row[r0 + i] * N;
            if (vec) {
                if (col_in[0])
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sL + (uint32_t)(lo_at + i * T2) * 8u),
                                 "l"(glo + grow + X2[0])
                                 : "memory");
            } else {
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    if (col_in[k])
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sL + (uint32_t)(lo_at + i * T2 + k) * 8u),
                                     "l"(glo + grow + X2[k])
                                     : "memory");
            }
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const bool own_w = a.w_in != a.psi;   // the launch starts from an iterate of its own
    if (own_w) {
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            const float2 *g = win + (int64_t)x_row[r0 + i] * N;
            if (vec) {
                const float4 v = *reinterpret_cast<const float4 *>(g + X2[0]);
                P[i][0] = make_float2(v.x, v.y);
                P[i][1] = make_float2(v.z, v.w);
            } else {
                P[i][0] = g[X2[0]];
                P[i][1] = g[X2[1]];
            }
        }
    }
    // coefficients of the region's rows and of this lane's columns
    for (int i = threadIdx.x; i <= RS; i += blockDim.x) {
        const int X1 = wrap(x1_0 + i);
        const float e = i < RS ? dt * a.eps[po + X1] : 0.f;
        const float j = -dt * a.J[po + (X1 == 0 ? N - 1 : X1 - 1)];
        rowc[i] = make_float2(e, j);
    }
    if (threadIdx.x < 32) zero[threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
    float2 ec[2], nJc[3];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float v = dt * a.eps[po + X2[k]];
        ec[k] = make_float2(v, v);
    }
#pragma unroll
    for (int k = 0; k <= 2; ++k) {   // bond left of column 2 lane + k
        const int X = k < 2 ? (X2[k] == 0 ? N - 1 : X2[k] - 1) : X2[1];
        const float v = -dt * a.J[po + X];
        nJc[k] = make_float2(v, v);
    }
    unsigned diag = 0;
    if (a.dtU != 0.f) {
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            const int X1 = x_row[r0 + i];
            diag |= (X1 == X2[0] ? 1u << (2 * i) : 0u) | (X1 == X2[1] ? 2u << (2 * i) : 0u);
        }
    }
    const bool any_diag = __any_sync(0xffffffffu, diag != 0);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    if (!own_w) {
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            const float4 q = Q[(r0 + i) * 32 + lane];
            P[i][0] = make_float2(q.x, q.y);
            P[i][1] = make_float2(q.z, q.w);
        }
    }

    const float2 dU = make_float2(a.dtU, a.dtU);
    const int from_left = (lane + 31) & 31, from_right = (lane + 1) & 31;
    const int n_mid = a.final ? a.n_stages - 1 : a.n_stages;   // stages that update the iterate
    const float4 *Ql = Q + r0 * 32 + lane;
    // publish the warp's first and last rows; the rows above and below it
    float4 u4, d4;
    auto exchange = [&](int par) {
        float4 *eb = edge + (par * W + warp) * 2 * 32;
        eb[lane] = make_float4(P[0][0].x, P[0][0].y, P[0][1].x, P[0][1].y);
        eb[32 + lane] = make_float4(P[RL - 1][0].x, P[RL - 1][0].y, P[RL - 1][1].x, P[RL - 1][1].y);
        __syncthreads();
        u4 = warp > 0 ? edge[(par * W + warp - 1) * 2 * 32 + 32 + lane] : zero[lane];
        d4 = warp < W - 1 ? edge[(par * W + warp + 1) * 2 * 32 + lane] : zero[lane];
    };
    auto mid = [&](auto diag_tag, float inv_j) {
        float2 prev[2] = {make_float2(u4.x, u4.y), make_float2(u4.z, u4.w)};
        float2 rc = rowc[r0];
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            const float2 rn = rowc[r0 + i + 1];
            float2 y0, y1;
            reg_stencil_row<decltype(diag_tag)::value>(P, i, prev, d4, rc, rn, ec, nJc, dU, diag, from_left, from_right,
                                                       y0, y1);
            rc = rn;
            prev[0] = P[i][0];
            prev[1] = P[i][1];
            const float4 q = Ql[i * 32];
            P[i][0] = make_float2(fmaf(inv_j, y0.y, q.x), fmaf(-inv_j, y0.x, q.y));
            P[i][1] = make_float2(fmaf(inv_j, y1.y, q.z), fmaf(-inv_j, y1.x, q.w));
        }
    };
#pragma unroll 1
    for (int d = 1; d <= n_mid; ++d) {
        exchange(d & 1);
        const float inv_j = 1.0f / (float)(a.j0 - d + 1);
        if (any_diag)
            mid(std::true_type(), inv_j);
        else
            mid(std::false_type(), inv_j);
    }
    if (!a.final) {
        // the tile of the launch's last iterate
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            if (!row_in(r0 + i)) continue;
            float2 *g = a.w_out + base + (int64_t)x_row[r0 + i] * N;
            if (vec) {
                if (col_in[0])
                    *reinterpret_cast<float4 *>(g + X2[0]) = make_float4(P[i][0].x, P[i][0].y, P[i][1].x, P[i][1].y);
            } else {
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    if (col_in[k]) g[X2[k]] = P[i][k];
            }
        }
        return;
    }
    // the final stage: psi(t+dt) = psi + (-i) y on the tile, rounding error carried in lo
    exchange(a.n_stages & 1);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    float2 prev[2] = {make_float2(u4.x, u4.y), make_float2(u4.z, u4.w)};
    float2 rc = rowc[r0];
#pragma unroll
    for (int i = 0; i < RL; ++i) {
        const float2 rn = rowc[r0 + i + 1];
        float2 y0, y1;
        reg_stencil_row<true>(P, i, prev, d4, rc, rn, ec, nJc, dU, diag, from_left, from_right, y0, y1);
        rc = rn;
        prev[0] = P[i][0];
        prev[1] = P[i][1];
        if (!row_in(r0 + i)) continue;
        const float4 q = Ql[i * 32];
        float2 h[2] = {make_float2(q.x, q.y), make_float2(q.z, q.w)};
        const float2 inc[2] = {make_float2(y0.y, -y0.x), make_float2(y1.y, -y1.x)};
        const int64_t g = base + (int64_t)x_row[r0 + i] * N;
        float2 l[2] = {};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (!col_in[k]) continue;
            if (a.compensated) {
                l[k] = los[lo_at + i * T2 + k];
                compensated_add2(h[k], l[k], inc[k]);
            } else {
                h[k].x += inc[k].x;
                h[k].y += inc[k].y;
            }
        }
        if (vec) {
            if (col_in[0]) {
                if (a.compensated)
                    *reinterpret_cast<float4 *>(a.lo + g + X2[0]) = make_float4(l[0].x, l[0].y, l[1].x, l[1].y);
                *reinterpret_cast<float4 *>(a.w_out + g + X2[0]) = make_float4(h[0].x, h[0].y, h[1].x, h[1].y);
            }
        } else {
#pragma unroll
            for (int k = 0; k < 2; ++k)
                if (col_in[k]) {
                    if (a.compensated) a.lo[g + X2[k]] = l[k];
                    a.w_out[g + X2[k]] = h[k];
                }
        }
    }
}

// The register tiles on a wider region: 64 rows x 32 CL columns (tile
// (64 - 2D) x (32 CL - 2D)), every lane owning CL adjacent columns, so a
// smaller share of the region is halo and neighbours along x2 are mostly in
// the lane.  psi rows in shared memory are lane-major (column pair k/2 of
// lane l at float4 slot (k/2)*32 + l), as in the full-row kernel.
template <int D, int CL>
__global__ void __launch_bounds__(256, 2) taylor_tiled_wide_kernel(const __grid_constant__ TiledArgs a) {
    constexpr int RR = 64, RC = 32 * CL, T1 = RR - 2 * D, T2 = RC - 2 * D, RL = 8;
    static_assert(CL % 2 == 0, "column pairs");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *Q = reinterpret_cast<float4 *>(smem_raw);            // [RR][RC / 2] lane-major pairs
    float4 *edge = Q + RR * (RC / 2);                             // [2 parity][8 warps][2][RC / 2]
    float4 *zero = edge + 2 * 8 * 2 * (RC / 2);                   // [RC / 2]
    float4 *rowc = zero + RC / 2;                                 // [RR + 1]
    int *x_row = reinterpret_cast<int *>(rowc + RR + 1);          // [RR]

    const TileItem item = tile_item(a);
    const int r = item.r;
    const int N = a.tab.N[r];
    const int x1_0 = item.ty * T1 - D, x2_0 = item.tx * T2 - D;
    const int64_t base = a.tab.st_off[r];
    const int64_t po = a.tab.par_off[r];
    const float dt = a.dt;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r0 = warp * RL;

    for (int i = threadIdx.x; i <= RR; i += blockDim.x) {
        const int X1 = ((x1_0 + i) % N + N) % N;
        if (i < RR) x_row[i] = X1;
        const float e = i < RR ? dt * a.eps[po + X1] : 0.f;
        const float j = -dt * a.J[po + (X1 + N - 1) % N];
        rowc[i] = make_float4(e, e, j, j);
    }
    for (int q = threadIdx.x; q < RC / 2; q += blockDim.x) zero[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    int X2[CL];
    float2 ec[CL], nJc[CL + 1];
#pragma unroll
    for (int k = 0; k < CL; ++k) {
        X2[k] = ((x2_0 + CL * lane + k) % N + N) % N;
        const float v = dt * a.eps[po + X2[k]];
        ec[k] = make_float2(v, v);
    }
#pragma unroll
    for (int k = 0; k <= CL; ++k) {
        const int X = ((x2_0 + CL * lane + k - 1) % N + N) % N;   // bond left of column CL lane + k
        const float v = -dt * a.J[po + X];
        nJc[k] = make_float2(v, v);
    }
    __syncthreads();
    const float2 *win = a.w_in + base, *gpsi = a.psi + base;
    const uint32_t sQ = smem_u32(Q);
    for (int i = warp; i < RR; i += 8) {
        const int64_t grow = (int64_t)x_row[i] * N;
#pragma unroll
        for (int k = 0; k < CL; ++k) {
            const uint32_t slot = (uint32_t)(i * (RC / 2) + (k / 2) * 32 + lane);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sQ + slot * 16u + 8u * (k & 1)),
                         "l"(gpsi + grow + X2[k])
                         : "memory");
        }
    }
    float2 P[RL][CL];
#pragma unroll
    for (int i = 0; i < RL; ++i) {
        const int64_t grow = (int64_t)x_row[r0 + i] * N;
#pragma unroll
        for (int k = 0; k < CL; ++k) P[i][k] = win[grow + X2[k]];
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    const float2 dU = make_float2(a.dtU, a.dtU);
    const int from_left = (lane + 31) & 31, from_right = (lane + 1) & 31;
#pragma unroll 1
    for (int d = 1; d <= a.n_stages; ++d) {
        const int par = d & 1;
        const int j = a.j0 - d + 1;
        const bool last_final = a.final && d == a.n_stages;   // j == 1
        const float inv_j = 1.0f / (float)j;
        float4 *eb = edge + (par * 8 + warp) * 2 * (RC / 2);
#pragma unroll
        for (int k = 0; k < CL; k += 2) {
            eb[(k / 2) * 32 + lane] = make_float4(P[0][k].x, P[0][k].y, P[0][k + 1].x, P[0][k + 1].y);
            eb[RC / 2 + (k / 2) * 32 + lane] =
                make_float4(P[RL - 1][k].x, P[RL - 1][k].y, P[RL - 1][k + 1].x, P[RL - 1][k + 1].y);
        }
        __syncthreads();
        const float4 *us = warp > 0 ? edge + (par * 8 + warp - 1) * 2 * (RC / 2) + RC / 2 : zero;
        const float4 *ds = warp < 7 ? edge + (par * 8 + warp + 1) * 2 * (RC / 2) : zero;
        float2 prev[CL];
#pragma unroll
        for (int k = 0; k < CL; k += 2) {
            const float4 u4 = us[(k / 2) * 32 + lane];
            prev[k] = make_float2(u4.x, u4.y);
            prev[k + 1] = make_float2(u4.z, u4.w);
        }
        float4 rc = rowc[r0];
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            float2 c[CL];
#pragma unroll
            for (int k = 0; k < CL; ++k) c[k] = P[i][k];
            const float2 lft = shfl2(c[CL - 1], from_left), rgt = shfl2(c[0], from_right);
            float2 nb[CL];
            if (i < RL - 1) {
#pragma unroll
                for (int k = 0; k < CL; ++k) nb[k] = P[i + 1][k];
            } else {
#pragma unroll
                for (int k = 0; k < CL; k += 2) {
                    const float4 d4 = ds[(k / 2) * 32 + lane];
                    nb[k] = make_float2(d4.x, d4.y);
                    nb[k + 1] = make_float2(d4.z, d4.w);
                }
            }
            const float4 rn = rowc[r0 + i + 1];
            const float2 er = make_float2(rc.x, rc.y), jup = make_float2(rc.z, rc.w), jdn = make_float2(rn.z, rn.w);
            rc = rn;
            const int X1w = x_row[r0 + i];
            float2 y[CL];
#pragma unroll
            for (int k = 0; k < CL; ++k) {
                const float2 l = (k == 0) ? lft : c[k - 1];
                const float2 rr = (k == CL - 1) ? rgt : c[k + 1];
                float2 t = __fmul2_rn(ec[k], c[k]);
                t = __ffma2_rn(er, c[k], t);
                t = __ffma2_rn(jup, prev[k], t);
                t = __ffma2_rn(jdn, nb[k], t);
                t = __ffma2_rn(nJc[k], l, t);
                t = __ffma2_rn(nJc[k + 1], rr, t);
                if (X1w == X2[k]) t = __ffma2_rn(dU, c[k], t);   // dt U on x1 = x2
                y[k] = t;
            }
#pragma unroll
            for (int k = 0; k < CL; ++k) prev[k] = c[k];
            const int ri = r0 + i;
#pragma unroll
            for (int k = 0; k < CL; k += 2) {
                const float4 q = Q[ri * (RC / 2) + (k / 2) * 32 + lane];
                if (!last_final) {
                    P[i][k] = make_float2(fmaf(inv_j, y[k].y, q.x), fmaf(-inv_j, y[k].x, q.y));
                    P[i][k + 1] = make_float2(fmaf(inv_j, y[k + 1].y, q.z), fmaf(-inv_j, y[k + 1].x, q.w));
                } else if (ri >= D && ri < D + T1 && x1_0 + ri < N) {
                    // psi(t+dt) = psi + (-i) y on the tile, rounding error carried in lo
#pragma unroll
                    for (int h2 = 0; h2 < 2; ++h2) {
                        const int ck = CL * lane + k + h2;
                        if (ck < D || ck >= D + T2 || x2_0 + ck >= N) continue;
                        const int64_t g = base + (int64_t)X1w * N + X2[k + h2];
                        const float2 yk = y[k + h2];
                        float2 hv = h2 ? make_float2(q.z, q.w) : make_float2(q.x, q.y);
                        const float2 inc = make_float2(yk.y, -yk.x);
                        if (a.compensated) {
                            float2 l = a.lo[g];
                            compensated_add(hv.x, l.x, inc.x);
                            compensated_add(hv.y, l.y, inc.y);
                            a.lo[g] = l;
                        } else {
                            hv.x += inc.x;
                            hv.y += inc.y;
                        }
                        a.w_out[g] = hv;
                    }
                }
            }
        }
    }
    if (!a.final) {
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            const int ri = r0 + i;
            if (ri < D || ri >= D + T1 || x1_0 + ri >= N) continue;
            const int64_t grow = base + (int64_t)x_row[ri] * N;
#pragma unroll
            for (int k = 0; k < CL; ++k) {
                const int ck = CL * lane + k;
                if (ck >= D && ck < D + T2 && x2_0 + ck < N) a.w_out[grow + X2[k]] = P[i][k];
            }
        }
    }
}

using TiledKernel = void (*)(TiledArgs);

struct TiledShape {
    int TMAX, D;
    TiledKernel kern;
    size_t smem;
    bool fixed_tile;   // the register kernels: tile TMAX (rows) x TMAX2 (columns) exactly
    int TMAX2;
    int threads = 256;
    // odd depths: the same with a halo of D columns (see settle_columns)
    TiledKernel kern_flush = nullptr;
    size_t smem_flush = 0;
    int T2_flush = 0;
};

template <int TMAX, int D>
TiledShape tiled_shape() {
    constexpr int RS = TMAX + 2 * D;
    TiledShape s;
    s.TMAX = TMAX;
    s.D = D;
    s.kern = taylor_tiled_kernel<TMAX, D>;
    s.smem = sizeof(float2) * 3 * (size_t)RS * RS + sizeof(float) * (4 * (size_t)RS + 2) +
             sizeof(int) * 2 * (size_t)RS;
    s.fixed_tile = false;
    s.TMAX2 = TMAX;
    return s;
}

template <int D, int W = 8>
TiledShape tiled_reg_shape() {
    using Tile = RegTile<D, W, false>;
    TiledShape s;
    s.TMAX = Tile::T;
    s.TMAX2 = Tile::T2;
    s.D = D;
    s.kern = taylor_tiled_reg_kernel<D, W, false>;
    s.smem = Tile::smem;
    s.fixed_tile = true;
    s.threads = 32 * W;
    if constexpr (D % 2 == 1) {
        s.kern_flush = taylor_tiled_reg_kernel<D, W, true>;
        s.T2_flush = RegTile<D, W, true>::T2;
        s.smem_flush = RegTile<D, W, true>::smem;
    }
    return s;
}

template <int D, int CL>
TiledShape tiled_wide_shape() {
    constexpr int RC = 32 * CL;
    TiledShape s;
    s.TMAX = 64 - 2 * D;
    s.TMAX2 = RC - 2 * D;
    s.D = D;
    s.kern = taylor_tiled_wide_kernel<D, CL>;
    s.smem = sizeof(float4) * (64 * (RC / 2) + 2 * 8 * 2 * (RC / 2) + RC / 2 + 65) + sizeof(int) * 64;
    s.fixed_tile = true;
    return s;
}

// 0: regions of at most 64 x 64 (two 32-lane column passes per row);
// 3..10: the iterate in registers at depths 4, 8, 2, 7, 6, 5, 3 and 1;
// 11: registers on 64 x 128 regions at depth 8; 13, 14: registers on 96 x 64
// regions (12 warps) at depths 8 and 7 (tiles: 2D less, along x2 at odd depths
// 2D + 2 less)
bool tiled_shape_for(int idx, TiledShape &s) {
    switch (idx) {
        case 0: s = tiled_shape<56, 4>(); return true;
        case 3: s = tiled_reg_shape<4>(); return true;
        case 4: s = tiled_reg_shape<8>(); return true;
        case 5: s = tiled_reg_shape<2>(); return true;
        case 6: s = tiled_reg_shape<7>(); return true;
        case 7: s = tiled_reg_shape<6>(); return true;
        case 8: s = tiled_reg_shape<5>(); return true;
        case 9: s = tiled_reg_shape<3>(); return true;
        case 10: s = tiled_reg_shape<1>(); return true;
        case 11: s = tiled_wide_shape<8, 4>(); return true;
        case 13: s = tiled_reg_shape<8, 12>(); return true;
        case 14: s = tiled_reg_shape<7, 12>(); return true;
        default: return false;
    }
}

}  // namespace

// At an odd depth the halo of whole column pairs costs two columns of the tile
// and saves half the copies of lattices of even N.  Odd N has no aligned pairs
// to copy, so there (every size odd) the tiles keep the two columns; and so
// they do where that needs fewer tiles by more than the 15% that the copies
// are worth (K = 14, 64 x N = 512: 5.97 against 5.07 ms).  7 x N = 771, K = 19, 37
// steps: 8.96 ms with pairs, 7.86 without.  Returns the cost against a tile of pairs.
static double settle_columns(const ctqw_hamiltonian *h, TiledShape &f) {
    if (!f.kern_flush) return 1.0;
    double pairs = 0.0, flush = 0.0;
    bool all_odd = true;
    for (size_t g = 0; g < h->group_N.size(); ++g) {
        const int N = h->group_N[g];
        const double rows = (double)h->group_count[g] * ((N + f.TMAX - 1) / f.TMAX);
        pairs += rows * ((N + f.TMAX2 - 1) / f.TMAX2);
        flush += rows * ((N + f.T2_flush - 1) / f.T2_flush);
        all_odd = all_odd && N % 2 == 1;
    }
    if (!all_odd && 1.15 * flush >= pairs) return 1.0;
    f.kern = f.kern_flush;
    f.smem = f.smem_flush;
    f.TMAX2 = f.T2_flush;
    return all_odd ? 1.0 : 1.15;
}

bool tiled_supported(const ctqw_hamiltonian *h, int dtype, int shape) {
    TiledShape s;
    return dtype == CTQW_C64 && h->m == 2 && tiled_shape_for(shape, s);
}

int tiled_depth(int shape) {
    TiledShape s;
    return tiled_shape_for(shape, s) ? s.D : 0;
}

// The register tiles' depth (and region) for this handle and order: the least
// time by a model over the depths 1..8.  A launch takes kLaunch, and its tiles
// run in rounds of three blocks an SM, each of them a fixed part (loads,
// coefficients, the compensated update) and a part for every stage; the last
// round takes half a round and the rest by how full it is.  So deeper launches
// are fewer but leave a smaller tile, the next shallower depth may cover the
// lattice with fewer tiles, and where the tiles do not fill the SMs the launches
// are what counts.  The constants, in warp instructions, are fitted to 450
// calls at every depth (N = 20..1150, also ragged, 3 to 10000 tiles, K = 3..20): the
// choice is 0.3% above the best depth on average, 12% at most.  By the number of
// tiles alone it was 1.2%, up to 47% where they do not fill the SMs (10 steps of R
// x N, K: 7 x 277, 7 299 us, now 224; 6 x 318, 17 606 and 481; 6 x 501, 8 498 and 437).
// The 96 x 64 regions (depth 7 and 8 only, two blocks an SM) run at 0.94 of the
// rate a region point.
static constexpr double kTileFixed = 1180.0, kTileStage = 170.0, kLaunch = 1000.0, kTallRate = 0.94;

int tiled_default_shape(const ctqw_hamiltonian *h, int K) {
    static const int by_depth[9] = {4, 10, 5, 9, 3, 8, 7, 6, 4};   // 64 x 64 regions
    int best = by_depth[8], n_sm = 152;
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, h->device);
    double best_cost = 0.0;
    auto consider = [&](int shape) {
        TiledShape f;
        if (!tiled_shape_for(shape, f)) return;
        const double rate = settle_columns(h, f);
        int64_t tiles = 0;
        for (size_t g = 0; g < h->group_N.size(); ++g) {
            const int N = h->group_N[g];
            tiles += (int64_t)h->group_count[g] * ((N + f.TMAX - 1) / f.TMAX) * ((N + f.TMAX2 - 1) / f.TMAX2);
        }
        const int launches = (K + f.D - 1) / f.D;
        const bool tall = f.threads > 256;   // two blocks an SM, else three
        const int64_t at_once = (tall ? 2 : 3) * n_sm, rest = tiles % at_once;
        const double rounds = (double)(tiles / at_once) + (rest ? 0.5 + 0.5 * (double)rest / (double)at_once : 0.0);
        const double cost = launches * kLaunch +
                            rate * rounds / (tall ? kTallRate : 1.0) * (launches * kTileFixed + kTileStage * K);
        if (best_cost == 0.0 || cost < best_cost) {
            best = shape;
            best_cost = cost;
        }
    };
    const int few = (K + 7) / 8, even8 = (K + few - 1) / few;
    for (int d = 8; d >= 1; --d) {
        // only depths that split the stages evenly: another one does the same
        // launches on smaller tiles
        const int launches = (K + d - 1) / d;
        if ((K + launches - 1) / launches == d) consider(by_depth[d]);
    }
    if (even8 == 8) consider(13);
    if (even8 == 7) consider(14);
    return best;
}

// A round of blocks (24 warps an SM) beside the clusters takes 4.45 ns for each
// instruction of a tile's warp (1180 a launch and 216 a stage, from the counters
// of the 64 x 64 tiles at depths 8 and 4: 2918 and 2049), and a fifth more at odd N,
// whose copies are of 8 bytes, where a step is several launches.  So the best
// share of R x N, K measured (realizations on the tiles, and what others cost): 1024 x
// 256, 16: 94 (64 +2.5%, 109 +2.4%); 300 x 240, 5: 30 (15 +3%); 600 x 192, 16: 25 (2 +3%);
// 356 x 237, 12: 26 (41 +4%); 181 x 221, 12: 16 (31 +4%); 286 x 187, 4: 10 (0 +5%).
// With all SMs to themselves the tiles take 5.3 ns.
double tiled_round_us(const ctqw_hamiltonian *h, int K, int *blocks, int *resident) {
    constexpr double kInstructionUs = 4.45e-3, kFixed = 1180.0, kStage = 216.0;
    TiledShape f;
    tiled_shape_for(tiled_default_shape(h, K), f);
    double rate = settle_columns(h, f);
    if (h->Nmax % 2 && K > f.D) rate *= 1.2;
    *blocks = ((h->Nmax + f.TMAX - 1) / f.TMAX) * ((h->Nmax + f.TMAX2 - 1) / f.TMAX2);
    *resident = f.threads > 256 ? 2 : 3;
    const int launches = (K + f.D - 1) / f.D;
    return kInstructionUs * rate / (f.threads > 256 ? kTallRate : 1.0) * (launches * kFixed / K + kStage);
}

int launch_taylor_tiled_range(const ctqw_hamiltonian *h, int shape, const void *w_in, const void *psi,
                              void *w_out, void *lo, double dt, int j0, int n_stages, int final,
                              int compensated, int r0, int R_run, cudaStream_t s) {
    const bool whole = r0 == 0 && R_run == h->R;
    if (!whole && (h->group_N.size() != 1 || r0 < 0 || R_run < 0 || r0 + R_run > h->R)) {
        ctqw_set_error("tiled path: realizations %d..%d of %d (a range needs one size group)", r0,
                       r0 + R_run, h->R);
        return CTQW_EINVAL;
    }
    if (R_run == 0) return CTQW_OK;
    TiledShape f;
    if (!tiled_shape_for(shape, f)) {
        ctqw_set_error("tiled path: unknown shape %d", shape);
        return CTQW_EUNSUPPORTED;
    }
    settle_columns(h, f);
    if (n_stages < 1 || n_stages > f.D || (final && j0 != n_stages)) {
        ctqw_set_error("tiled path: %d stages from j0=%d with depth %d", n_stages, j0, f.D);
        return CTQW_EINVAL;
    }
    TiledArgs a;
    a.tab = real_table(h);
    a.eps = h->eps32;
    a.J = h->J32;
    a.w_in = (const float2 *)w_in;
    a.psi = (const float2 *)psi;
    a.w_out = (float2 *)w_out;
    a.lo = (float2 *)lo;
    a.dt = (float)dt;
    a.dtU = (float)(dt * h->U);
    a.j0 = j0;
    a.n_stages = n_stages;
    a.final = final;
    a.compensated = compensated;
    // (with a few sites the 16-byte copies of a block are of few addresses: at N = 2
    // a launch takes 27 us instead of 11, at N = 6 up to 12% more, at N = 8 no more)
    a.aligned16 = (((uintptr_t)w_in | (uintptr_t)psi | (uintptr_t)w_out | (uintptr_t)lo) & 15) == 0 && h->Nmax > 6;
    CTQW_CUDA_TRY(cudaFuncSetAttribute((const void *)f.kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)f.smem));
    const int G = (int)h->group_N.size();
    a.flat.n = 0;
    if (f.fixed_tile && G > 1) {
        // one launch over every group, largest N first (see FlatGroups)
        a.list = h->by_group_d;
        a.T = f.TMAX;
        int off = h->R;
        int64_t items = 0;
        for (int g = G - 1; g >= 0; --g) {   // groups are stored in ascending N
            const int N = h->group_N[g], cnt = h->group_count[g];
            const int ty = (N + f.TMAX - 1) / f.TMAX, tx = (N + f.TMAX2 - 1) / f.TMAX2;
            off -= cnt;
            const int n = a.flat.n;
            if (n > 0 && a.flat.tiles_y[n - 1] == ty && a.flat.tiles_x[n - 1] == tx) {
                a.flat.list_off[n - 1] = off;   // the group before it joins its range of the list
            } else {
                a.flat.item_off[n] = items;
                a.flat.list_off[n] = off;
                a.flat.tiles_y[n] = ty;
                a.flat.tiles_x[n] = tx;
                ++a.flat.n;
            }
            items += (int64_t)cnt * ty * tx;
            bool flush = g == 0;
            if (!flush && a.flat.n == kMaxFlatGroups) {   // unless the next group joins the last range
                const int Nn = h->group_N[g - 1];
                flush = (Nn + f.TMAX - 1) / f.TMAX != ty || (Nn + f.TMAX2 - 1) / f.TMAX2 != tx;
            }
            if (!flush) continue;
            if (items > 0x7fffffffLL) {
                ctqw_set_error("tiled path: %lld tiles in one launch", (long long)items);
                return CTQW_EUNSUPPORTED;
            }
            a.flat.item_off[a.flat.n] = items;
            f.kern<<<(unsigned)items, f.threads, f.smem, s>>>(a);
            CTQW_CUDA_TRY(cudaGetLastError());
            a.flat.n = 0;
            items = 0;
        }
        return CTQW_OK;
    }
    // one size group: a range is a slice of its (ascending) realization list
    int off = whole ? 0 : r0;
    for (size_t g = 0; g < h->group_N.size(); ++g) {
        const int N = h->group_N[g], cnt = whole ? h->group_count[g] : R_run;
        // as few tiles per side as the compiled maximum allows, of equal size
        const int tiles = (N + f.TMAX - 1) / f.TMAX;             // along x1 (and x2 if square)
        const int tiles2 = (N + f.TMAX2 - 1) / f.TMAX2;          // along x2
        a.T = f.fixed_tile ? f.TMAX : (N + tiles - 1) / tiles;
        a.list = h->by_group_d + off;
        f.kern<<<dim3((unsigned)tiles2, (unsigned)tiles, (unsigned)cnt), f.threads, f.smem, s>>>(a);
        CTQW_CUDA_TRY(cudaGetLastError());
        off += cnt;
    }
    return CTQW_OK;
}

int launch_taylor_tiled(const ctqw_hamiltonian *h, int shape, const void *w_in, const void *psi,
                        void *w_out, void *lo, double dt, int j0, int n_stages, int final,
                        int compensated, cudaStream_t s) {
    return launch_taylor_tiled_range(h, shape, w_in, psi, w_out, lo, dt, j0, n_stages, final, compensated, 0,
                                     h->R, s);
}

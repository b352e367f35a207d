// Fused, cluster-resident Taylor propagation for two particles in complex FP32,
// full-row layout.
//
// One thread-block cluster owns one realization at a time for all steps of
// the launch (the order-K Taylor polynomial of Algorithm 3, Sec. 2.3, applied
// n_steps times).  The grid holds only as many clusters as are resident at
// once, and each takes realization after realization, so the SMs a cluster
// holds stay its own until the launch ends.  They come from a counter in the
// call's own workspace (one in the handle would be shared by calls that overlap
// on it), or, where there is one for each cluster or no room for the counter,
// in turn.  The counter is for clusters of unequal speed, which share their SMs
// with others or with the tiles of the second stream: 20 steps of 600 x N = 200
// 10.6 ms with it and 11.2 in turn on one stream, and in turn up to 17.8 with
// the tiles; with SMs of their own (1024 x N = 256, 50 steps) 47.9 either way.
// The N x N tile is split into row slabs, one per CTA; every warp owns RL
// whole rows and each lane CL adjacent columns of them (N <= 32 CL), so a warp
// covers full rows: neighbours along x2 are in the lane's registers or one
// 64-bit rotate-shuffle away.  The rotation runs over the lanes that hold
// columns and wraps from column N-1 to 0, which is the ring's bond and is
// multiplied by J[N-1] = 0 on an open chain; rings therefore need CL and RL
// to divide N, open chains pad rows and columns with zeros behind bonds that
// are zero.
// Neighbours along x1 are in registers except for the warp's first and last
// rows, which come from the adjacent warps through shared memory (an mbarrier
// of the CTA's warps) or, at the slab's edges, are pushed by the neighbour
// CTAs straight into this CTA's shared memory with st.async on an mbarrier
// (bounded waits).
//
// Arithmetic: the same polynomial in Horner form with A = -i dt H applied to
// (re, im) pairs with FFMA2:
//   w_K = psi + (A/K) psi,  w_j = psi + (A/j) w_{j+1},  psi(t+dt) = psi + A w_2,
// (forward FP32 summation would drop every term below half an ulp of the
// running sum).  The diagonal dt*(eps_x1 + eps_x2) enters as two FFMA2 with
// a per-row and a per-column pair; dt*U on x1 = x2 is added for the one lane
// of a row that owns the diagonal.  The increment A w_2 is added to the state
// with its rounding error carried in a second FP32 word (lo), so hi + lo
// holds the state to ~2^-48 relative.  lo sits in shared memory for the
// launch and in a state-sized buffer between launches.
//
// What bounds it: the FP32 pipe takes 14 cycles an amplitude and warp (6
// FFMA2 of two cycles, 2 FFMA); everything else is latency.  psi of the step
// stays in registers beside the iterate (reading it from shared memory every
// stage took half of that pipe), and the exchange of edge rows is hidden: a
// stage publishes its edge rows, computes the rows between them into spare
// registers, and only then waits for the neighbours' rows.  Two stages
// alternate between the two register sets of the inner rows, so nothing is
// moved between them.  Measured against psi in shared memory and a block
// barrier a stage (K = 16, site-updates/s, one stream): N = 64 1.17e12 ->
// 1.23e12, N = 128 1.27e12 -> 1.33e12, N = 192 1.01e12 -> 1.23e12, N = 256
// 9.1e11 -> 1.11e12; N = 100, on the register tiles before, 4.4e11 -> 7.6e11;
// one realization of N = 64, 10 steps: 129 us -> 73 us.
//
// (At 4 columns a lane 16 warps leave 128 registers, and a thread spills 56 bytes,
// 100 with switching noise; the other widths spill nothing.)
//
// Control flow: the stages of a step are a first one (from psi), middle ones
// in pairs and a final one, with no per-stage dispatch.  A row tests the few
// columns that the diagonal x1 = x2 can meet it in; a step loop compiled per
// offset of the diagonal had the warps of an SM run different copies of it
// and wait for instructions.
//
// Observables are not formed here.  At every snap_every-th step inside the
// launch the kernel stores the state to a snapshot slot (row-major, the
// layout of psi), and the host reduces the snapshots in FP64 with the
// observables kernel; a launch covers the steps between a sample and the
// sample after its last snapshot.  Keeping that work out of the kernel
// leaves the registers of the Horner loop to the stencil.
#include <algorithm>
#include <type_traits>

#include "ctqw_internal.cuh"
#include "fused_common.cuh"
#include "switching.cuh"

namespace {

using namespace fused;

constexpr int kMaxK = 30;

struct RowsArgs {
    const double *eps;
    const double *J;
    RealTable tab;
    float2 *psi;            // state in (start of the launch) and out (end)
    float2 *lo;             // carried rounding error, in and out
    float2 *snap;           // snapshot slots (states), or null
    double dt;
    float dtU;
    int N, W;               // lattice sites; warps a CTA
    int vec;                // rows of every buffer can be accessed 16 bytes at a time
    int K;
    long long n_steps;      // steps of this launch
    int snap_every;         // snapshot after every snap_every-th step (< n_steps), 0: none
    long long snap_stride;  // amplitudes per snapshot slot
    int compensated;
    int *status;
    unsigned long long wait_limit_ns;
    int test_timeout;
    int r0, R_run;          // realizations r0 .. r0 + R_run - 1
    int *work;              // counter they are taken from, zero at the launch; null: cluster by cluster in turn
    // switching noise: the law, the number of the first step, and the
    // parameters to leave the updated values in
    SwitchLaw law;
    unsigned long long step0;
    double *eps_out, *J_out;
    float *eps32_out, *J32_out;
    float inv_j[kMaxK + 1];
};

// y = dt H of one row of a warp from its values c and the rows up and dn.
// rc, rn: (dt eps, -dt J above) of the row and of the one below it.  dt U on
// x1 = x2: row I of the warp meets it in the lane's column I + d, d = x1 - x2
// of the lane's first column and the warp's first row, a multiple of
// gcd(4, CL); dU holds dt U for the d of this lane and zeros for the others.
template <int CL, int I>
__device__ __forceinline__ void stencil_row(const pair_t (&ec)[CL], const pair_t (&nJc)[CL + 1], float2 rc, float2 rn,
                                            const pair_t (&up)[CL], const pair_t (&c)[CL], const pair_t (&dn)[CL],
                                            const pair_t (&dU)[4], int from_left, int from_right,
                                            pair_t (&y)[CL]) {
    const pair_t er = pack2(rc.x, rc.x), jup = pack2(rc.y, rc.y), jdn = pack2(rn.y, rn.y);
    const pair_t lft = __shfl_sync(0xffffffffu, c[CL - 1], from_left), rgt = __shfl_sync(0xffffffffu, c[0], from_right);
#pragma unroll
    for (int k = 0; k < CL; ++k) y[k] = mul2(ec[k], c[k]);
#pragma unroll
    for (int k = 0; k < CL; ++k) y[k] = fma2(er, c[k], y[k]);
#pragma unroll
    for (int k = 0; k < CL; ++k) y[k] = fma2(jup, up[k], y[k]);
#pragma unroll
    for (int k = 0; k < CL; ++k) y[k] = fma2(jdn, dn[k], y[k]);
#pragma unroll
    for (int k = 0; k < CL; ++k) y[k] = fma2(nJc[k], k == 0 ? lft : c[k == 0 ? 0 : k - 1], y[k]);
#pragma unroll
    for (int k = 0; k < CL; ++k) y[k] = fma2(nJc[k + 1], k == CL - 1 ? rgt : c[k == CL - 1 ? k : k + 1], y[k]);
    constexpr int G = CL % 4 == 0 ? 4 : 2;
#pragma unroll
    for (int k = I % G; k < CL; k += G) y[k] = fma2(dU[(k - I + 2) / 2], c[k], y[k]);
}

// out <- Q + (-i / j) y
template <int CL>
__device__ __forceinline__ void horner_row(pair_t (&out)[CL], const pair_t (&Q)[CL], const pair_t (&y)[CL], float inv_j) {
#pragma unroll
    for (int k = 0; k < CL; ++k) out[k] = horner2(Q[k], y[k], inv_j);
}

// CL columns per lane (N <= 32 CL), 4 rows a warp, up to MAXW warps a CTA.
// SWITCH: the Hamiltonian update of switching noise after every step.  Every
// CTA keeps the realization's parameters in shared memory and redraws all N
// sites (the draws depend on nothing but the counter), so nothing is
// exchanged for it.  256 realizations of N = 256, 50 steps of K = 16: 29.2 ms
// on the tiles with an update launch a step, 18.3 ms here.
template <int CL, int MAXW, bool SWITCH>
__global__ void __launch_bounds__(32 * MAXW, 1) taylor_fused_rows_kernel(const __grid_constant__ RowsArgs a) {
    constexpr int RL = 4;
    constexpr int RQ = 16 * CL;       // float4 (column pairs) a row in shared memory, lane-major
    const int N = a.N, W = a.W, SR = RL * W;
    const int units = (N + RL - 1) / RL;              // warps' row blocks of the lattice
    const int C = (units + W - 1) / W;                // CTAs per cluster
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *halo = reinterpret_cast<float4 *>(smem_raw);    // [2 parity][2: above, below][RQ]
    float4 *edge = halo + 2 * 2 * RQ;                       // [2 parity][W][2: first, last][RQ]
    float4 *los = edge + 2 * W * 2 * RQ;                    // [SR][RQ] carried error
    float2 *rowc = reinterpret_cast<float2 *>(los + SR * RQ);   // [SR + 1] (dt eps, -dt J of the bond above)
    double *par = reinterpret_cast<double *>(rowc + SR + 2);    // SWITCH: [2][N] eps, J
    __shared__ __align__(8) unsigned long long mbar[2][2];      // halo rows: [parity][above, below]
    __shared__ __align__(8) unsigned long long mbar_edge;       // the CTA's warps have published a stage
    __shared__ __align__(8) unsigned long long mbar_never;
    __shared__ int next_r;

    const int rank = (int)cluster_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int unit = rank * W + warp;
    const bool active = unit < units;                       // the last CTA may have idle warps
    const int my_warps = min(W, units - rank * W);          // warps of this CTA that hold rows
    const bool top = warp == 0, bottom = warp == my_warps - 1;
    const int lrow0 = warp * RL;
    const int x1_0 = unit * RL;
    const int x2_0 = lane * CL;
    const int lanes = (N + CL - 1) / CL;                    // lanes that hold columns
    const int from_left = lane == 0 ? lanes - 1 : lane - 1, from_right = lane + 1 >= lanes ? 0 : lane + 1;

    pair_t P[RL][CL], Q[RL][CL], T[2][CL], ec[CL], nJc[CL + 1];
    // this warp's and lane's coefficients from the parameters (every warp
    // reads rowc, so the caller orders this behind the last stage that did)
    auto coefficients = [&](const double *eps, const double *J) {
        const double dt = a.dt;
        for (int q = threadIdx.x; q <= SR; q += blockDim.x) {
            const int x1 = rank * SR + q;
            const float e = x1 < N ? (float)(dt * eps[x1]) : 0.f;
            // the bond above row x1 (x1 = N: the ring's, below the last row)
            const float j = x1 <= N ? (float)(-dt * J[x1 == 0 ? N - 1 : x1 - 1]) : 0.f;
            rowc[q] = make_float2(e, j);
        }
#pragma unroll
        for (int k = 0; k < CL; ++k) {
            const float v = x2_0 + k < N ? (float)(dt * eps[x2_0 + k]) : 0.f;
            ec[k] = pack2(v, v);
        }
#pragma unroll
        for (int k = 0; k <= CL; ++k) {   // left of column x2_0 + k (N: the ring's)
            const int x = x2_0 + k;
            const float v = x2_0 < N && x <= N ? (float)(-dt * J[x == 0 ? N - 1 : x - 1]) : 0.f;
            nJc[k] = pack2(v, v);
        }
    };
    // coefficients and state of realization r
    auto load_realization = [&](const int r) {
        const int64_t po = a.tab.par_off[r];
        if (SWITCH) {
            for (int i = threadIdx.x; i < N; i += blockDim.x) {
                par[i] = a.eps[po + i];
                par[N + i] = a.J[po + i];
            }
            __syncthreads();
            coefficients(par, par + N);
        } else {
            coefficients(a.eps + po, a.J + po);
        }
        const int64_t base = a.tab.st_off[r];
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            const int64_t g = base + (int64_t)(x1_0 + i) * N + x2_0;
#pragma unroll
            for (int k = 0; k < CL; k += 2) {
                float4 h = make_float4(0.f, 0.f, 0.f, 0.f), l = h;
                if (x1_0 + i < N && x2_0 + k < N) {
                    if (a.vec) {
                        h = *reinterpret_cast<const float4 *>(a.psi + g + k);
                        l = *reinterpret_cast<const float4 *>(a.lo + g + k);
                    } else {
                        const float2 h0 = a.psi[g + k], l0 = a.lo[g + k];
                        h.x = h0.x; h.y = h0.y; l.x = l0.x; l.y = l0.y;
                        if (x2_0 + k + 1 < N) {
                            const float2 h1 = a.psi[g + k + 1], l1 = a.lo[g + k + 1];
                            h.z = h1.x; h.w = h1.y; l.z = l1.x; l.w = l1.y;
                        }
                    }
                }
                Q[i][k] = pack2(h.x, h.y);
                Q[i][k + 1] = pack2(h.z, h.w);
                los[(lrow0 + i) * RQ + k * 16 + lane] = l;
            }
        }
    };
    auto store_rows = [&](float2 *dst, const int r, bool with_lo) {
        const int64_t base = a.tab.st_off[r];
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            const int64_t g = base + (int64_t)(x1_0 + i) * N + x2_0;
#pragma unroll
            for (int k = 0; k < CL; k += 2) {
                if (x1_0 + i >= N || x2_0 + k >= N) continue;
                const float4 l = with_lo ? los[(lrow0 + i) * RQ + k * 16 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
                if (a.vec) {
                    *reinterpret_cast<ulonglong2 *>(dst + g + k) = make_ulonglong2(Q[i][k], Q[i][k + 1]);
                    if (with_lo) *reinterpret_cast<float4 *>(a.lo + g + k) = l;
                } else {
                    dst[g + k] = unpack2(Q[i][k]);
                    if (with_lo) a.lo[g + k] = make_float2(l.x, l.y);
                    if (x2_0 + k + 1 < N) {
                        dst[g + k + 1] = unpack2(Q[i][k + 1]);
                        if (with_lo) a.lo[g + k + 1] = make_float2(l.z, l.w);
                    }
                }
            }
        }
    };

    const int rank_up = (rank + C - 1) % C, rank_dn = (rank + 1) % C;
    const uint32_t send_up = map_rank(smem_u32(halo + RQ + lane), rank_up);    // their "row below" slot
    const uint32_t send_up_mb = map_rank(smem_u32(&mbar[0][1]), rank_up);
    const uint32_t send_dn = map_rank(smem_u32(halo + lane), rank_dn);         // their "row above" slot
    const uint32_t send_dn_mb = map_rank(smem_u32(&mbar[0][0]), rank_dn);
    const uint32_t mb_edge = smem_u32(&mbar_edge), mb_halo = smem_u32(&mbar[0][0]);
    bool dead = false;

    if (threadIdx.x == 0) {
        for (int q = 0; q < 2; ++q)
            for (int sd = 0; sd < 2; ++sd) mbar_init(smem_u32(&mbar[q][sd]), 1);
        mbar_init(mb_edge, my_warps > 0 ? my_warps : 1);
        mbar_init(smem_u32(&mbar_never), 1);
        next_r = a.r0 + (int)blockIdx.x / C - (int)gridDim.x / C;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cluster_barrier();
    if (a.test_timeout && threadIdx.x == 0 && blockIdx.x == 0)
        (void)mbar_wait_bounded(smem_u32(&mbar_never), 0, 1000000ull, a.status);

    const long long n_steps = a.n_steps;
    const int K = a.K;
    // this cluster's next realization, which CTA 0 reads from its counter (or
    // counts on by itself) and the others from CTA 0.  Every warp of the cluster
    // is done with the last one's shared memory when it returns.
    auto next = [&]() -> int {
        if (rank == 0 && threadIdx.x == 0) next_r = a.work ? a.r0 + atomicAdd(a.work, 1) : next_r + (int)gridDim.x / C;
        cluster_barrier();
        const int r = ld_shared_cluster_s32(map_rank(smem_u32(&next_r), 0));
        cluster_barrier();
        return r;
    };
    // edge rows of the warp and of its neighbours, by parity (with one CTA the
    // slab's edges are each other's neighbours)
    const bool push_up = C > 1 && top, push_dn = C > 1 && bottom;
    float4 *edge_own = edge + warp * 2 * RQ + lane;
    const float4 *above = push_up ? halo + lane : edge + ((top ? my_warps : warp) - 1) * 2 * RQ + RQ + lane;
    const float4 *below = push_dn ? halo + RQ + lane : edge + (bottom ? 0 : warp + 1) * 2 * RQ + lane;
    const int above_stride = push_up ? 2 * RQ : 2 * W * RQ, below_stride = push_dn ? 2 * RQ : 2 * W * RQ;
    // dt U for the lane's column that lies d = -2, 0, 2 or 4 beyond the row's
    // index in the warp, where that column is on the diagonal x1 = x2
    pair_t dU[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        const float v = x1_0 - x2_0 == 2 * d - 2 ? a.dtU : 0.f;
        dU[d] = pack2(v, v);
    }
    const float2 *rcw = rowc + lrow0;
    {
        // the stage counter runs on across realizations: the halo slots and
        // their mbarrier phases continue without a reset, and a neighbour can
        // never be more than one stage ahead
        unsigned tc = 0;
        // the warp's first and last rows to its neighbours: shared memory, and
        // from the slab's edges the neighbour CTAs (each edge warp arms the
        // barrier it will wait on itself, whose previous phase it has seen)
        auto publish = [&](const pair_t (&first)[CL], const pair_t (&last)[CL]) {
            const int par = tc & 1;
            ulonglong2 *eb = reinterpret_cast<ulonglong2 *>(edge_own + par * (2 * W * RQ));
#pragma unroll
            for (int k = 0; k < CL; k += 2) {
                eb[k * 16] = make_ulonglong2(first[k], first[k + 1]);
                eb[RQ + k * 16] = make_ulonglong2(last[k], last[k + 1]);
            }
            if (push_up) {
                if (lane == 0) mbar_expect_tx(mb_halo + par * 16, RQ * 16);
#pragma unroll
                for (int k = 0; k < CL; k += 2)
                    st_async16(send_up + par * (2 * RQ * 16) + k * 256, first[k], first[k + 1], send_up_mb + par * 16);
            }
            if (push_dn) {
                if (lane == 0) mbar_expect_tx(mb_halo + par * 16 + 8, RQ * 16);
#pragma unroll
                for (int k = 0; k < CL; k += 2)
                    st_async16(send_dn + par * (2 * RQ * 16) + k * 256, last[k], last[k + 1], send_dn_mb + par * 16);
            }
            __syncwarp();
            mbar_arrive_lane0(mb_edge, lane);
        };
        auto wait_edges = [&]() {
            if (!dead) dead = !mbar_wait_bounded(mb_edge, tc & 1, a.wait_limit_ns, a.status);
            if (push_up || push_dn) {
                const int par = tc & 1;
                const uint32_t phase = (tc >> 1) & 1;
                if (push_up && !dead) dead = !mbar_wait_bounded(mb_halo + par * 16, phase, a.wait_limit_ns, a.status);
                if (push_dn && !dead) dead = !mbar_wait_bounded(mb_halo + par * 16 + 8, phase, a.wait_limit_ns, a.status);
            }
        };
        auto load_row = [&](pair_t (&v)[CL], const float4 *src) {
#pragma unroll
            for (int k = 0; k < CL; k += 2) {
                const ulonglong2 f = *reinterpret_cast<const ulonglong2 *>(src + k * 16);
                v[k] = f.x;
                v[k + 1] = f.y;
            }
        };
        // the row above the warp's first and below its last row
        auto load_above = [&](pair_t (&v)[CL]) { load_row(v, above + (tc & 1) * above_stride); };
        auto load_below = [&](pair_t (&v)[CL]) { load_row(v, below + (tc & 1) * below_stride); };
#define CTQW_ROW(i, up, c, dn) \
    stencil_row<CL, i>(ec, nJc, rcw[i], rcw[(i) + 1], up, c, dn, dU, from_left, from_right, y)
        // one middle stage: the edge rows in place, the inner rows from one register set to the other
#define CTQW_MID(I1, I2, O1, O2)                    \
    {                                               \
        pair_t y[CL], nb[CL];                       \
        publish(P[0], P[3]);                        \
        CTQW_ROW(1, P[0], I1, I2);                  \
        horner_row<CL>(O1, Q[1], y, inv_j);         \
        CTQW_ROW(2, I1, I2, P[3]);                  \
        horner_row<CL>(O2, Q[2], y, inv_j);         \
        wait_edges();                               \
        load_above(nb);                             \
        CTQW_ROW(0, nb, P[0], I1);                  \
        horner_row<CL>(P[0], Q[0], y, inv_j);       \
        load_below(nb);                             \
        CTQW_ROW(3, I2, P[3], nb);                  \
        horner_row<CL>(P[3], Q[3], y, inv_j);       \
        ++tc;                                       \
    }
        // psi(t+dt) = psi + A w_2, the rounding error carried in lo
        auto update = [&](int i, const pair_t (&y)[CL]) {
#pragma unroll
            for (int k = 0; k < CL; k += 2) {
                const float2 y0 = unpack2(y[k]), y1 = unpack2(y[k + 1]);
                float2 h0 = unpack2(Q[i][k]), h1 = unpack2(Q[i][k + 1]);
                const float2 s0 = make_float2(y0.y, -y0.x), s1 = make_float2(y1.y, -y1.x);
                if (a.compensated) {
                    float4 *lp = los + (lrow0 + i) * RQ + k * 16 + lane;
                    const float4 l4 = *lp;
                    float2 l0 = make_float2(l4.x, l4.y), l1 = make_float2(l4.z, l4.w);
                    compensated_add2(h0, l0, s0);
                    compensated_add2(h1, l1, s1);
                    *lp = make_float4(l0.x, l0.y, l1.x, l1.y);
                } else {
                    h0 = make_float2(h0.x + s0.x, h0.y + s0.y);
                    h1 = make_float2(h1.x + s1.x, h1.y + s1.y);
                }
                Q[i][k] = pack2(h0.x, h0.y);
                Q[i][k + 1] = pack2(h1.x, h1.y);
            }
        };
        const int r_end = a.r0 + a.R_run;
        for (int r = next(); r < r_end; r = next()) {
            load_realization(r);
            if (SWITCH)
                cluster_barrier();   // every CTA has read the parameters that CTA 0 overwrites when it is done
            else
                __syncthreads();
            if (!active) continue;
            for (long long step = 0; step < n_steps; ++step) {
                if (K > 1) {
                    // the first stage: w_K from psi, which stays in place
                    const float inv_j = a.inv_j[K];
                    pair_t y[CL], nb[CL];
                    publish(Q[0], Q[3]);
                    CTQW_ROW(1, Q[0], Q[1], Q[2]);
                    horner_row<CL>(P[1], Q[1], y, inv_j);
                    CTQW_ROW(2, Q[1], Q[2], Q[3]);
                    horner_row<CL>(P[2], Q[2], y, inv_j);
                    wait_edges();
                    load_above(nb);
                    CTQW_ROW(0, nb, Q[0], Q[1]);
                    horner_row<CL>(P[0], Q[0], y, inv_j);
                    load_below(nb);
                    CTQW_ROW(3, Q[2], Q[3], nb);
                    horner_row<CL>(P[3], Q[3], y, inv_j);
                    ++tc;
                } else {
#pragma unroll
                    for (int i = 0; i < RL; ++i) {
#pragma unroll
                        for (int k = 0; k < CL; ++k) P[i][k] = Q[i][k];
                    }
                }
                int j = K - 1;
#pragma unroll 1
                while (j >= 2) {
                    float inv_j = a.inv_j[j];
                    CTQW_MID(P[1], P[2], T[0], T[1]);
                    if (--j < 2) {
#pragma unroll
                        for (int k = 0; k < CL; ++k) {
                            P[1][k] = T[0][k];
                            P[2][k] = T[1][k];
                        }
                        break;
                    }
                    inv_j = a.inv_j[j];
                    CTQW_MID(T[0], T[1], P[1], P[2]);
                    --j;
                }
                {
                    pair_t y[CL], nb[CL];
                    publish(P[0], P[3]);
                    CTQW_ROW(1, P[0], P[1], P[2]);
                    update(1, y);
                    CTQW_ROW(2, P[1], P[2], P[3]);
                    update(2, y);
                    wait_edges();
                    load_above(nb);
                    CTQW_ROW(0, nb, P[0], P[1]);
                    update(0, y);
                    load_below(nb);
                    CTQW_ROW(3, P[2], P[3], nb);
                    update(3, y);
                    ++tc;
                }
                if (SWITCH) {
                    // the Hamiltonian update: the warps with rows have read the
                    // coefficients of this step when they get here
                    const int threads = 32 * my_warps;
                    asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
                    for (int i = threadIdx.x; i < N; i += threads)
                        (void)switch_site(a.law, a.step0 + step, r, i, N, par[i], par[N + i]);
                    asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
                    coefficients(par, par + N);
                    asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
                }
                // a snapshot step: the new state to its slot, row-major like psi
                if (a.snap_every > 0 && step + 1 < n_steps && (step + 1) % a.snap_every == 0)
                    store_rows(a.snap + ((step + 1) / a.snap_every - 1) * a.snap_stride, r, false);
            }
            store_rows(a.psi, r, true);
            if (SWITCH && rank == 0) {
                const int64_t po = a.tab.par_off[r];
                for (int i = threadIdx.x; i < N; i += 32 * my_warps) {
                    a.eps_out[po + i] = par[i];
                    a.J_out[po + i] = par[N + i];
                    a.eps32_out[po + i] = (float)par[i];
                    a.J32_out[po + i] = (float)par[N + i];
                }
            }
        }
#undef CTQW_MID
#undef CTQW_ROW
    }
    cluster_barrier();   // no CTA leaves while a neighbour may still push into it
}

using RowsKernel = void (*)(RowsArgs);

struct RowsShape {
    int N, C, W, threads;
    size_t smem;
    RowsKernel kern, kern_switch;
};

constexpr int kRowsShapes = 3;

// Columns per lane for the lattice: the fewest that cover it, and on a ring
// divide it (0: none does).
int rows_columns(int N, int periodic) {
    for (int CL = 2; CL <= 8; CL += 2)
        if (N <= 32 * CL && (!periodic || (N % CL == 0 && N % 4 == 0))) return CL;
    return 0;
}

// Most warps a CTA: what one SM's registers hold (128 a thread for 16, 255
// for 8), so smaller CTAs share an SM.
int rows_max_warps(int CL) { return CL <= 4 ? 16 : 8; }

// The kernel for the lattice with at most maxw warps a CTA, evened out over
// the CTAs of the cluster.
bool rows_shape_for(int N, int periodic, int maxw, RowsShape &f) {
    const int CL = rows_columns(N, periodic);
    if (CL == 0 || maxw < 1) return false;
    switch (CL) {
        case 2: f.kern = taylor_fused_rows_kernel<2, 16, false>; f.kern_switch = taylor_fused_rows_kernel<2, 16, true>; break;
        case 4: f.kern = taylor_fused_rows_kernel<4, 16, false>; f.kern_switch = taylor_fused_rows_kernel<4, 16, true>; break;
        case 6: f.kern = taylor_fused_rows_kernel<6, 8, false>; f.kern_switch = taylor_fused_rows_kernel<6, 8, true>; break;
        default: f.kern = taylor_fused_rows_kernel<8, 8, false>; f.kern_switch = taylor_fused_rows_kernel<8, 8, true>; break;
    }
    f.N = N;
    const int units = (N + 3) / 4;
    f.C = (units + maxw - 1) / maxw;
    if (f.C > 16) return false;
    f.W = (units + f.C - 1) / f.C;
    f.C = (units + f.W - 1) / f.W;
    f.threads = 32 * f.W;
    f.smem = sizeof(float4) * 16 * CL * (size_t)(4 + 4 * f.W + 4 * f.W) + sizeof(float2) * (size_t)(4 * f.W + 2);
    return true;
}

// The same layout with switching noise: room for the parameters.
void with_switching(RowsShape &f) {
    f.kern = f.kern_switch;
    f.smem += sizeof(double) * 2 * (size_t)f.N;
}

// The kernels are shared by layouts of different sizes: the limit is always
// the device's, so that calls for two handles cannot undo each other's.
int set_rows_attributes(RowsKernel kern) {
    CTQW_CUDA_TRY(cudaFuncSetAttribute((const void *)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024 - 1024));
    CTQW_CUDA_TRY(cudaFuncSetAttribute((const void *)kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    return CTQW_OK;
}

int rows_residency(const RowsShape &f, int *clusters, int *per_sm) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)f.C);
    cfg.blockDim = dim3((unsigned)f.threads);
    cfg.dynamicSmemBytes = f.smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)f.C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    CTQW_CUDA_TRY(cudaOccupancyMaxActiveClusters(clusters, (const void *)f.kern, &cfg));
    CTQW_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, (const void *)f.kern, f.threads, f.smem));
    return CTQW_OK;
}

// Layout `shape` of the handle: 0 the planned one, 1 at most half and 2 three
// quarters of the most warps a CTA.
bool rows_shape_of(const ctqw_hamiltonian *h, int shape, RowsShape &f) {
    if (shape < 0 || shape >= kRowsShapes) return false;
    const int most = rows_max_warps(rows_columns(h->Nmax, h->periodic));
    return rows_shape_for(h->Nmax, h->periodic, shape == 0 ? h->rows_W : (shape == 1 ? most / 2 : most * 3 / 4), f);
}

}  // namespace

bool fused_rows_supported(const ctqw_hamiltonian *h, int dtype) { return dtype == CTQW_C64 && h->rows_clusters > 0; }

bool fused_rows_switching_supported(const ctqw_hamiltonian *h, int dtype) {
    return dtype == CTQW_C64 && h->rows_switch_clusters > 0;
}

// With many realizations the largest CTAs win by a little (fewest rows cross
// between SMs: N = 128, R = 4096: 1.33e12 site-updates/s against 1.28e12 with
// 8 warps).  With few, a realization spread over more SMs takes its stages
// faster.  A stage measured a + b w microseconds with w warps on the SM:
// (a, b) = (0.33, 0.011), (0.40, 0.034), (0.41, 0.035), (0.54, 0.042) for 2,
// 4, 6, 8 columns a lane (N = 128, R = 1: 0.94, 0.65, 0.56 with 16, 8, 4
// warps a CTA; N = 256: 0.88, 0.71 with 8, 4).  So: the time of the full
// rounds of resident clusters plus the last one, which has its SMs to itself
// as far as they go.
int plan_fused_rows(ctqw_hamiltonian *h) {
    RowsShape planned;
    if (h->m != 2 || !h->uniform || !rows_shape_for(h->Nmax, h->periodic, 16, planned)) return CTQW_OK;
    static const double a_of[5] = {0, 0.33, 0.40, 0.41, 0.54}, b_of[5] = {0, 0.011, 0.034, 0.035, 0.042};
    const int CL = rows_columns(h->Nmax, h->periodic);
    const double a = a_of[CL / 2], b = b_of[CL / 2];
    double best = 0.0;
    for (int maxw = rows_max_warps(CL); maxw >= rows_max_warps(CL) / 4; maxw /= 2) {
        RowsShape f;
        if (!rows_shape_for(h->Nmax, h->periodic, maxw, f)) continue;
        CTQW_TRY(set_rows_attributes(f.kern));
        int clusters = 0, per_sm = 0;
        CTQW_TRY(rows_residency(f, &clusters, &per_sm));
        if (clusters < 1 || per_sm < 1) continue;
        const int rounds = h->R / clusters, rest = h->R % clusters;
        const int alone = std::max(1, clusters / per_sm);   // clusters that find SMs of their own
        double t = rounds * (a + b * f.W * per_sm);
        if (rest) t += a + b * f.W * std::min(per_sm, (rest + alone - 1) / alone);
        if (best == 0.0 || t < 0.97 * best) {
            best = t;
            planned = f;
            h->rows_W = f.W;
            h->rows_C = f.C;
            h->rows_clusters = clusters;
            h->rows_per_sm = per_sm;
            h->rows_stage_us = a + b * f.W * per_sm;
        }
    }
    if (h->rows_clusters > 0) {
        with_switching(planned);
        int per_sm = 0;
        CTQW_TRY(set_rows_attributes(planned.kern));
        CTQW_TRY(rows_residency(planned, &h->rows_switch_clusters, &per_sm));
    }
    return CTQW_OK;
}

int fused_rows_split(const ctqw_hamiltonian *h, int shape, int K, int *R_tiled) {
    *R_tiled = 0;
    if (shape != 0 || h->rows_clusters < 1 || h->group_N.size() != 1 ||
        !tiled_supported(h, CTQW_C64, tiled_default_shape(h, K)))
        return CTQW_OK;
    const int clusters = h->rows_clusters, per_sm = h->rows_per_sm;
    int n_sm = 0;
    CTQW_CUDA_TRY(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, h->device));
    const int used = std::min(n_sm, (clusters * h->rows_C + per_sm - 1) / per_sm);
    const int idle = n_sm - used;
    if (idle * 16 < n_sm) return CTQW_OK;   // under 1/16 of the SMs idle: not worth a second stream
    // few SMs idle (clusters of 5 CTAs leave 12): at the launch the tiles may hold
    // an SM that a cluster needs, so only shares that take well under the clusters'
    // time (of 581 x N = 145 21 on the tiles: 60 steps 7.34 to 8 ms instead of 7.55;
    // 24 of 640 x 156: no gain; clusters of 6 leave 14: no such loss)
    const double margin = idle * 12 < n_sm ? 1.6 : 1.0;
    // two CTAs an SM: tiles that hold half an SM when the clusters are launched
    // keep some of them out for the whole launch (20 steps of K = 16, one stream
    // and with 8% on the tiles: 600 x N = 200 10.5 and 12.0 to 13.7 ms, 350 x 196
    // 6.3 and 6.8 to 8.3, 200 x 200 3.7 and 3.5 to 4.8)
    if (per_sm > 1) return CTQW_OK;
    // the rounds of resident clusters with the least time of the longer part, a
    // stage: so many rounds of clusters, against so many rounds of tile blocks on
    // the SMs left over
    int blocks = 0;   // of a realization, and resident on an SM
    int resident = 1;
    const double round_us = tiled_round_us(h, K, &blocks, &resident);
    const int most = (h->R + clusters - 1) / clusters;
    int R_f = h->R;
    double best = most * h->rows_stage_us;
    for (int rounds = std::max(1, most / 2); rounds < most; ++rounds) {
        const int64_t all = (int64_t)(h->R - rounds * clusters) * blocks, at_once = idle * resident;
        double tile_rounds = (double)(all / at_once);
        if (all % at_once) tile_rounds += 0.6 + 0.4 * (double)(all % at_once) / at_once;   // fewer blocks an SM, a little sooner
        const double t = std::max(rounds * h->rows_stage_us, margin * tile_rounds * round_us);
        if (t < best) {
            best = t;
            R_f = rounds * clusters;
        }
    }
    *R_tiled = h->R - R_f;
    return CTQW_OK;
}

static int launch_rows(const ctqw_hamiltonian *h, void *psi, void *lo, void *snap, int snap_every, double dt, int K,
                       int64_t n_steps, int compensated, int shape, int test_timeout, int r0, int R_run, int *work,
                       const SwitchLaw *law, int64_t step0, cudaStream_t s) {
    RowsShape f;
    if (!rows_shape_of(h, shape, f)) {
        ctqw_set_error("fused path: unsupported size N=%d or shape %d", h->Nmax, shape);
        return CTQW_EUNSUPPORTED;
    }
    if (K > kMaxK) {
        ctqw_set_error("fused path: K=%d above %d", K, kMaxK);
        return CTQW_EUNSUPPORTED;
    }
    if (r0 < 0 || R_run < 0 || r0 + R_run > h->R) {
        ctqw_set_error("fused path: realizations %d..%d outside 0..%d", r0, r0 + R_run, h->R);
        return CTQW_EINVAL;
    }
    if (R_run == 0) return CTQW_OK;
    RowsArgs a;
    a.eps = h->eps64;
    a.J = h->J64;
    a.tab = real_table(h);
    a.psi = (float2 *)psi;
    a.lo = (float2 *)lo;
    a.snap = (float2 *)snap;
    a.snap_every = snap ? snap_every : 0;
    a.snap_stride = h->total_amp;
    a.dt = dt;
    a.dtU = (float)(dt * h->U);
    a.N = h->Nmax;
    a.W = f.W;
    // even rows, and states that start on 16 bytes (N^2 amplitudes each)
    a.vec = h->Nmax % 2 == 0 && (((uintptr_t)psi | (uintptr_t)lo | (uintptr_t)snap) & 15) == 0;
    a.K = K;
    a.n_steps = n_steps;
    a.compensated = compensated;
    a.status = h->status_d;
    a.test_timeout = test_timeout;
    a.wait_limit_ns = 2000000000ull;
    a.r0 = r0;
    a.R_run = R_run;
    a.step0 = (unsigned long long)step0;
    if (law) {
        a.law = *law;
        a.eps_out = h->eps64;
        a.J_out = h->J64;
        a.eps32_out = h->eps32;
        a.J32_out = h->J32;
        with_switching(f);
    }
    a.inv_j[0] = 0.f;
    for (int j = 1; j <= kMaxK; ++j) a.inv_j[j] = (float)(1.0 / j);
    CTQW_TRY(set_rows_attributes(f.kern));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)f.C);
    cfg.blockDim = dim3((unsigned)f.threads);
    cfg.dynamicSmemBytes = f.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)f.C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = law ? h->rows_switch_clusters : h->rows_clusters, per_sm = 0;
    if (shape != 0) CTQW_TRY(rows_residency(f, &clusters, &per_sm));
    if (clusters < 1) {
        ctqw_set_error("fused path: no cluster of %d CTAs x %d threads fits", f.C, f.threads);
        return CTQW_EUNSUPPORTED;
    }
    // one cluster per resident slot
    cfg.gridDim = dim3((unsigned)(std::min(R_run, clusters) * f.C));
    a.work = R_run > clusters ? work : nullptr;
    if (a.work) CTQW_CUDA_TRY(cudaMemsetAsync(a.work, 0, sizeof(int), s));
    CTQW_CUDA_TRY(cudaLaunchKernelEx(&cfg, f.kern, a));
    return CTQW_OK;
}

int launch_taylor_fused_rows(const ctqw_hamiltonian *h, void *psi, void *lo, void *snap, int snap_every, double dt,
                             int K, int64_t n_steps, int compensated, int shape, int test_timeout, int r0,
                             int R_run, int *work, cudaStream_t s) {
    return launch_rows(h, psi, lo, snap, snap_every, dt, K, n_steps, compensated, shape, test_timeout, r0, R_run, work,
                       nullptr, 0, s);
}

int launch_taylor_fused_rows_switching(const ctqw_hamiltonian *h, void *psi, void *lo, double dt, int K,
                                       int64_t step0, int64_t n_steps, int compensated, const SwitchLaw &law,
                                       int *work, cudaStream_t s) {
    return launch_rows(h, psi, lo, nullptr, 0, dt, K, n_steps, compensated, 0, 0, 0, h->R, work, &law, step0, s);
}

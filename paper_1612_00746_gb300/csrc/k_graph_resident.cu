// Two particles on a small graph in complex FP32: all steps between two
// samples in one launch, the Horner iterate on chip.
//
// One launch per stage reads, per amplitude, its neighbours and their hoppings
// through L1 and L2 (136 bytes on a torus, near 20 TB/s) and streams two states
// through HBM; that L1 and L2 traffic bounded it.  Here a cluster of CTAs owns
// one realization: CTA k holds the rows x_1 of its share of nodes, all x_2, of
// two iterates (read and written in turn, one cluster barrier a stage).  A
// thread owns one or two columns x_2 of consecutive rows: the links of particle
// 2 and their hoppings stay in its registers for the whole launch, the links
// of particle 1 are the same for a whole warp and come from a small table by
// broadcast, and those to the row before and after are in its registers too.
// Rows of another CTA are read from its shared memory.  psi and its carried
// error pass through global memory (L2) once a stage and once a step, each
// amplitude by its own thread only, in [r][s] order (the state's own order has
// the realizations fastest; a transpose at either end of the launch).
//
// What bounds it is shared memory: about 23 wavefronts a warp, row and column,
// of the 26 to 31 clocks that takes (on one CTA a realization; with clusters
// the other CTA's rows and the barrier add a few).  10 steps of K = 16, samples
// at 0, 5, 10, one launch a stage -> this kernel: 15 x 15 torus, 1000
// realizations 56.1 -> 37.9 ms (1.44e11 -> 2.14e11 site-updates/s), 76 of them
// 7.50 -> 3.87, one 2.20 -> 1.53; 16 x 16, 300 27.2 -> 14.1; 10 x 10, 600 7.98
// -> 3.97; 8 x 8, 1500 8.24 -> 3.34, 20 1.29 -> 0.56; 3 x 3, 1500 1.11 -> 0.46;
// ring of 225, 300 17.3 -> 8.5.  Wider threads (4 columns, 128 registers, 16
// warps) took 33.7 ms where 2 columns and 20 warps take 33.4; 2 columns and 16
// warps 35.3; particle 1's other links two at a time 34.3.
#include <algorithm>
#include <cstdlib>
#include <type_traits>

#include "fused_common.cuh"
#include "graph_internal.cuh"

namespace {

using namespace fused;

constexpr int kMaxK = 30;
// 96 registers a thread hold two columns of up to 4 links each; up to 8 need 128
constexpr int max_threads(int deg) { return deg <= 4 ? 640 : 512; }
constexpr size_t kMaxSmem = 227 * 1024;

struct ResidentArgs {
    GraphView g;
    const float *eps, *w;   // [N][Rp], [nnz][Rp]
    float2 *psi, *lo;       // [r][D]
    int CL, rows, CW, G;    // CTAs a realization, rows a CTA, threads a row, rows at a time
    int64_t n_steps;
    int K;
    float U;
    float coef[kMaxK + 1];  // dt / j
};

// What particle 1 needs at a row: hoppings (negated) to the rows before and
// after it where the same thread owns those (their amplitudes are then in its
// registers), the on-site energy, and n | 16 (row before linked) | 32 (row
// after linked), n the number of other links; those follow in their own table.
struct RowHead {
    float Jprev, Jnext, e;
    uint32_t bits;
};
struct RowLink {
    uint32_t at;   // address of the other row, in the cluster's window
    float J;
};

// (and 1 KB, which lanes past the last column may read)
inline size_t table_bytes(int rows, int deg) { return (size_t)rows * (sizeof(RowHead) + deg * sizeof(RowLink)) + 1024; }

__device__ __forceinline__ float2 lds2(uint32_t a) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}
template <bool CLUSTER>
__device__ __forceinline__ float2 ld_row(uint32_t a) {
    float2 v;
    if (CLUSTER)
        asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    else
        v = lds2(a);
    return v;
}
__device__ __forceinline__ void sts2(uint32_t a, float2 v) {
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void axpy(float2 &y, float J, float2 v) {
    y.x = fmaf(J, v.x, y.x);
    y.y = fmaf(J, v.y, y.y);
}

// DEG: links a node at most; NC: columns a thread, 32 apart; CLUSTER: more
// than one CTA a realization.
template <int DEG, int NC, bool CLUSTER>
__global__ void __launch_bounds__(max_threads(DEG), 1) graph_resident_kernel(const __grid_constant__ ResidentArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int N = a.g.N;
    const int rank = CLUSTER ? (int)cluster_rank() : 0;
    const int64_t r = a.g.r_begin + blockIdx.x / a.CL;
    const int row0 = rank * a.rows, n_rows = max(0, min(a.rows, N - row0));
    // a lane past the last column reads on into the next row, or the tables;
    // what it makes of that is not stored
    const uint32_t bytes = (uint32_t)a.rows * N * 8, buf = smem_u32(smem);
    RowHead *heads = (RowHead *)(smem + 2 * (size_t)bytes);
    RowLink *links = (RowLink *)(heads + a.rows);
    const int64_t Rp = a.g.Rp;
    // rows first .. last - 1 of group grp
    const int grp = threadIdx.x / a.CW, tx = threadIdx.x - grp * a.CW;
    const int first = n_rows * grp / a.G, last = n_rows * (grp + 1) / a.G;
    const int col = (tx & ~31) * NC + (tx & 31);   // and col + 32, ...

    for (int row = first + tx; row < last; row += a.CW) {
        RowHead h{0.f, 0.f, a.eps[(int64_t)(row0 + row) * Rp + r], 0};
        int n = 0;
        for (int k = a.g.row_ptr[row0 + row]; k < a.g.row_ptr[row0 + row + 1]; ++k) {
            const int c = a.g.col[k], owner = c / a.rows, at = c - owner * a.rows;
            const float J = -a.w[(int64_t)k * Rp + r];
            if (owner == rank && at == row - 1 && row > first && !(h.bits & 16u)) {
                h.Jprev = J;
                h.bits |= 16u;
            } else if (owner == rank && at == row + 1 && row + 1 < last && !(h.bits & 32u)) {
                h.Jnext = J;
                h.bits |= 32u;
            } else {
                const uint32_t p = buf + (uint32_t)at * N * 8;
                links[row * DEG + n++] = RowLink{owner == rank ? p : map_rank(p, (uint32_t)owner), J};
            }
        }
        h.bits |= (uint32_t)n;
        heads[row] = h;
    }

    bool own[NC];
    float e2[NC];
    uint32_t off[NC][DEG];
    float J2[NC][DEG];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        own[c] = col + 32 * c < N;
        const int x = own[c] ? col + 32 * c : N - 1;
        e2[c] = a.eps[(int64_t)x * Rp + r];
        const int k0 = a.g.row_ptr[x], k1 = a.g.row_ptr[x + 1];
#pragma unroll
        for (int d = 0; d < DEG; ++d) {   // padded with zero hoppings to itself
            const bool link = k0 + d < k1;
            off[c][d] = (uint32_t)(link ? a.g.col[k0 + d] : x) * 8;
            J2[c][d] = link ? -a.w[(int64_t)(k0 + d) * Rp + r] : 0.f;
        }
    }
    const int64_t mine = r * a.g.D + (int64_t)(row0 + first) * N + col;
    for (int row = first; row < last; ++row)
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (own[c]) sts2(buf + (uint32_t)(row * N + col + 32 * c) * 8, a.psi[mine + (row - first) * N + 32 * c]);

    auto sync = [&]() {
        if (CLUSTER)
            cluster_barrier();
        else
            __syncthreads();
    };
    // One stage over the thread's rows, from the buffer at offset flip to the
    // other one.  A row's table entry, centre and psi are read a row ahead, the
    // first row's entry and psi before the barrier that ends a stage.
    RowHead h{};
    float2 qn[NC];
    float2 *const psi0 = a.psi + mine, *const lo0 = a.lo + mine;
    auto ahead = [&](const float2 *psi) {
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (own[c]) qn[c] = psi[32 * c];
    };
    auto stage = [&](uint32_t flip, auto final, float coef) {
        constexpr bool kFinal = decltype(final)::value;
        if (first >= last) return;
        uint32_t at = buf + flip + (uint32_t)first * N * 8;               // the row
        uint32_t to = buf + (bytes - flip) + (uint32_t)(first * N + col) * 8;   // where its result goes
        uint32_t link = smem_u32(links + first * DEG);
        const uint32_t shift = flip + (uint32_t)col * 8;
        float2 *psi = psi0, *lo = lo0;
        float2 prev[NC], cur[NC], next[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            next[c] = prev[c] = cur[c] = lds2(at + (uint32_t)(col + 32 * c) * 8);
        }
        int diag = col - (row0 + first);   // 0 or -32 c where the two particles meet
#pragma unroll 1
        for (int row = first; row < last; ++row) {
            const RowHead hh = h;
            h = heads[row + 1 < last ? row + 1 : first];
            float2 y[NC], lw[NC], q[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) q[c] = qn[c];
            if (kFinal) {
#pragma unroll
                for (int c = 0; c < NC; ++c)
                    if (own[c]) lw[c] = lo[32 * c];
            }
            if (row + 1 < last) {
                ahead(psi + N);
#pragma unroll
                for (int c = 0; c < NC; ++c) next[c] = lds2(at + (uint32_t)(N + col + 32 * c) * 8);
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                float v = hh.e + e2[c];
                if (diag == -32 * c) v += a.U;
                y[c] = make_float2(v * cur[c].x, v * cur[c].y);
            }
#pragma unroll
            for (int c = 0; c < NC; ++c)
#pragma unroll
                for (int d = 0; d < DEG; ++d) axpy(y[c], J2[c][d], lds2(at + off[c][d]));
            if (hh.bits & 16u)
#pragma unroll
                for (int c = 0; c < NC; ++c) axpy(y[c], hh.Jprev, prev[c]);
            if (hh.bits & 32u)
#pragma unroll
                for (int c = 0; c < NC; ++c) axpy(y[c], hh.Jnext, next[c]);
            for (uint32_t d = 0; d < (hh.bits & 15u); ++d) {
                const float2 l = lds2(link + d * 8);
                const uint32_t p = __float_as_uint(l.x) + shift;
#pragma unroll
                for (int c = 0; c < NC; ++c) axpy(y[c], l.y, ld_row<CLUSTER>(p + 256 * c));
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                if (own[c]) {
                    if (!kFinal) {   // psi + coef (-i) y
                        sts2(to + 256 * c, make_float2(fmaf(coef, y[c].y, q[c].x), fmaf(-coef, y[c].x, q[c].y)));
                    } else {         // (psi, lo) += -i dt y
                        compensated_add2(q[c], lw[c], make_float2(coef * y[c].y, -coef * y[c].x));
                        psi[32 * c] = q[c];
                        lo[32 * c] = lw[c];
                        sts2(to + 256 * c, q[c]);
                    }
                }
                prev[c] = cur[c];
                cur[c] = next[c];
            }
            psi += N;
            if (kFinal) lo += N;
            at += (uint32_t)N * 8;
            to += (uint32_t)N * 8;
            link += DEG * (uint32_t)sizeof(RowLink);
            --diag;
        }
        ahead(psi0);
    };
    sync();
    if (first < last) {
        h = heads[first];
        ahead(psi0);
    }
    uint32_t flip = 0;
    for (int64_t step = 0; step < a.n_steps; ++step) {
        for (int j = a.K; j >= 2; --j) {
            stage(flip, std::false_type{}, a.coef[j]);
            flip = bytes - flip;
            sync();
        }
        stage(flip, std::true_type{}, a.coef[1]);
        flip = bytes - flip;
        sync();   // also: no CTA leaves while another reads its rows
    }
}

// out[c][r] = in[r][c] for one 32 x 32 tile: n_r rows of stride in_ld, n_c
// columns.
__global__ void __launch_bounds__(256) graph_transpose_kernel(const float2 *__restrict__ in, int64_t in_ld,
                                                              float2 *__restrict__ out, int64_t out_ld, int n_r,
                                                              int n_c) {
    __shared__ float2 t[32][33];
    const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32, lane = threadIdx.x & 31, y = threadIdx.x >> 5;
    for (int k = y; k < 32; k += 8)
        if (r0 + k < n_r && c0 + lane < n_c) t[k][lane] = in[(int64_t)(r0 + k) * in_ld + c0 + lane];
    __syncthreads();
    for (int k = y; k < 32; k += 8)
        if (c0 + k < n_c && r0 + lane < n_r) out[(int64_t)(c0 + k) * out_ld + r0 + lane] = t[lane][k];
}

using ResidentKernel = void (*)(const ResidentArgs);

struct ResidentShape {
    ResidentKernel kern = nullptr;
    int deg = 0, nc = 0, CW = 0;
};

ResidentShape resident_shape(int N, int max_deg, int CL) {
    ResidentShape f;
    f.deg = max_deg <= 2 ? 2 : max_deg <= 4 ? 4 : max_deg <= 6 ? 6 : 8;
    if (max_deg > 8) return f;
    f.nc = N > 32 ? 2 : 1;
    f.CW = ((N + f.nc - 1) / f.nc + 31) / 32 * 32;
    if (f.CW > max_threads(f.deg)) return f;
#define PICK(DEG) (f.nc == 2 ? KERN(DEG, 2) : KERN(DEG, 1))
#define KERN(DEG, NC) (CL > 1 ? graph_resident_kernel<DEG, NC, true> : graph_resident_kernel<DEG, NC, false>)
    f.kern = f.deg == 2 ? PICK(2) : f.deg == 4 ? PICK(4) : f.deg == 6 ? PICK(6) : PICK(8);
#undef KERN
#undef PICK
    return f;
}

cudaLaunchConfig_t resident_config(cudaLaunchAttribute *attr, int CL, int threads, size_t smem) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)CL);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

}  // namespace

// The plan of least time by a model in clocks a stage, fitted on tori of 64 to
// 324 nodes and on rings with chords, 8 to 1500 realizations, every CL that
// fits: 17 a warp, row and column on an SM (the shared-memory pipe), per row
// of a thread 100 + 60 for each link read there + 400 for each in another CTA,
// and a barrier.  It is within 20 % of what those took.  None where one launch
// a stage is faster: that takes some 5 us and 24 links + 40 bytes an amplitude
// at 19.6 TB/s (links of the mean node: only here every node is padded to the
// most links), measured the same way; so graphs of many or uneven links that
// cluster CTAs cannot hold near each other stay there (127 x 222 nodes of 0 to 8
// links, 2.9 on average, K = 17, 5 steps: 5.1 ms with a launch a stage, 6.3 here).
int plan_graph_resident(ctqw_graph *g, const int32_t *row_ptr, const int32_t *col, int max_deg) {
    g->res_CL = 0;
    if (g->m != 2) return CTQW_OK;
    double least = ((24.0 * row_ptr[g->N] / g->N + 40.0) * g->D * g->R / 19.6e12 + 5e-6) * 1.92e9;
    int n_sm = 0;
    CTQW_CUDA_TRY(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, g->device));
    bool enough = false;   // realizations for every SM already
    for (int CL = 1; CL <= 16 && !enough; CL += CL < 8 ? 1 : 2) {
        const ResidentShape f = resident_shape(g->N, max_deg, CL);
        if (!f.kern) return CTQW_OK;
        const int rows = (g->N + CL - 1) / CL;
        const size_t smem = 2 * (size_t)rows * g->N * 8 + table_bytes(rows, f.deg);
        if (smem > kMaxSmem || (CL > 1 && rows < 2)) continue;
        enough = (int64_t)g->R * CL >= 4 * n_sm && g->res_CL > 0;
        CTQW_CUDA_TRY(cudaFuncSetAttribute((const void *)f.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem));
        CTQW_CUDA_TRY(cudaFuncSetAttribute((const void *)f.kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        double here = 0.0, away = 0.0;   // links a row, read from this CTA and from others
        for (int x = 0; x < g->N; ++x)
            for (int k = row_ptr[x]; k < row_ptr[x + 1]; ++k) {
                if (col[k] / rows != x / rows) away += 1.0 / g->N;
                else if (std::abs(col[k] - x) != 1) here += 1.0 / g->N;
            }
        const int most = std::min(max_threads(f.deg) / f.CW, rows);
        for (int G = most; G >= 1 && G > most / 8; G /= 2) {
            auto cost_of = [&](int clusters) {
                const double per_sm = std::max(1.0, (double)std::min(clusters, g->R) * CL / n_sm);
                const double stage = 17.0 * per_sm * rows * (f.CW / 32) * f.nc +
                                     (100.0 + 60.0 * here + 400.0 * away) * ((rows + G - 1) / G) + (CL == 1 ? 300.0 : 1700.0);
                return stage * ((g->R + clusters - 1) / clusters);
            };
            // ask for the residency only of what could be the best
            const int per_sm_most = std::min(2048 / (f.CW * G), (int)(kMaxSmem / smem));
            bool hopeful = false;
            for (int q = 1; q <= per_sm_most; ++q) hopeful |= cost_of(std::max(1, n_sm * q / CL)) < least;
            if (!hopeful) continue;
            cudaLaunchAttribute attr[1];
            cudaLaunchConfig_t cfg = resident_config(attr, CL, f.CW * G, smem);
            int clusters = 0;
            if (cudaOccupancyMaxActiveClusters(&clusters, (const void *)f.kern, &cfg) != cudaSuccess) {
                cudaGetLastError();   // a size this device does not take
                continue;
            }
            if (clusters < 1) continue;
            const double cost = cost_of(clusters);
            if (cost < least) {
                least = cost;
                g->res_CL = CL;
                g->res_G = G;
                g->res_deg = max_deg;
            }
        }
    }
    return CTQW_OK;
}

int launch_graph_resident(const ctqw_graph *g, int rb, int re, void *psi, void *lo, double dt, int K, int64_t n_steps,
                          cudaStream_t s) {
    const ResidentShape f = resident_shape(g->N, g->res_deg, g->res_CL);
    ResidentArgs a;
    a.g = graph_view(g, rb, re);
    a.eps = g->eps32;
    a.w = g->w32;
    a.psi = (float2 *)psi;
    a.lo = (float2 *)lo;
    a.CL = g->res_CL;
    a.rows = (g->N + a.CL - 1) / a.CL;
    a.CW = f.CW;
    a.G = g->res_G;
    a.n_steps = n_steps;
    a.K = K;
    a.U = (float)g->U;
    for (int j = 1; j <= K; ++j) a.coef[j] = (float)(dt / j);
    const size_t smem = 2 * (size_t)a.rows * g->N * 8 + table_bytes(a.rows, f.deg);
    CTQW_CUDA_TRY(cudaFuncSetAttribute((const void *)f.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem));
    CTQW_CUDA_TRY(cudaFuncSetAttribute((const void *)f.kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = resident_config(attr, a.CL, f.CW * a.G, smem);
    cfg.gridDim = dim3((unsigned)((re - rb) * a.CL));
    cfg.stream = s;
    CTQW_CUDA_TRY(cudaLaunchKernelEx(&cfg, f.kern, a));
    return CTQW_OK;
}

int launch_graph_to_rows(const ctqw_graph *g, int rb, int re, const void *psi, void *psi_t, cudaStream_t s) {
    const int n = re - rb, D = (int)g->D;
    for (int s0 = 0; s0 < D; s0 += 65535 * 32) {
        const int m = std::min(D - s0, 65535 * 32);
        graph_transpose_kernel<<<dim3((unsigned)((n + 31) / 32), (unsigned)((m + 31) / 32)), 256, 0, s>>>(
            (const float2 *)psi + (int64_t)s0 * g->Rp + rb, g->Rp, (float2 *)psi_t + (int64_t)rb * g->D + s0, g->D, m, n);
        CTQW_CUDA_TRY(cudaGetLastError());
    }
    return CTQW_OK;
}

int launch_graph_from_rows(const ctqw_graph *g, int rb, int re, const void *psi_t, void *psi, cudaStream_t s) {
    const int n = re - rb, D = (int)g->D;
    for (int r0 = 0; r0 < n; r0 += 65535 * 32) {
        const int m = std::min(n - r0, 65535 * 32);
        graph_transpose_kernel<<<dim3((unsigned)((D + 31) / 32), (unsigned)((m + 31) / 32)), 256, 0, s>>>(
            (const float2 *)psi_t + (int64_t)(rb + r0) * g->D, g->D, (float2 *)psi + rb + r0, g->Rp, m, D);
        CTQW_CUDA_TRY(cudaGetLastError());
    }
    return CTQW_OK;
}

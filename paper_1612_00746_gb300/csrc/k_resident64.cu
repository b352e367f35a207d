// FP64 propagation of small two-particle states, resident on chip: a cluster
// of CTAs owns one realization for all steps of the launch (the polynomial of
// Algorithm 3, Sec. 2.3, in Horner form, as launch_horner_f64).
//
// One launch per term costs about 4 microseconds however little it does; at
// N = 64 and 8 realizations the FP64 pipes need 0.6 for it.  Here a term is a
// stage between two cluster barriers: every CTA holds a slab of rows of the
// iterate in shared memory (two copies, read and written in turn) with one
// row of its neighbours on either side, each thread computes its amplitudes
// and the threads of the slab's first and last rows also store theirs into
// the neighbour CTAs.  psi of the step and the diagonal stay in registers.
// 12 FP64 operations an amplitude: 10 for dt H w, 2 to add it to psi; the FP64
// pipe (2 operations a clock and SM) and the barrier take about equal parts.
// 8 realizations of N = 64, K = 12, 200 steps sampled every 10: 10.4 ms with
// a launch per term (15.0 ms in the forward order), 4.4 ms here.
#include <algorithm>
#include <cmath>

#include "ctqw_internal.cuh"
#include "fused_common.cuh"

namespace {

using namespace fused;

constexpr int kThreads = 256;

struct ResidentArgs {
    RealTable tab;
    const double *eps, *J;
    double2 *psi;
    double dt;
    int N, SR, C;            // sites, rows a CTA (fewer in the last), CTAs a cluster
    int K;
    long long n_steps;
    double inv_j[31];
};

static __device__ __forceinline__ void st_cluster(uint32_t addr, double2 v) {
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(addr), "d"(v.x), "d"(v.y) : "memory");
}

// EPT: amplitudes a thread.
template <int EPT>
__global__ void __launch_bounds__(kThreads) resident_f64_kernel(const __grid_constant__ ResidentArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = a.N, SR = a.SR, C = a.C;
    const int rank = (int)cluster_rank();
    const int r = (int)blockIdx.x / C;
    const int row0 = rank * SR, rows = min(SR, N - row0);
    // rows 1 .. rows are the slab's, 0 and rows + 1 its neighbours'
    double2 *buf[2];
    buf[0] = reinterpret_cast<double2 *>(smem_raw);
    buf[1] = buf[0] + (SR + 2) * N;
    double *js = reinterpret_cast<double *>(buf[1] + (SR + 2) * N);   // [N] -dt J of the bond right of x
    const int64_t po = a.tab.par_off[r], base = a.tab.st_off[r];
    const double dt = a.dt;
    double2 *psi = a.psi + base;
    for (int x = threadIdx.x; x < N; x += kThreads) js[x] = -dt * a.J[po + x];
    for (int e = threadIdx.x; e < (rows + 2) * N; e += kThreads) {
        const int i = e / N, x2 = e - i * N;
        int x1 = row0 + i - 1;
        x1 = x1 < 0 ? N - 1 : (x1 >= N ? x1 - N : x1);
        buf[0][e] = psi[(int64_t)x1 * N + x2];
    }
    // where the first and last rows go: the row below the slab above and the
    // row above the slab below
    const int up = (rank + C - 1) % C, dn = (rank + 1) % C;
    const int rows_up = min(SR, N - up * SR);
    uint32_t to_up[2], to_dn[2];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        to_up[b] = map_rank(smem_u32(buf[b] + (rows_up + 1) * N), up);
        to_dn[b] = map_rank(smem_u32(buf[b]), dn);
    }
    __syncthreads();
    // the thread's amplitudes: place in the slab, psi, diagonal
    int at[EPT], x2s[EPT], rw[EPT];
    double2 q[EPT];
    double v[EPT];
#pragma unroll
    for (int k = 0; k < EPT; ++k) {
        const int e = threadIdx.x + k * kThreads;
        const bool in = e < rows * N;
        const int i = in ? e / N : 0, x2 = in ? e - i * N : 0;
        rw[k] = in ? i : -1;
        x2s[k] = x2;
        at[k] = (i + 1) * N + x2;
        q[k] = buf[0][at[k]];
        v[k] = dt * (a.eps[po + row0 + i] + a.eps[po + x2]) + (row0 + i == x2 ? dt * a.tab.U : 0.0);
    }
    cluster_barrier();   // every slab is in place before a neighbour stores into it
    int cur = 0;
    for (long long step = 0; step < a.n_steps; ++step) {
#pragma unroll 1
        for (int j = a.K; j >= 1; --j) {
            const double2 *w = buf[cur];
            double2 *o = buf[cur ^ 1];
            const double c = a.inv_j[j];
#pragma unroll
            for (int k = 0; k < EPT; ++k) {
                if (rw[k] < 0) continue;
                const int x2 = x2s[k], x1 = row0 + rw[k];
                const int left = x2 == 0 ? at[k] + N - 1 : at[k] - 1, right = x2 == N - 1 ? at[k] - N + 1 : at[k] + 1;
                const double jl = js[x2 == 0 ? N - 1 : x2 - 1], jr = js[x2];
                const double ju = js[x1 == 0 ? N - 1 : x1 - 1], jd = js[x1];
                const double2 wc = w[at[k]], wu = w[at[k] - N], wd = w[at[k] + N], wl = w[left], wr = w[right];
                double yr = v[k] * wc.x, yi = v[k] * wc.y;
                yr = fma(ju, wu.x, yr);
                yi = fma(ju, wu.y, yi);
                yr = fma(jd, wd.x, yr);
                yi = fma(jd, wd.y, yi);
                yr = fma(jl, wl.x, yr);
                yi = fma(jl, wl.y, yi);
                yr = fma(jr, wr.x, yr);
                yi = fma(jr, wr.y, yi);
                const double2 n = make_double2(fma(c, yi, q[k].x), fma(-c, yr, q[k].y));
                o[at[k]] = n;
                if (rw[k] == 0) st_cluster(to_up[cur ^ 1] + (uint32_t)x2 * 16u, n);
                if (rw[k] == rows - 1) st_cluster(to_dn[cur ^ 1] + (uint32_t)x2 * 16u, n);
                if (j == 1) q[k] = n;
            }
            cur ^= 1;
            cluster_barrier();
        }
    }
#pragma unroll
    for (int k = 0; k < EPT; ++k)
        if (rw[k] >= 0) psi[(int64_t)(row0 + rw[k]) * N + x2s[k]] = q[k];
}

using ResidentKernel = void (*)(ResidentArgs);

struct ResidentShape {
    int C, SR, ept;
    size_t smem;
    ResidentKernel kern;
};

bool resident_shape(int N, int C_max, ResidentShape &f) {
    f.SR = (N + C_max - 1) / C_max;
    f.C = (N + f.SR - 1) / f.SR;
    const int need = (f.SR * N + kThreads - 1) / kThreads;
    if (need <= 1) { f.ept = 1; f.kern = resident_f64_kernel<1>; }
    else if (need <= 2) { f.ept = 2; f.kern = resident_f64_kernel<2>; }
    else if (need <= 3) { f.ept = 3; f.kern = resident_f64_kernel<3>; }
    else if (need <= 4) { f.ept = 4; f.kern = resident_f64_kernel<4>; }
    else if (need <= 6) { f.ept = 6; f.kern = resident_f64_kernel<6>; }
    else if (need <= 8) { f.ept = 8; f.kern = resident_f64_kernel<8>; }
    else return false;
    f.smem = sizeof(double2) * 2 * (size_t)(f.SR + 2) * N + sizeof(double) * N;
    return f.smem <= 226 * 1024;
}

}  // namespace

// A stage takes about 0.5 us of barrier and latency and 0.0029 us for every
// amplitude on the busiest SM (12 operations, 2 a clock); a launch per term
// about 4.1 us and 2.6e-5 us an amplitude.  Clusters of 16 fit 7 of the GPCs
// (19 SMs each), smaller ones spread over all SMs, evenly while 120 of them suffice.  Measured, us a stage
// (per term; 4, 8, 16 CTAs): N = 32, R = 8: 4.12; 1.19, 0.86, 0.89; N = 64,
// R = 8: 4.13; 3.56, 2.02, 1.63; N = 64, R = 32: 8.22; 3.58, 3.26, 3.92;
// N = 128, R = 1: 4.12; -, 6.83, 3.60; N = 128, R = 16: 10.4; -, 12.8, 10.2.
int resident_f64_ctas(const ctqw_hamiltonian *h) {
    if (h->m != 2 || !h->uniform) return 0;
    const int N = h->Nmax, R = h->R;
    double best = 4.1 + 2.6e-5 * R * (double)N * N;
    int ctas = 0;
    for (int C_max : {16, 8, 4}) {
        ResidentShape f;
        if (!resident_shape(N, C_max, f)) continue;
        const double share = f.C > 8 ? std::ceil((R + 6) / 7 * f.C / 19.0) : std::max(std::ceil(R * (double)f.C / 148.0), R > 120 / f.C ? 2.0 : 1.0);
        const double t = 0.5 + 0.0029 * f.SR * N * share;
        if (t < best) {
            best = t;
            ctas = C_max;
        }
    }
    return ctas;
}

int launch_resident_f64(const ctqw_hamiltonian *h, int C_max, void *psi, double dt, int K, int64_t n_steps,
                        cudaStream_t s) {
    ResidentShape f;
    if (!resident_shape(h->Nmax, C_max, f)) {
        ctqw_set_error("resident FP64 path: N = %d does not fit %d CTAs", h->Nmax, C_max);
        return CTQW_EUNSUPPORTED;
    }
    ResidentArgs a;
    a.tab = real_table(h);
    a.eps = h->eps64;
    a.J = h->J64;
    a.psi = (double2 *)psi;
    a.dt = dt;
    a.N = h->Nmax;
    a.SR = f.SR;
    a.C = f.C;
    a.K = K;
    a.n_steps = n_steps;
    a.inv_j[0] = 0.0;
    for (int j = 1; j <= 30; ++j) a.inv_j[j] = 1.0 / j;
    CTQW_CUDA_TRY(cudaFuncSetAttribute((const void *)f.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024));
    CTQW_CUDA_TRY(cudaFuncSetAttribute((const void *)f.kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(h->R * f.C));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = f.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)f.C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    CTQW_CUDA_TRY(cudaLaunchKernelEx(&cfg, f.kern, a));
    return CTQW_OK;
}

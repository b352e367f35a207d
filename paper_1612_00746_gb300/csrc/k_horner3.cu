// Two Horner stages per launch for three particles in complex FP32.
//
// One launch per stage streams the iterate and psi in and the next iterate
// out, 24 bytes a site-update, and ran at 0.72 of HBM.  Here a block owns some
// consecutive x2 of one realization over all x3 and walks x1: plane x1 = t of
// the input iterate arrives in shared memory by cp.async a turn ahead, the
// first stage is formed on plane t - 1 and the second on plane t - 2, so the
// iterate between the two never leaves the SM: 12 bytes a site-update.  The
// neighbours along x1 are in registers, those along x2 mostly too (a thread
// owns several rows), those along x3 in shared memory, double buffered so that
// one barrier a plane orders everything.  Every stage loses one row of the
// block at either end; the rows shared with the next block come from L2.
// What bounds it now is instructions (about 50 a point and stage).  10 steps of
// K = 16 without samples, one launch a stage -> this kernel: 16 x N = 160
// 56.6 -> 36.5 ms, 40 x N = 100 42.3 -> 20.8, 100 x N = 64 23.4 -> 14.1,
// 200 x N = 40 19.7 -> 8.6, 100 x N = 12 1.70 -> 1.21: faster at every size
// that fits, so those all take it.
//   w_j = psi + (-i dt / j) H w_{j+1}; the last stage of a step also adds its
// increment to psi with the rounding error carried in lo.
#include <algorithm>

#include "ctqw_internal.cuh"
#include "fused_common.cuh"

namespace {

constexpr int kMaxThreads = 512;

struct PairArgs {
    RealTable tab;
    const int32_t *list;
    const float *eps, *J;
    const float2 *in;        // w_{j+1} (psi itself in the first stages of a step)
    const float2 *psi;
    float2 *out;             // w_{j-1}, or the new state
    float2 *lo;              // carried error, in place (FINAL)
    float U;
    float c1, c2;            // dt / j and dt / (j - 1)
    int groups, chunk;       // threads' row groups a block, x1 planes a block
};

__device__ __forceinline__ void copy8(uint32_t dst, const float2 *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

// Thread (x3, group g) owns kRL rows of the block's at its x3, so the
// neighbours along x2 are mostly its own registers.
// SAME: the input iterate is psi.  FINAL: the second stage is j = 1 and its
// update is compensated.
template <bool SAME, bool FINAL, int kRL>
__global__ void __launch_bounds__(kMaxThreads, 1) horner3_pair_kernel(const __grid_constant__ PairArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int r = a.list[blockIdx.z];
    const int N = a.tab.N[r];
    const int64_t base = a.tab.st_off[r], po = a.tab.par_off[r];
    const int rows = kRL * a.groups, plane = rows * N;
    float2 *A = reinterpret_cast<float2 *>(smem_raw);     // [3][rows][N] the input iterate: planes t - 1, t, t + 1
    float2 *B = A + 3 * plane;                            // [2][rows][N] the iterate between the stages
    float2 *S = B + 2 * plane;                            // [3][rows][N] psi: planes t - 2, t - 1, t (not if SAME)
    float *es = reinterpret_cast<float *>(S + (SAME ? 0 : 3 * plane)); // [N] eps
    float *js = es + N;                                   // [N] J
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        es[i] = a.eps[po + i];
        js[i] = a.J[po + i];
    }
    __syncthreads();
    const int x2_0 = (int)blockIdx.x * (rows - 4) - 2;
    const int first = blockIdx.y * a.chunk, last = min(first + a.chunk, N);   // planes this block writes
    const float U = a.U;
    auto wrap = [N](int x) {
        x = x < 0 ? x + N : x;
        x = x >= N ? x - N : x;
        return x < 0 || x >= N ? (x % N + N) % N : x;   // more rows than sites
    };
    const bool live = (int)threadIdx.x < a.groups * N;    // the block is rounded up to whole warps
    const int g = live ? (int)threadIdx.x / N : 0, x3 = live ? (int)threadIdx.x - g * N : 0;
    const int row0 = g * kRL;
    const int at = row0 * N + x3;                         // this thread's first point in a plane of the block
    const int dl = x3 == 0 ? N - 1 : -1, dr = x3 + 1 == N ? 1 - N : 1;
    const int d_up = g > 0 ? -N : 0, d_dn = g + 1 < a.groups ? N : 0;   // the block's border rows read themselves
    const float jl3 = js[x3 == 0 ? N - 1 : x3 - 1], jr3 = js[x3];
    int off[kRL];
    float e23[kRL], j2[kRL + 1];   // j2[k]: the bond above row k
    unsigned keep = 0;
#pragma unroll
    for (int k = 0; k < kRL; ++k) {
        const int x2 = wrap(x2_0 + row0 + k);
        off[k] = x2 * N + x3;
        e23[k] = es[x2] + es[x3] + (x2 == x3 ? U : 0.f);
        j2[k] = js[x2 == 0 ? N - 1 : x2 - 1];
        if (k == kRL - 1) j2[kRL] = js[x2];
        // rows 2 .. rows - 3, and of the last block those inside the lattice
        if (live && row0 + k >= 2 && row0 + k < rows - 2 && x2_0 + row0 + k < N) keep |= 1u << k;
    }
    const int x2_first = wrap(x2_0 + row0);   // rows follow it, wrapping at N
    const int NN = N * N;
    const float2 *in0 = a.in + base, *psi0 = a.psi + base;
    const uint32_t sA = fused::smem_u32(A + at), sS = fused::smem_u32(S + at);
    // plane t of the input into slot s; psi, needed two planes later, lags one behind
    auto fetch = [&](int t, int s, bool with_psi) {
        const int64_t p = (int64_t)wrap(t) * NN, pq = (int64_t)wrap(t - 1) * NN;
        const int sq = s == 0 ? 2 : s - 1;
#pragma unroll
        for (int k = 0; k < kRL; ++k) {
            copy8(sA + 8u * (s * plane + k * N), in0 + p + off[k]);
            if (!SAME && with_psi) copy8(sS + 8u * (sq * plane + k * N), psi0 + pq + off[k]);
        }
    };
    if (live) fetch(first - 2, 0, false);
    asm volatile("cp.async.commit_group;" ::: "memory");
    // planes t - 2 and t - 1 of the input, t - 3 and t - 2 of the middle iterate
    const float2 z = make_float2(0.f, 0.f);
    float2 ap[kRL], ac[kRL], bp[kRL], bc[kRL];
#pragma unroll
    for (int k = 0; k < kRL; ++k) ap[k] = ac[k] = bp[k] = bc[k] = z;
    // (H w) of row k: W the plane's copy at the thread's first point, c its
    // rows' values with the row above the first and below the last, up and dn
    // along x1
    auto apply = [&](int k, const float2 *W, float2 up2, float2 c, float2 dn2, float2 up1, float2 dn1, float e1,
                     float jl1, float jr1, int x1) {
        float v = e1 + e23[k];
        int d = x1 - x2_first;
        if (d < 0) d += N;
        if (d == k) v += U;          // x1 = x2
        if (x1 == x3) v += U;
        const float2 l3 = W[k * N + dl], r3 = W[k * N + dr];
        float2 y = make_float2(v * c.x, v * c.y);
        y.x = fmaf(-jl3, l3.x, y.x);
        y.y = fmaf(-jl3, l3.y, y.y);
        y.x = fmaf(-jr3, r3.x, y.x);
        y.y = fmaf(-jr3, r3.y, y.y);
        y.x = fmaf(-j2[k], up2.x, y.x);
        y.y = fmaf(-j2[k], up2.y, y.y);
        y.x = fmaf(-j2[k + 1], dn2.x, y.x);
        y.y = fmaf(-j2[k + 1], dn2.y, y.y);
        y.x = fmaf(-jl1, up1.x, y.x);
        y.y = fmaf(-jl1, up1.y, y.y);
        y.x = fmaf(-jr1, dn1.x, y.x);
        y.y = fmaf(-jr1, dn1.y, y.y);
        return y;
    };
    // t: the plane whose input has arrived; its slot in A, and psi's on the same plane
    int tA = 0;
    for (int t = first - 2; t <= last + 1; ++t) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();   // this plane's input and the last turn's middle iterate are everybody's
        const int nA = tA == 2 ? 0 : tA + 1, pA = tA == 0 ? 2 : tA - 1;
        if (live && t <= last) fetch(t + 1, nA, true);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const int x1o = t - 2;   // the plane the second stage writes
        float2 l[kRL];
        if (FINAL && x1o >= first) {
            const float2 *pl = a.lo + base + (int64_t)x1o * NN;
#pragma unroll
            for (int k = 0; k < kRL; ++k)
                if (keep >> k & 1) l[k] = pl[off[k]];
        }
        const float2 *An = A + tA * plane + at, *Ac = A + pA * plane + at;
        float2 *Bn = B + ((t + 1) & 1) * plane + at;
        const float2 *Bc = B + (t & 1) * plane + at;
        float2 an[kRL], bn[kRL];
#pragma unroll
        for (int k = 0; k < kRL; ++k) an[k] = An[k * N];
        if (t >= first) {
            // first stage on plane t - 1
            const int x1 = wrap(t - 1);
            const float e1 = es[x1], jl1 = js[x1 == 0 ? N - 1 : x1 - 1], jr1 = js[x1];
            const float2 top = Ac[d_up], bot = Ac[(kRL - 1) * N + d_dn];
            const float2 *q = S + pA * plane + at;      // plane t - 1
#pragma unroll
            for (int k = 0; k < kRL; ++k) {
                const float2 y = apply(k, Ac, k == 0 ? top : ac[k == 0 ? 0 : k - 1], ac[k],
                                       k == kRL - 1 ? bot : ac[k == kRL - 1 ? k : k + 1], ap[k], an[k], e1, jl1, jr1, x1);
                const float2 h = SAME ? ac[k] : q[k * N];
                bn[k] = make_float2(fmaf(a.c1, y.y, h.x), fmaf(-a.c1, y.x, h.y));
            }
        } else {
#pragma unroll
            for (int k = 0; k < kRL; ++k) bn[k] = z;
        }
        if (x1o >= first) {
            // second stage on plane t - 2
            const float e1 = es[x1o], jl1 = js[x1o == 0 ? N - 1 : x1o - 1], jr1 = js[x1o];
            const float2 top = Bc[d_up], bot = Bc[(kRL - 1) * N + d_dn];
            const float2 *q = S + nA * plane + at;      // plane t - 2
            float2 *po_ = a.out + base + (int64_t)x1o * NN, *pl = a.lo + (FINAL ? base + (int64_t)x1o * NN : 0);
#pragma unroll
            for (int k = 0; k < kRL; ++k) {
                const float2 y = apply(k, Bc, k == 0 ? top : bc[k == 0 ? 0 : k - 1], bc[k],
                                       k == kRL - 1 ? bot : bc[k == kRL - 1 ? k : k + 1], bp[k], bn[k], e1, jl1, jr1, x1o);
                float2 h = SAME ? ap[k] : q[k * N];
                if (!(keep >> k & 1)) continue;
                if (FINAL) {
                    fused::compensated_add(h.x, l[k].x, a.c2 * y.y);
                    fused::compensated_add(h.y, l[k].y, -a.c2 * y.x);
                    pl[off[k]] = l[k];
                } else {
                    h = make_float2(fmaf(a.c2, y.y, h.x), fmaf(-a.c2, y.x, h.y));
                }
                po_[off[k]] = h;
            }
        }
#pragma unroll
        for (int k = 0; k < kRL; ++k) {
            if (live) Bn[k * N] = bn[k];
            ap[k] = ac[k];
            ac[k] = an[k];
            bp[k] = bc[k];
            bc[k] = bn[k];
        }
        tA = nA;
    }
}

using PairKernel = void (*)(PairArgs);

// How a lattice is cut up: rows a thread and row groups a block, and x1 planes
// a block.
struct PairCut {
    int rl = 0, groups = 0, chunk = 0;
};

size_t pair_smem(int N, int rows) { return sizeof(float2) * 8 * (size_t)rows * N + sizeof(float) * 2 * N; }

// The cut of least time: a block fills an SM, so blocks run in rounds of one
// per SM; one that writes c planes walks c + 4, and keeps all but four of its
// rows.  A plane costs its rows a thread times (400 + threads), measured: the
// chain of a thread's rows shows beside the instructions of all.  5 and 6 rows
// a thread are what 128 registers hold.
// (64-bit pairs and the names of the planes rotated over three copies of the
// loop body, which save the moves between planes, spilled and were slower:
// 55 ms against 43 ms on 16 x N = 160, 10 steps of K = 16.)
PairCut pair_cut(int N, int64_t members, int n_sm) {
    PairCut best;
    int64_t least = 0;
    for (int rl = 6; rl >= 5; --rl) {
        const int most = std::min((N + 4 + rl - 1) / rl, kMaxThreads / N);
        for (int groups = most; groups >= 2 && groups >= most - 2; --groups) {
            const int rows = rl * groups, tiles = (N + rows - 5) / (rows - 4);
            if (N < rl || pair_smem(N, rows) > 226 * 1024) continue;
            for (int chunks = 1; chunks == 1 || chunks * 8 <= N; ++chunks) {
                const int chunk = (N + chunks - 1) / chunks;
                const int64_t blocks = members * tiles * ((N + chunk - 1) / chunk);
                const int64_t cost = (blocks + n_sm - 1) / n_sm * (chunk + 4) * rl * (400 + groups * N);
                if (best.rl == 0 || cost < least) {
                    least = cost;
                    best.rl = rl;
                    best.groups = groups;
                    best.chunk = chunk;
                }
            }
        }
    }
    return best;
}

template <int RL>
PairKernel pair_kernel(bool same, bool final) {
    return same ? (final ? horner3_pair_kernel<true, true, RL> : horner3_pair_kernel<true, false, RL>)
                : (final ? horner3_pair_kernel<false, true, RL> : horner3_pair_kernel<false, false, RL>);
}

}  // namespace

bool horner3_pair_supported(const ctqw_hamiltonian *h) {
    if (h->m != 3) return false;
    for (int N : h->group_N)   // two row groups: 8 of 12 rows are kept
        if (pair_cut(N, 1, 152).rl == 0) return false;
    return true;
}

int launch_horner3_pair(const ctqw_hamiltonian *h, const void *in, const void *psi, void *out, void *lo, double c1,
                        double c2, cudaStream_t s) {
    PairArgs a;
    a.tab = real_table(h);
    a.eps = h->eps32;
    a.J = h->J32;
    a.in = (const float2 *)in;
    a.psi = (const float2 *)psi;
    a.out = (float2 *)out;
    a.lo = (float2 *)lo;
    a.U = (float)h->U;
    a.c1 = (float)c1;
    a.c2 = (float)c2;
    const bool same = in == psi, final = lo != nullptr;
    int n_sm = 0, off = 0;
    CTQW_CUDA_TRY(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, h->device));
    for (size_t g = 0; g < h->group_N.size(); ++g) {
        const int N = h->group_N[g], cnt = h->group_count[g];
        const PairCut cut = pair_cut(N, cnt, n_sm);
        const int rows = cut.rl * cut.groups, tiles = (N + rows - 5) / (rows - 4), chunks = (N + cut.chunk - 1) / cut.chunk;
        a.groups = cut.groups;
        a.chunk = cut.chunk;
        const PairKernel k = cut.rl == 5 ? pair_kernel<5>(same, final) : pair_kernel<6>(same, final);
        CTQW_CUDA_TRY(cudaFuncSetAttribute((const void *)k, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024));
        const int threads = (cut.groups * N + 31) / 32 * 32;
        for (int done = 0; done < cnt; done += 65535) {
            const int part = std::min(cnt - done, 65535);
            a.list = h->by_group_d + off + done;
            k<<<dim3((unsigned)tiles, (unsigned)chunks, (unsigned)part), threads, pair_smem(N, rows), s>>>(a);
            CTQW_CUDA_TRY(cudaGetLastError());
        }
        off += cnt;
    }
    return CTQW_OK;
}

// One-body reduced density matrix averaged over the realizations of each
// size group (the partial trace of Sec. 2's <rho> = (1/R) sum_i |Psi_i><Psi_i|
// over all particles but one, averaged over which particle is kept):
//
//   rho1(x, x') = (1/R_g) (1/m) sum_r sum_j sum_k psi_r(x_j = x, k) conj(psi_r(x_j = x', k)),
//
// k running over the other m-1 coordinates.  For particle j the amplitude
// psi(x_j = x, k) sits at (k / K_lo) S_hi + x S_x + (k % K_lo) in the
// row-major N^m tile (x_m fastest): S_x = N^(m-1-j), K_lo = S_x,
// S_hi = N^(m-j).  One launch per particle and size group; a block owns a
// 32 x 64 tile of (x, x') and a chunk of realizations, walks k in chunks of
// 32 (16 in FP64) through shared memory, forms the products in the state's type (FP32
// for c64) per chunk and accumulates the chunks in FP64 registers, then
// adds its tile to the FP64 output with one atomic per element.
//
// rho1 is Hermitian: only the tiles that reach the diagonal or above it are
// computed, and an element above it also fills its conjugate below.  The
// amplitude's place needs a division only for the middle particles of three;
// as 64-bit divisions for every load they were half the instructions.  What
// bounds it is shared memory in FP32 (12 passes for 32 FMAs) and the FP64 pipe
// in FP64.  Every tile and 64-bit divisions -> this, FP32: 740 x N = 303 20.0 ->
// 11.5 ms, 906 x N = 134 3.91 -> 2.77, 53 x N = 759 20.5 -> 11.2; FP64: 40 x N = 256
// 28.3 -> 10.6, 200 x N = 100 12.4 -> 6.2.
#include "ctqw_internal.cuh"
#include "stencil.cuh"

namespace {

constexpr int kTX = 64;   // x' per block
constexpr int kTY = 32;   // x per block
constexpr int kRCH = 8;   // realizations per block, at most

// k per chunk (FP64 states: half, to stay within 48 KB of static shared memory)
template <typename T> struct Chunk { static constexpr int value = 32; };
template <> struct Chunk<double> { static constexpr int value = 16; };

template <typename T>
__global__ void __launch_bounds__(256) rho1_term_kernel(RealTable tab, const int32_t *__restrict__ list,
                                                        int n_real, const cplx_t<T> *__restrict__ psi,
                                                        double *__restrict__ rho, int64_t rho_off, int N,
                                                        int64_t n_k, int64_t S_x, int64_t K_lo,
                                                        int64_t S_hi, int rch, int k_parts, double scale) {
    using C = cplx_t<T>;
    constexpr int kKC = Chunk<T>::value;
    __shared__ C A[kTY][kKC + 1];     // psi(x, k) for the block's x rows
    __shared__ C B[kKC][kTX + 1];     // psi(x', k), k-major
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 32 x 8
    const int x0 = blockIdx.y * kTY, xp0 = blockIdx.x * kTX;
    if (xp0 + kTX <= x0) return;   // all of it below the diagonal
    const bool x_contig = S_x == 1, one_run = K_lo == n_k;   // k in one run: x S_x + k
    double accr[4][2], acci[4][2];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 2; ++c) accr[q][c] = acci[q][c] = 0.0;

    const int zr = blockIdx.z / k_parts, zk = blockIdx.z - zr * k_parts;
    const int rbeg = zr * rch, rend = min(n_real, rbeg + rch);
    // this block's k, whole chunks
    const int64_t chunks = (n_k + kKC - 1) / kKC;
    const int64_t k_beg = chunks * zk / k_parts * kKC, k_end = min(n_k, chunks * (zk + 1) / k_parts * kKC);
    for (int rr = rbeg; rr < rend; ++rr) {
        const C *p = psi + tab.st_off[list[rr]];
        auto at = [&](int x, int64_t k) -> C {
            if (x_contig) return p[k * S_hi + x];
            if (one_run) return p[(int64_t)x * S_x + k];
            const unsigned hi = (unsigned)k / (unsigned)K_lo;   // N^(m-1) below 2^31
            return p[(int64_t)hi * S_hi + (int64_t)x * S_x + (k - (int64_t)hi * K_lo)];
        };
        for (int64_t k0 = k_beg; k0 < k_end; k0 += kKC) {
            // tiles of psi: consecutive threads along the contiguous index
            for (int e = threadIdx.x; e < kTY * kKC; e += blockDim.x) {
                const int i = x_contig ? e % kTY : e / kKC, kk = x_contig ? e / kTY : e % kKC;
                const int x = x0 + i;
                const int64_t k = k0 + kk;
                A[i][kk] = (x < N && k < n_k) ? at(x, k) : C{};
            }
            for (int e = threadIdx.x; e < kTX * kKC; e += blockDim.x) {
                const int i = x_contig ? e % kTX : e / kKC, kk = x_contig ? e / kTX : e % kKC;
                const int x = xp0 + i;
                const int64_t k = k0 + kk;
                B[kk][i] = (x < N && k < n_k) ? at(x, k) : C{};
            }
            __syncthreads();
            T sr[4][2], si[4][2];
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int c = 0; c < 2; ++c) sr[q][c] = si[q][c] = T(0);
#pragma unroll 8
            for (int kk = 0; kk < kKC; ++kk) {
                const C b0 = B[kk][tx], b1 = B[kk][tx + 32];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const C a = A[ty + 8 * q][kk];
                    // a conj(b)
                    sr[q][0] += a.x * b0.x + a.y * b0.y;
                    si[q][0] += a.y * b0.x - a.x * b0.y;
                    sr[q][1] += a.x * b1.x + a.y * b1.y;
                    si[q][1] += a.y * b1.x - a.x * b1.y;
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    accr[q][c] += (double)sr[q][c];
                    acci[q][c] += (double)si[q][c];
                }
            __syncthreads();
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int x = x0 + ty + 8 * q;
        if (x >= N) continue;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int xp = xp0 + tx + 32 * c;
            if (xp >= N || xp < x) continue;
            double *o = rho + 2 * (rho_off + (int64_t)x * N + xp);
            atomicAdd(o, scale * accr[q][c]);
            atomicAdd(o + 1, scale * acci[q][c]);
            if (xp == x) continue;
            o = rho + 2 * (rho_off + (int64_t)xp * N + x);
            atomicAdd(o, scale * accr[q][c]);
            atomicAdd(o + 1, scale * -acci[q][c]);
        }
    }
}

}  // namespace

int launch_one_body_density(const ctqw_hamiltonian *h, int dtype, const void *psi, double *rho,
                            cudaStream_t s) {
    RealTable t = real_table(h);
    const int m = h->m;
    int n_sm = 0;
    CTQW_CUDA_TRY(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, h->device));
    int off = 0;
    for (size_t g = 0; g < h->group_N.size(); ++g) {
        const int N = h->group_N[g], cnt = h->group_count[g];
        int64_t n_k = 1;
        for (int j = 1; j < m; ++j) n_k *= N;
        const double scale = 1.0 / ((double)cnt * (double)m);
        // A block walks up to 8 realizations; fewer, and then a part of k only,
        // while the blocks do not fill the SMs twice over two rounds (4 x N = 250
        // in FP64: 20 blocks, 7.3 ms, now 1.8)
        int64_t tiles = 0;
        for (int y = 0; y < N; y += kTY)
            for (int x = 0; x < N; x += kTX) tiles += x + kTX > y;
        int rch = kRCH, k_parts = 1;
        auto blocks = [&]() { return tiles * ((cnt + rch - 1) / rch) * k_parts; };
        while (rch > 1 && blocks() < 4 * n_sm) rch /= 2;
        while (k_parts < 64 && n_k / k_parts >= 128 && blocks() < 4 * n_sm) k_parts *= 2;
        while ((int64_t)((cnt + rch - 1) / rch) * k_parts > 65535) {   // the grid's limit
            if (k_parts > 1) k_parts /= 2;
            else rch *= 2;
        }
        const dim3 grid((unsigned)((N + kTX - 1) / kTX), (unsigned)((N + kTY - 1) / kTY),
                        (unsigned)((cnt + rch - 1) / rch * k_parts));
        for (int j = 0; j < m; ++j) {
            int64_t S_x = 1;
            for (int l = j + 1; l < m; ++l) S_x *= N;
            const int64_t K_lo = S_x, S_hi = S_x * N;
            if (dtype == CTQW_C64)
                rho1_term_kernel<float><<<grid, 256, 0, s>>>(t, h->by_group_d + off, cnt, (const float2 *)psi,
                                                             rho, h->joint_off[g], N, n_k, S_x, K_lo, S_hi,
                                                             rch, k_parts, scale);
            else
                rho1_term_kernel<double><<<grid, 256, 0, s>>>(t, h->by_group_d + off, cnt,
                                                              (const double2 *)psi, rho, h->joint_off[g], N,
                                                              n_k, S_x, K_lo, S_hi, rch, k_parts, scale);
            CTQW_CUDA_TRY(cudaGetLastError());
        }
        off += cnt;
    }
    return CTQW_OK;
}

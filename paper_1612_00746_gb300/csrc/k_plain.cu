// Per-term propagation kernels: the structure of Algorithms 2 and 3 with
// one launch per Taylor term (or RK4 stage) over all realizations at once
// (the realization x node loop collapsed into one grid, Sec. 2.2).  These
// are the plain path: every term streams the iterate and psi through HBM.
#include <algorithm>

#include "ctqw_internal.cuh"
#include "stencil.cuh"

namespace {

// k = -i H in;  next = psi + a k (when next != null);  acc = (first ? psi : acc) + b k.
template <typename T, int M>
__global__ void __launch_bounds__(256) rk4_stage_kernel(RealTable tab, const int32_t *__restrict__ list,
                                                        const T *__restrict__ eps,
                                                        const T *__restrict__ J,
                                                        const cplx_t<T> *__restrict__ in,
                                                        cplx_t<T> *__restrict__ next,
                                                        const cplx_t<T> *__restrict__ psi,
                                                        cplx_t<T> *__restrict__ acc, T a, T b,
                                                        int first) {
    Site<M> p;
    if (!site_of<M>(tab, list, p)) return;
    const int64_t s = p.s;
    const int64_t base = tab.st_off[p.r];
    const int64_t po = tab.par_off[p.r];
    cplx_t<T> y = apply_h<T, M>(in + base, s, p.x, p.N, eps + po, J + po, (T)tab.U);
    cplx_t<T> k = mk<T>(y.y, -y.x);   // -i H in
    cplx_t<T> q = psi[base + s];
    if (next) next[base + s] = mk<T>(q.x + a * k.x, q.y + a * k.y);
    cplx_t<T> c = first ? q : acc[base + s];
    acc[base + s] = mk<T>(c.x + b * k.x, c.y + b * k.y);
}

}  // namespace

int launch_rk4_stage(const ctqw_hamiltonian *h, int dtype, const void *in, void *next,
                     const void *psi, void *acc, double a, double b, int first, cudaStream_t s) {
    RealTable t = real_table(h);
    return for_each_group(h, [&](dim3 grid, dim3 block, const int32_t *list) {
        if (dtype == CTQW_C64) {
            auto k = h->m == 2 ? rk4_stage_kernel<float, 2> : rk4_stage_kernel<float, 3>;
            k<<<grid, block, 0, s>>>(t, list, h->eps32, h->J32, (const float2 *)in, (float2 *)next,
                                     (const float2 *)psi, (float2 *)acc, (float)a, (float)b, first);
        } else {
            auto k = h->m == 2 ? rk4_stage_kernel<double, 2> : rk4_stage_kernel<double, 3>;
            k<<<grid, block, 0, s>>>(t, list, h->eps64, h->J64, (const double2 *)in, (double2 *)next,
                                     (const double2 *)psi, (double2 *)acc, a, b, first);
        }
    });
}

// ---------------------------------------------------------------- FP64 per-term path
// One Horner stage of Algorithm 3's polynomial (Sec. 2.3), w_j = psi + (A/j) w_{j+1},
// A = -i dt H; with j = 1 that is the new state itself, which may overwrite
// psi in place (a thread reads psi at its own amplitude only).
//
// The FP64 pipe bounds it: GB300 issues 2 FP64 operations a clock and SM.
// One launch per term in the forward order of Algorithm 3 spends 21 of them
// an amplitude (13 with fused multiply-adds) and moves 64 bytes; this form
// spends 11 for two particles (one add for the diagonal, ten fused
// multiply-adds into psi, the coefficients scaled by dt / j once a thread and
// row) and moves 48.  It also rounds at the state's own magnitude 5 times a
// step instead of K: against 80-bit arithmetic 200 steps of N = 64, K = 12 end
// 1.5e-15 off, the forward sum 4.2e-15.  4 realizations of N = 4096, K = 16,
// 5 steps: 187.8 ms forward, 106.7 ms here (5.0e10 site-updates/s, 0.88 of the
// FP64 pipe); RK4 on 16 x N = 256, 100 steps: 17.0 ms -> 11.7 ms.
namespace {

// Two particles: a block's thread row owns `rows` lattice rows x1 of up to
// 256 columns x2, each thread walking down one column with w at x1 - 1, x1
// and x1 + 1 in registers (the next one loaded a row ahead).
constexpr int kF64Rows = 16;   // lattice rows a thread row walks at most

__global__ void __launch_bounds__(256) horner2_f64_kernel(RealTable tab, const int32_t *__restrict__ list,
                                                          const double *__restrict__ eps,
                                                          const double *__restrict__ J, const double2 *in,
                                                          const double2 *psi, double2 *out, double coef, int rows) {
    __shared__ double2 rowc[8 * kF64Rows + 1];   // coef (eps, -J of the bond above) of the block's rows
    const int r = list[blockIdx.z];
    const int N = tab.N[r];
    const int64_t po = tab.par_off[r], base = tab.st_off[r];
    const int b0 = blockIdx.x * blockDim.y * rows;   // the block's first row
    for (int q = threadIdx.y * blockDim.x + threadIdx.x; q <= (int)blockDim.y * rows; q += blockDim.x * blockDim.y) {
        const int x1 = b0 + q < N ? b0 + q : (b0 + q) % N;
        rowc[q] = make_double2(coef * eps[po + x1], -coef * J[po + (x1 == 0 ? N - 1 : x1 - 1)]);
    }
    __syncthreads();
    const int x2 = blockIdx.y * blockDim.x + threadIdx.x;
    const int x1_0 = b0 + threadIdx.y * rows, x1_e = min(x1_0 + rows, N);
    if (x2 >= N || x1_0 >= x1_e) return;
    const int xl = x2 == 0 ? N - 1 : x2 - 1, xr = x2 == N - 1 ? 0 : x2 + 1;
    const double e2 = coef * eps[po + x2], jl = -coef * J[po + xl], jr = -coef * J[po + x2];
    const double cU = coef * tab.U;
    const double2 *w = in + base;
    double2 up = w[(int64_t)(x1_0 == 0 ? N - 1 : x1_0 - 1) * N + x2], c = w[(int64_t)x1_0 * N + x2];
    double2 dn = w[(int64_t)(x1_0 + 1 == N ? 0 : x1_0 + 1) * N + x2];
    double2 l = w[(int64_t)x1_0 * N + xl], rt = w[(int64_t)x1_0 * N + xr];
    double2 q = psi[base + (int64_t)x1_0 * N + x2];
    const double2 *rc = rowc + threadIdx.y * rows;
    for (int x1 = x1_0; x1 < x1_e; ++x1, ++rc) {
        double2 nn = dn, l2 = l, rt2 = rt, q2 = q;
        if (x1 + 1 < x1_e) {   // the next row's values, a row ahead
            const int64_t row = (int64_t)(x1 + 1) * N;
            nn = w[(int64_t)(x1 + 2 == N ? 0 : x1 + 2) * N + x2];
            l2 = w[row + xl];
            rt2 = w[row + xr];
            q2 = psi[base + row + x2];
        }
        const double2 r0 = rc[0];
        const double jup = r0.y, jdn = rc[1].y;
        double v = r0.x + e2;
        if (x1 == x2) v += cU;
        // psi - i (coef H w): the real part takes +, the imaginary part -
        double yr = fma(v, c.y, q.x), yi = fma(-v, c.x, q.y);
        yr = fma(jup, up.y, yr);
        yi = fma(-jup, up.x, yi);
        yr = fma(jdn, dn.y, yr);
        yi = fma(-jdn, dn.x, yi);
        yr = fma(jl, l.y, yr);
        yi = fma(-jl, l.x, yi);
        yr = fma(jr, rt.y, yr);
        yi = fma(-jr, rt.x, yi);
        out[base + (int64_t)x1 * N + x2] = make_double2(yr, yi);
        up = c;
        c = dn;
        dn = nn;
        l = l2;
        rt = rt2;
        q = q2;
    }
}

// Three particles: one amplitude a thread.
__global__ void __launch_bounds__(256) horner3_f64_kernel(RealTable tab, const int32_t *__restrict__ list,
                                                          const double *__restrict__ eps,
                                                          const double *__restrict__ J, const double2 *in,
                                                          const double2 *psi, double2 *out, double coef) {
    Site<3> p;
    if (!site_of<3>(tab, list, p)) return;
    const int64_t base = tab.st_off[p.r], po = tab.par_off[p.r];
    const double2 y = apply_h<double, 3>(in + base, p.s, p.x, p.N, eps + po, J + po, tab.U);
    const double2 q = psi[base + p.s];
    out[base + p.s] = make_double2(fma(coef, y.y, q.x), fma(-coef, y.x, q.y));
}

}  // namespace

int launch_horner_f64(const ctqw_hamiltonian *h, const void *in, const void *psi, void *out, double coef,
                      cudaStream_t s) {
    RealTable t = real_table(h);
    if (h->m == 3)
        return for_each_group(h, [&](dim3 grid, dim3 block, const int32_t *list) {
            horner3_f64_kernel<<<grid, block, 0, s>>>(t, list, h->eps64, h->J64, (const double2 *)in,
                                                      (const double2 *)psi, (double2 *)out, coef);
        });
    int off = 0;
    for (size_t g = 0; g < h->group_N.size(); ++g) {
        const int N = h->group_N[g], cnt = h->group_count[g];
        const int tx = N >= 256 ? 256 : ((N + 31) / 32) * 32, ty = 256 / tx;
        const int64_t cols = (N + tx - 1) / tx;
        // longer walks scale and reload less, but the FP64 pipes of all SMs
        // have to get work: at least six blocks an SM, or one row a thread.  No
        // more rows than give every thread row some of them (1953 x N = 11 with
        // switching noise, 19 steps of K = 12: 8.3 ms with 16, 5.5 with 2)
        int rows = std::min(kF64Rows, (N + ty - 1) / ty);
        while (rows > 1 && (int64_t)((N + ty * rows - 1) / (ty * rows)) * cols * cnt < 912) rows /= 2;
        for (int done = 0; done < cnt; done += 65535) {
            const int part = cnt - done < 65535 ? cnt - done : 65535;
            horner2_f64_kernel<<<dim3((unsigned)((N + ty * rows - 1) / (ty * rows)), (unsigned)cols, (unsigned)part),
                                 dim3((unsigned)tx, (unsigned)ty), 0, s>>>(
                t, h->by_group_d + off + done, h->eps64, h->J64, (const double2 *)in, (const double2 *)psi,
                (double2 *)out, coef, rows);
            CTQW_CUDA_TRY(cudaGetLastError());
        }
        off += cnt;
    }
    return CTQW_OK;
}

// ---------------------------------------------------------------- FP32 per-term path
// Horner form of the same order-K polynomial (Sec. 2.3), one launch per stage:
//   w_K = psi + (A/K) psi,  w_j = psi + (A/j) w_{j+1},  psi(t+dt) = psi + A w_2,
// A = -i dt H.  In FP32 the forward sum drops every term below half an ulp
// of the running sum, which truncates the series; Horner keeps each term at
// its own scale.  The final stage adds A w_2 to the state with its rounding
// error carried in a second FP32 word (lo).
namespace {

template <int M>
__global__ void __launch_bounds__(256) horner_stage_kernel(RealTable tab, const int32_t *__restrict__ list,
                                                           const float *__restrict__ eps,
                                                           const float *__restrict__ J,
                                                           const float2 *__restrict__ in,
                                                           const float2 *__restrict__ psi,
                                                           float2 *__restrict__ out, float coef) {
    Site<M> p;
    if (!site_of<M>(tab, list, p)) return;
    const int64_t s = p.s;
    const int64_t base = tab.st_off[p.r];
    const int64_t po = tab.par_off[p.r];
    const float2 y = apply_h<float, M>(in + base, s, p.x, p.N, eps + po, J + po, (float)tab.U);
    const float2 q = psi[base + s];
    out[base + s] = make_float2(fmaf(coef, y.y, q.x), fmaf(-coef, y.x, q.y));   // q + coef (-i) y
}

template <int M>
__global__ void __launch_bounds__(256) horner_final_kernel(RealTable tab, const int32_t *__restrict__ list,
                                                           const float *__restrict__ eps,
                                                           const float *__restrict__ J,
                                                           const float2 *__restrict__ w2,
                                                           float2 *__restrict__ psi,
                                                           float2 *__restrict__ lo, float dt) {
    Site<M> p;
    if (!site_of<M>(tab, list, p)) return;
    const int64_t s = p.s;
    const int64_t base = tab.st_off[p.r];
    const int64_t po = tab.par_off[p.r];
    const float2 y = apply_h<float, M>(w2 + base, s, p.x, p.N, eps + po, J + po, (float)tab.U);
    const float sx = dt * y.y, sy = -dt * y.x;   // -i dt H w2
    float2 h = psi[base + s], l = lo[base + s];
    // TwoSum then FastTwoSum per component
    auto add = [](float &hi, float &lw, float v) {
        const float t = __fadd_rn(hi, v);
        const float bb = __fsub_rn(t, hi);
        const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bb)), __fsub_rn(v, bb));
        const float e = __fadd_rn(err, lw);
        const float h2 = __fadd_rn(t, e);
        lw = __fsub_rn(e, __fsub_rn(h2, t));
        hi = h2;
    };
    add(h.x, l.x, sx);
    add(h.y, l.y, sy);
    psi[base + s] = h;
    lo[base + s] = l;
}

// The same two kernels for three particles, walking along x1: a block owns
// kRows3 slabs x1, one x2 and up to 256 x3 of one realization, and each
// thread keeps w at x1 - 1, x1, x1 + 1 of its (x2, x3) in registers (the
// next slab's value loaded one slab ahead), takes the x3 neighbours from
// the adjacent lanes and the x2 neighbours from L2: per amplitude 4 loads
// of w and psi against 8 for the one-amplitude-per-thread kernels.  The
// stencil is that of apply_h, term for term.
constexpr int kRows3 = 32;

template <bool FINAL>
__global__ void __launch_bounds__(256) horner3_rows_kernel(RealTable tab, const int32_t *__restrict__ list,
                                                           const float *__restrict__ eps,
                                                           const float *__restrict__ J,
                                                           const float2 *__restrict__ in,
                                                           const float2 *__restrict__ psi,
                                                           float2 *__restrict__ out, float2 *__restrict__ lo,
                                                           float coef, int x3_chunks) {
    const int r = list[blockIdx.z];
    const int N = tab.N[r];
    const int x3c = blockIdx.x % x3_chunks, x1c = blockIdx.x / x3_chunks;
    const int x3 = x3c * blockDim.x + threadIdx.x, x2 = blockIdx.y;
    const bool live = x3 < N;
    const int lane = threadIdx.x & 31;
    const int x1_0 = x1c * kRows3, rows = min(kRows3, N - x1_0);
    const int64_t base = tab.st_off[r];
    const int64_t po = tab.par_off[r];
    const float2 *w = in + base;
    const float2 *q_ = FINAL ? nullptr : psi + base;   // the stage's psi (not read by the final stage)
    const float *e_ = eps + po, *j_ = J + po;
    const float U = (float)tab.U;
    auto wrap = [N](int x) { return x < 0 ? x + N : (x >= N ? x - N : x); };
    const int x2l = wrap(x2 - 1), x2r = wrap(x2 + 1), x3l = wrap(x3 - 1), x3r = wrap(x3 + 1);
    const float e2 = e_[x2], jl2 = j_[x2l], jr2 = j_[x2];
    const float e3 = live ? e_[x3] : 0.f, jl3 = live ? j_[x3l] : 0.f, jr3 = live ? j_[x3] : 0.f;
    const bool own_l = lane > 0 && x3 > 0, own_r = lane < 31 && x3 + 1 < N;
    auto at = [&](int x1, int xx2, int xx3) { return ((int64_t)x1 * N + xx2) * N + xx3; };
    const float2 z = make_float2(0.f, 0.f);
    float2 w_up = z, w_c = z, w_dn = z;
    if (live) {
        w_up = w[at(wrap(x1_0 - 1), x2, x3)];
        w_c = w[at(x1_0, x2, x3)];
        w_dn = w[at(wrap(x1_0 + 1), x2, x3)];
    }
    for (int i = 0; i < rows; ++i) {
        const int x1 = x1_0 + i;
        const int64_t sidx = at(x1, x2, x3);
        float2 w_nn = z;
        if (live && i + 1 < rows) w_nn = w[at(wrap(x1 + 2), x2, x3)];
        float2 a3l = make_float2(__shfl_sync(0xffffffffu, w_c.x, (lane + 31) & 31),
                                 __shfl_sync(0xffffffffu, w_c.y, (lane + 31) & 31));
        float2 a3r = make_float2(__shfl_sync(0xffffffffu, w_c.x, (lane + 1) & 31),
                                 __shfl_sync(0xffffffffu, w_c.y, (lane + 1) & 31));
        if (live) {
            if (!own_l) a3l = w[sidx - x3 + x3l];
            if (!own_r) a3r = w[sidx - x3 + x3r];
            const float2 a2l = w[sidx + (int64_t)(x2l - x2) * N], a2r = w[sidx + (int64_t)(x2r - x2) * N];
            const int x1m = wrap(x1 - 1);
            float v = 0.f;
            v += e_[x1];
            v += e2;
            v += e3;
            v += U * (float)((x1 == x2) + (x1 == x3) + (x2 == x3));
            float yr = v * w_c.x, yi = v * w_c.y;
            yr -= jl3 * a3l.x + jr3 * a3r.x;
            yi -= jl3 * a3l.y + jr3 * a3r.y;
            yr -= jl2 * a2l.x + jr2 * a2r.x;
            yi -= jl2 * a2l.y + jr2 * a2r.y;
            const float jl1 = j_[x1m], jr1 = j_[x1];
            yr -= jl1 * w_up.x + jr1 * w_dn.x;
            yi -= jl1 * w_up.y + jr1 * w_dn.y;
            if (!FINAL) {
                const float2 q = q_[sidx];
                out[base + sidx] = make_float2(fmaf(coef, yi, q.x), fmaf(-coef, yr, q.y));   // q + coef (-i) y
            } else {
                const float sx = coef * yi, sy = -coef * yr;   // -i dt H w2
                float2 hh = out[base + sidx], l = lo[base + sidx];
                auto add = [](float &hi, float &lw, float v2) {
                    const float t = __fadd_rn(hi, v2);
                    const float bb = __fsub_rn(t, hi);
                    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bb)), __fsub_rn(v2, bb));
                    const float e = __fadd_rn(err, lw);
                    const float h2 = __fadd_rn(t, e);
                    lw = __fsub_rn(e, __fsub_rn(h2, t));
                    hi = h2;
                };
                add(hh.x, l.x, sx);
                add(hh.y, l.y, sy);
                out[base + sidx] = hh;
                lo[base + sidx] = l;
            }
        }
        w_up = w_c;
        w_c = w_dn;
        w_dn = w_nn;
    }
}

// One launch per size group of horner3_rows_kernel: (x1 chunks x x3 chunks, x2, realizations).
template <bool FINAL>
int launch_horner3_rows(const ctqw_hamiltonian *h, const void *in, const void *psi, void *out, void *lo, double coef,
                        cudaStream_t s) {
    RealTable t = real_table(h);
    int off = 0;
    for (size_t g = 0; g < h->group_N.size(); ++g) {
        const int N = h->group_N[g], cnt = h->group_count[g];
        const int tx = N >= 256 ? 256 : ((N + 31) / 32) * 32;
        const int x3_chunks = (N + tx - 1) / tx;
        const unsigned gx = (unsigned)(((N + kRows3 - 1) / kRows3) * x3_chunks);
        for (int done = 0; done < cnt; done += 65535) {
            const int part = cnt - done < 65535 ? cnt - done : 65535;
            horner3_rows_kernel<FINAL><<<dim3(gx, (unsigned)N, (unsigned)part), tx, 0, s>>>(
                t, h->by_group_d + off + done, h->eps32, h->J32, (const float2 *)in, (const float2 *)psi,
                (float2 *)out, (float2 *)lo, (float)coef, x3_chunks);
            CTQW_CUDA_TRY(cudaGetLastError());
        }
        off += cnt;
    }
    return CTQW_OK;
}

}  // namespace

int launch_horner_stage(const ctqw_hamiltonian *h, const void *in, const void *psi, void *out,
                        double coef, cudaStream_t s) {
    if (h->m == 3) return launch_horner3_rows<false>(h, in, psi, out, nullptr, coef, s);
    RealTable t = real_table(h);
    return for_each_group(h, [&](dim3 grid, dim3 block, const int32_t *list) {
        horner_stage_kernel<2><<<grid, block, 0, s>>>(t, list, h->eps32, h->J32, (const float2 *)in,
                                                      (const float2 *)psi, (float2 *)out, (float)coef);
    });
}

int launch_horner_final(const ctqw_hamiltonian *h, const void *w2, void *psi, void *lo, double dt,
                        cudaStream_t s) {
    if (h->m == 3) return launch_horner3_rows<true>(h, w2, nullptr, psi, lo, dt, s);
    RealTable t = real_table(h);
    return for_each_group(h, [&](dim3 grid, dim3 block, const int32_t *list) {
        horner_final_kernel<2><<<grid, block, 0, s>>>(t, list, h->eps32, h->J32, (const float2 *)w2,
                                                      (float2 *)psi, (float2 *)lo, (float)dt);
    });
}

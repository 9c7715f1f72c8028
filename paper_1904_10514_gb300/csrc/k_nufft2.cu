// Type-2 direction of the latitude NUFFT (Sec. 3.2.2): from the latitude
// Fourier coefficients of every column (m, map) to values at the 4 Nside + 1
// latitude nodes.  It is the exact transpose of the analysis NUFFT of
// k_nufft.cu (deconvolution, M-point FFT, half-grid spreading with folded
// mirrors), used by hpx_synthesize and, with the synthesis coefficients as
// input, by hpx_sh_synthesis.  The inputs and outputs are those of
// nufft_adj_kernel (k_adjoint.cu):
//     even m:  y_r = w_r sum_j X_j cos(j theta_r)   (w_r = 2 on rings, 1 at poles)
//     odd m:   y_r = sum_j X_j sin(j theta_r)
// with X_j = bvec[b][m][j & 1][j >> 1] (odd m: the conj(i/2)-scaled sine
// coefficients of the analysis' right-hand-side convention).
//
// Two kernels, the transposes of lat_fft_pair and spread_rb.  6 maps, Nside 256, lmax
// 400: 163 us as one radix-2 FFT and one strided column per block (the form left for
// small grids in few columns), now 12 + 25 us.
//   ifft_pair_kernel  one block per pair of orders (m even, m + 1) and map:
//       the transposed truncation puts the deconvolved coefficients c_j on j = 0..p;
//       the transposed symmetric extension of the half grid folds them into the
//       two-sided spectra U_j = c_j, U_{-j} = s c_j, U_0 = (1 + s) c_0 (s = +1 for
//       even m, -1 for odd m), so the half grid is v(t) = IFFT(U)(t) for
//       0 < t < M/2 and half of it at t = 0 and t = M/2.  The even order's grid
//       is symmetric and the odd order's antisymmetric, so one inverse FFT of
//       the sum of the two spectra gives both: v_m = (z(t) + z(M - t))/2,
//       v_{m+1} = (z(t) - z(M - t))/2.  Output: U[b][m][t], t = 0..M/2.
//       The FFT's rounding errors are those of the sum and fall on both orders alike, so
//       the even order enters times `even`, a power of two (1/2 in the synthesis, whose
//       even orders carry the rings' weight 2; halfInv = 1 / (2 even) takes it out).
//   interp_rb_kernel  the transpose of the half-grid spreading: node r takes the
//       grid points tstart[r] .. tstart[r] + E - 1 with the spreading weights of
//       (grid point, node) (table hwn, one per parity of m).  A block takes 32
//       nodes of one map and loops over all orders 32 at a time (lane = order,
//       warp = 4 nodes, weights in registers), staging each order tile's grid
//       window through shared memory, and writes 32 contiguous orders per node
//       row of Y.
#include "fft_ip.cuh"
#include "plan.h"

namespace hpx {

template <class T, int LOGM, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) ifft_pair_kernel(const cplx<T>* __restrict__ bvec, cplx<T>* __restrict__ U,
                                                             const T* __restrict__ dec, const cplx<T>* __restrict__ tw,
                                                             int p, int L, int P2, int ldu, T even, T halfInv) {
    constexpr int M = 1 << LOGM, R = ip::out_radix(LOGM, NT);
    constexpr int H = M >> 1;
    extern __shared__ unsigned char smem_raw[];
    cplx<T>* buf = reinterpret_cast<cplx<T>*>(smem_raw);   // slots(M)
    const int m0 = 2 * blockIdx.x, m1 = m0 + 1;
    const int b = blockIdx.y;
    const int tid = threadIdx.x;
    const bool has1 = m1 <= L;
    const cplx<T>* in0 = bvec + ((int64_t)b * (p + 1) + m0) * 2 * P2;
    const cplx<T>* in1 = in0 + 2 * P2;
    // even c0_j + c1_j (lower half) or even c0_j - c1_j (upper half), c1 = conj(i/2) v deconvolved
    auto both = [&](int j, T sg) {
        const int o = (j & 1) * P2 + (j >> 1);
        const T d = dec[j];
        cplx<T> v = scale(in0[o], even * d);
        if (has1) {
            const cplx<T> w = in1[o];
            const T hd = sg * T(0.5) * d;
            v = mk<T>(v.r + hd * w.i, v.i - hd * w.r);
        }
        return v;
    };
    // j = t + r M/16, t < M/16: r <= 4 can hold j <= p = M/4, r >= 12 j >= M - p
    auto ld = [&](int j, int r) {
        if (r > 4 && r < 12) return mk<T>(T(0), T(0));
        if (j == 0) return scale(in0[0], T(2) * even * dec[0]);
        if (j <= p) return both(j, T(1));
        if (j >= M - p) return both(M - j, T(-1));
        return mk<T>(T(0), T(0));
    };
    ip::transform<T, LOGM, NT, true, R, R, true, true>(
        buf, tw, tid, ld, [&](int k, int, int, cplx<T> v) { buf[ip::slot(k)] = v; });
    __syncthreads();
    cplx<T>* out0 = U + ((int64_t)b * (L + 1) + m0) * ldu;
    cplx<T>* out1 = out0 + ldu;
    for (int t = tid; t <= H; t += NT) {
        const cplx<T> z = buf[ip::slot(t)], zr = buf[ip::slot((M - t) & (M - 1))];
        cplx<T> v0 = scale(add(z, zr), halfInv);
        if (t == 0 || t == H) v0 = scale(v0, T(0.5));
        out0[t] = v0;
        if (has1) out1[t] = scale(sub(z, zr), T(0.5));
    }
}

// 32 nodes x 32 orders of one map per block (FP64, and runs wider than the
// register-blocked form below takes): the grid window of the 32 orders is staged in
// shared memory, lane = order, warp = 4 nodes.  nrw: odd row stride of the window.
template <class T>
__global__ void __launch_bounds__(256) interp_kernel(const cplx<T>* __restrict__ U, cplx<T>* __restrict__ Y,
                                                     const int* __restrict__ tstart, const T* __restrict__ hwn, int E,
                                                     int H, int p, int Q, int L, int ldu, int nrw) {
    extern __shared__ unsigned char smem_raw[];
    cplx<T>* out = reinterpret_cast<cplx<T>*>(smem_raw);   // [32 nodes][33]
    cplx<T>* us = out + 32 * 33;                           // [32 orders][nrw]
    const int r0 = blockIdx.x * 32, m0 = blockIdx.y * 32, b = blockIdx.z;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int T0 = tstart[r0];
    const cplx<T>* ub = U + (int64_t)b * (L + 1) * ldu;
    for (int ml = warp; ml < 32; ml += 8)
        for (int tt = lane; tt < nrw; tt += 32) {
            const int m = m0 + ml, t = T0 + tt;
            us[ml * nrw + tt] = (m <= L && t <= H) ? ub[(int64_t)m * ldu + t] : mk<T>(T(0), T(0));
        }
    __syncthreads();
    const int odd = lane & 1;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int r = r0 + 4 * warp + j;
        T ar = T(0), ai = T(0);
        if (r < Q) {
            const cplx<T>* ur = us + lane * nrw + (tstart[r] - T0);
            const T* w = hwn + 2 * r + odd;
            for (int e = 0; e < E; ++e) {
                const T we = w[(size_t)e * 2 * Q];
                ar += we * ur[e].r;
                ai += we * ur[e].i;
            }
        }
        out[(4 * warp + j) * 33 + lane] = mk<T>(ar, ai);
    }
    __syncthreads();
    for (int rl = warp; rl < 32; rl += 8) {
        const int r = r0 + rl, m = m0 + lane;
        if (r < Q && m <= L) Y[((int64_t)b * Q + r) * (p + 1) + m] = out[rl * 33 + lane];
    }
}

__device__ __forceinline__ void cp_async_commit2() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait2() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// EW: taps per node at most, DM: spread of tstart over 4 consecutive nodes at
// most, NS: order tiles in flight.  nrw: grid points per staged row (rounded
// up to an odd stride against bank conflicts).
template <int EW, int DM, int NS>
__global__ void __launch_bounds__(256, 2) interp_rb_kernel(const cplx<float>* __restrict__ U,
                                                           cplx<float>* __restrict__ Y,
                                                           const int* __restrict__ tstart,
                                                           const float* __restrict__ hwn, int E, int H, int p,
                                                           int Q, int L, int ldu, int nrw) {
    constexpr int W = EW + DM;
    extern __shared__ unsigned char smem_raw[];
    cplx<float>* out = reinterpret_cast<cplx<float>*>(smem_raw);   // [32 nodes][33]
    cplx<float>* us0 = out + 32 * 33;                              // NS x [32 orders][nrw]
    const int r0 = blockIdx.x * 32, b = blockIdx.y;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int T0 = tstart[r0];
    const int rf = min(r0 + 4 * warp, Q - 1);
    const int base = tstart[rf] - T0;   // window start of this warp's nodes, relative to T0
    const int par = lane & 1;           // order tiles start at multiples of 32
    float w[4][W];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int r = r0 + 4 * warp + j;
        const int off = (r < Q) ? tstart[r] - tstart[rf] : 0;
#pragma unroll
        for (int q = 0; q < W; ++q) {
            const int e = q - off;
            w[j][q] = (r < Q && e >= 0 && e < E) ? hwn[((size_t)e * Q + r) * 2 + par] : 0.f;
        }
    }
    const cplx<float>* ub = U + (int64_t)b * (L + 1) * ldu;
    auto fetch = [&](int m0, cplx<float>* us) {
        for (int ml = warp; ml < 32; ml += 8) {
            const int m = m0 + ml;
            const cplx<float>* row = ub + (int64_t)m * ldu + T0;
            for (int tt = lane; tt < nrw; tt += 32) {
                const bool ok = m <= L && T0 + tt <= H;
                cp_async8(us + ml * nrw + tt, ok ? row + tt : ub, ok ? 8 : 0);
            }
        }
        cp_async_commit2();
    };
    const int ntiles = (L + 32) / 32;
#pragma unroll
    for (int q = 0; q < NS - 1; ++q) {
        if (q < ntiles) fetch(32 * q, us0 + q * 32 * nrw);
        else cp_async_commit2();
    }
    for (int it = 0; it < ntiles; ++it) {
        const int m0 = 32 * it;
        cplx<float>* us = us0 + (it % NS) * 32 * nrw;
        if (it + NS - 1 < ntiles) fetch(m0 + 32 * (NS - 1), us0 + ((it + NS - 1) % NS) * 32 * nrw);
        else cp_async_commit2();
        cp_async_wait2<NS - 1>();
        __syncthreads();
        float ar[4] = {0.f, 0.f, 0.f, 0.f}, ai[4] = {0.f, 0.f, 0.f, 0.f};
        const cplx<float>* ur = us + lane * nrw + base;
#pragma unroll
        for (int q = 0; q < W; ++q) {
            const cplx<float> v = ur[q];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                ar[j] += w[j][q] * v.r;
                ai[j] += w[j][q] * v.i;
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) out[(4 * warp + j) * 33 + lane] = mk<float>(ar[j], ai[j]);
        __syncthreads();
        for (int idx = tid; idx < 32 * 32; idx += 256) {
            const int rl = idx >> 5, ml = idx & 31;
            const int r = r0 + rl, m = m0 + ml;
            if (r < Q && m <= L) Y[((int64_t)b * Q + r) * (p + 1) + m] = out[rl * 33 + ml];
        }
    }
}

// Returns false at nside 2 (16 grid points) and for small batches of small grids; the
// caller then runs nufft_adj_kernel.
template <class T>
bool launch_nufft2(const hpx_plan_s* P, cudaStream_t s, T even) {
    const auto& g = P->g;
    const auto& t = P->t;
    constexpr int EW = 12, DM = 4, NS = 3;
    constexpr bool F = sizeof(T) == 4;
    int logM = 0;
    while ((1 << logM) < g.M) ++logM;
    // small grids in few columns: one block per column does all of it (nufft_adj_kernel)
    // in a wave or so, in 8 to 10 us where the two kernels here, each with its own
    // latency, take 13 to 20.  FP32: up to 512 points and 600 columns of them (Nside 64,
    // 1 map: 10 against 20 us; 32 maps, lmax 33: 23 against 19); FP64, bound by its pipe:
    // up to a fourth of that (Nside 64, 1 map: 25 against 44; Nside 32, 8 maps: 42 / 40)
    if (logM < 5 || (g.M <= 512 && (int64_t)g.B * (g.L + 1) * g.M <= (F ? 4 : 1) * (int64_t)P->sms * 512)) return false;
    const size_t smem1 = (size_t)ip::slots(g.M) * sizeof(cplx<T>);
    dim3 grid1((g.L + 2) / 2, g.B);
    auto run1 = [&](auto kern, int threads) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem1);
        kern<<<grid1, threads, smem1, s>>>((const cplx<T>*)P->bvec, (cplx<T>*)P->U, (const T*)t.dec,
                                           (const cplx<T>*)t.twx, g.p, g.L, g.P2, P->ldu, even, T(0.5) / even);
    };
    // the shapes of the analysis' grid FFT (k_nufft.cu)
    if (logM == 5) run1(ifft_pair_kernel<T, 5, 32, 1>, 32);
    else if (logM == 6) run1(ifft_pair_kernel<T, 6, 32, 1>, 32);
    else if (logM == 7) run1(ifft_pair_kernel<T, 7, 32, 1>, 32);
    else if (logM == 8) run1(ifft_pair_kernel<T, 8, 32, 1>, 32);
    else if (logM == 9) run1(ifft_pair_kernel<T, 9, 32, 1>, 32);
    else if (logM == 10) run1(ifft_pair_kernel<T, 10, 64, 1>, 64);
    else if (logM == 11) run1(ifft_pair_kernel<T, 11, 128, F ? 8 : 1>, 128);
    else if (logM == 12) run1(ifft_pair_kernel<T, 12, 256, F ? 4 : 1>, 256);
    else if (logM == 13) run1(ifft_pair_kernel<T, 13, 256, F ? 2 : 1>, 256);
    else if constexpr (F) run1(ifft_pair_kernel<T, 14, 512, 1>, 512);
    if constexpr (F) {
        if (t.interpE <= EW && t.interpD <= DM) {
            const int nrw = (t.interpRows - t.interpE + EW + DM) | 1;   // first window start .. last window end
            const size_t smem2 = (size_t)(32 * 33 + NS * 32 * nrw) * sizeof(cplx<float>);
            auto kern2 = interp_rb_kernel<EW, DM, NS>;
            allow_shared(kern2);
            dim3 grid2((g.Q + 31) / 32, g.B);
            kern2<<<grid2, 256, smem2, s>>>((const cplx<float>*)P->U, (cplx<float>*)P->Y, t.tstart,
                                            (const float*)t.hwn, t.interpE, g.M / 2, g.p, g.Q, g.L, P->ldu, nrw);
            return true;
        }
    }
    const int nrw = t.interpRows | 1;
    const size_t smem2 = (size_t)(32 * 33 + 32 * nrw) * sizeof(cplx<T>);
    allow_shared(interp_kernel<T>);
    dim3 grid2((g.Q + 31) / 32, (g.L + 32) / 32, g.B);
    interp_kernel<T><<<grid2, 256, smem2, s>>>((const cplx<T>*)P->U, (cplx<T>*)P->Y, t.tstart, (const T*)t.hwn,
                                               t.interpE, g.M / 2, g.p, g.Q, g.L, P->ldu, nrw);
    return true;
}

template bool launch_nufft2<float>(const hpx_plan_s*, cudaStream_t, float);
template bool launch_nufft2<double>(const hpx_plan_s*, cudaStream_t, double);

}  // namespace hpx

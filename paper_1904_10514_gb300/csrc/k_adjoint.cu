// The exact adjoint (transpose) of the analysis, hpx_synthesize: every stage of
// Algorithm 1 transposed and applied in reverse order.  Inner products: plain
// sum_i f_i g_i on maps, plain Re(x conj y) on the intermediate complex arrays,
// and sum_l [Re(a_l0 conj b_l0) + 2 sum_{m>0} Re(a_lm conj b_lm)] on alm (so the
// input alm are weighted by 1 at m = 0 and 2 at m > 0 first).  The analysis
// returns real a_l0 and a_l^p, so the imaginary parts of those inputs are
// dropped, as the exact transpose of a real-valued output does.
//
//   rot_adj    transposed Givens sweeps (Sec. 3.3): each sweep appends a zero
//              carry and applies the rotations in reverse order, top down; the
//              sweeps run in reverse order as a register wavefront.
//   dense_adj  beta -> b:  D^T (latitude least squares and Legendre change of basis)
//   nufft_adj  b -> y: deconvolution, inverse M-point FFT and interpolation from the
//              fine grid to the DFS nodes (the transposed ES spreading, Sec. 3.2.2)
//   ring_back  y -> ring samples: transposed shift/Nyquist/padding and inverse
//              DFT per ring pair (Sec. 3.1)
//   pole_adj   adds the transposed pole fit (Sec. 3.2.1) to the 3 rings per cap
#include <algorithm>

#include "ring_blue.cuh"
#include "plan.h"
#include "plan_math.h"
#include "sweep.cuh"

namespace hpx {

// ---------------------------------------------------------------- rot_adj
// One transposed pass of K sweeps.  The chain has n_in elements on entry and
// n_in + K on exit.  Stage k (undoing the pass's forward stage K-1-k) handles
// rotation index i = n_in + 2k - t at time t, from the top of its chain down:
//     (carry, out_i) = (c_i a - s_i carry, s_i a + c_i carry),  a = input w_{i-1},
// then emits the carry as out_0 at i = 0.  Idle slots hold (0, 0) (clearing the
// carry before the stage starts) and the emission slot holds (1, 0).
template <class T, int K>
__device__ __forceinline__ void sweep_pass_adj(T* chain, int64_t ldc, int n_in, const cplx<T>* __restrict__ A,
                                               int coff) {
    T carry[K], pipe[K];
#pragma unroll
    for (int k = 0; k < K; ++k) { carry[k] = T(0); pipe[k] = T(0); }
    const int steps = n_in + 2 * K - 1;
    for (int t = 0; t < steps; ++t) {
        const T x0 = (t < n_in) ? chain[(int64_t)(n_in - 1 - t) * ldc] : T(0);
        const cplx<T>* row = A + (int64_t)t * 32 + coff;
#pragma unroll
        for (int k = K - 1; k >= 0; --k) {
            const T x = (k == 0) ? x0 : pipe[k - 1];
            const cplx<T> cs = row[k];
            const T o = cs.i * x + cs.r * carry[k];
            carry[k] = cs.r * x - cs.i * carry[k];
            pipe[k] = o;
        }
        const int j = n_in + 2 * K - 2 - t;
        if (j >= 0 && j < n_in + K) chain[(int64_t)j * ldc] = pipe[K - 1];
    }
}

template <class T, int KMAX>
__global__ void __launch_bounds__(128) rot_adj_kernel(const T* __restrict__ alm, T* __restrict__ beta2,
                                                      const int64_t* __restrict__ skOff,
                                                      const cplx<T>* __restrict__ skewT, int nq, int P2, int L,
                                                      int p, int B, int64_t nalm, int ngroups, int nitems,
                                                      T wpos, bool dropim) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= nitems) return;
    const int g = warp % ngroups;
    const int c = (warp / ngroups) & 1;
    const int m = L - warp / (2 * ngroups);
    const int m0 = m & 1;
    const int S = (m - m0) >> 1;
    const int ncol = 2 * B;
    const int col = 32 * g + lane;
    if (col >= ncol) return;
    const int par = (m0 + c) & 1;
    const int q0 = (m0 == 1 && c == 1) ? 1 : 0;
    T* chain = beta2 + (((int64_t)m * 2 + par) * P2 + q0) * ncol + col;
    const int64_t ldc = ncol;
    // order-m chain from the weighted input coefficients
    int n = chain_len(m, c, L);
    const int b = col >> 1, ri = col & 1;
    const T w = (m == 0) ? T(1) : wpos;
    const bool drop = dropim && ri == 1 && (m == 0 || m == p);
    const T* in = alm + (int64_t)b * nalm * 2 + ri;
    const int64_t base = (int64_t)m * (2 * L + 1 - m) / 2 + m + c;
    for (int i = 0; i < n; ++i) chain[(int64_t)i * ldc] = drop ? T(0) : w * in[(base + 2 * i) * 2];
    // forward passes: F full passes of KMAX at s = 0, KMAX, ..., then the binary
    // digits of the remainder r (16, 8, 4, 2, 1 below KMAX); undo them in reverse.
    const int F = S / KMAX, r = S % KMAX;
    auto block = [&](int s_lo, int K) {
        const int e = 32 - (s_lo & 31) - K;
        return skewT + (skOff[(size_t)(m0 * 2 + c) * nq + (s_lo >> 5)] + e) * 32;
    };
    auto coff = [&](int s_lo, int K) { return 32 - (s_lo & 31) - K; };
#define HPX_SUBPASS_ADJ(KK)                                                               \
    if (KK < KMAX && (r & KK)) {                                                          \
        const int s_lo = F * KMAX + (r & ~(2 * KK - 1));                                  \
        sweep_pass_adj<T, KK>(chain, ldc, n, block(s_lo, KK), coff(s_lo, KK));          \
        n += KK;                                                                          \
    }
    HPX_SUBPASS_ADJ(1)
    HPX_SUBPASS_ADJ(2)
    HPX_SUBPASS_ADJ(4)
    HPX_SUBPASS_ADJ(8)
    HPX_SUBPASS_ADJ(16)
#undef HPX_SUBPASS_ADJ
    for (int f = F - 1; f >= 0; --f) {
        const int s_lo = f * KMAX;
        sweep_pass_adj<T, KMAX>(chain, ldc, n, block(s_lo, KMAX), coff(s_lo, KMAX));
        n += KMAX;
    }
}

// FP32: the same transposed pass with the angle rows and the chain inputs of
// step t staged through a per-warp ring of shared memory RB - 1 steps ahead
// (8-byte copies of the 32 angles, one 4-byte copy per lane).  Every lane of
// the warp runs it (lanes without a column neither load nor store chain values).
// The outputs go to indices above every input still to be read, so the
// prefetch never reads a value this pass has rewritten.
template <int K, int RB>
__device__ __forceinline__ void sweep_pass_adj_staged(float* chain, int64_t ldc, int n_in, bool live,
                                                      const cplx<float>* __restrict__ A, int coff,
                                                      cplx<float>* ring) {
    constexpr int SL = SweepRing<RB>::kSlot;
    const int lane = threadIdx.x & 31;
    float carry[K], pipe[K];
#pragma unroll
    for (int k = 0; k < K; ++k) { carry[k] = 0.f; pipe[k] = 0.f; }
    const int steps = n_in + 2 * K - 1;
    auto issue = [&](int t) {
        if (t < steps) {
            cplx<float>* slot = ring + (t % RB) * SL;
            cp_async8(slot + lane, A + (int64_t)t * 32 + lane, 8);
            const bool have = live && t < n_in;
            cp_async4(reinterpret_cast<float*>(slot + 32) + lane,
                      have ? chain + (int64_t)(n_in - 1 - t) * ldc : (const float*)A, have ? 4 : 0);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int q = 0; q < RB - 1; ++q) issue(q);
    for (int t = 0; t < steps; ++t) {
        __syncwarp();
        issue(t + RB - 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(RB - 1) : "memory");
        __syncwarp();
        const cplx<float>* slot = ring + (t % RB) * SL;
        const float x0 = reinterpret_cast<const float*>(slot + 32)[lane];
        const cplx<float>* row = slot + coff;
        auto rotate = [&](int k, cplx<float> cs, float x) {
            const float o = cs.i * x + cs.r * carry[k];
            carry[k] = cs.r * x - cs.i * carry[k];
            pipe[k] = o;
        };
        if constexpr (K == 1) {
            rotate(0, row[0], x0);
        } else {
#pragma unroll
            for (int k = K - 2; k >= 0; k -= 2) {   // two stages per 16-byte read (coff is even)
                cplx<float> ca, cb;
                load2(row + k, ca, cb);
                rotate(k + 1, cb, pipe[k]);
                rotate(k, ca, k == 0 ? x0 : pipe[k - 1]);
            }
        }
        const int j = n_in + 2 * K - 2 - t;
        if (live && j >= 0 && j < n_in + K) chain[(int64_t)j * ldc] = pipe[K - 1];
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
}

// rot_adj_kernel for FP32 with the staged passes: one real column per lane and G
// orders of one parity and chain per warp, as rot_staged_real_kernel of the forward
// sweeps: sweep S0 + q is undone for the orders i > q, q descending, then the first
// S0 sweeps of all of them (warps of 2 per block; the whole warp stays in the
// passes).  8 maps, Nside 2048: 73 ms with one order per warp, now 40.4 ms
template <int KMAX>
__global__ void __launch_bounds__(64, 8) rot_adj_staged_kernel(const float* __restrict__ alm, float* __restrict__ beta2,
                                                              const int64_t* __restrict__ skOff,
                                                              const cplx<float>* __restrict__ skewT, int nq, int P2,
                                                              int L, int p, int B, int64_t nalm, int G, int ngroups,
                                                              int nitems, float wpos, bool dropim) {
    constexpr int RB = 8;
    constexpr int SL = SweepRing<RB>::kSlot;
    __shared__ __align__(16) cplx<float> rings[2][RB * SL];
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= nitems) return;   // whole warps leave together
    cplx<float>* ring = rings[(threadIdx.x >> 5) & 1];
    const int g = warp % ngroups;
    const int c = (warp / ngroups) & 1, m0 = (warp / (2 * ngroups)) & 1;
    const int S0 = G * (L / 2 / G - warp / (4 * ngroups));
    if (m0 + 2 * S0 > L) return;
    const int W = 32 / G, o = lane / W;
    const int m = m0 + 2 * (S0 + o);
    const int ncol = 2 * B;
    const int col = 32 * g + lane - o * W;
    const bool live = col < ncol && m <= L;
    const int par = (m0 + c) & 1;
    const int q0 = (m0 == 1 && c == 1) ? 1 : 0;
    float* chain = live ? beta2 + (((int64_t)m * 2 + par) * P2 + q0) * ncol + col : beta2;
    const int64_t ldc = ncol;
    if (live) {   // order-m chain from the weighted input coefficients
        const int n = chain_len(m, c, L);
        const int b = col >> 1, ri = col & 1;
        const float w = (m == 0) ? 1.f : wpos;
        const bool drop = dropim && ri == 1 && (m == 0 || m == p);
        const float* in = alm + (int64_t)b * nalm * 2 + ri;
        const int64_t base = (int64_t)m * (2 * L + 1 - m) / 2 + m + c;
        for (int i = 0; i < n; ++i) chain[(int64_t)i * ldc] = drop ? 0.f : w * in[(base + 2 * i) * 2];
    }
    __syncwarp();
    auto block = [&](int s_lo, int K) {
        const int e = 32 - (s_lo & 31) - K;
        return skewT + (skOff[(size_t)(m0 * 2 + c) * nq + (s_lo >> 5)] + e) * 32;
    };
    auto coff = [&](int s_lo, int K) { return 32 - (s_lo & 31) - K; };
    for (int q = G - 2; q >= 0; --q) {
        if (m0 + 2 * (S0 + q + 1) > L) continue;
        sweep_pass_adj_staged<1, RB>(chain, ldc, chain_len(m0 + 2 * (S0 + q + 1), c, L), live && o > q,
                                     block(S0 + q, 1), coff(S0 + q, 1), ring);
    }
    int n = chain_len(m0 + 2 * S0, c, L);
    const int F = S0 / KMAX, r = S0 % KMAX;
#define HPX_SUBPASS_ADJ(KK)                                                                        \
    if (KK < KMAX && (r & KK)) {                                                                   \
        const int s_lo = F * KMAX + (r & ~(2 * KK - 1));                                           \
        sweep_pass_adj_staged<KK, RB>(chain, ldc, n, live, block(s_lo, KK), coff(s_lo, KK), ring); \
        n += KK;                                                                                   \
    }
    HPX_SUBPASS_ADJ(1)
    HPX_SUBPASS_ADJ(2)
    HPX_SUBPASS_ADJ(4)
    HPX_SUBPASS_ADJ(8)
    HPX_SUBPASS_ADJ(16)
#undef HPX_SUBPASS_ADJ
    for (int f = F - 1; f >= 0; --f) {
        const int s_lo = f * KMAX;
        sweep_pass_adj_staged<KMAX, RB>(chain, ldc, n, live, block(s_lo, KMAX), coff(s_lo, KMAX), ring);
        n += KMAX;
    }
}

// ---------------------------------------------------------------- dense_adj
namespace {
constexpr int AK = 64;   // output rows (k) per block
constexpr int AC = 32;   // columns (m, map) per block
constexpr int AQ = 16;   // reduction chunk (q)
}  // namespace

template <class T>
__global__ void __launch_bounds__(256) dense_adj_kernel(const T* __restrict__ D, const cplx<T>* __restrict__ beta,
                                                        cplx<T>* __restrict__ bvec, int P2, int p, int L, int B) {
    __shared__ T Ds[AQ][AK + 1];
    __shared__ cplx<T> Bs[AQ][AC];
    const int mpar = blockIdx.z >> 1, par = blockIdx.z & 1;
    const int nmp = (L >= mpar) ? (L - mpar) / 2 + 1 : 0;
    const int ncols = nmp * B;
    const int c0 = blockIdx.x * AC, k0 = blockIdx.y * AK;
    if (c0 >= ncols) return;
    const T* Dm = D + ((size_t)(mpar * 2 + par) * P2) * P2;
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    T accr[4][2], acci[4][2];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < 2; ++c) { accr[a][c] = T(0); acci[a][c] = T(0); }
    for (int qb = 0; qb < P2; qb += AQ) {
        for (int e = tid; e < AQ * AK; e += 256) {
            const int qq = e / AK, kk = e % AK;
            const int q = qb + qq, k = k0 + kk;
            Ds[qq][kk] = (q < P2 && k < P2) ? Dm[(size_t)q * P2 + k] : T(0);
        }
        for (int e = tid; e < AQ * AC; e += 256) {
            const int qq = e / AC, cc = e % AC;
            const int q = qb + qq, col = c0 + cc;
            const int l = 2 * q + par;
            cplx<T> v = mk<T>(T(0), T(0));
            if (col < ncols && q < P2 && l <= L && l >= mpar) {
                const int b = col % B, mi = col / B;
                const int m = 2 * mi + mpar;
                v = beta[(((int64_t)m * 2 + par) * P2 + q) * B + b];
            }
            Bs[qq][cc] = v;
        }
        __syncthreads();
#pragma unroll
        for (int qq = 0; qq < AQ; ++qq) {
            T a[4];
#pragma unroll
            for (int rr = 0; rr < 4; ++rr) a[rr] = Ds[qq][tx * 4 + rr];
            cplx<T> bb[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) bb[c] = Bs[qq][ty * 2 + c];
#pragma unroll
            for (int rr = 0; rr < 4; ++rr)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    accr[rr][c] += a[rr] * bb[c].r;
                    acci[rr][c] += a[rr] * bb[c].i;
                }
        }
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int col = c0 + ty * 2 + c;
        if (col >= ncols) continue;
        const int b = col % B, mi = col / B;
        const int m = 2 * mi + mpar;
        cplx<T>* out = bvec + (((int64_t)b * (p + 1) + m) * 2 + par) * P2;
#pragma unroll
        for (int rr = 0; rr < 4; ++rr) {
            const int k = k0 + tx * 4 + rr;
            if (k < P2) out[k] = mk<T>(accr[rr][c], acci[rr][c]);
        }
    }
}

// ---------------------------------------------------------------- nufft_adj
template <class T>
__global__ void __launch_bounds__(512) nufft_adj_kernel(const cplx<T>* __restrict__ bvec, cplx<T>* __restrict__ Y,
                                                        const int* __restrict__ nrowptr,
                                                        const int* __restrict__ nent, const T* __restrict__ nentw,
                                                        const T* __restrict__ dec, const cplx<T>* __restrict__ tw,
                                                        int twlen, int M, int logM, int p, int Q, int P2) {
    extern __shared__ unsigned char smem_raw[];
    cplx<T>* u = reinterpret_cast<cplx<T>*>(smem_raw);
    const int m = blockIdx.x, b = blockIdx.y;
    const int tid = threadIdx.x, nt = blockDim.x;
    const bool odd = (m & 1) != 0;
    const cplx<T>* in = bvec + ((int64_t)b * (p + 1) + m) * 2 * P2;
    for (int j = tid; j < M; j += nt) {
        cplx<T> v = mk<T>(T(0), T(0));
        if (j <= p) {
            v = in[(j & 1) * P2 + (j >> 1)];
            if (odd) v = mk<T>(T(0.5) * v.i, T(-0.5) * v.r);   // conj(i/2) v
            v = scale(v, dec[j]);
        }
        u[j] = v;
    }
    __syncthreads();
    block_fft(u, M, logM, tw, twlen, true);
    cplx<T>* out = Y + (int64_t)b * Q * (p + 1) + m;
    for (int r = tid; r < Q; r += nt) {
        T ar = T(0), ai = T(0);
        const int e1 = nrowptr[r + 1];
        for (int e = nrowptr[r]; e < e1; ++e) {
            const int code = nent[e];
            const int t = code & ((1 << 30) - 1);
            T w = nentw[e];
            if (odd && (code >> 30)) w = -w;
            const cplx<T> v = u[t];
            ar += w * v.r;
            ai += w * v.i;
        }
        out[(int64_t)r * (p + 1)] = mk<T>(ar, ai);
    }
}

template <class T>
__global__ void pole_adj_kernel(const cplx<T>* __restrict__ Y, T* __restrict__ maps, const int* __restrict__ poleN,
                                const int* __restrict__ poleS, const double* __restrict__ w, int npole, int p,
                                int Q, int64_t npix) {
    const int b = blockIdx.x;
    const cplx<T>* Yb = Y + (int64_t)b * Q * (p + 1);
    const T vn = Yb[0].r;
    const T vs = Yb[(int64_t)(Q - 1) * (p + 1)].r;
    T* f = maps + (int64_t)b * npix;
    for (int k = threadIdx.x; k < npole; k += blockDim.x) {
        f[poleN[k]] += (T)w[k] * vn;
        f[poleS[k]] += (T)w[k] * vs;
    }
}

// ---------------------------------------------------------------- rings, backwards
// Both directions that end in maps finish with an inverse DFT per ring pair: the
// north and south rings packed as z = f_N + i f_S, conj(z) = DFT(conj(Z)) with conj(Z_k)
// formed on the fly from the pair's rows of Y (BackInput), on the in-place passes of
// fft_ip.cuh (Bluestein rings of 4096 points and more: ring_blue.cuh), the pixels written straight from
// registers by the last pass (plain rings) or the radix-4 step (Bluestein rings).
//
// adjoint (SYN = false): Z = H_N + i H_S with H the Hermitian extension of
//     conj(ph_m) y_m (the transposed shift, Nyquist split and padding of Sec. 3.1);
// synthesis (SYN = true): Z_k = sum of F_m e^{i m phi0} over m = k mod n, m in [-L, L],
//     F_m = Y_m (Y_m / 2 for even m: ring weight 2), F_{-m} = conj(F_m).  With
//     phi0 = pi / n every phase is +-e^{i pi k / n}: (-1)^q for m = k + q n and
//     m = k - q n, so a rotation is made once per k; phi0 = 0: none.
// Bound by the shared-memory passes and, in the synthesis, the reads of the aliased
// orders.  Synthesis of 32 maps at Nside 512: 1266 us (plain and short rings, radix-2
// passes) + 321 us (Bluestein rings, whole convolutions) before, 728 us now.
template <class T, bool SYN>
struct BackInput {
    const cplx<T>*rowN, *rowS, *ph;
    int n, L;
    bool equator, sh;

    __device__ __forceinline__ cplx<T> operator()(int k) const {
        const cplx<T> zero = mk<T>(T(0), T(0));
        if constexpr (!SYN) {
            const int h = n >> 1, m = k <= h ? k : n - k;
            if (m > L) return zero;
            const cplx<T> w = conjg(ph[m]);
            const cplx<T> zn = mul(w, rowN[m]);
            const cplx<T> zs = equator ? zero : mul(w, rowS[m]);
            if (m == 0 || m == h) return mk<T>(zn.r, -zs.r);
            if (k <= h) return mk<T>(T(0.5) * (zn.r - zs.i), T(-0.5) * (zn.i + zs.r));   // conj(zn/2 + i zs/2)
            return mk<T>(T(0.5) * (zn.r + zs.i), T(-0.5) * (-zn.i + zs.r));              // conj(conj(zn)/2 + i conj(zs)/2)
        } else {
            cplx<T> cN = zero, cS = zero;
            T sg = T(1);
            auto take = [&](int m, bool cj) {   // +-F_m or +-conj(F_m) of both rings
                const T f = (m & 1) ? sg : T(0.5) * sg;
                cplx<T> v = rowN[m];
                if (m == 0) v.i = T(0);
                cN.r += f * v.r;
                cN.i += cj ? -(f * v.i) : f * v.i;
                if (!equator) {
                    v = rowS[m];
                    if (m == 0) v.i = T(0);
                    cS.r += f * v.r;
                    cS.i += cj ? -(f * v.i) : f * v.i;
                }
            };
            for (int m = k; m <= L; m += n) {
                take(m, false);
                if (sh) sg = -sg;
            }
            sg = sh ? T(-1) : T(1);
            for (int m = n - k; m <= L; m += n) {
                take(m, true);
                if (sh) sg = -sg;
            }
            if (sh) {
                T sn, cs;
                if constexpr (sizeof(T) == 4) sincospif((float)k / (float)n, &sn, &cs);
                else sincospi((double)k / (double)n, &sn, &cs);
                const cplx<T> w = mk<T>(cs, sn);
                cN = mul(w, cN);
                cS = mul(w, cS);
            }
            return mk<T>(cN.r - cS.i, -(cN.i + cS.r));
        }
    }
};

// Bluestein rings: four quarter transforms (ring_blue.cuh) of 2^LOGQ points, or one
// convolution of the whole ring of 2^LOGN points.
template <class T, int LOGQ, int NTQ, class V>
__device__ __forceinline__ void ring_back_quarters(cplx<T>* buf, T* f, int sN, int sS, int n,
                                                   const cplx<T>* __restrict__ ch, const cplx<T>* __restrict__ bh,
                                                   const cplx<T>* __restrict__ tw, V in) {
    const RingQuarters<T> R = quarter_transforms<T, LOGQ, NTQ, true>(buf, n, ch, bh, tw, in);
    const int jq = n >> 2;
    for (int q = threadIdx.x; q < jq; q += 4 * NTQ) {
        cplx<T> z[4];
        R.combine(q, n, z);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            f[sN + q + r * jq] = z[r].r;
            f[sS + q + r * jq] = -z[r].i;
        }
    }
}

template <class T, int LOGN, int NT, class V>
__device__ __forceinline__ void ring_back_whole(cplx<T>* buf, T* f, int sN, int sS, int n,
                                                const cplx<T>* __restrict__ ch, const cplx<T>* __restrict__ bh,
                                                const cplx<T>* __restrict__ tw, V in) {
    ip::convolve<T, LOGN, NT, true>(
        buf, tw, threadIdx.x, [&](int k) { return k < n ? mul(in(k), ch[k]) : mk<T>(T(0), T(0)); },
        [&](int k) { return bh[k]; },
        [&](int k, cplx<T> v) {
            if (k < n) {
                const cplx<T> z = mul(v, ch[k]);
                f[sN + k] = z.r;
                f[sS + k] = -z.i;
            }
        });
}

// Rings of n = 2^LOGN points.
template <class T, int LOGN, int NT, class V>
__device__ __forceinline__ void ring_back_plain(cplx<T>* buf, T* f, int sN, int sS, const cplx<T>* __restrict__ tw,
                                                V in) {
    constexpr int R = ip::out_radix(LOGN, NT);
    ip::transform<T, LOGN, NT, false, R, R, true, true>(
        buf, tw, threadIdx.x, [&](int k, int) { return in(k); },
        [&](int k, int, int, cplx<T> v) {
            f[sN + k] = v.r;
            if (sN != sS) f[sS + k] = -v.i;
        });
}

// One transform length per launch (KIND 0: rings of 2^LOGN points, KIND 2: Bluestein
// rings as quarters of 2^LOGN points).
template <class T, bool SYN, int LOGN, int NT, int MINB, int KIND>
__global__ void __launch_bounds__(KIND ? 4 * NT : NT, MINB) ring_back_kernel(
    const cplx<T>* __restrict__ Y, T* __restrict__ maps, const int* __restrict__ nphi_t,
    const int* __restrict__ startN_t, const int* __restrict__ startS_t, const int* __restrict__ shifted_t,
    const int64_t* __restrict__ shOff_t, const int64_t* __restrict__ ch4Off_t, const int64_t* __restrict__ bh4Off_t,
    const cplx<T>* __restrict__ shift, const cplx<T>* __restrict__ chirp4, const cplx<T>* __restrict__ bhat4,
    const cplx<T>* __restrict__ tw, int p, int L, int Q, int64_t npix, const int* __restrict__ ringlist) {
    extern __shared__ unsigned char smem_raw[];
    cplx<T>* buf = reinterpret_cast<cplx<T>*>(smem_raw);
    const int i = ringlist[blockIdx.y], b = blockIdx.x;
    const int n = nphi_t[i], sN = startN_t[i], sS = startS_t[i];
    const BackInput<T, SYN> in{Y + ((int64_t)b * Q + (i + 1)) * (p + 1), Y + ((int64_t)b * Q + (Q - 2 - i)) * (p + 1),
                               shift + shOff_t[i], n, L, sN == sS, shifted_t[i] != 0};
    T* f = maps + (int64_t)b * npix;
    if constexpr (KIND == 2)
        ring_back_quarters<T, LOGN, NT>(buf, f, sN, sS, n, chirp4 + ch4Off_t[i], bhat4 + bh4Off_t[i], tw, in);
    else
        ring_back_plain<T, LOGN, NT>(buf, f, sN, sS, tw, in);
}

// Every transform of at most 2048 points in one launch of 128 threads per ring
// pair; below 512 points radix-2 passes of run-time length, which keep more of the threads
// busy than radix-16 ones (Nside 16, 1 map: 12.7 us with radix 16, now 10.7, FP64 28.1 and
// 19.3; Nside 64 and more: the same).
template <class T, bool SYN>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 6 : 3) ring_back_short_kernel(
    const cplx<T>* __restrict__ Y, T* __restrict__ maps, const int* __restrict__ nphi_t,
    const int* __restrict__ startN_t, const int* __restrict__ startS_t, const int* __restrict__ shifted_t,
    const int* __restrict__ pow2_t, const int* __restrict__ logn_t, const int* __restrict__ logL_t,
    const int64_t* __restrict__ shOff_t, const int64_t* __restrict__ chOff_t, const int64_t* __restrict__ bhOff_t,
    const cplx<T>* __restrict__ shift, const cplx<T>* __restrict__ chirp, const cplx<T>* __restrict__ bhat,
    const cplx<T>* __restrict__ tw, const cplx<T>* __restrict__ twx, int twlen, int p, int L, int Q, int64_t npix, const int* __restrict__ ringlist) {
    extern __shared__ unsigned char smem_raw[];
    cplx<T>* buf = reinterpret_cast<cplx<T>*>(smem_raw);
    const int i = ringlist[blockIdx.y], b = blockIdx.x;
    const int n = nphi_t[i], sN = startN_t[i], sS = startS_t[i];
    const BackInput<T, SYN> in{Y + ((int64_t)b * Q + (i + 1)) * (p + 1), Y + ((int64_t)b * Q + (Q - 2 - i)) * (p + 1),
                               shift + shOff_t[i], n, L, sN == sS, shifted_t[i] != 0};
    T* f = maps + (int64_t)b * npix;
    const cplx<T>*ch = chirp + chOff_t[i], *bh = bhat + bhOff_t[i];
    if (pow2_t[i]) {
        switch (logn_t[i]) {
            case 11: ring_back_plain<T, 11, 128>(buf, f, sN, sS, twx, in); return;
            case 10: ring_back_plain<T, 10, 128>(buf, f, sN, sS, twx, in); return;
            case 9: ring_back_plain<T, 9, 128>(buf, f, sN, sS, twx, in); return;
            default: break;
        }
    } else {
        switch (logL_t[i]) {
            case 11: ring_back_whole<T, 11, 128>(buf, f, sN, sS, n, ch, bh, twx, in); return;
            case 10: ring_back_whole<T, 10, 128>(buf, f, sN, sS, n, ch, bh, twx, in); return;
            case 9: ring_back_whole<T, 9, 128>(buf, f, sN, sS, n, ch, bh, twx, in); return;
            default: break;
        }
    }
    const int tid = threadIdx.x;
    if (pow2_t[i]) {
        for (int k = tid; k < n; k += 128) buf[k] = in(k);
        __syncthreads();
        block_fft(buf, n, logn_t[i], tw, twlen, false);
    } else {
        const int N = 1 << logL_t[i];
        for (int k = tid; k < N; k += 128) buf[k] = k < n ? mul(in(k), ch[k]) : mk<T>(T(0), T(0));
        __syncthreads();
        block_fft(buf, N, logL_t[i], tw, twlen, false);
        for (int k = tid; k < N; k += 128) buf[k] = mul(buf[k], bh[k]);
        __syncthreads();
        block_fft(buf, N, logL_t[i], tw, twlen, true);
        for (int k = tid; k < n; k += 128) buf[k] = mul(buf[k], ch[k]);
        __syncthreads();
    }
    for (int k = tid; k < n; k += 128) {
        const cplx<T> v = buf[k];
        f[sN + k] = v.r;
        if (sN != sS) f[sS + k] = -v.i;
    }
}

template <class T, bool SYN>
void launch_ring_back(const hpx_plan_s* P, T* maps, cudaStream_t s) {
    const auto& g = P->g;
    const auto& t = P->t;
    const cplx<T>*Y = (const cplx<T>*)P->Y, *shift = (const cplx<T>*)t.shift, *tw = (const cplx<T>*)t.twid;
    for (const auto& c : P->ringClasses) {
        dim3 grid(g.B, c.count);
        const int* list = P->ringList + c.first;
        constexpr bool F = sizeof(T) == 4;
        if (c.N < kRingCtMin) {
            auto kern = ring_back_short_kernel<T, SYN>;
            const size_t smem = (size_t)ip::slots(c.N) * sizeof(cplx<T>);
            allow_shared(kern);
            kern<<<grid, 128, smem, s>>>(Y, maps, t.nphi, t.startN, t.startS, t.shifted, t.pow2, t.logn, t.logL,
                                         t.shOff, t.chOff, t.bhOff, shift, (const cplx<T>*)t.chirp,
                                         (const cplx<T>*)t.bhat, tw, (const cplx<T>*)t.twx, g.Lmax, g.p, g.L, g.Q, g.npix,
                                         list);
            continue;
        }
        const size_t smem = (size_t)(c.blue ? 4 * ip::slots(c.N / 4) : ip::slots(c.N)) * sizeof(cplx<T>);
        auto run = [&](auto kern, int threads) {
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            kern<<<grid, threads, smem, s>>>(Y, maps, t.nphi, t.startN, t.startS, t.shifted, t.shOff, t.ch4Off,
                                             t.bh4Off, shift, (const cplx<T>*)t.chirp4, (const cplx<T>*)t.bhat4,
                                             (const cplx<T>*)t.twx, g.p, g.L, g.Q, g.npix, list);
        };
        if (c.N == 4096) {
            if (c.blue) run(ring_back_kernel<T, SYN, 10, 64, F ? 4 : 2, 2>, 256);
            else run(ring_back_kernel<T, SYN, 12, 256, F ? 4 : 2, 0>, 256);
        } else if (c.N == 8192) {
            if (c.blue) run(ring_back_kernel<T, SYN, 11, 128, F ? 2 : 1, 2>, 512);
            else run(ring_back_kernel<T, SYN, 13, 256, F ? 2 : 1, 0>, 256);
        } else if constexpr (F) {   // nside 2048 (FP32 only)
            run(ring_back_kernel<T, SYN, 12, 256, 1, 2>, 1024);
        }
    }
}

template <class T>
void launch_adjoint(const hpx_plan_s* P, const T* alm, T* maps, cudaStream_t s, T wpos) {
    const auto& g = P->g;
    const auto& t = P->t;
    if (P->fusedM && !P->use_tc) {   // the plan's operators, transposed
        launch_operator_cols<T>(P, P->fusedM, sizeof(T) == 4 && g.B <= 8, alm, s, wpos, true);
    } else {   // (operators stored as FP16 pairs hold 22 bits: the sweeps keep FP32 throughout)
        const int ngroups = (2 * g.B + 31) / 32;
        constexpr int KMAX = sizeof(T) == 4 ? 32 : 16;
        if constexpr (sizeof(T) == 4) {   // angle rows and inputs staged ahead of use
            const int G = sweep_orders_per_warp(g.B, g.L, P->sms), sitems = (g.L / 2 / G + 1) * 4 * ngroups;
            rot_adj_staged_kernel<32><<<(sitems * 32 + 63) / 64, 64, 0, s>>>(
                (const float*)alm, (float*)P->beta, t.skOff, (const cplx<float>*)t.skewT, t.nq, g.P2, g.L, g.p, g.B,
                g.nalm, G, ngroups, sitems, (float)wpos, true);
        } else {
            const int nitems = (g.L + 1) * 2 * ngroups, blocks = (nitems * 32 + 127) / 128;
            rot_adj_kernel<T, KMAX><<<blocks, 128, 0, s>>>(alm, (T*)P->beta, t.skOff, (const cplx<T>*)t.skewT, t.nq,
                                                           g.P2, g.L, g.p, g.B, g.nalm, ngroups, nitems, wpos, true);
        }
        const int nmp = g.L / 2 + 1;
        dim3 grid((nmp * g.B + AC - 1) / AC, (g.P2 + AK - 1) / AK, 4);
        if (sizeof(T) == 8 || !launch_dense_adj_big(P, s, t.D))
            dense_adj_kernel<T><<<grid, 256, 0, s>>>((const T*)t.D, (const cplx<T>*)P->beta, (cplx<T>*)P->bvec, g.P2,
                                                     g.p, g.L, g.B);
    }
    {
        int logM = 0;
        while ((1 << logM) < g.M) ++logM;
        const size_t smem = (size_t)g.M * sizeof(cplx<T>);
        dim3 grid(g.L + 1, g.B);
        if (!launch_nufft2<T>(P, s, T(1))) {
            allow_shared(nufft_adj_kernel<T>);
            nufft_adj_kernel<T><<<grid, 512, smem, s>>>((const cplx<T>*)P->bvec, (cplx<T>*)P->Y, t.nrowptr, t.nent,
                                                    (const T*)t.nentw, (const T*)t.dec, (const cplx<T>*)t.twid,
                                                    g.Lmax, g.M, logM, g.p, g.Q, g.P2);
        }
    }
    {
        launch_ring_back<T, false>(P, maps, s);
        pole_adj_kernel<T><<<g.B, 128, 0, s>>>((const cplx<T>*)P->Y, maps, t.poleN, t.poleS, t.polew, t.npole,
                                               g.p, g.Q, g.npix);
    }
}

// ---------------------------------------------------------------- synthesis
// Spherical-harmonic synthesis f(pixel) = sum_{l,m} a_l^m Y_l^m (real maps: m < 0
// from a_l^{-m} = (-1)^m conj(a_l^m)), the inverse direction of the analysis:
//   1. the transposed Givens sweeps (rot_adj_kernel, unweighted) take order m to
//      order-0/1 Legendre coefficients (the sweeps are orthogonal: R^-1 = R^T);
//   2. dense_adj_kernel with the table Es maps those to the coefficients X_j of
//      F_m(t) = (1/sqrt(2 pi)) sum_l a_l^m Pbar_l^m(cos t) = sum_j X_j cos|sin(j t);
//   3. nufft_adj_kernel evaluates the cosine / sine series at the latitude nodes
//      (type-2 NUFFT; for even m it returns w_r F_m(t_r) with w_r = 2 on rings);
//   4. ring_back_kernel folds the orders into the nphi frequencies of each ring,
//      F_m e^{i m phi0} summed over m = n mod nphi (m in [-lmax, lmax]), and
//      transforms back to the ring's pixels (N and S rings packed as one complex
//      sequence; Bluestein for the polar rings).
template <class T>
void launch_sh_synthesis(const hpx_plan_s* P, const T* alm, T* maps, cudaStream_t s, cudaEvent_t* ev) {
    const auto& g = P->g;
    const auto& t = P->t;
    if (ev) cudaEventRecord(ev[0], s);
    if (sizeof(T) == 4 && P->synT) {
        launch_synth_tc(P, (const float*)alm, s);   // the same operators on the tensor cores
    } else if (P->synM) {
        // the sweeps and Es composed per (m, c)
        launch_operator_cols<T>(P, P->synM, P->synQuad, alm, s, T(1), false);
    } else {
        const int ngroups = (2 * g.B + 31) / 32;
        constexpr int KMAX = sizeof(T) == 4 ? 32 : 16;
        if constexpr (sizeof(T) == 4) {
            const int G = sweep_orders_per_warp(g.B, g.L, P->sms), sitems = (g.L / 2 / G + 1) * 4 * ngroups;
            rot_adj_staged_kernel<32><<<(sitems * 32 + 63) / 64, 64, 0, s>>>(
                (const float*)alm, (float*)P->beta, t.skOff, (const cplx<float>*)t.skewT, t.nq, g.P2, g.L, g.p, g.B,
                g.nalm, G, ngroups, sitems, 1.f, false);
        } else {
            const int nitems = (g.L + 1) * 2 * ngroups, blocks = (nitems * 32 + 127) / 128;
            rot_adj_kernel<T, KMAX><<<blocks, 128, 0, s>>>(alm, (T*)P->beta, t.skOff, (const cplx<T>*)t.skewT, t.nq,
                                                           g.P2, g.L, g.p, g.B, g.nalm, ngroups, nitems, T(1), false);
        }
        const int nmp = g.L / 2 + 1;
        dim3 grid((nmp * g.B + AC - 1) / AC, (g.P2 + AK - 1) / AK, 4);
        if (sizeof(T) == 8 || !launch_dense_adj_big(P, s, t.Es))
            dense_adj_kernel<T><<<grid, 256, 0, s>>>((const T*)t.Es, (const cplx<T>*)P->beta, (cplx<T>*)P->bvec, g.P2,
                                                     g.p, g.L, g.B);
    }
    if (ev) cudaEventRecord(ev[1], s);
    {
        int logM = 0;
        while ((1 << logM) < g.M) ++logM;
        const size_t smem = (size_t)g.M * sizeof(cplx<T>);
        dim3 grid(g.L + 1, g.B);
        if (!launch_nufft2<T>(P, s, T(0.5))) {
            allow_shared(nufft_adj_kernel<T>);
            nufft_adj_kernel<T><<<grid, 512, smem, s>>>((const cplx<T>*)P->bvec, (cplx<T>*)P->Y, t.nrowptr, t.nent,
                                                        (const T*)t.nentw, (const T*)t.dec, (const cplx<T>*)t.twid,
                                                        g.Lmax, g.M, logM, g.p, g.Q, g.P2);
        }
    }
    if (ev) cudaEventRecord(ev[2], s);
    launch_ring_back<T, true>(P, maps, s);
    if (ev)
        for (int k = 3; k <= hpx_plan_s::kStages; ++k) cudaEventRecord(ev[k], s);
}

template void launch_sh_synthesis<float>(const hpx_plan_s*, const float*, float*, cudaStream_t, cudaEvent_t*);
template void launch_sh_synthesis<double>(const hpx_plan_s*, const double*, double*, cudaStream_t, cudaEvent_t*);

template void launch_adjoint<float>(const hpx_plan_s*, const float*, float*, cudaStream_t, float);
template void launch_adjoint<double>(const hpx_plan_s*, const double*, double*, cudaStream_t, double);

}  // namespace hpx

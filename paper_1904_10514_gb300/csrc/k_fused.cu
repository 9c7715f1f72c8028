// Per-order operators: the latitude least-squares solve, the change of basis to
// order-0/1 Legendre functions (operator D) and the m/2 Givens sweeps of
// Sec. 3.3 are all fixed linear maps, so for every order m and parity chain c
// their composition is one matrix
//     M_{m,c} = R_{m,c} D_par[rows of chain c],   N(m,c) x P2,
// with R_{m,c} the product of the sweeps.  The plan builds every M_{m,c} once,
// in FP64 on the GPU, by running the same register-wavefront sweeps over the
// columns of D (build_fused_kernel), and stores it rounded to the plan precision
// (n_alm x P2 entries in total, 8.6 GB in FP32 at lmax 2048).  The analysis then
// needs one multi-map contraction per (m, c) instead of the dense stage and the
// run-time sweeps (fused_apply_kernel):
//     a_{m+c+2i}^m[map] = sum_k M_{m,c}[i][k] * b[map][m][par][k].
#include <algorithm>

#include "plan.h"
#include "plan_math.h"
#include "sweep.cuh"

namespace hpx {

// Element (row i, column k) of a chain of n rows in the layout of fused_quad_kernel.
__host__ __device__ inline int64_t quad_elem(int n, int ldm, int i, int k) {
    const int g0 = i & ~31, cnt = n - g0 < 32 ? n - g0 : 32;
    return (int64_t)g0 * ldm + (int64_t)(k >> 2) * 4 * cnt + 4 * (i - g0) + (k & 3);
}

// ---------------------------------------------------------------- build (FP64)
// One warp per (m, chain c, group of 32 complex columns); complex column j holds
// the real columns 2j and 2j+1 of D.  The chain of each lane lives in `scratch`.
template <class T>
__global__ void __launch_bounds__(64) build_fused_kernel(const double* __restrict__ D, T* __restrict__ Mout,
                                                         const int64_t* __restrict__ moff,
                                                         const int64_t* __restrict__ skOff,
                                                         const cplx<double>* __restrict__ skew, int nq, int P2,
                                                         int ldm, int L, int m_lo, int m_cnt, int ngroups,
                                                         cplx<double>* __restrict__ scratch,
                                                         const int64_t* __restrict__ tcOff,
                                                         const int* __restrict__ tcFirst, bool quad) {
    constexpr int KMAX = 16;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int nitems = m_cnt * 2 * ngroups;
    if (warp >= nitems) return;
    const int g = warp % ngroups;
    const int c = (warp / ngroups) & 1;
    const int mi = warp / (2 * ngroups);
    const int m = m_lo + mi;
    const int m0 = m & 1;
    const int S = (m - m0) >> 1;
    const int ncplx = (P2 + 1) / 2;
    const int j = 32 * g + lane;
    if (j >= ncplx) return;
    const int par = (m0 + c) & 1;
    const int q0 = (m0 == 1 && c == 1) ? 1 : 0;
    cplx<double>* chain = scratch + ((int64_t)mi * 2 + c) * P2 * ncplx + j;
    const int64_t ldc = ncplx;
    const double* Dp = D + ((size_t)(m0 * 2 + par) * P2) * P2;
    int n = chain_len(m0, c, L);
    for (int i = 0; i < n; ++i) {
        const double* row = Dp + (size_t)(q0 + i) * P2;
        chain[(int64_t)i * ldc] = mk<double>(row[2 * j], (2 * j + 1 < P2) ? row[2 * j + 1] : 0.0);
    }
    int s0 = 0;
    auto block = [&](int s) {
        return skew + (skOff[(size_t)(m0 * 2 + c) * nq + (s >> 5)] + 2 * (s & 31)) * 32;
    };
    while (S - s0 >= KMAX && n > 0) {
        sweep_pass<double, KMAX>(chain, ldc, n, block(s0), s0 & 31);
        n -= KMAX;
        s0 += KMAX;
    }
#define HPX_SUBPASS(KK)                                                   \
    if (S - s0 >= KK && n > 0) {                                          \
        sweep_pass<double, KK>(chain, ldc, n, block(s0), s0 & 31);        \
        n -= KK;                                                          \
        s0 += KK;                                                         \
    }
    HPX_SUBPASS(8)
    HPX_SUBPASS(4)
    HPX_SUBPASS(2)
    HPX_SUBPASS(1)
#undef HPX_SUBPASS
    if (tcOff) {   // tensor-core layout (FP32 plans)
        for (int i = 0; i < n; ++i) {
            const cplx<double> v = chain[(int64_t)i * ldc];
            const int rp = (min(128, n - (i & ~127)) + 7) & ~7;
            T* out = Mout + tcOff[tcFirst[m * 2 + c] + (i >> 7)];
            out[tc_elem(rp, i & 127, 2 * j)] = (T)v.r;
            if (2 * j + 1 < P2) out[tc_elem(rp, i & 127, 2 * j + 1)] = (T)v.i;
        }
        return;
    }
    T* out = Mout + moff[(size_t)m * 2 + c] * ldm;
    if (quad) {   // groups of 32 rows, four k side by side (fused_quad_kernel)
        for (int i = 0; i < n; ++i) {
            const cplx<double> v = chain[(int64_t)i * ldc];
            out[quad_elem(n, ldm, i, 2 * j)] = (T)v.r;
            if (2 * j + 1 < P2) out[quad_elem(n, ldm, i, 2 * j + 1)] = (T)v.i;
        }
        return;
    }
    for (int i = 0; i < n; ++i) {
        const cplx<double> v = chain[(int64_t)i * ldc];
        out[(size_t)i * ldm + 2 * j] = (T)v.r;
        if (2 * j + 1 < P2) out[(size_t)i * ldm + 2 * j + 1] = (T)v.i;
    }
}

// ---------------------------------------------------------------- apply
namespace {
constexpr int kFusedRows = 64;   // rows per block of fused_rows_kernel
}  // namespace

// Block = one (m, c, tile of 8*TR rows) x 2*TC maps; TR*TC threads, each 8 rows x 2 maps.
// M rows are padded to ldm (a multiple of 4, zero filled) so that they load as
// 16-byte vectors.
template <class T, int TR, int TC>
__global__ void __launch_bounds__(TR* TC) fused_apply_kernel(const T* __restrict__ M, const int64_t* __restrict__ moff,
                                                             const int* __restrict__ tiles,
                                                             const cplx<T>* __restrict__ bvec,
                                                             cplx<T>* __restrict__ alm, int P2, int ldm, int p,
                                                             int L, int B, int64_t nalm) {
    constexpr int FR = 8 * TR, FC = 2 * TC, NT = TR * TC;
    constexpr int FK = sizeof(T) == 4 ? 16 : 8;   // k per stage
    constexpr int VA = 16 / sizeof(T);            // elements per 16-byte vector
    __shared__ __align__(16) T As[FK][FR + 4];
    __shared__ __align__(16) cplx<T> Bs[FK][FC];
    const int m = tiles[3 * blockIdx.x], c = tiles[3 * blockIdx.x + 1], i0 = tiles[3 * blockIdx.x + 2];
    const int m0 = m & 1;
    const int par = (m0 + c) & 1;
    const int nrows = chain_len(m, c, L);
    const int b0 = blockIdx.y * FC;
    const T* A = M + moff[(size_t)m * 2 + c] * ldm;
    const int tid = threadIdx.x;
    const int tr = tid % TR, tc = tid / TR;
    T accr[8][2], acci[8][2];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int q = 0; q < 2; ++q) { accr[r][q] = T(0); acci[r][q] = T(0); }

    for (int k0 = 0; k0 < P2; k0 += FK) {
        // A tile: FR rows x 16 k as 16-byte vectors, stored k-major
        for (int e = tid; e < FR * (FK / VA); e += NT) {
            const int rr = e % FR, kv = e / FR;   // a warp stores 32 consecutive rows: no bank conflicts
            const int i = i0 + rr, k = k0 + kv * VA;
            T v[VA];
            if (i < nrows && k < ldm) {
                if constexpr (sizeof(T) == 4) {
                    const float4 q4 = *reinterpret_cast<const float4*>(A + (size_t)i * ldm + k);
                    v[0] = q4.x; v[1] = q4.y; v[2] = q4.z; v[3] = q4.w;
                } else {
                    const double2 q2 = *reinterpret_cast<const double2*>(A + (size_t)i * ldm + k);
                    v[0] = q2.x; v[1] = q2.y;
                }
            } else {
#pragma unroll
                for (int q = 0; q < VA; ++q) v[q] = T(0);
            }
#pragma unroll
            for (int q = 0; q < VA; ++q) As[kv * VA + q][rr] = v[q];
        }
        // B tile: FC maps x 16 k (each map's column is contiguous in k)
        for (int e = tid; e < FC * FK; e += NT) {
            const int cc = e / FK, kk = e % FK;
            const int b = b0 + cc, k = k0 + kk;
            Bs[kk][cc] = (b < B && k < P2) ? bvec[(((int64_t)b * (p + 1) + m) * 2 + par) * P2 + k]
                                           : mk<T>(T(0), T(0));
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < FK; ++kk) {
            T a[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) a[r] = As[kk][tr * 8 + r];
            const cplx<T> x0 = Bs[kk][tc * 2], x1 = Bs[kk][tc * 2 + 1];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                accr[r][0] += a[r] * x0.r;
                acci[r][0] += a[r] * x0.i;
                accr[r][1] += a[r] * x1.r;
                acci[r][1] += a[r] * x1.i;
            }
        }
        __syncthreads();
    }
    const int64_t base = (int64_t)m * (2 * L + 1 - m) / 2 + m + c;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int b = b0 + tc * 2 + q;
        if (b >= B) continue;
        cplx<T>* out = alm + (int64_t)b * nalm + base;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int i = i0 + tr * 8 + r;
            if (i < nrows) out[2 * i] = mk<T>(accr[r][q], acci[r][q]);
        }
    }
}

// FP32 batches of at most 8 maps.  The operator is stored for it at plan time in
// groups of 32 rows of one chain (the last group of a chain has fewer, cnt), four k
// of all rows of a group side by side (quad_elem), so that lane = row reads 16 bytes
// of 512 contiguous ones per four k and every coefficient is one thread's sum over k
// in ascending order (the order of the 32-map form below, so a map's coefficients
// do not depend on the batch).  b sits in shared memory, read as broadcasts.  The
// bound is the operator's stream, 4 (nside + 1) n_alm bytes per call: blocks of four
// warps (128 rows) with eight loads in flight per lane.  Before, row-major M went
// through shared memory in tiles of 512 rows x 2 maps with 64 threads: analysis and
// C_l of one map at Nside 256 took 297 us, now 92; five at Nside 128 79.9, now 64.5.
// BLOCKED (the transposed synthesis of 5 to 8 maps, launch_fused): each 32 k are summed
// by themselves and then added, as few roundings as the lanes' sums of fused_rows_kernel.
template <int NB, bool BLOCKED = false>
__global__ void __launch_bounds__(128) fused_quad_kernel(const float* __restrict__ M, const int64_t* __restrict__ moff,
                                                         const int* __restrict__ tiles,
                                                         const cplx<float>* __restrict__ bvec,
                                                         cplx<float>* __restrict__ alm, int P2, int ldm, int p, int L,
                                                         int B, int64_t nalm) {
    constexpr int NC = 2 * NB;
    extern __shared__ __align__(16) float bq[];   // [ldm][NC]: k, then (map, part)
    const int m = tiles[3 * blockIdx.x], c = tiles[3 * blockIdx.x + 1], i0 = tiles[3 * blockIdx.x + 2];
    const int par = ((m & 1) + c) & 1;
    const int nrows = chain_len(m, c, L);
    const int b0 = blockIdx.y * NB;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < NB; ++q) {
        const cplx<float>* col = bvec + (((int64_t)min(b0 + q, B - 1) * (p + 1) + m) * 2 + par) * P2;
        for (int k = threadIdx.x; k < ldm; k += 128)
            reinterpret_cast<cplx<float>*>(bq)[k * NB + q] =
                b0 + q < B && k < P2 ? col[k] : mk<float>(0.f, 0.f);
    }
    __syncthreads();
    const int g0 = i0 + 32 * warp;   // this warp's group of rows
    const int cnt = min(32, nrows - g0);
    if (lane >= cnt) return;
    const float4* A = reinterpret_cast<const float4*>(M + (moff[(size_t)m * 2 + c] + g0) * ldm) + lane;
    float acc[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) acc[q] = 0.f;
    auto step = [&](const float4& a4, int k4) {
        const float a[4] = {a4.x, a4.y, a4.z, a4.w};
        const float4* x4 = reinterpret_cast<const float4*>(bq + k4 * 4 * NC);
#pragma unroll
        for (int h = 0; h < NC; ++h) {   // 4 NC values: k = h / (NC / 4) when NC >= 4
            const float4 v = x4[h];
            const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int id = 4 * h + e;
                acc[id % NC] = fmaf(a[id / NC], x[e], acc[id % NC]);
            }
        }
    };
    const int n4 = ldm >> 2;
    int k4 = 0;
    float sum[BLOCKED ? NC : 1];
    if constexpr (BLOCKED)
#pragma unroll
        for (int q = 0; q < NC; ++q) sum[q] = 0.f;
    for (; k4 + 8 <= n4; k4 += 8) {
        float4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldg(A + (int64_t)(k4 + u) * cnt);
#pragma unroll
        for (int u = 0; u < 8; ++u) step(v[u], k4 + u);
        if constexpr (BLOCKED)
#pragma unroll
            for (int q = 0; q < NC; ++q) {
                sum[q] += acc[q];
                acc[q] = 0.f;
            }
    }
    for (; k4 < n4; ++k4) step(__ldg(A + (int64_t)k4 * cnt), k4);
    if constexpr (BLOCKED)
#pragma unroll
        for (int q = 0; q < NC; ++q) acc[q] += sum[q];
    const int64_t at = (int64_t)m * (2 * L + 1 - m) / 2 + m + c + 2 * (int64_t)(g0 + lane);
#pragma unroll
    for (int q = 0; q < NB; ++q)
        if (b0 + q < B) alm[(int64_t)(b0 + q) * nalm + at] = mk<float>(acc[2 * q], acc[2 * q + 1]);
}

// FP64 batches (and the FP32 equal-weight analysis of small batches whose synthesis
// operators are row-major): a matrix-vector form.  A block takes 64 rows of one (m, c) and NB
// maps; a warp takes R rows at a time, its lanes split the k of a row (one 16-byte
// load per lane and row: 512 contiguous bytes of the operator per warp load, R loads
// in flight per lane), b sits in shared memory as 2 NB real columns, and the R x 2 NB
// partial sums of the lanes are combined by a butterfly that leaves each lane with
// one result.  Every sum has the same order whatever NB, R and the map's position
// are: lane l adds k = VA l + CH j + a for j, a ascending, the lanes combine over
// lane distance 16, 8, 4, 2, 1, then the last term k = nside.
// The bound is the FP64 pipe (2 FMA per SM and clock on this GPU), so no lane
// computes for a map or row that is not there beyond the tail of a group.  One map,
// Nside 512: analysis and C_l 5.11 -> 1.84 ms (this kernel about 4.2 -> 1.0, FMA floor
// 0.87); Nside 16: 107 -> 78 us.
// Tiles of 512 rows x 2 maps, always computed in full, before.
template <class T, int NB, int R>
__global__ void __launch_bounds__(256) fused_rows_kernel(const T* __restrict__ M, const int64_t* __restrict__ moff,
                                                         const int* __restrict__ tiles,
                                                         const cplx<T>* __restrict__ bvec, T* __restrict__ alm,
                                                         int P2, int ldm, int p, int L, int B, int64_t nalm) {
    constexpr int VA = 16 / sizeof(T), CH = 32 * VA;   // k per lane and load, k per warp load
    constexpr int NC = 2 * NB;
    constexpr int V = R * NC <= 16 ? 16 : R * NC <= 32 ? 32 : 64;   // sums per lane, rounded up
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* bs = reinterpret_cast<T*>(smem_raw);   // [NC][KP], then the NC values at k = K
    const int K = P2 - 1;                     // = nside; the term k = K is added last
    const int KP = (K + CH - 1) / CH * CH;
    T* bl = bs + NC * KP;
    const int m = tiles[3 * blockIdx.x], c = tiles[3 * blockIdx.x + 1];
    const int i0 = tiles[3 * blockIdx.x + 2] + kFusedRows * blockIdx.z;
    const int par = ((m & 1) + c) & 1;
    const int nrows = chain_len(m, c, L);
    if (i0 >= nrows) return;
    const int b0 = blockIdx.y * NB;
    const T* A = M + moff[(size_t)m * 2 + c] * ldm;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < NB; ++q) {
        const cplx<T>* col = bvec + (((int64_t)min(b0 + q, B - 1) * (p + 1) + m) * 2 + par) * P2;
        const bool have = b0 + q < B;
        for (int k = threadIdx.x; k < KP; k += 256) {
            const cplx<T> v = have && k < K ? col[k] : mk<T>(T(0), T(0));
            bs[(2 * q) * KP + k] = v.r;
            bs[(2 * q + 1) * KP + k] = v.i;
        }
        if (threadIdx.x == 0) {
            const cplx<T> v = have ? col[K] : mk<T>(T(0), T(0));
            bl[2 * q] = v.r;
            bl[2 * q + 1] = v.i;
        }
    }
    __syncthreads();
    const int iend = min(i0 + kFusedRows, nrows);
    for (int r0 = i0 + warp * R; r0 < iend; r0 += 8 * R) {
        T acc[V];
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = T(0);
        const T* row[R];
#pragma unroll
        for (int r = 0; r < R; ++r) row[r] = A + (int64_t)min(r0 + r, nrows - 1) * ldm;
#pragma unroll 2
        for (int k = lane * VA; k < K; k += CH) {   // ldm >= k + VA: rows are padded to 4
            T mv[R][VA];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if constexpr (sizeof(T) == 4) {
                    const float4 q4 = __ldg(reinterpret_cast<const float4*>(row[r] + k));
                    mv[r][0] = q4.x; mv[r][1] = q4.y; mv[r][2] = q4.z; mv[r][3] = q4.w;
                } else {
                    const double2 q2 = __ldg(reinterpret_cast<const double2*>(row[r] + k));
                    mv[r][0] = q2.x; mv[r][1] = q2.y;
                }
            }
#pragma unroll
            for (int col = 0; col < NC; ++col) {
                T x[VA];
                if constexpr (sizeof(T) == 4) {
                    const float4 q4 = *reinterpret_cast<const float4*>(bs + col * KP + k);
                    x[0] = q4.x; x[1] = q4.y; x[2] = q4.z; x[3] = q4.w;
                } else {
                    const double2 q2 = *reinterpret_cast<const double2*>(bs + col * KP + k);
                    x[0] = q2.x; x[1] = q2.y;
                }
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int a = 0; a < VA; ++a) acc[r * NC + col] = fma(mv[r][a], x[a], acc[r * NC + col]);
            }
        }
        // butterfly: each level halves the sums a lane holds, then plain adds
        int n = V;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const bool up = (lane & off) != 0;
            if (n > 1) {
                n >>= 1;
#pragma unroll
                for (int v = 0; v < V / 2; ++v)
                    if (v < n) {
                        const T give = up ? acc[v] : acc[v + n];
                        acc[v] = (up ? acc[v + n] : acc[v]) + __shfl_xor_sync(0xffffffffu, give, off);
                    }
            } else {
                acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], off);
            }
        }
        constexpr int PER = V > 32 ? V / 32 : 1;
        const int first = V >= 32 ? lane * PER : lane >> 1;   // V = 16: two lanes hold each sum
#pragma unroll
        for (int v = 0; v < PER; ++v) {
            const int id = first + v, r = id / NC, col = id - r * NC;
            const int i = r0 + r, b = b0 + (col >> 1);
            if (r < R && i < iend && b < B && (V >= 32 || (lane & 1) == 0)) {
                const int64_t base = (int64_t)m * (2 * L + 1 - m) / 2 + m + c;
                alm[((int64_t)b * nalm + base + 2 * i) * 2 + (col & 1)] =
                    fma(A[(int64_t)i * ldm + K], bl[col], acc[v]);
            }
        }
    }
}

// ---------------------------------------------------------------- transposed
// The transposed contraction X[map][m][par][k] = sum_i O_{m,c}[i][k] a_{m+c+2i}^m[map] of
// the same operators, 0 <= k < P2: the adjoint's first two stages (O = M, with the
// coefficients' weights and without the imaginary parts that the analysis never
// returns) and the synthesis' (O = S_{m,c} = R_{m,c} Es, built with Es, the
// Legendre-0/1 -> latitude-Fourier table, in place of D: X are then the cosine / sine
// coefficients of F_m).
struct CoefWeights {
    double pos;    // weight of the m > 0 coefficients (m = 0: 1)
    bool dropim;   // ignore the imaginary parts at m = 0 and m = p
};
template <class T>
__device__ __forceinline__ cplx<T> weighted(cplx<T> v, int m, int p, CoefWeights w) {
    if (m > 0) v = scale(v, (T)w.pos);
    if (w.dropim && (m == 0 || m == p)) v.i = T(0);
    return v;
}

// FP64 plans and FP32 plans off the tensor cores.  A block takes one (m, c), NB maps
// and 32 lanes x 16 bytes of k; its four warps take 32 rows each of every 128, the
// coefficients of the rows sit in shared memory (read as broadcasts), each lane sums
// its k over the warp's rows, and the four partial sums are added in warp order at
// the end.  QUAD: the operator is in the groups of fused_quad_kernel, else row-major.
// P2 = Nside + 1 is one past a multiple of the tiles from Nside 128 (FP32) or 64 (FP64)
// on: the last blocks of the grid take that k, a warp each, instead of a tile of one.
// FP32 is bound by the latency of the tiles' loads, FP64 by the FP64 pipe.  6 maps,
// Nside 256, lmax 400 (synthesis): 96 us as matrix-matrix tiles, 65 us with a tile for
// the last k, now 48 us (in groups of 32 rows).
template <class T, int NB, bool QUAD>
__global__ void __launch_bounds__(128) operator_cols_kernel(const T* __restrict__ M, const int64_t* __restrict__ moff,
                                                            const cplx<T>* __restrict__ alm,
                                                            cplx<T>* __restrict__ bvec, int P2, int ldm, int p, int L,
                                                            int B, int64_t nalm, int nkt, CoefWeights w) {
    constexpr int VA = 16 / sizeof(T), NC = 2 * NB, KT = 32 * VA;
    __shared__ __align__(16) T as[128][NC];
    __shared__ T red[3][VA * NC][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, b0 = blockIdx.y * NB;
    const int ntile = 2 * (L + 1) * nkt;
    if ((int)blockIdx.x >= ntile) {   // the k past the tiles, one (m, c) per warp, lane = row
        const int mc = 4 * (blockIdx.x - ntile) + warp, m = mc >> 1, c = mc & 1, k = nkt * KT;
        if (m > L) return;
        const int n = chain_len(m, c, L), par = ((m & 1) + c) & 1;
        const T* A = M + moff[(size_t)m * 2 + c] * ldm;
        const cplx<T>* in = alm + (int64_t)b0 * nalm + (int64_t)m * (2 * L + 1 - m) / 2 + m + c;
        cplx<T> acc[NB];
#pragma unroll
        for (int q = 0; q < NB; ++q) acc[q] = mk<T>(T(0), T(0));
        for (int i = lane; i < n; i += 32) {
            const int g0 = i & ~31;
            const T v = QUAD ? A[(int64_t)g0 * ldm + (int64_t)(k >> 2) * 4 * min(32, n - g0) + 4 * lane]
                             : A[(int64_t)i * ldm + k];
#pragma unroll
            for (int q = 0; q < NB; ++q)
                if (b0 + q < B) {
                    const cplx<T> x = weighted<T>(in[q * nalm + 2 * i], m, p, w);
                    acc[q].r = fma(v, x.r, acc[q].r);
                    acc[q].i = fma(v, x.i, acc[q].i);
                }
        }
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            for (int o = 16; o > 0; o >>= 1) {
                acc[q].r += __shfl_xor_sync(0xffffffffu, acc[q].r, o);
                acc[q].i += __shfl_xor_sync(0xffffffffu, acc[q].i, o);
            }
            if (lane == 0 && b0 + q < B) bvec[(((int64_t)(b0 + q) * (p + 1) + m) * 2 + par) * P2 + k] = acc[q];
        }
        return;
    }
    const int kt = blockIdx.x % nkt, mc = blockIdx.x / nkt;
    const int m = mc >> 1, c = mc & 1;
    const int par = ((m & 1) + c) & 1;
    const int n = chain_len(m, c, L);
    const int k = kt * KT + lane * VA;
    const bool on = k < P2;   // ldm >= k + VA: rows are padded to 4
    const T* A = M + moff[(size_t)m * 2 + c] * ldm;
    const int64_t base = (int64_t)m * (2 * L + 1 - m) / 2 + m + c;
    T acc[VA][NC];
#pragma unroll
    for (int a = 0; a < VA; ++a)
#pragma unroll
        for (int q = 0; q < NC; ++q) acc[a][q] = T(0);
    for (int r0 = 0; r0 < n; r0 += 128) {
        for (int e = threadIdx.x; e < 128 * NB; e += 128) {
            const int q = e >> 7, i = r0 + (e & 127);
            cplx<T> v = mk<T>(T(0), T(0));
            if (i < n && b0 + q < B) v = weighted<T>(alm[(int64_t)(b0 + q) * nalm + base + 2 * i], m, p, w);
            as[e & 127][2 * q] = v.r;
            as[e & 127][2 * q + 1] = v.i;
        }
        __syncthreads();
        const int g0 = r0 + 32 * warp, cnt = min(32, n - g0);
        if (on && cnt > 0) {
            // row i of the group: stride between rows and first element
            const T* row = QUAD ? A + (int64_t)g0 * ldm + (int64_t)(k >> 2) * 4 * cnt : A + (int64_t)g0 * ldm + k;
            const int64_t step = QUAD ? 4 : ldm;
            auto one = [&](int i, const T (&v)[VA]) {
                const T* x = as[32 * warp + i];
#pragma unroll
                for (int q = 0; q < NC; ++q)
#pragma unroll
                    for (int a = 0; a < VA; ++a) acc[a][q] = fma(v[a], x[q], acc[a][q]);
            };
            auto load = [&](int i, T (&v)[VA]) {
                if constexpr (sizeof(T) == 4) {
                    const float4 f = __ldg(reinterpret_cast<const float4*>(row + i * step));
                    v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
                } else {
                    const double2 f = __ldg(reinterpret_cast<const double2*>(row + i * step));
                    v[0] = f.x; v[1] = f.y;
                }
            };
            int i = 0;
            for (; i + 8 <= cnt; i += 8) {
                T v[8][VA];
#pragma unroll
                for (int u = 0; u < 8; ++u) load(i + u, v[u]);
#pragma unroll
                for (int u = 0; u < 8; ++u) one(i + u, v[u]);
            }
            for (; i < cnt; ++i) {
                T v[VA];
                load(i, v);
                one(i, v);
            }
        }
        __syncthreads();
    }
    if (warp > 0)
#pragma unroll
        for (int a = 0; a < VA; ++a)
#pragma unroll
            for (int q = 0; q < NC; ++q) red[warp - 1][a * NC + q][lane] = acc[a][q];
    __syncthreads();
    if (warp > 0 || !on) return;
#pragma unroll
    for (int u = 0; u < 3; ++u)
#pragma unroll
        for (int a = 0; a < VA; ++a)
#pragma unroll
            for (int q = 0; q < NC; ++q) acc[a][q] += red[u][a * NC + q][lane];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
        if (b0 + q >= B) continue;
        cplx<T>* out = bvec + (((int64_t)(b0 + q) * (p + 1) + m) * 2 + par) * P2 + k;
#pragma unroll
        for (int a = 0; a < VA; ++a)
            if (k + a < P2) out[a] = mk<T>(acc[a][2 * q], acc[a][2 * q + 1]);
    }
}

template <class T>
void launch_operator_cols(const hpx_plan_s* P, const void* M, bool quad, const T* alm, cudaStream_t s, T wpos,
                          bool dropim) {
    const auto& g = P->g;
    const int kt = 32 * 16 / sizeof(T);
    const bool tail = g.P2 > kt && g.P2 % kt == 1;
    const int nkt = tail ? g.P2 / kt : (g.P2 + kt - 1) / kt;
    // maps per block as launch_fused: FP32 as many as possible (8), FP64 no absent ones
    const int nb = sizeof(T) == 4 ? (g.B > 4 ? 8 : g.B > 2 ? 4 : g.B)
                                  : (g.B + (g.B + 3) / 4 - 1) / ((g.B + 3) / 4);
    auto run = [&](auto kern, int NB) {
        dim3 grid((g.L + 1) * 2 * nkt + (tail ? (g.L + 2) / 2 : 0), (g.B + NB - 1) / NB);
        kern<<<grid, 128, 0, s>>>((const T*)M, P->fusedOff, (const cplx<T>*)alm, (cplx<T>*)P->bvec, g.P2,
                                  P->fused_ldm, g.p, g.L, g.B, g.nalm, nkt, CoefWeights{(double)wpos, dropim});
    };
    if constexpr (sizeof(T) == 4) {
        if (quad) {
            if (nb == 1) run(operator_cols_kernel<T, 1, true>, 1);
            else if (nb == 2) run(operator_cols_kernel<T, 2, true>, 2);
            else if (nb == 4) run(operator_cols_kernel<T, 4, true>, 4);
            else run(operator_cols_kernel<T, 8, true>, 8);
            return;
        }
    }
    if (nb == 1) run(operator_cols_kernel<T, 1, false>, 1);
    else if (nb == 2) run(operator_cols_kernel<T, 2, false>, 2);
    else if (nb == 4) run(operator_cols_kernel<T, 4, false>, 4);
    else if constexpr (sizeof(T) == 4) run(operator_cols_kernel<T, 8, false>, 8);
    else run(operator_cols_kernel<T, 3, false>, 3);
}

template void launch_operator_cols<float>(const hpx_plan_s*, const void*, bool, const float*, cudaStream_t, float, bool);
template void launch_operator_cols<double>(const hpx_plan_s*, const void*, bool, const double*, cudaStream_t, double,
                                           bool);

// Rows per block of the apply kernels (the plan builds its tile list with this).
int fused_tile_rows(bool fp64) { return fp64 ? kFusedRows : 128; }

template <class T>
void launch_fused(const hpx_plan_s* P, T* alm, cudaStream_t s, const void* Msyn) {
    const auto& g = P->g;
    const int ldm = P->fused_ldm;
    const T* M = (const T*)(Msyn ? Msyn : P->fusedM);
    if constexpr (sizeof(T) == 4) {
        if (g.B > 8) {
            dim3 grid(P->fused_ntiles, (g.B + 31) / 32);
            fused_apply_kernel<T, 16, 16><<<grid, 256, 0, s>>>(M, P->fusedOff, P->fusedTiles,
                                                               (const cplx<T>*)P->bvec, (cplx<T>*)alm, g.P2, ldm,
                                                               g.p, g.L, g.B, g.nalm);
            return;
        }
    }
    if constexpr (sizeof(T) == 4) {
        if (!Msyn || P->synQuad) {
            auto run = [&](auto kern, int NB) {   // each operator read once: all maps in one block
                const size_t smem = (size_t)2 * NB * ldm * sizeof(float);
                allow_shared(kern);
                kern<<<P->fused_ntiles, 128, smem, s>>>(M, P->fusedOff, P->fusedTiles, (const cplx<float>*)P->bvec,
                                                        (cplx<float>*)alm, g.P2, ldm, g.p, g.L, g.B, g.nalm);
            };
            if (Msyn) run(fused_quad_kernel<8, true>, 8);
            else if (g.B == 1) run(fused_quad_kernel<1>, 1);
            else if (g.B == 2) run(fused_quad_kernel<2>, 2);
            else if (g.B <= 4) run(fused_quad_kernel<4>, 4);
            else run(fused_quad_kernel<8>, 8);
            return;
        }
    }
    // maps per block: FP32 reads each operator once (up to 8 maps); FP64 computes for
    // as few absent maps as possible (groups of at most 4, of equal size)
    const int nb = sizeof(T) == 4 ? (g.B > 4 ? 8 : g.B > 2 ? 4 : g.B)
                                  : (g.B + (g.B + 3) / 4 - 1) / ((g.B + 3) / 4);
    constexpr int per = sizeof(T) == 4 ? 2 : 1;   // blocks of 64 rows per tile of the plan's list
    auto run = [&](auto kern, int NB) {
        constexpr int CH = 32 * 16 / sizeof(T);
        const size_t smem = (size_t)2 * NB * ((g.P2 - 1 + CH - 1) / CH * CH + 1) * sizeof(T);
        allow_shared(kern);
        dim3 grid(P->fused_ntiles, (g.B + NB - 1) / NB, per);
        kern<<<grid, 256, smem, s>>>(M, P->fusedOff, P->fusedTiles, (const cplx<T>*)P->bvec, alm, g.P2, ldm, g.p,
                                     g.L, g.B, g.nalm);
    };
    if (nb == 1) run(fused_rows_kernel<T, 1, 8>, 1);
    else if (nb == 2) run(fused_rows_kernel<T, 2, 8>, 2);
    else if (nb == 4) run(fused_rows_kernel<T, 4, 4>, 4);
    else if constexpr (sizeof(T) == 4) run(fused_rows_kernel<T, 8, 4>, 8);
    else run(fused_rows_kernel<T, 3, 4>, 3);
}

// Builds the per-order operators of a plan (called once by hpx_plan_ex).
// D64 / skew64 are FP64 device copies of D and of the skewed sweep angles.  form: 0
// row-major, 1 the tensor-core tiles, 2 the groups of fused_quad_kernel.
template <class T>
int build_fused(hpx_plan_s* P, const double* D64, const cplx<double>* skew64, cudaStream_t s, void* out,
                int form) {
    const auto& g = P->g;
    const int ncplx = (g.P2 + 1) / 2;
    const int ngroups = (ncplx + 31) / 32;
    const int chunk = 64;
    cplx<double>* scratch = nullptr;
    const size_t sbytes = (size_t)chunk * 2 * g.P2 * ncplx * sizeof(cplx<double>);
    if (cudaMalloc(&scratch, sbytes) != cudaSuccess) return -1;
    for (int m_lo = 0; m_lo <= g.L; m_lo += chunk) {
        const int m_cnt = std::min(chunk, g.L + 1 - m_lo);
        const int nitems = m_cnt * 2 * ngroups;
        const int blocks = (nitems * 32 + 63) / 64;
        build_fused_kernel<T><<<blocks, 64, 0, s>>>(D64, (T*)out, P->fusedOff, P->t.skOff, skew64, P->t.nq,
                                                    g.P2, P->fused_ldm, g.L, m_lo, m_cnt, ngroups, scratch,
                                                    form == 1 ? P->tcOff : nullptr, P->tcFirst, form == 2);
    }
    const cudaError_t e = cudaStreamSynchronize(s);
    cudaFree(scratch);
    return e == cudaSuccess ? 0 : -1;
}

template void launch_fused<float>(const hpx_plan_s*, float*, cudaStream_t, const void*);
template void launch_fused<double>(const hpx_plan_s*, double*, cudaStream_t, const void*);
template int build_fused<float>(hpx_plan_s*, const double*, const cplx<double>*, cudaStream_t, void*, int);
template int build_fused<double>(hpx_plan_s*, const double*, const cplx<double>*, cudaStream_t, void*, int);

}  // namespace hpx

// Latitude least-squares solve and change of basis to order-0/1 normalised
// Legendre functions (Sec. 3.2.2 and the first half of Sec. 3.3).
//
// For every column (map, m) the LS solution of the truncated normal equations
// T g = b (T = F^* F restricted to the m = 4 Nside + 1 latitude modes, split by
// the DFS parity of m into a cosine and a sine system) is followed by the
// projection of the resulting latitude series onto Pbar_l^0 (m even) or Pbar_l^1
// (m odd), scaled by sqrt(2 pi).  Both maps are fixed and shared by all columns
// and maps, so the plan premultiplies them (FP64) into one dense operator per
// (parity of m, parity of l):  beta = D b.  This kernel is that multi-column
// contraction:  beta[m][par][q][b][re/im] = sum_k D[m&1][par][q][k] * bvec[b][m][par][k].
// The output is column-contiguous (all maps of one (m, par, q) side by side) for
// the rotation sweeps, which process one real column per lane.
#include "plan.h"

namespace hpx {

// FP32: tiles of 128 rows x 64 complex columns, 256 threads, 8 rows x 4 complex columns
// per thread (64 FMA per k against 4 + 2 shared-memory vector loads), the next 16 k of
// both operands in registers while the current ones are multiplied.  Every
// result is one thread's sum over k in ascending order.  ADJ: the transposed operator,
// rows = k of D, reduction over q (beta -> bvec, the adjoint's direction).
// The bound is the FP32 pipe.  8 maps, Nside 2048: 46.4 ms (64 x 32 tiles, 4 x 2 per
// thread) to 27.3 ms forward, 47.6 to 27.6 ms transposed (41 TFLOP/s).
namespace {
constexpr int DR = 128, DC = 64, DK = 16;   // rows, complex columns, reduction chunk
}  // namespace

template <bool ADJ>
__global__ void __launch_bounds__(256, 2) dense_big_kernel(const float* __restrict__ D, const cplx<float>* __restrict__ in,
                                                           cplx<float>* __restrict__ out, int P2, int p, int L, int B) {
    __shared__ __align__(16) float As[2][DK][DR + 4];
    __shared__ __align__(16) cplx<float> Bs[2][DK][DC + 2];
    const int mpar = blockIdx.z >> 1, par = blockIdx.z & 1;
    const int nmp = (L >= mpar) ? (L - mpar) / 2 + 1 : 0;
    const int ncols = nmp * B;
    const int c0 = blockIdx.x * DC, q0 = blockIdx.y * DR;
    if (c0 >= ncols) return;
    const float* Dm = D + ((size_t)(mpar * 2 + par) * P2) * P2;
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;   // rows 4 tx + {0..3, 64..67}, columns 4 ty ..
    // loads of a chunk: A 8 values, B 4 complex values per thread
    float ra[8];
    cplx<float> rb[4];
    // column of B this thread loads (the same for all chunks), and its address
    const cplx<float>* bcol[4];
    int bk[4], bc[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int id = tid + 256 * e;
        // forward: 16 consecutive k of one column are contiguous; adjoint: consecutive columns are
        bk[e] = ADJ ? id / DC : id % DK;
        bc[e] = ADJ ? id % DC : id / DK;
        const int col = c0 + bc[e];
        const int b = col % B, m = 2 * (col / B) + mpar;
        bcol[e] = col < ncols ? (ADJ ? in + (((int64_t)m * 2 + par) * P2) * B + b
                                     : in + (((int64_t)b * (p + 1) + m) * 2 + par) * P2)
                              : nullptr;
    }
    auto load = [&](int k0) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int id = tid + 256 * e;
            // forward: A[k][row] = D[row][k] (k contiguous); adjoint: D[k][row] (row contiguous)
            const int kk = ADJ ? id / DR : id % DK, rr = ADJ ? id % DR : id / DK;
            const int k = k0 + kk, r = q0 + rr;
            ra[e] = (k < P2 && r < P2) ? Dm[ADJ ? (size_t)k * P2 + r : (size_t)r * P2 + k] : 0.f;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int k = k0 + bk[e];
            bool ok = bcol[e] != nullptr && k < P2;
            if (ADJ) ok = ok && 2 * k + par <= L && 2 * k + par >= mpar;
            rb[e] = ok ? bcol[e][ADJ ? (int64_t)k * B : k] : mk<float>(0.f, 0.f);
        }
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int id = tid + 256 * e;
            As[buf][ADJ ? id / DR : id % DK][ADJ ? id % DR : id / DK] = ra[e];
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) Bs[buf][bk[e]][bc[e]] = rb[e];
    };
    float accr[8][4], acci[8][4];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) { accr[r][c] = 0.f; acci[r][c] = 0.f; }
    load(0);
    store(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = 0; k0 < P2; k0 += DK) {
        const bool more = k0 + DK < P2;
        if (more) load(k0 + DK);
#pragma unroll
        for (int kk = 0; kk < DK; ++kk) {
            const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][kk][4 * tx]);
            const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][kk][64 + 4 * tx]);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float4 b0 = *reinterpret_cast<const float4*>(&Bs[buf][kk][4 * ty]);
            const float4 b1 = *reinterpret_cast<const float4*>(&Bs[buf][kk][4 * ty + 2]);
            const float xr[4] = {b0.x, b0.z, b1.x, b1.z}, xi[4] = {b0.y, b0.w, b1.y, b1.w};
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    accr[r][c] = fmaf(a[r], xr[c], accr[r][c]);
                    acci[r][c] = fmaf(a[r], xi[c], acci[r][c]);
                }
        }
        if (more) {
            store(buf ^ 1);
            __syncthreads();
            buf ^= 1;
        }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int col = c0 + 4 * ty + c;
        if (col >= ncols) continue;
        const int b = col % B, m = 2 * (col / B) + mpar;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int q = q0 + (r < 4 ? 4 * tx + r : 60 + 4 * tx + r);
            if (q >= P2) continue;
            const cplx<float> v = mk<float>(accr[r][c], acci[r][c]);
            if (ADJ) out[(((int64_t)b * (p + 1) + m) * 2 + par) * P2 + q] = v;
            else out[(((int64_t)m * 2 + par) * P2 + q) * B + b] = v;
        }
    }
}

// The large tiles only where they give every SM two blocks (below, the smaller tiles
// spread the work over more of them); both sum in the same order.
static bool dense_big(const hpx_plan_s* P, dim3& grid) {
    const auto& g = P->g;
    grid = dim3(((g.L / 2 + 1) * g.B + DC - 1) / DC, (g.P2 + DR - 1) / DR, 4);
    return (int64_t)grid.x * grid.y * 4 >= 2 * P->sms;
}

bool launch_dense_adj_big(const hpx_plan_s* P, cudaStream_t s, const void* Dmat) {
    const auto& g = P->g;
    dim3 grid;
    if (!dense_big(P, grid)) return false;
    dense_big_kernel<true><<<grid, 256, 0, s>>>((const float*)Dmat, (const cplx<float>*)P->beta,
                                                (cplx<float>*)P->bvec, g.P2, g.p, g.L, g.B);
    return true;
}

namespace {
constexpr int TQ = 64;   // rows (q) per block
constexpr int TC = 32;   // columns (map, m) per block
constexpr int TK = 16;   // k per stage
}  // namespace

template <class T>
__global__ void __launch_bounds__(256) dense_kernel(const T* __restrict__ D,
                                                    const cplx<T>* __restrict__ bvec,
                                                    cplx<T>* __restrict__ beta, int P2, int p, int L,
                                                    int B) {
    __shared__ T Ds[TK][TQ + 1];
    __shared__ cplx<T> Bs[TK][TC + 1];   // padded: the loads below store 16 consecutive k of one column
    const int mpar = blockIdx.z >> 1, par = blockIdx.z & 1;
    const int nmp = (L >= mpar) ? (L - mpar) / 2 + 1 : 0;
    const int ncols = nmp * B;
    const int c0 = blockIdx.x * TC, q0 = blockIdx.y * TQ;
    if (c0 >= ncols) return;
    const T* Dm = D + ((size_t)(mpar * 2 + par) * P2) * P2;
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;   // 4 rows x 2 columns per thread
    T accr[4][2], acci[4][2];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < 2; ++c) { accr[a][c] = T(0); acci[a][c] = T(0); }

    for (int k0 = 0; k0 < P2; k0 += TK) {
        for (int e = tid; e < TQ * TK; e += 256) {
            const int qq = e / TK, kk = e % TK;
            const int q = q0 + qq, k = k0 + kk;
            Ds[kk][qq] = (q < P2 && k < P2) ? Dm[(size_t)q * P2 + k] : T(0);
        }
        for (int e = tid; e < TC * TK; e += 256) {
            const int cc = e / TK, kk = e % TK;
            const int col = c0 + cc, k = k0 + kk;
            cplx<T> v = mk<T>(T(0), T(0));
            if (col < ncols && k < P2) {
                const int b = col % B, mi = col / B;
                const int m = 2 * mi + mpar;
                v = bvec[(((int64_t)b * (p + 1) + m) * 2 + par) * P2 + k];
            }
            Bs[kk][cc] = v;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            T a[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) a[r] = Ds[kk][tx * 4 + r];
            cplx<T> bb[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) bb[c] = Bs[kk][ty * 2 + c];
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    accr[r][c] += a[r] * bb[c].r;
                    acci[r][c] += a[r] * bb[c].i;
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
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int q = q0 + tx * 4 + r;
            if (q < P2) beta[(((int64_t)m * 2 + par) * P2 + q) * B + b] = mk<T>(accr[r][c], acci[r][c]);
        }
    }
}

template <class T>
void launch_dense(const hpx_plan_s* P, cudaStream_t s, const void* Dmat) {
    const auto& g = P->g;
    const int nmp = g.L / 2 + 1;
    if constexpr (sizeof(T) == 4) {
        dim3 big;
        if (dense_big(P, big)) {
            dense_big_kernel<false><<<big, 256, 0, s>>>((const float*)(Dmat ? Dmat : P->t.D),
                                                        (const cplx<float>*)P->bvec, (cplx<float>*)P->beta, g.P2,
                                                        g.p, g.L, g.B);
            return;
        }
    }
    dim3 grid((nmp * g.B + TC - 1) / TC, (g.P2 + TQ - 1) / TQ, 4);
    dense_kernel<T><<<grid, 256, 0, s>>>((const T*)(Dmat ? Dmat : P->t.D), (const cplx<T>*)P->bvec, (cplx<T>*)P->beta,
                                         g.P2, g.p, g.L, g.B);
}

template void launch_dense<float>(const hpx_plan_s*, cudaStream_t, const void*);
template void launch_dense<double>(const hpx_plan_s*, cudaStream_t, const void*);

}  // namespace hpx

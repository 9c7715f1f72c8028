// Step 2 (Sec. 3.2): DFS doubling in latitude and the right-hand side of the
// least-squares inverse NUFFT-II, b = F^* y (the type-1 NUFFT of Sec. 3.2.2).
//
// For longitude wavenumber m the DFS data (remark of Sec. 3.2.1) are y_r at the
// latitudes theta_r (r = 0..4 Nside: poles and rings) and (-1)^m y_r at
// 2 pi - theta_r (interior r).  The type-1 sums
//     B_j = sum_nodes y_nu e^{-i j theta_nu},   j = 0..p,
// are computed with an exponential-of-semicircle (ES) kernel: the node values are
// spread onto a uniform grid of M = 8 Nside points on [0, 2 pi) (a gather over a
// precomputed sparse table, accumulated in shared memory), the grid is
// transformed by an M-point FFT in shared memory, and each mode is divided by
// the kernel's Fourier transform (table `dec`, FP64-built).
//
// By the DFS parity the LS problem splits (even m: cosine basis, odd m: sine
// basis); the outputs are the normal-equation right-hand sides
//     even m:  b_j = sum_r w_r y_r cos(j theta_r)          = B_j
//     odd m:   b_j = sum_{interior r} y_r sin(j theta_r)   = (i/2) B_j
// stored as bvec[b][m][j & 1][j >> 1].
//
// nufft_kernel does the whole step per column (used by the allocation-free
// entry point); plans run it as a spreading and a grid-FFT kernel below.
#include "fft_ip.cuh"
#include "fp16pair.cuh"
#include "plan.h"

namespace hpx {

template <class T, int E>
__global__ void __launch_bounds__(512, (E <= 16 ? 2 : 1)) nufft_kernel(
    const cplx<T>* __restrict__ Y, cplx<T>* __restrict__ bvec, const int* __restrict__ nstart,
    const T* __restrict__ swts, int nsw, const T* __restrict__ dec, const cplx<T>* __restrict__ tw, int twlen, int M,
    int logM, int p, int Q, int P2) {
    extern __shared__ unsigned char smem_raw[];
    cplx<T>* u = reinterpret_cast<cplx<T>*>(smem_raw);   // M
    cplx<T>* y = u + M + M / 16;                           // Q (after the padded grid)
    const int m = blockIdx.x;
    const int b = blockIdx.y;
    const int tid = threadIdx.x, nt = blockDim.x;
    const cplx<T>* col = Y + (int64_t)b * Q * (p + 1) + m;
    for (int r = tid; r < Q; r += nt) y[r] = col[(int64_t)r * (p + 1)];
    __syncthreads();
    const bool odd = (m & 1) != 0;
    // gather-spread: grid point t sees the DFS nodes nstart[t] .. nstart[t]+nsw-1
    // (cyclically; node nu <= 4 Nside is theta_nu, beyond it is the mirror of
    // ring 8 Nside - nu, whose data carry the sign (-1)^m); M = 8 Nside nodes.
    const int half = M >> 1;
    for (int t = tid; t < M; t += nt) {
        T ar = T(0), ai = T(0);
        int nu = nstart[t];
        for (int e = 0; e < nsw; ++e) {
            const T w = swts[(size_t)e * M + t];
            const bool mir = nu > half;
            const cplx<T> v = y[mir ? M - nu : nu];
            const T ws = (odd && mir) ? -w : w;
            ar += ws * v.r;
            ai += ws * v.i;
            nu = (nu + 1 == M) ? 0 : nu + 1;
        }
        u[pad(t)] = mk<T>(ar, ai);
    }
    __syncthreads();
    block_fft_pad<T, E>(u, logM, tw, twlen, false);
    cplx<T>* out = bvec + ((int64_t)b * (p + 1) + m) * 2 * P2;
    for (int j = tid; j <= p; j += nt) {
        cplx<T> v = scale(u[pad(j)], dec[j]);
        if (odd) v = mk<T>(T(-0.5) * v.i, T(0.5) * v.r);
        out[(j & 1) * P2 + (j >> 1)] = v;
    }
    // the odd-parity block has one slot fewer (j = p + 1 would be index p/2)
    if (tid == 0) out[P2 + (P2 - 1)] = mk<T>(T(0), T(0));
}

// ---------------------------------------------------------------------------
// The same step as two kernels (the analysis path of plans):
//
// The spreading.  The grid values obey u[M - t] = (-1)^m u[t], so only the half
// grid t = 0..M/2 is spread, with every mirrored node folded into its latitude
// node (weights hwts, one per parity of m).  With e the half grid of an even
// order m and o that of m + 1, the sequence the grid FFT transforms for the two
// of them is z_t = e_t + o_t for t <= M/2 and z_{M-t} = e_t - o_t, and in FP32
// its leaky first difference dz_t = z_t - rho z_{t-1} (cyclic; kPrewhiten below).
// The spreading kernels have both orders in neighbouring lanes and the
// neighbouring grid points in shared memory, so they write dz itself,
// U[b][m / 2][t], t < M: the grid FFT reads one value per element where it would
// read four and combine them (rho = 0: z itself).
//
// Order of the values of a pair in U: dz_t at t for t <= M/2, then dz_{M-t} at M/2 + t
// for 0 < t < M/2, so that a tile of grid points is one aligned run in either half
// (grid_index).
//
// The staged tile zs: rows of 34 grid points t0 - 1 .. t0 + 32, even rows e + o, odd
// rows e - o of the pair.  spread_value: element (row ml, grid point t0 + lane) of the
// output; zrow the row, other the row of its odd partner (read at t = 0 only:
// z_{-1} = z_{M-1} = e_1 - o_1).
constexpr int kZS = 35;   // row stride of the staged tile (odd: no bank conflicts)
__device__ __forceinline__ int grid_index(int i, int M) { return i <= M / 2 ? i : M + M / 2 - i; }
template <class T>
__device__ __forceinline__ cplx<T> spread_value(const cplx<T>* zrow, const cplx<T>* other, int lane, int t, bool odd,
                                                T rho) {
    const cplx<T> z = zrow[lane + 1];
    const cplx<T> zp = odd ? zrow[lane + 2] : t == 0 ? other[2] : zrow[lane];
    return mk<T>(fma(-rho, zp.r, z.r), fma(-rho, zp.i, z.i));
}
// e + o (even lanes) or e - o (odd lanes) from this lane's order and its partner's
template <class T>
__device__ __forceinline__ cplx<T> pair_value(T ar, T ai, int lane) {
    const T pr = __shfl_xor_sync(0xffffffffu, ar, 1), pi = __shfl_xor_sync(0xffffffffu, ai, 1);
    return (lane & 1) ? mk<T>(pr - ar, pi - ai) : mk<T>(ar + pr, ai + pi);
}

// spread_kernel: 32 grid points x 32 consecutive orders of one map per block: the
// ring coefficients of the latitude nodes it needs are read row by row (32 orders
// = contiguous), the taps per grid point are summed from shared memory, and
// the tile is written transposed, as contiguous segments of U.  FP64, and FP32
// kernels wider than the register-blocked form takes.
template <class T>
__global__ void __launch_bounds__(256) spread_kernel(const cplx<T>* __restrict__ Y, cplx<T>* __restrict__ U,
                                                     const int* __restrict__ hstart, const T* __restrict__ hwts,
                                                     int E, int H, int p, int Q, int L, T rho) {
    extern __shared__ unsigned char smem_raw[];
    cplx<T>* zs = reinterpret_cast<cplx<T>*>(smem_raw);   // [32 rows][kZS]
    cplx<T>* ys = zs + 32 * kZS;                          // [rows][32 orders]
    const int t0 = blockIdx.x * 32, m0 = blockIdx.y * 32, b = blockIdx.z;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int R0 = hstart[max(t0 - 1, 0)];
    const int nr = hstart[min(t0 + 32, H)] + E - R0;
    const cplx<T>* yb = Y + (int64_t)b * Q * (p + 1);
    for (int idx = tid; idx < nr * 32; idx += 256) {
        const int r = idx >> 5, ml = idx & 31;
        const int m = m0 + ml;
        ys[idx] = (m <= L) ? yb[(int64_t)(R0 + r) * (p + 1) + m] : mk<T>(T(0), T(0));
    }
    __syncthreads();
    const int odd = (m0 + lane) & 1;
    auto point = [&](int tl) {   // tl = -1 .. 32
        const int t = t0 + tl;
        T ar = T(0), ai = T(0);
        if (t >= 0 && t <= H) {
            const cplx<T>* yr = ys + (hstart[t] - R0) * 32 + lane;
            const T* w = hwts + 2 * t + odd;
            for (int e = 0; e < E; ++e) {
                const T we = w[(size_t)e * 2 * (H + 1)];
                const cplx<T> v = yr[32 * e];
                ar += we * v.r;
                ai += we * v.i;
            }
        }
        zs[lane * kZS + tl + 1] = pair_value<T>(ar, ai, lane);
    };
#pragma unroll
    for (int j = 0; j < 4; ++j) point(4 * warp + j);
    if (warp == 0) point(-1);
    if (warp == 7) point(32);
    __syncthreads();
    const int t = t0 + lane, up = warp & 1;   // warp w: rows w, w + 8, ..
    if (up ? t == 0 || t >= H : t > H) return;
    cplx<T>* row = U + ((int64_t)b * ((L + 2) / 2) + (m0 + warp) / 2) * (2 * H) + up * H + t;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const cplx<T>* zr = zs + (warp + 8 * k) * kZS;
        if (((m0 + warp + 8 * k) & ~1) <= L)
            row[(int64_t)k * 8 * H] = spread_value<T>(zr, zr + kZS, lane, t, up, rho);
    }
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Register-blocked form for FP32 (at most EW taps, consecutive groups of 4 grid
// points starting at most DM latitude nodes apart): a block takes 32 grid points
// of one map and loops over all orders 32 at a time.  Warp w owns grid points
// t0 + 4w .. t0 + 4w + 3 and lane l order m0 + l; the thread keeps its 4 x EW
// weights (for the parity of its order) in registers, aligned to a common
// window of EW + DM latitude nodes, so every node value read from shared
// memory feeds four grid points.  The two points next to the tile that the
// differences need are summed by two of the eight warps, another two for every
// tile of orders, with weights from shared memory.  (A ninth warp for them made one
// of the four schedulers carry three warps of a block: 1.46 ms at Nside 1024 x 32
// maps.)  The node values of the orders 32 .. 32 (NS-1) ahead are in flight
// (cp.async into a ring of NS buffers) while the current ones are used.  Bound by the
// shared-memory pipe (68%); with the differences it takes 1.15 ms at Nside 1024 x 32
// maps where writing the two half grids took 1.05, for 0.59 ms less in the grid FFT.
template <int EW, int DM, int NS>
__global__ void __launch_bounds__(256, 2) spread_rb_kernel(const cplx<float>* __restrict__ Y,
                                                           cplx<float>* __restrict__ U,
                                                           const int* __restrict__ hstart,
                                                           const float* __restrict__ hwts, int E, int H, int p,
                                                           int Q, int L, int nrw, float rho) {
    constexpr int W = EW + DM;
    extern __shared__ unsigned char smem_raw[];
    cplx<float>* zs = reinterpret_cast<cplx<float>*>(smem_raw);   // [32 rows][kZS]
    cplx<float>* ys0 = zs + 32 * kZS;                              // NS x [nrw rows][32 orders]
    __shared__ float we[2][EW][2];   // weights of the tile's neighbours t0 - 1 and t0 + 32, per parity
    const int t0 = blockIdx.x * 32, b = blockIdx.y;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tlo = max(t0 - 1, 0), thi = min(t0 + 32, H);
    const int R0 = hstart[tlo];
    const int tf = min(t0 + 4 * warp, H);
    const int base = hstart[tf] - R0;                              // window start, relative to R0
    const int par = lane & 1;           // m0 is a multiple of 32
    float w[4][W];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int t = t0 + 4 * warp + j;
        const int off = (t <= H) ? hstart[t] - hstart[tf] : 0;
#pragma unroll
        for (int q = 0; q < W; ++q) {
            const int e = q - off;
            w[j][q] = (t <= H && e >= 0 && e < E) ? hwts[((size_t)e * (H + 1) + t) * 2 + par] : 0.f;
        }
    }
    if (tid < 4 * EW) {   // neighbours outside the half grid: zero
        const int s = tid / (2 * EW), e = (tid >> 1) % EW, t = s ? t0 + 32 : t0 - 1;
        we[s][e][tid & 1] = (t >= 0 && t <= H && e < E) ? hwts[((size_t)e * (H + 1) + t) * 2 + (tid & 1)] : 0.f;
    }
    const int base2 = hstart[thi] - R0;
    // this thread's first row of node values and first output row (rows warp + 8 i)
    const cplx<float>* ysrc = Y + (int64_t)b * Q * (p + 1) + (int64_t)(R0 + warp) * (p + 1) + lane;
    auto fetch = [&](int m0, cplx<float>* ys) {
        const cplx<float>* src = ysrc + m0;
        cplx<float>* dst = ys + warp * 32 + lane;
        if (m0 + 31 <= L && R0 + nrw <= Q) {   // whole tile
            for (int r = warp; r < nrw; r += 8, src += 8 * (int64_t)(p + 1), dst += 256) cp_async8(dst, src, 8);
        } else {
            const bool in = m0 + lane <= L;
            for (int r = warp; r < nrw; r += 8, src += 8 * (int64_t)(p + 1), dst += 256) {
                const bool ok = in && R0 + r < Q;
                cp_async8(dst, ok ? src : Y, ok ? 8 : 0);
            }
        }
        cp_async_commit();
    };
    const int up = warp & 1, t = t0 + lane;
    const bool out = up ? t > 0 && t < H : t <= H;
    cplx<float>* row = U + ((int64_t)b * ((L + 2) / 2) + warp / 2) * (2 * H) + up * H + t;
    const int ntiles = (L + 32) / 32;
    // one commit group per tile (empty past the last), so that waiting until at
    // most NS - 1 groups are pending means tile it has landed
#pragma unroll
    for (int q = 0; q < NS - 1; ++q) {
        if (q < ntiles) fetch(32 * q, ys0 + q * nrw * 32);
        else cp_async_commit();
    }
    for (int it = 0; it < ntiles; ++it) {
        const int m0 = 32 * it;
        cplx<float>* ys = ys0 + (it % NS) * nrw * 32;
        // buffer (it + NS - 1) % NS was last read in iteration it - 1, before the
        // barrier that ended its sums
        if (it + NS - 1 < ntiles) fetch(m0 + 32 * (NS - 1), ys0 + ((it + NS - 1) % NS) * nrw * 32);
        else cp_async_commit();
        cp_async_wait<NS - 1>();
        __syncthreads();
        const cplx<float>* yr = ys + base * 32 + lane;
        float ar[4] = {0.f, 0.f, 0.f, 0.f}, ai[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < W; ++q) {
            const cplx<float> v = yr[32 * q];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                ar[j] += w[j][q] * v.r;
                ai[j] += w[j][q] * v.i;
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) zs[lane * kZS + 4 * warp + j + 1] = pair_value<float>(ar[j], ai[j], lane);
        const int turn = (warp - it) & 7;
        if ((turn & 3) == 0) {   // warp it mod 8: t0 - 1, warp it + 4 mod 8: t0 + 32
            const int s = turn >> 2;
            const cplx<float>* ye = ys + (s ? base2 : 0) * 32 + lane;
            float er = 0.f, ei = 0.f;
#pragma unroll
            for (int e = 0; e < EW; ++e) {
                const float f = we[s][e][par];
                const cplx<float> v = ye[32 * e];
                er += f * v.r;
                ei += f * v.i;
            }
            zs[lane * kZS + (s ? 33 : 0)] = pair_value<float>(er, ei, lane);
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; ++k) {   // rows warp + 8 k: pairs m0/2 + warp/2 + 4 k
            const cplx<float>* zr = zs + (warp + 8 * k) * kZS;
            if (out && ((m0 + warp + 8 * k) & ~1) <= L)
                row[(int64_t)k * 8 * H] = spread_value<float>(zr, zr + kZS, lane, t, up, rho);
        }
        row += (int64_t)32 * H;
    }
}

// The FP32 grid FFT of 4096 points and more transforms the leaky first difference
// dz_t = z_t - rho z_{t-1} (cyclic, one rounding: a fused multiply-add):
//
// An FP32 FFT leaves every output with an absolute error of about 2^-24 times the
// norm of its input, which for a smooth grid (a steep spectrum: most of the power
// at low latitude frequencies) swamps the small modes near j = p that carry the
// highest degrees.  The norm of dz is mostly that of the grid's high-frequency
// part, and Z_j = DFT(dz)_j / (1 - rho e^{-2 pi i j / M}).  The division is exact
// algebra; it amplifies rounding errors by at most 1 / (1 - rho) = 8 at j = 0 (a
// rough grid, e.g. white noise, loses up to a factor of about 5 there), while a
// smooth grid keeps the high modes about ten times more accurately.
//
// The table of a and b, 1 / (1 - rho e^{-2 pi i j / M}) = a - i b, 0 <= j <= p = M/4 (plan
// time; per mode and call the sine, cosine and quotient cost more than the FFT's
// butterflies), without cancellation:
// 1 - rho e^{-i x} = (1 - rho) + 2 rho sin^2(x/2) + i rho sin x, x = 2 pi j / M.
__global__ void prewhiten_kernel(cplx<float>* __restrict__ pw, int M) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j > M / 4) return;
    float sn, cs;
    sincospif((float)j / (float)M, &sn, &cs);   // sin, cos of x/2
    const float a = (1.f - kPrewhiten) + 2.f * kPrewhiten * sn * sn;
    const float b = 2.f * kPrewhiten * sn * cs;
    const float inv = 1.f / (a * a + b * b);
    pw[j] = mk<float>(a * inv, b * inv);
}
void launch_prewhiten_table(void* pw, int M) {
    prewhiten_kernel<<<(M / 4 + 256) / 256, 256>>>((cplx<float>*)pw, M);
}

template <class T>
bool prewhitens(int M) { return sizeof(T) == 4 && M >= kPrewhitenMin; }

template <class T>
void launch_spread(const hpx_plan_s* P, cudaStream_t s) {
    const auto& g = P->g;
    const auto& t = P->t;
    const int H = g.M / 2;
    const T rho = prewhitens<T>(g.M) ? T(kPrewhiten) : T(0);
    constexpr int EW = 12, DM = 4, NS = 4;
    if constexpr (sizeof(T) == 4) {
        if (t.spreadH <= EW && t.spreadD <= DM) {
            // rows a block needs: its first window start .. the last window end
            const int nrw = t.spreadRows - t.spreadH + EW + DM;
            const size_t smem = (size_t)(32 * kZS + NS * 32 * nrw) * sizeof(cplx<float>);
            auto kern = spread_rb_kernel<EW, DM, NS>;
            allow_shared(kern);
            dim3 grid((H + 32) / 32, g.B);
            kern<<<grid, 256, smem, s>>>((const cplx<float>*)P->Y, (cplx<float>*)P->U, t.hstart, (const float*)t.hwts,
                                         t.spreadH, H, g.p, g.Q, g.L, nrw, rho);
            return;
        }
    }
    const size_t smem = (size_t)(32 * kZS + 32 * t.spreadRows) * sizeof(cplx<T>);
    allow_shared(spread_kernel<T>);
    dim3 grid((H + 32) / 32, (g.L + 32) / 32, g.B);
    spread_kernel<T><<<grid, 256, smem, s>>>((const cplx<T>*)P->Y, (cplx<T>*)P->U, t.hstart, (const T*)t.hwts,
                                             t.spreadH, H, g.p, g.Q, g.L, rho);
}

// The largest magnitudes of the two columns of a block into bscale (non-negative
// floats order like their bits).
__device__ __forceinline__ void column_maxima(float* bscale, int64_t i0, bool has1, float mx0, float mx1, int tid) {
    for (int o = 16; o > 0; o >>= 1) {
        mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, o));
        mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, o));
    }
    if ((tid & 31) == 0) {
        atomicMax(reinterpret_cast<int*>(bscale) + i0, __float_as_int(mx0));
        if (has1) atomicMax(reinterpret_cast<int*>(bscale) + i0 + 1, __float_as_int(mx1));
    }
}

// The grid FFT of the shortest grid (nside 2, M = 16): one block of 32 threads per
// pair of orders, the sum z of the two grids from U, and
//     B_m(j) = (Z_j + Z_{M-j}) / 2,   B_{m+1}(j) = (Z_j - Z_{M-j}) / 2
// (the grid of an even order is symmetric, that of an odd one antisymmetric),
// deconvolved and stored as normal-equation right-hand sides.
template <class T>
__global__ void __launch_bounds__(32) lat_fft_small_kernel(const cplx<T>* __restrict__ U, cplx<T>* __restrict__ bvec,
                                                           const T* __restrict__ dec, const cplx<T>* __restrict__ tw,
                                                           int twlen, int M, int logM, int p, int L, int P2,
                                                           float* __restrict__ bscale) {
    __shared__ cplx<T> u[16 + 1];
    const int m0 = 2 * blockIdx.x, b = blockIdx.y, tid = threadIdx.x;
    const bool has1 = m0 + 1 <= L;
    const cplx<T>* z = U + ((int64_t)b * ((L + 2) / 2) + blockIdx.x) * M;
    for (int t = tid; t < M; t += 32) u[pad(t)] = z[grid_index(t, M)];
    __syncthreads();
    block_fft_pad<T, 16>(u, logM, tw, twlen, false);
    cplx<T>* out0 = bvec + ((int64_t)b * (p + 1) + m0) * 2 * P2;
    cplx<T>* out1 = out0 + 2 * P2;
    float mx0 = 0.f, mx1 = 0.f;
    for (int j = tid; j <= p; j += 32) {
        const cplx<T> a = u[pad(j)], c = u[pad((M - j) & (M - 1))];
        const T dj = T(0.5) * dec[j];
        const cplx<T> v0 = scale(add(a, c), dj), v = scale(sub(a, c), dj);
        out0[(j & 1) * P2 + (j >> 1)] = v0;
        mx0 = fmaxf(mx0, fmaxf(fabsf((float)v0.r), fabsf((float)v0.i)));
        if (has1) {
            const cplx<T> v1 = mk<T>(T(-0.5) * v.i, T(0.5) * v.r);   // i/2 B_{m+1}(j)
            out1[(j & 1) * P2 + (j >> 1)] = v1;
            mx1 = fmaxf(mx1, fmaxf(fabsf((float)v1.r), fabsf((float)v1.i)));
        }
    }
    if (tid == 0) {   // the odd-parity block has one slot fewer (j = p + 1 would be index p/2)
        out0[P2 + (P2 - 1)] = mk<T>(T(0), T(0));
        if (has1) out1[P2 + (P2 - 1)] = mk<T>(T(0), T(0));
    }
    if (bscale) column_maxima(bscale, (int64_t)b * (L + 1) + m0, has1, mx0, mx1, tid);
}

// The grid FFT for M = 2^LOGM >= 32 points (fft_ip.cuh), one block per pair of
// orders and map, the same outputs: the first pass reads dz (or z) from U, the last
// one computes only the outputs that hold modes j <= p = M/4 and j >= M - p; the modes
// M - j go to shared memory (zhi), the thread that holds Z_j reads its partner
// there and forms both right-hand sides.  PW: pw[j] = (a, b), 1 / (1 - rho e^{-2 pi i j
// / M}) = a - i b (prewhiten_kernel).
// What bounds it is the shared-memory and L1 pipe (64% at 8192 points) at 40% issue, not
// DRAM (25%).  32 maps: Nside 1024 2.10 -> 1.32 ms, of which the packing of b 0.43;
// Nside 512 x 64 maps 0.88 -> 0.61 ms (before: four loads and the combination of two
// half grids per element, two barriers per pass, sine, cosine and quotient per mode).
template <class T, int LOGM, int NT, int MINB, bool PW>
__global__ void __launch_bounds__(NT, MINB) lat_fft_pair_kernel(
    const cplx<T>* __restrict__ U, cplx<T>* __restrict__ bvec, const T* __restrict__ dec,
    const cplx<T>* __restrict__ pw, const cplx<T>* __restrict__ tw, int p, int L, int P2,
    float* __restrict__ bscale, unsigned char* __restrict__ bpk) {
    constexpr int M = 1 << LOGM, R = ip::out_radix(LOGM, NT), NG1 = M / R, G1 = (NG1 + NT - 1) / NT;
    constexpr int LO = R == 2 ? 1 : R / 4 + 1, HI = R == 2 ? 1 : 3 * R / 4;
    extern __shared__ unsigned char smem_raw[];
    cplx<T>* u = reinterpret_cast<cplx<T>*>(smem_raw);   // slots(M)
    constexpr bool REUSE = LOGM == 13 && NT == 256;        // (all of u is read before the outputs come)
    cplx<T>* zhi = REUSE ? u + ip::slots(M) - M / 4 - 1 : u + ip::slots(M);    // Z_{M-j}, j = 0..p
    // blocks of one pair of orders and consecutive maps run together (map
    // index fastest), so the packed b of a pair's 32 maps, which share every
    // 128-byte line of the B layout, is written while its lines are in L2
    const int b = blockIdx.x;
    const int m0 = 2 * blockIdx.y;
    const int tid = threadIdx.x;
    const bool has1 = m0 + 1 <= L;
    const cplx<T>* src = U + ((int64_t)b * gridDim.y + blockIdx.y) * M;
    cplx<T> lo[G1][LO];
    auto undo = [&](cplx<T> v, cplx<T> w) {   // undoes the difference
        if constexpr (PW) {
            hide(w);   // (the sign of w.i else changes which product is fused)
            v = mul(v, w);
        }
        return v;
    };
    ip::transform<T, LOGM, NT, false, LO, HI, true, false>(
        u, tw, tid, [&](int t, int r) { return src[r < 8 || (r == 8 && t == M / 2) ? t : M + M / 2 - t]; },
        [&](int j, int q, int gg, cplx<T> v) {
            // (the ranges of gg and q are known at compile time)
            if (q < LO && gg * NT + q * NG1 <= M / 4) {
                lo[gg][q] = undo(v, PW ? conjg(pw[min(j, p)]) : v);
            }
            if (gg * NT + NT - 1 + q * NG1 >= 3 * M / 4 && j >= M - p) zhi[M - j] = undo(v, PW ? pw[M - j] : v);
        });
    __syncthreads();
    // right-hand sides of mode j from Z_j and its partner: B_m(j) and i/2 B_{m+1}(j)
    auto modes = [&](int j, cplx<T> a, cplx<T>& v0, cplx<T>& v1) {
        const cplx<T> c = j == 0 ? a : zhi[j];
        const T dj = dec[j];
        v0 = scale(add(a, c), T(0.5) * dj);
        const cplx<T> v = scale(sub(a, c), T(0.5) * dj);
        v1 = mk<T>(T(-0.5) * v.i, T(0.5) * v.r);
    };
    float mx0 = 0.f, mx1 = 0.f;   // largest magnitudes
    auto mag = [&](cplx<T> v) { return fmaxf(fabsf((float)v.r), fabsf((float)v.i)); };
    auto each = [&](auto put) {
#pragma unroll
        for (int gg = 0; gg < G1; ++gg)
#pragma unroll
            for (int q = 0; q < LO; ++q) {
                const int j = tid + gg * NT + q * NG1;
                if (gg * NT + q * NG1 > M / 4 || (NG1 % NT != 0 && tid + gg * NT >= NG1) || j > p) continue;
                cplx<T> v0, v1;
                modes(j, lo[gg][q], v0, v1);
                mx0 = fmaxf(mx0, mag(v0));
                mx1 = fmaxf(mx1, mag(v1));
                put(j, v0, v1);
            }
    };
    if constexpr (sizeof(T) == 4) {
        if (bpk) {   // FP16 pairs for the tensor cores, scaled per column by its largest magnitude
            __shared__ float2 red32[32];
            // the values by (column, parity of j, k = j >> 1) into the FFT buffer,
            // which is free now; one spare slot every 8 k, so that the packing below,
            // where lane g reads k = 8 g + e, spreads over the banks
            cplx<float>* vb = u;
            const int LD = P2 + (P2 >> 3) + 1;
            auto vidx = [&](int col, int par, int k) { return (col * 2 + par) * LD + k + (k >> 3); };
            each([&](int j, cplx<T> v0, cplx<T> v1) {
                vb[vidx(0, j & 1, j >> 1)] = v0;
                vb[vidx(1, j & 1, j >> 1)] = v1;
            });
            const float2 mx = block_max2(make_float2(mx0, mx1), red32);   // (its barrier also publishes vb)
            if (tid == 0) {
                bscale[(int64_t)b * (L + 1) + m0] = mx.x;
                if (has1) bscale[(int64_t)b * (L + 1) + m0 + 1] = mx.y;
            }
            auto val = [&](int col, int par, int k) {   // zero past the column
                return (k < P2 && 2 * k + par <= p) ? vb[vidx(col, par, k)] : mk<float>(0.f, 0.f);
            };
            pack_column(bpk, b, m0, L, P2, pow2_scale(mx.x, 13), [&](int par, int k) { return val(0, par, k); },
                        tid, NT);
            if (has1)
                pack_column(bpk, b, m0 + 1, L, P2, pow2_scale(mx.y, 13),
                            [&](int par, int k) { return val(1, par, k); }, tid, NT);
            return;
        }
    }
    cplx<T>* out0 = bvec + ((int64_t)b * (p + 1) + m0) * 2 * P2;
    cplx<T>* out1 = out0 + 2 * P2;
    each([&](int j, cplx<T> v0, cplx<T> v1) {
        out0[(j & 1) * P2 + (j >> 1)] = v0;
        if (has1) out1[(j & 1) * P2 + (j >> 1)] = v1;
    });
    if (tid == 0) {   // the odd-parity block has one slot fewer (j = p + 1 would be index p/2)
        out0[P2 + (P2 - 1)] = mk<T>(T(0), T(0));
        if (has1) out1[P2 + (P2 - 1)] = mk<T>(T(0), T(0));
    }
    if (bscale) column_maxima(bscale, (int64_t)b * (L + 1) + m0, has1, mx0, mx1, tid);
}

// The packed form of b (fp16pair.cuh) from bvec and the column maxima in
// bscale: one block of 256 threads per (map tile, order, parity), two K-chunks
// per step; thread = (chunk, group of 8 k, map), so that the 8 lanes of a
// 128-byte line of the packed layout are adjacent in a warp (full-line stores)
// and each thread reads 64 contiguous bytes of its map's column.
__global__ void __launch_bounds__(256) pack_b_tiles_kernel(const cplx<float>* __restrict__ bvec,
                                                           unsigned char* __restrict__ bpk,
                                                           const float* __restrict__ bscale, int p, int L, int P2,
                                                           int B) {
    const int m = blockIdx.x, par = blockIdx.y, mt = blockIdx.z;
    const int nch = (P2 + 31) >> 5;
    const int t = threadIdx.x, n = t & 31, kg = (t >> 5) & 3, cl = t >> 7;
    const int b = mt * 32 + n;
    if (b >= B) return;   // columns past the batch stay zero
    const float sc = pow2_scale(bscale[(int64_t)b * (L + 1) + m], 13);
    const cplx<float>* col = bvec + (((int64_t)b * (p + 1) + m) * 2 + par) * P2;
    unsigned char* half = packed_half(bpk, b, m, par, L, nch);
    const int offr = packed_col_offset(b);
    for (int ch = cl; ch < nch; ch += 2) {
        const int g8 = ch * 4 + kg;
        pack_group(half, offr, g8, sc, [&](int k) { return k < P2 ? col[k] : mk<float>(0.f, 0.f); });
    }
}

bool packs_b(const hpx_plan_s* P) {
    return P->bpk && P->precision == HPX_FP32 && ((P->fusedM && P->use_tc) || (!P->fusedM && P->dTC));
}

template <class T>
void launch_lat_fft(const hpx_plan_s* P, cudaStream_t s, bool packed) {
    const auto& g = P->g;
    packed = packed && sizeof(T) == 4 && P->bpk && P->bscale;
    // packed b: either written by the grid-FFT kernel itself, or (P->packSep, and
    // grids below 4096 points, whose columns are shorter than a full line's worth of
    // blocks in flight) FP32 b with the column maxima as atomic maxima of the
    // float bits, then one pass of pack_b_tiles_kernel
    int logM = 0;
    while ((1 << logM) < g.M) ++logM;
    const bool inFft = packed && !P->packSep && logM >= 12;
    if (packed && !inFft) cudaMemsetAsync(P->bscale, 0, (size_t)g.B * (g.L + 1) * sizeof(float), s);
    float* bsc = packed ? P->bscale : nullptr;
    if (logM < 5) {
        lat_fft_small_kernel<T><<<dim3((g.L + 2) / 2, g.B), 32, 0, s>>>(
            (const cplx<T>*)P->U, (cplx<T>*)P->bvec, (const T*)P->t.dec, (const cplx<T>*)P->t.twid, g.Lmax, g.M,
            logM, g.p, g.L, g.P2, bsc);
    } else {
        auto run = [&](auto kern, int threads) {
            const size_t smem =
                (size_t)(ip::slots(g.M) + (logM == 13 && threads == 256 ? 0 : g.p + 1)) * sizeof(cplx<T>);
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            kern<<<dim3(g.B, (g.L + 2) / 2), threads, smem, s>>>(
                (const cplx<T>*)P->U, (cplx<T>*)P->bvec, (const T*)P->t.dec, (const cplx<T>*)P->t.pw,
                (const cplx<T>*)P->t.twc, g.p, g.L, g.P2, bsc, inFft ? P->bpk : nullptr);
        };
        // 16 elements per thread, at least a warp; 32 at 8192 points, where the last two
        // passes run on them in registers (with 512 threads and four passes: 1.61 ms
        // at 32 maps of Nside 1024)
        constexpr bool F = sizeof(T) == 4;
        if (logM == 5) run(lat_fft_pair_kernel<T, 5, 32, 1, false>, 32);
        else if (logM == 6) run(lat_fft_pair_kernel<T, 6, 32, 1, false>, 32);
        else if (logM == 7) run(lat_fft_pair_kernel<T, 7, 32, 1, false>, 32);
        else if (logM == 8) run(lat_fft_pair_kernel<T, 8, 32, 1, false>, 32);
        else if (logM == 9) run(lat_fft_pair_kernel<T, 9, 32, 1, false>, 32);
        else if (logM == 10) run(lat_fft_pair_kernel<T, 10, 64, 1, false>, 64);
        else if (logM == 11) run(lat_fft_pair_kernel<T, 11, 128, F ? 8 : 1, false>, 128);
        else if (logM == 12) run(lat_fft_pair_kernel<T, 12, 256, F ? 4 : 1, F>, 256);
        else if (logM == 13) run(lat_fft_pair_kernel<T, 13, 256, F ? 3 : 1, F>, 256);
        else if constexpr (F) run(lat_fft_pair_kernel<T, 14, 1024, 1, F>, 1024);
    }
    if (packed && !inFft)
        pack_b_tiles_kernel<<<dim3(g.L + 1, 2, (g.B + 31) / 32), 256, 0, s>>>(
            (const cplx<float>*)P->bvec, P->bpk, P->bscale, g.p, g.L, g.P2, g.B);
}

template void launch_spread<float>(const hpx_plan_s*, cudaStream_t);
template void launch_spread<double>(const hpx_plan_s*, cudaStream_t);
template void launch_lat_fft<float>(const hpx_plan_s*, cudaStream_t, bool);
template void launch_lat_fft<double>(const hpx_plan_s*, cudaStream_t, bool);

template <class T>
void launch_nufft(const hpx_plan_s* P, cudaStream_t s) {
    const auto& g = P->g;
    const auto& t = P->t;
    int logM = 0;
    while ((1 << logM) < g.M) ++logM;
    const size_t smem = (size_t)(g.M + g.M / 16 + g.Q) * sizeof(cplx<T>);
    auto kern = g.M > 16 * 512 ? nufft_kernel<T, 32> : nufft_kernel<T, 16>;
    allow_shared(kern);
    dim3 grid(g.L + 1, g.B);
    kern<<<grid, 512, smem, s>>>((const cplx<T>*)P->Y, (cplx<T>*)P->bvec, t.nstart, (const T*)t.swts, t.spreadE,
                                 (const T*)t.dec, (const cplx<T>*)t.twid, g.Lmax, g.M, logM, g.p, g.Q, g.P2);
}

template void launch_nufft<float>(const hpx_plan_s*, cudaStream_t);
template void launch_nufft<double>(const hpx_plan_s*, cudaStream_t);

}  // namespace hpx

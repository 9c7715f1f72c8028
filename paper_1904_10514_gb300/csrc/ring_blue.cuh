// The DFT of a ring of n = 4j points (j not a power of two) as four Bluestein
// transforms of j points side by side, with t = 4u + s:
//     Z[q + r j] = sum_s (-i)^{s r} W^{s q} Y_s[q],   W = e^{-2 pi i / n}, q < j, r < 4,
// Y_s the DFT of the subsequence z[4u + s].  Each Y_s is a chirp-z convolution of
// NQ = 2^LOGQ >= 2j points (fft_ip.cuh) on NTQ threads of the block: against one
// convolution of the whole ring a quarter of the transformed-kernel table and two
// levels less per transform.  chirp4 (j points) and bhat4 (NQ points, 1 / NQ folded
// in) are FP64-built.
#pragma once
#include "fft_ip.cuh"

namespace hpx {

// The four Y_s in shared memory, quarter s at s QS, element q at slot(q).
template <class T>
struct RingQuarters {
    cplx<T>* buf;
    int QS;

    static __device__ __forceinline__ cplx<T> root(int q, int n) {   // W^q
        T sn, cs;
        if constexpr (sizeof(T) == 4) sincospif(-2.f * (float)q / (float)n, &sn, &cs);
        else sincospi(-2.0 * (double)q / (double)n, &sn, &cs);
        return mk<T>(cs, sn);
    }
    // Z[q + r j], r = 0..3
    __device__ __forceinline__ void combine(int q, int n, cplx<T> (&z)[4]) const {
        const cplx<T> w1 = root(q, n);
        const cplx<T> w2 = mul(w1, w1), w3 = mul(w1, w2);
        const cplx<T>* y = buf + ip::slot(q);
        const cplx<T> t0 = y[0], t1 = mul(w1, y[QS]), t2 = mul(w2, y[2 * QS]), t3 = mul(w3, y[3 * QS]);
        const cplx<T> a = add(t0, t2), b = sub(t0, t2), c = add(t1, t3), d = sub(t1, t3);
        z[0] = add(a, c);
        z[1] = mk<T>(b.r + d.i, b.i - d.r);   // b - i d
        z[2] = sub(a, c);
        z[3] = mk<T>(b.r - d.i, b.i + d.r);   // b + i d
#pragma unroll
        for (int r = 0; r < 4; ++r) hide(z[r]);
    }
    // Z in natural order in the free tail of each quarter (2j <= NQ); read with at()
    __device__ __forceinline__ int tail(int n) const { return ip::slots(n >> 2); }
    __device__ __forceinline__ void natural(int n, int tid, int nt) const {
        const int jq = n >> 2, S0 = tail(n);
        for (int q = tid; q < jq; q += nt) {
            cplx<T> z[4];
            combine(q, n, z);
#pragma unroll
            for (int r = 0; r < 4; ++r) buf[r * QS + S0 + q] = z[r];
        }
        __syncthreads();
    }
    __device__ __forceinline__ cplx<T> at(int k, int n) const {
        const int jq = n >> 2;
        const int r = (k >= jq) + (k >= 2 * jq) + (k >= 3 * jq);
        return buf[r * QS + tail(n) + (k - r * jq)];
    }
};

// The quarter transforms of the sequence in(k), k < n, by 4 NTQ threads (EX: as
// ip::transform).  Ends with a barrier.
template <class T, int LOGQ, int NTQ, bool EX, class IN>
__device__ __forceinline__ RingQuarters<T> quarter_transforms(cplx<T>* buf, int n, const cplx<T>* __restrict__ ch,
                                                              const cplx<T>* __restrict__ bh,
                                                              const cplx<T>* __restrict__ tw, IN in) {
    constexpr int NQ = 1 << LOGQ, QS = ip::slots(NQ);
    const int jq = n >> 2;
    const int s = threadIdx.x / NTQ, ltid = threadIdx.x - s * NTQ;
    cplx<T>* qb = buf + s * QS;
    ip::convolve<T, LOGQ, NTQ, EX>(
        qb, tw, ltid, [&](int u) { return u < jq ? mul(in(4 * u + s), ch[u]) : mk<T>(T(0), T(0)); },
        [&](int u) { return bh[u]; },
        [&](int u, cplx<T> v) {
            if (u < jq) qb[ip::slot(u)] = mul(v, ch[u]);
        });
    __syncthreads();
    return RingQuarters<T>{buf, QS};
}

}  // namespace hpx

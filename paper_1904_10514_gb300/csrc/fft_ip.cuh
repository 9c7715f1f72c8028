// Shared-memory FFT passes with compile-time shapes, in place between barriers.
//
// A transform of N = 2^LOGN points (LOGN >= 5) is decimation in time with register
// passes of radix 16, ..., 16 and a last one of 2, 4, 8 or 16: the radices, twiddle
// products and order of operations of the Stockham passes in common.cuh, so both
// give the same bits.  Twiddles come from the compact tables (twc_offset, common.cuh).  What differs is where the values live: element with pass
// digits d_0 (of the first pass), d_1, ... sits at position d_0 + 16 d_1 + 256 d_2 ...
// at slot(position), so
//   * every pass but the first reads and writes the same positions (one barrier
//     per pass where a Stockham pass over one buffer needs two),
//   * the first pass takes its inputs straight from ld() and the last one hands its
//     outputs, natural order, to st() from registers,
//   * in a convolution the last forward pass, the product with the transformed
//     kernel and the first inverse pass work on the same 16 elements
//     k + r N/16 of thread k, in registers.
// An input whose second half is zero and an output whose second half is not wanted
// (both halves of a chirp-z convolution) leave out those operations.
#pragma once
#include "common.cuh"

namespace hpx {
namespace ip {

// One spare slot every 16 and every 256 elements, 8 where bit 12 is set and 20 where
// bit 13 is: the 8-byte accesses of the passes are free of bank conflicts, but for the
// first pass's stores at 512 to 2048 points (two to four ways).
__host__ __device__ constexpr int slot(int i) {
    return i + (i >> 4) + (i >> 8) + ((i >> 9) & 24) + ((i >> 11) & 4);
}
__host__ __device__ constexpr int slots(int n) { return slot(n - 1) + 1; }   // of an n-point transform

__host__ __device__ constexpr int npass(int logn) { return (logn + 3) / 4; }
// radix of pass i (from 0); its span (product of the radices before it) is 16^i
__host__ __device__ constexpr int radix(int logn, int i) {
    return i < npass(logn) - 1 || logn % 4 == 0 ? 16 : 1 << (logn % 4);
}

// Position of the run of 16 that first-pass group t (inputs t + r N/16) fills.
template <int LOGN>
__device__ __forceinline__ int run_base(int t) {
    int base = 0;
#pragma unroll
    for (int i = npass(LOGN) - 1; i >= 1; --i) {
        const int R = radix(LOGN, i);
        base += (t % R) << (4 * i);
        t /= R;
    }
    return base;
}

// First pass: ld(i, r) gives input i = t + r N/16 (HALF: those with r >= 8 are zero
// and not read).
template <class T, int LOGN, int NT, bool INV, bool HALF, class LD>
__device__ __forceinline__ void first_pass(cplx<T>* a, int tid, LD ld) {
    constexpr int NG = (1 << LOGN) / 16, G = (NG + NT - 1) / NT;
#pragma unroll
    for (int gg = 0; gg < G; ++gg) {
        const int t = tid + gg * NT;
        if (NG % NT != 0 && t >= NG) break;
        cplx<T> x[16];
#pragma unroll
        for (int r = 0; r < (HALF ? 8 : 16); ++r) x[r] = ld(t + r * NG, r);
        reg_dft<T, 16, INV, HALF>(x);
        cplx<T>* to = a + slot(run_base<LOGN>(t));
#pragma unroll
        for (int r = 0; r < 16; ++r) to[r] = x[r];
    }
}

// Pass I of span S = 16^I and radix R over the whole transform, in place, after a
// barrier; the first group's twiddles are read ahead of it.
template <class T, int LOGN, int I, int NT, bool INV, bool EX>
__device__ __forceinline__ void inner_pass(cplx<T>* a, const cplx<T>* __restrict__ tw, int tid) {
    constexpr int N = 1 << LOGN, R = radix(LOGN, I), S = 1 << (4 * I), NG = N / R, G = (NG + NT - 1) / NT;
    PassTwiddles<T, R, S, INV, EX> t;
    t.fetch(tid & (S - 1), tw);
    __syncthreads();
#pragma unroll
    for (int gg = 0; gg < G; ++gg) {
        const int k = tid + gg * NT;
        if (NG % NT != 0 && k >= NG) break;
        const int j = k & (S - 1);
        if (gg > 0 && NT % S != 0) t.fetch(j, tw);
        cplx<T>* e = a + slot((k / S) * (S * R) + j);
        cplx<T> x[R];
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = e[slot(r * S)];
        t.apply(x);
        reg_dft<T, R, INV>(x);
#pragma unroll
        for (int q = 0; q < R; ++q) e[slot(q * S)] = x[q];
    }
}

// The passes between the first and the last.
template <class T, int LOGN, int NT, bool INV, bool EX, int I = 1>
__device__ __forceinline__ void inner_passes(cplx<T>* a, const cplx<T>* __restrict__ tw, int tid) {
    if constexpr (I < npass(LOGN) - 1) {
        inner_pass<T, LOGN, I, NT, INV, EX>(a, tw, tid);
        inner_passes<T, LOGN, NT, INV, EX, I + 1>(a, tw, tid);
    }
}

__host__ __device__ constexpr int last_radix(int logn) { return radix(logn, npass(logn) - 1); }
// outputs per thread and round of transform()'s last step (q of its st), M / this apart
__host__ __device__ constexpr int out_radix(int logn, int nt) { return logn == 13 && nt == 256 ? 32 : last_radix(logn); }

// Last pass, after a barrier: outputs j + q S (S = N / R, group j = tid + gg NT) to
// st(index, q, gg, value) for q < LO or q >= HI.  PRE: the first group's twiddles are
// read ahead of the barrier.
template <class T, int LOGN, int NT, bool INV, int LO, int HI, bool PRE, bool EX, class ST>
__device__ __forceinline__ void last_pass(const cplx<T>* a, const cplx<T>* __restrict__ tw, int tid,
                                          ST st) {
    constexpr int N = 1 << LOGN, R = last_radix(LOGN), S = N / R, G = (S + NT - 1) / NT;
    PassTwiddles<T, R, S, INV, EX> t;
    if constexpr (PRE) t.fetch(min(tid, S - 1), tw);
    __syncthreads();
#pragma unroll
    for (int gg = 0; gg < G; ++gg) {
        const int j = tid + gg * NT;
        if (S % NT != 0 && j >= S) break;
        if (!PRE || gg > 0) t.fetch(j, tw);
        const cplx<T>* e = a + slot(j);
        cplx<T> x[R];
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = e[slot(r * S)];
        t.apply(x);
        reg_dft<T, R, INV>(x);
#pragma unroll
        for (int q = 0; q < R; ++q)
            if (q < LO || q >= HI) st(j + q * S, q, gg, x[q]);
    }
}

// The last two passes of LOGN = 13 (radix 16, span 256, and radix 2) on the 32
// elements j + 256 r of thread j < 256, in registers, after a barrier and with another
// one behind the reads (st may store anywhere in a): outputs j + 256 q, q < LO or
// q >= HI, to st(index, q, 0, value).
template <class T, int NT, bool INV, int LO, int HI, bool EX, class ST>
__device__ __forceinline__ void last_passes_8192(const cplx<T>* a, const cplx<T>* __restrict__ tw,
                                                 int tid, ST st) {
    static_assert(NT == 256, "one thread per j");
    const cplx<T>* e = a + slot(tid);
    PassTwiddles<T, 16, 256, INV, EX> t;
    t.fetch(tid, tw);
    __syncthreads();
    cplx<T> x[16], y[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) x[r] = e[slot(256 * r)];
#pragma unroll
    for (int r = 0; r < 16; ++r) y[r] = e[slot(4096 + 256 * r)];
    __syncthreads();
    t.apply(x);
    reg_dft<T, 16, INV>(x);
    t.apply(y);
    reg_dft<T, 16, INV>(y);
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const int k = tid + 256 * q;
        cplx<T> z[2] = {x[q], y[q]};
        PassTwiddles<T, 2, 4096, INV, EX> t2;
        t2.fetch(k, tw);
        t2.apply(z);
        reg_dft<T, 2, INV>(z);
        if (q < LO || q >= HI) st(k, q, 0, z[0]);
        if (q + 16 < LO || q + 16 >= HI) st(k + 4096, q + 16, 0, z[1]);
    }
}

// The whole transform: ld(i, r) as first_pass, st(index, q, gg, value) as last_pass.
// st may store to the positions of a (natural order): a thread only produces
// positions that it alone has read.  Ends without a barrier.
// EX: twiddles from the rows of all powers (tw = twx, else twc).
template <class T, int LOGN, int NT, bool INV, int LO, int HI, bool PRE, bool EX, class LD, class ST>
__device__ __forceinline__ void transform(cplx<T>* a, const cplx<T>* __restrict__ tw, int tid, LD ld,
                                          ST st) {
    first_pass<T, LOGN, NT, INV, false>(a, tid, ld);
    if constexpr (LOGN == 13 && NT == 256) {
        inner_pass<T, LOGN, 1, NT, INV, EX>(a, tw, tid);
        last_passes_8192<T, NT, INV, LO, HI, EX>(a, tw, tid, st);
    } else {
        inner_passes<T, LOGN, NT, INV, EX>(a, tw, tid);
        last_pass<T, LOGN, NT, INV, LO, HI, PRE, EX>(a, tw, tid, st);
    }
}

// Cyclic convolution of N = 2^LOGN points by NT >= N/16 threads: input ld(i), zero for
// i >= N/2 (not read there), transformed kernel ker(i); st(i, value) receives the
// outputs i < N/2.  The barriers are the block's: side-by-side convolutions run
// their passes in step.  Ends without one.  EX as transform().
template <class T, int LOGN, int NT, bool EX, class LD, class KER, class ST>
__device__ __forceinline__ void convolve(cplx<T>* a, const cplx<T>* __restrict__ tw, int tid, LD ld,
                                         KER ker, ST st) {
    constexpr int N = 1 << LOGN, R = radix(LOGN, npass(LOGN) - 1), NG = N / 16, D = 16 / R;
    static_assert(NT >= NG, "the turn keeps one group per thread");
    first_pass<T, LOGN, NT, false, true>(a, tid, [&](int i, int) { return ld(i); });
    inner_passes<T, LOGN, NT, false, EX>(a, tw, tid);
    const bool on = NG == NT || tid < NG;
    __syncthreads();
    cplx<T> y[16];
    if (on) {
        const cplx<T>* e = a + slot(tid);
#pragma unroll
        for (int i = 0; i < D; ++i) {   // last-pass group j = tid + i N/16
            cplx<T> x[R];
#pragma unroll
            for (int q = 0; q < R; ++q) x[q] = e[slot((i + q * D) * NG)];
            PassTwiddles<T, R, N / R, false, EX> t;
            t.fetch(tid + i * NG, tw);
            t.apply(x);
            reg_dft<T, R, false>(x);
#pragma unroll
            for (int q = 0; q < R; ++q) {
                y[i + q * D] = mul(x[q], ker(tid + (i + q * D) * NG));
                hide(y[i + q * D]);
            }
        }
        reg_dft<T, 16, true>(y);
    }
    __syncthreads();   // every thread has read its positions
    if (on) {
        cplx<T>* to = a + slot(run_base<LOGN>(tid));
#pragma unroll
        for (int r = 0; r < 16; ++r) to[r] = y[r];
    }
    inner_passes<T, LOGN, NT, true, EX>(a, tw, tid);
    last_pass<T, LOGN, NT, true, R / 2, R, false, EX>(a, tw, tid, [&](int i, int, int, cplx<T> v) { st(i, v); });
}

}  // namespace ip
}  // namespace hpx

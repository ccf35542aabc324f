// fft32_core.cuh -- one vector's fp32 transform: the Stockham passes of a
// register-resident FFT over threads that exchange through shared memory
// (fft32.cu and small.cu; the structure is described in fft32.cu).
#pragma once

#include "common.cuh"
#include "dft.cuh"
#include "fft32_tables.cuh"

namespace fm {

// shared-memory slot of element a of a transform of length 2^LOGN: one slot of
// padding per E, so that E-strided stores of W interleaved vectors hit every
// bank (the stride E W + W is W modulo 16 eight-byte slots)
template <int LOGN> __device__ __forceinline__ constexpr int padded(int a) { return a + (a >> FftPlan<LOGN>::LOGE); }

// barrier of the threads taking part: the whole CTA (NB = 0) or the first NB
// threads (named barrier 1; NB a multiple of 32)
template <int NB> __device__ __forceinline__ void part_sync()
{
    if constexpr (NB == 0)
        __syncthreads();
    else
        asm volatile("bar.sync 1, %0;" ::"n"(NB) : "memory");
}

// times the table's twiddle (its conjugate for the inverse)
template <bool INV> __device__ __forceinline__ float2 mul_tw(float2 a, const float2 *__restrict__ tw)
{
    float2 w = __ldg(tw);
    if (INV) w.y = -w.y;
    return cmul(a, w);
}

// In: v[q] = x[j + q TV].  Out: v[q] = X[j + q TV].
// Element i of vector c (of W) lives at sm[padded(i W + c)] between passes.
// tw: the pass tables of length N (FftPlan's layout, after the natural table).
// Every thread taking part must call this (it holds barriers).
template <int LOGN, int W, bool INV, int NB = 0>
__device__ __forceinline__ void fft_vec(float2 (&v)[FftPlan<LOGN>::E], float2 *sm, int c, int j,
                                        const float2 *__restrict__ tw)
{
    using P = FftPlan<LOGN>;
    constexpr int E = P::E;
    // Padded addresses split into one base a thread and compile-time offsets
    // (immediates of the loads and stores): exact, since TV W and E divide one
    // another and the base stays below TV W (and W and E do).
    constexpr int TVW = P::TV * W;
    float2 *rd = sm + padded<LOGN>(j * W + c);  // x[j]
    auto load = [&](int q) { return rd[padded<LOGN>(q * TVW)]; };
    Dft<E, INV, float2>::run(v);  // pass 0: Ns = 1, no twiddles; outputs at E j + r
    part_sync<NB>();              // the buffer may still be read by an earlier pass
    {
        float2 *wr = sm + j * (E * W + W) + padded<LOGN>(c);
#pragma unroll
        for (int r = 0; r < E; ++r) wr[padded<LOGN>(r * W)] = v[r];
    }
    part_sync<NB>();
    // middle passes: radix E, Ns = E, E^2
#pragma unroll
    for (int p = 1; p + 1 < P::NPASS; ++p) {
        const int NS = 1 << (P::LOGE * p);
#pragma unroll
        for (int r = 0; r < E; ++r) v[r] = load(r);
        const int k = j & (NS - 1);
        const float2 *t = tw + P::N + P::pass_off(p) + k;
#pragma unroll
        for (int r = 1; r < E; ++r) v[r] = mul_tw<INV>(v[r], t + (r - 1) * NS);
        Dft<E, INV, float2>::run(v);
        part_sync<NB>();
        float2 *wr = sm + padded<LOGN>(((j - k) * E + k) * W + c);
#pragma unroll
        for (int r = 0; r < E; ++r) wr[padded<LOGN>(r * NS * W)] = v[r];
        part_sync<NB>();
    }
    // last pass: radix RL, Ns = NSL, butterfly b = j + m TV (< NSL), twiddle W_n^(r b)
    const float2 *t = tw + P::N + P::pass_off(P::NPASS - 1) + j;
#pragma unroll
    for (int m = 0; m < P::ML; ++m) {
        float2 x[P::RL];
#pragma unroll
        for (int r = 0; r < P::RL; ++r) {
            x[r] = load(m + r * P::ML);
            if (r > 0) x[r] = mul_tw<INV>(x[r], t + (r - 1) * P::NSL + m * P::TV);
        }
        Dft<P::RL, INV, float2>::run(x);
        // output r of butterfly m is X[j + TV (m + r ML)]
#pragma unroll
        for (int r = 0; r < P::RL; ++r) v[m + r * P::ML] = x[r];
    }
}

// signed integer frequency of index j + q TV as a float (q a compile-time
// constant: no select); exact, and so are the squares and products below
// 2^24 that the KS multiplier takes of it
template <int LOGN> __device__ __forceinline__ float freq_of(float jf, int q)
{
    using P = FftPlan<LOGN>;
    return jf + (float)(q * P::TV - (q >= P::E / 2 ? P::N : 0));
}

}  // namespace fm

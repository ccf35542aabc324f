// fft32_tables.cuh -- pass structure and twiddle tables of the
// register-resident FFTs (fft32.cu; fft64.cu shares the tables' layout), for
// the kernels and for the host code that fills the tables (runtime.cu,
// noalloc.cu).
//
// A table for length n holds the natural table exp(-2 pi i t / n), t = 0 ..
// n - 1, and after it one block per Stockham pass p >= 1 with the twiddles in
// the order a warp reads them: entry [r - 1][k] = W^(r k) with k = 0 .. Ns - 1
// consecutive, so a load of 32 neighbouring threads covers one or two cache
// lines (taken from the natural table, the 16 threads of a pass with Ns = 16
// gathered from up to 16 lines).
#pragma once

#include <math.h>

#include <vector>

#include "common.cuh"

namespace fm {

// elements a thread holds (the radix of all passes but the last) for n = 2^logn
__host__ __device__ constexpr int fft_log_e(int logn) { return logn <= 8 ? 4 : 5; }

// n = 2^LOGN split into radix-E passes and one last radix RL
template <int LOGN> struct FftPlan {
    static constexpr int N = 1 << LOGN;
    static constexpr int LOGE = fft_log_e(LOGN), E = 1 << LOGE;  // elements per thread
    static constexpr int TV = N / E;                             // threads per vector
    static constexpr int NPASS = (LOGN + LOGE - 1) / LOGE;       // passes (all radix E but the last)
    static constexpr int LOGRL = LOGN - LOGE * (NPASS - 1);      // log2 of the last radix
    static constexpr int RL = 1 << LOGRL;
    static constexpr int ML = E / RL;   // butterflies per thread in the last pass
    static constexpr int NSL = N / RL;  // stride of the last pass outputs (= ML TV)
    static_assert(NPASS >= 2, "at least two passes");
    // first entry of pass p's block after the natural table: (E - 1) E^q
    // entries for each earlier pass q = 1 .. p - 1
    __host__ __device__ static constexpr int pass_off(int p) { return (1 << (LOGE * p)) - E; }
};

// fp64 (fft64.cu): radix 8 throughout
constexpr int kFft64LogE = 3;

// elements of a table: the natural one and the blocks of passes 1 .. (their
// sizes sum to n - E)
inline int fft_table_elems(int n, int loge) { return 2 * n - (1 << loge); }
inline int fft32_table_elems(int n) { return fft_table_elems(n, fft_log_e(ilog2((unsigned)n))); }

// exp(-2 pi i e / n) within about an ulp of either part, n a power of two from
// 4 up, 0 <= e < n.  The angle is brought to the first octant in integers and
// kept as a sum of two doubles (pi = M_PI + 1.2246e-16): the rounding of 2 pi
// e / n, up to 4e-16 at the far end of the circle, is six times the rounding of
// the entries (2.3e-16 against 4.7e-17 rms) and was most of the fp64
// transform's error (kappa_E of 64^2 / 256^2 / 1024^2 4.0 / 5.1 / 5.9e-16 rms,
// now 3.3 / 4.0 / 4.8e-16).
template <typename V> inline V unit_root(int e, int n)
{
    const int q = (int)((long)e * 4 / n);  // quadrant
    int r = e - q * (n / 4);               // 0 .. n/4 - 1
    const bool swap = 8 * (long)r > n;
    if (swap) r = n / 4 - r;
    const double p = M_PI * r, lo = fma(M_PI, (double)r, -p) + 1.2246467991473532e-16 * r;
    const double a = p * 2 / n, al = lo * 2 / n;  // exact scalings
    double c = cos(a) - al * sin(a), s = sin(a) + al * cos(a);
    if (swap) {
        const double t = c;
        c = s;
        s = t;
    }
    V v;  // cos and -sin of q pi / 2 + the octant's angle
    v.x = (decltype(v.x))(q == 0 ? c : q == 1 ? -s : q == 2 ? -c : s);
    v.y = (decltype(v.y))(q == 0 ? -s : q == 1 ? -c : q == 2 ? s : c);
    return v;
}

// fills fft_table_elems(n, loge) entries (FP64 on the host, rounded once)
template <typename V> inline void fft_fill_table(int n, int loge, V *t)
{
    auto w = [n](long e) { return unit_root<V>((int)(e % n), n); };
    for (int i = 0; i < n; ++i) *t++ = w(i);
    const int logn = ilog2((unsigned)n), np = (logn + loge - 1) / loge;
    for (int p = 1; p < np; ++p) {
        const int ns = 1 << (loge * p), radix = p + 1 < np ? 1 << loge : n / ns;
        for (int r = 1; r < radix; ++r)
            for (int k = 0; k < ns; ++k) *t++ = w((long)r * k * (n / (ns * radix)));
    }
}
inline void fft32_fill_table(int n, float2 *t) { fft_fill_table(n, fft_log_e(ilog2((unsigned)n)), t); }

}  // namespace fm

// noise.cu -- randomised-shear noise maps (Sec. 1): the FP64 accumulation of
// the bands over realisations, the per-pixel unbiased variance and S/N, and
// the elementwise helpers of the exact expected variance.
#include "common.cuh"

namespace fm {

// The inputs of one noise call into the library's buffers: the generator's
// seed (read there by the row FFT) and, where d1 is given, the two shear maps
// as `words` vectors V, so that a recorded graph reads neither the caller's
// pointers nor a seed fixed at its recording.
template <typename V>
__global__ void __launch_bounds__(256) k_noise_stage(const V *__restrict__ g1, const V *__restrict__ g2,
                                                     V *__restrict__ d1, V *__restrict__ d2, long words, uint64_t seed,
                                                     uint64_t *__restrict__ dseed)
{
    pdl_entry();
    const long i0 = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i0 == 0) *dseed = seed;
    for (long i = i0; i < words; i += (long)gridDim.x * blockDim.x) {
        d1[i] = g1[i];
        d2[i] = g2[i];
    }
}

int launch_noise_stage(const void *g1, const void *g2, void *d1, void *d2, size_t bytes, uint64_t seed,
                       uint64_t *dseed, cudaStream_t s)
{
    if (!d1) bytes = 0;
    const bool wide = ((reinterpret_cast<uintptr_t>(g1) | reinterpret_cast<uintptr_t>(g2) | bytes) & 15) == 0;
    const long words = (long)(bytes / (wide ? 16 : 4));
    const unsigned g = (unsigned)(words / 256 + 1 > 152 * 8 ? 152 * 8 : words / 256 + 1);
    if (wide)
        FM_LAUNCH(0, k_noise_stage<float4>, g, 256, 0, s, (const float4 *)g1, (const float4 *)g2, (float4 *)d1,
                  (float4 *)d2, words, seed, dseed);
    else
        FM_LAUNCH(0, k_noise_stage<uint32_t>, g, 256, 0, s, (const uint32_t *)g1, (const uint32_t *)g2, (uint32_t *)d1,
                  (uint32_t *)d2, words, seed, dseed);
    return FM_OK;
}

// f(the vector at p of every realisation), in order, kAccLoads of them
// loaded ahead (4 / 8 / 16 at two CTAs an SM, R = 256 of 1024^2: 5701 / 5599 /
// 5784 us)
constexpr int kAccLoads = 8;
template <typename V, typename T, typename F>
__device__ __forceinline__ void for_realisations(const T *__restrict__ p, int nb, long bs, F &&f)
{
    int b = 0;
    for (; b + kAccLoads <= nb; b += kAccLoads) {
        V v[kAccLoads];
#pragma unroll
        for (int k = 0; k < kAccLoads; ++k) v[k] = __ldcs(reinterpret_cast<const V *>(p + (b + k) * bs));
#pragma unroll
        for (int k = 0; k < kAccLoads; ++k) f(v[k]);
    }
    for (; b < nb; ++b) f(__ldcs(reinterpret_cast<const V *>(p + b * bs)));
}

// two neighbouring FP64 sums, as one 16-byte word where they are aligned
// (`wide`; the caller's own sums need not be); streaming, as they are next
// used a batch later
__device__ __forceinline__ void add_sums(double *p, double a, double b, bool first, bool wide)
{
    if (wide) {
        double2 v = make_double2(0.0, 0.0);
        if (!first) v = __ldcs(reinterpret_cast<const double2 *>(p));
        __stcs(reinterpret_cast<double2 *>(p), make_double2(v.x + a, v.y + b));
    } else {
        p[0] = first ? a : p[0] + a;
        p[1] = first ? b : p[1] + b;
    }
}

// S1 += sum_b w, S2 += sum_b w^2 over a batch of `nb` (<= 32) realisations'
// pyramids ([nb][J][n][n], bands 0..J-2 used).  The batch's partial sums are
// formed in the element type (at most 32 terms) and added once to the FP64
// running sums: GB300's FP64 rate is a small fraction of its FP32 rate, so
// the FP64 work is two additions per band pixel per batch.  The pyramids are
// read once with streaming (evict-first) loads, so they do not push the chunk
// pipeline's intermediates out of L2.  The first batch writes the sums
// (`first`) instead of adding to zeroed ones.  Bound by HBM: 32 realisations
// of 6 bands of 1024^2 and their sums, 1 GB, in 171 us; R = 100 with the sums'
// zeroing, their scalar accesses and the S/N's map after the last batch 2427,
// now 2299 us.
template <typename T, typename V>
__global__ void __launch_bounds__(256) k_noise_accum(const T *__restrict__ pyr, int nb, long pyr_bs, long nn,
                                                     int bands, double *__restrict__ s1, double *__restrict__ s2,
                                                     int first, int wide)
{
    pdl_entry();
    constexpr int VW = sizeof(V) / sizeof(T);
    const long nq = bands * nn / VW;  // nn % 4 == 0 (n a power of two >= 4)
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < nq; i += (long)gridDim.x * blockDim.x) {
        const long e = i * VW;  // band-major element index: band * nn + pixel
        T a[VW], q[VW];
#pragma unroll
        for (int u = 0; u < VW; ++u) a[u] = q[u] = (T)0;
        for_realisations<V>(pyr + e, nb, pyr_bs, [&](const V &v) {
            const T *w = reinterpret_cast<const T *>(&v);
#pragma unroll
            for (int u = 0; u < VW; ++u) {
                a[u] += w[u];
                q[u] = fma(w[u], w[u], q[u]);
            }
        });
#pragma unroll
        for (int u = 0; u < VW; u += 2) {
            add_sums(s1 + e + u, (double)a[u], (double)a[u + 1], first, wide);
            add_sums(s2 + e + u, (double)q[u], (double)q[u + 1], first, wide);
        }
    }
}

// accum = 1 (fp32 maps): the running sums are fp32 with Kahan compensation
// (Kahan 1965): per element a sum s and a compensation c, the true sum being
// s - c; a batch's partial sum a enters as y = a - c, t = s + y,
// c = (t - s) - y, s = t.  The arrays are s1, c1, s2, c2, each nb floats.
__global__ void __launch_bounds__(256) k_noise_accum_kahan(const float *__restrict__ pyr, int nb, long pyr_bs,
                                                           long nn, int bands, float *__restrict__ acc, int first)
{
    pdl_entry();
    const long ne = bands * nn;
    const long nq = ne / 4;
    float4 *s1 = reinterpret_cast<float4 *>(acc), *c1 = s1 + nq, *s2 = c1 + nq, *c2 = s2 + nq;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < nq; i += (long)gridDim.x * blockDim.x) {
        float a[4] = {0.f, 0.f, 0.f, 0.f}, q[4] = {0.f, 0.f, 0.f, 0.f};
        for_realisations<float4>(pyr + i * 4, nb, pyr_bs, [&](const float4 &v) {
            const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                a[u] += w[u];
                q[u] = fmaf(w[u], w[u], q[u]);
            }
        });
        float4 S1 = make_float4(0.f, 0.f, 0.f, 0.f), C1 = S1, S2 = S1, C2 = S1;
        if (!first) {
            S1 = s1[i];
            C1 = c1[i];
            S2 = s2[i];
            C2 = c2[i];
        }
        float *ps1 = &S1.x, *pc1 = &C1.x, *ps2 = &S2.x, *pc2 = &C2.x;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float y1 = __fsub_rn(a[u], pc1[u]);
            const float t1 = __fadd_rn(ps1[u], y1);
            pc1[u] = __fsub_rn(__fsub_rn(t1, ps1[u]), y1);
            ps1[u] = t1;
            const float y2 = __fsub_rn(q[u], pc2[u]);
            const float t2 = __fadd_rn(ps2[u], y2);
            pc2[u] = __fsub_rn(__fsub_rn(t2, ps2[u]), y2);
            ps2[u] = t2;
        }
        s1[i] = S1;
        c1[i] = C1;
        s2[i] = S2;
        c2[i] = C2;
    }
}

// acc: FP64 s1, s2 (accum 0) or fp32 s1, c1, s2, c2 (accum 1), bands * nn each;
// first: they are written, not added to; beside: a full batch of maps runs
// beside it, so it takes three CTAs an SM instead of sixteen and leaves the
// maps' kernels room.  A short batch ends before a narrow accumulation does:
// there it is wide.  1024^2, wide / four / three / two / one CTA an SM: R = 256
// 5763 / 5754 / 5651 / 5599 / 6402 us, R = 100 2326 / 2314 / 2299 / 2298 / 2526;
// 512^2, R = 100 545 / 542 / 536 / 558 / 603.
int launch_noise_accum(const void *pyr, int nb, long pyr_bs, long nn, int bands, void *acc, int precision, int accum,
                       bool first, bool beside, cudaStream_t s)
{
    long g = (bands * nn / 4 + 255) / 256;
    const long gmax = 152L * (beside ? 3 : 16);
    if (g > gmax) g = gmax;
    double *s1 = static_cast<double *>(acc), *s2 = s1 + (long)bands * nn;
    const int wide = (reinterpret_cast<uintptr_t>(acc) & 15) == 0;
    if (accum == 1)
        FM_LAUNCH(FM_K_NOISE_ACCUM, k_noise_accum_kahan, (unsigned)g, 256, 0, s, (const float *)pyr, nb, pyr_bs, nn,
                  bands, static_cast<float *>(acc), (int)first);
    else if (precision == FM_F64)
        FM_LAUNCH(FM_K_NOISE_ACCUM, (k_noise_accum<double, double2>), (unsigned)g, 256, 0, s, (const double *)pyr,
                  nb, pyr_bs, nn, bands, s1, s2, (int)first, wide);
    else
        FM_LAUNCH(FM_K_NOISE_ACCUM, (k_noise_accum<float, float4>), (unsigned)g, 256, 0, s, (const float *)pyr, nb,
                  pyr_bs, nn, bands, s1, s2, (int)first, wide);
    return FM_OK;
}

// S1 and S2 of element i in FP64: the FP64 sums, or s - c of the Kahan pairs
template <bool KAHAN>
__device__ __forceinline__ void noise_sums(const void *acc, long nelem, long i, double &a, double &q)
{
    if constexpr (KAHAN) {
        const float *f = static_cast<const float *>(acc);
        a = (double)f[i] - (double)f[nelem + i];
        q = (double)f[2 * nelem + i] - (double)f[3 * nelem + i];
    } else {
        const double *d = static_cast<const double *>(acc);
        a = d[i];
        q = d[nelem + i];
    }
}

__device__ __forceinline__ double snr_of(double w, double v) { return w / sqrt(v); }
// fp32 result: w / sqrt(v) with v in FP64.  FP64 square root and division
// are some 40 instructions of a pipe that takes one warp in 16 to 32 cycles,
// so the usual case runs in fp32 pairs: v is split by its bits into hi (24
// leading bits) + lo, y = rsqrt(hi) gets the residual e = 1 - v y^2 from
// exact products (fma), and w y (1 + e / 2) is rounded once: its error is
// that of the rounding plus 3/8 e^2 < 2^-43.  Values near the ends of the
// fp32 range (and zeros, infinities, NaN) take the FP64 form.
__device__ __forceinline__ float snr_of(float w, double v)
{
    const uint32_t vh = (uint32_t)__double2hiint(v), vl = (uint32_t)__double2loint(v);
    const int ex = (int)(vh >> 20) - 1023;  // sign and exponent: negative v fails the test below
    const float aw = fabsf(w);
    if (ex >= -64 && ex <= 64 && aw >= 5.421011e-20f && aw <= 1.844674e19f) {  // 2^-64 .. 2^64
        const float hi = __uint_as_float((uint32_t)(ex + 127) << 23 | (vh & 0xfffffu) << 3 | vl >> 29);
        const float lo = (float)(vl & 0x1fffffffu) * __uint_as_float((uint32_t)(ex - 52 + 127) << 23);
        const float y = rsqrtf(hi);
        const float p = __fmul_rn(hi, y), pe = __fmaf_rn(hi, y, -p);  // hi y = p + pe
        const float e = __fmaf_rn(-p, y, 1.f) - __fmul_rn(__fmaf_rn(lo, y, pe), y);
        const float r = __fmul_rn(w, y), re = __fmaf_rn(w, y, -r);
        return __fadd_rn(r, __fmaf_rn(r, 0.5f * e, re));
    }
    return (float)((double)w / sqrt(v));
}

// VW neighbouring elements a thread (nelem is a multiple of VW)
template <typename T, bool KAHAN, int VW>
__global__ void __launch_bounds__(256) k_noise_final(const void *__restrict__ acc, const T *__restrict__ wdata,
                                                     double *__restrict__ var, T *__restrict__ snr, long nelem,
                                                     double invR, double invR1)
{
    pdl_entry();
    struct alignas(VW * sizeof(T)) Vec {
        T e[VW];
    };
    struct alignas(16) Var {
        double e[2];
    };
    for (long i = (blockIdx.x * (long)blockDim.x + threadIdx.x) * VW; i < nelem;
         i += (long)gridDim.x * blockDim.x * VW) {
        double v[VW], s1[VW], s2[VW];
        if constexpr (VW == 2 && !KAHAN) {
            const double *d = static_cast<const double *>(acc);
            const Var a = *reinterpret_cast<const Var *>(d + i), q = *reinterpret_cast<const Var *>(d + nelem + i);
            s1[0] = a.e[0];
            s1[1] = a.e[1];
            s2[0] = q.e[0];
            s2[1] = q.e[1];
        } else {
#pragma unroll
            for (int u = 0; u < VW; ++u) noise_sums<KAHAN>(acc, nelem, i + u, s1[u], s2[u]);
        }
#pragma unroll
        for (int u = 0; u < VW; ++u) {
            const double a = s1[u], q = s2[u];
            v[u] = (q - a * a * invR) * invR1;
            // v < 0 (rounding) by its bits, without an FP64 comparison; NaN stays
            const uint32_t vh = (uint32_t)__double2hiint(v[u]);
            if (vh >= 0x80000000u && vh <= 0xfff00000u) v[u] = 0;
        }
        if constexpr (VW == 1) {
            var[i] = v[0];
        } else {
#pragma unroll
            for (int u = 0; u < VW; u += 2) *reinterpret_cast<Var *>(var + i + u) = Var{{v[u], v[u + 1]}};
        }
        if (snr) {
            Vec w = *reinterpret_cast<const Vec *>(wdata + i);
#pragma unroll
            for (int u = 0; u < VW; ++u) w.e[u] = snr_of(w.e[u], v[u]);
            *reinterpret_cast<Vec *>(snr + i) = w;
        }
    }
}

template <typename T, bool KAHAN, int VW>
static int final_launch(const void *acc, const T *wdata, double *var, T *snr, long nelem, int R, cudaStream_t s)
{
    long g = (nelem / VW + 255) / 256;
    if (g > 152L * 32) g = 152L * 32;
    FM_LAUNCH(FM_K_NOISE_FINAL, (k_noise_final<T, KAHAN, VW>), (unsigned)g, 256, 0, s, acc, wdata, var, snr, nelem,
              1.0 / R, 1.0 / (R - 1));
    return FM_OK;
}

// Bound by HBM: 16 bytes of sums read and 8 (and 4 + 4 for the S/N) written
// an element.  6 bands of 1024^2 with S/N: 269 -> 42 us (FP64
// square root, division and comparison before).
int launch_noise_finalize(const void *acc, const void *wdata, double *var, void *snr, long nelem, int R,
                          int precision, int accum, cudaStream_t s)
{
    // two elements a thread where every array allows the wide accesses (the
    // caller's pointers need not be aligned beyond their type)
    auto al = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
    const bool wide = nelem % 2 == 0 && al(acc) && al(wdata) && al(var) && al(snr);
    if (precision == FM_F64) {
        const double *w = static_cast<const double *>(wdata);
        double *o = static_cast<double *>(snr);
        return wide ? final_launch<double, false, 2>(acc, w, var, o, nelem, R, s)
                    : final_launch<double, false, 1>(acc, w, var, o, nelem, R, s);
    }
    const float *w = static_cast<const float *>(wdata);
    float *o = static_cast<float *>(snr);
    if (accum == 1)
        return wide ? final_launch<float, true, 2>(acc, w, var, o, nelem, R, s)
                    : final_launch<float, true, 1>(acc, w, var, o, nelem, R, s);
    return wide ? final_launch<float, false, 2>(acc, w, var, o, nelem, R, s)
                : final_launch<float, false, 1>(acc, w, var, o, nelem, R, s);
}

// ---- exact expected variance (periodic boundary) ----------------------------
// out[c][p] = (a[c][p]^2 + b[c][p]^2) f, f = 1 for c < h, fh for c = h and f0
// above (powers of two): |K_j|^2 from the two delta responses (the second half
// of the bands scaled up to the first's magnitude), |gamma|^2 from the shear.
// VW elements a thread; grid = (blocks, count).
template <typename T, int VW>
__global__ void __launch_bounds__(256) k_modulus2(const T *__restrict__ a, long a_bs, const T *__restrict__ b,
                                                  long b_bs, T *__restrict__ out, long nn, int h, T fh, T f0)
{
    pdl_entry();
    struct alignas(VW * sizeof(T)) Vec {
        T e[VW];
    };
    const int c = blockIdx.y;
    const T f = c < h ? (T)1 : c == h ? fh : f0;
    a += c * a_bs;
    b += c * b_bs;
    out += c * nn;
    for (long i = (blockIdx.x * (long)blockDim.x + threadIdx.x) * VW; i < nn; i += (long)gridDim.x * blockDim.x * VW) {
        Vec x = *reinterpret_cast<const Vec *>(a + i);
        const Vec y = *reinterpret_cast<const Vec *>(b + i);
#pragma unroll
        for (int u = 0; u < VW; ++u) x.e[u] = (x.e[u] * x.e[u] + y.e[u] * y.e[u]) * f;
        *reinterpret_cast<Vec *>(out + i) = x;
    }
}

// unit shear at pixel 0: gamma1 of map 0 and gamma2 of map 1 (arrays zeroed before)
template <typename T> __global__ void k_unit_shears(T *g1d, T *g2d, long nn)
{
    pdl_entry();
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        g1d[0] = (T)1;
        g2d[nn] = (T)1;
    }
}

template <typename T, int VW>
static int modulus2_impl(const T *a, long a_bs, const T *b, long b_bs, T *out, long nn, int count, int h, T fh, T f0,
                         cudaStream_t s)
{
    long g = (nn / VW + 255) / 256;
    if (g > 152L * 8) g = 152L * 8;
    FM_LAUNCH(0, (k_modulus2<T, VW>), dim3((unsigned)g, count), 256, 0, s, a, a_bs, b, b_bs, out, nn, h, fh, f0);
    return FM_OK;
}

int launch_modulus2(const void *a, long a_bs, const void *b, long b_bs, void *out, long nn, int count, int h,
                    double fh, double f0, int precision, cudaStream_t s)
{
    // 16-byte accesses (nn is a multiple of 16); the caller's shear may be aligned to its element only
    const bool al = ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0;
    if (precision == FM_F64) {
        const double *p = static_cast<const double *>(a), *q = static_cast<const double *>(b);
        double *o = static_cast<double *>(out);
        return al ? modulus2_impl<double, 2>(p, a_bs, q, b_bs, o, nn, count, h, fh, f0, s)
                  : modulus2_impl<double, 1>(p, a_bs, q, b_bs, o, nn, count, h, fh, f0, s);
    }
    const float *p = static_cast<const float *>(a), *q = static_cast<const float *>(b);
    float *o = static_cast<float *>(out);
    return al ? modulus2_impl<float, 4>(p, a_bs, q, b_bs, o, nn, count, h, (float)fh, (float)f0, s)
              : modulus2_impl<float, 1>(p, a_bs, q, b_bs, o, nn, count, h, (float)fh, (float)f0, s);
}

int launch_unit_shears(void *g1d, void *g2d, long nn, int precision, cudaStream_t s)
{
    const size_t es = precision == FM_F64 ? 8 : 4;
    FM_CUDA_TRY(cudaMemsetAsync(g1d, 0, 2 * nn * es, s));
    FM_CUDA_TRY(cudaMemsetAsync(g2d, 0, 2 * nn * es, s));
    if (precision == FM_F64)
        FM_LAUNCH(0, k_unit_shears<double>, 1, 32, 0, s, (double *)g1d, (double *)g2d, nn);
    else
        FM_LAUNCH(0, k_unit_shears<float>, 1, 32, 0, s, (float *)g1d, (float *)g2d, nn);
    return FM_OK;
}

}  // namespace fm

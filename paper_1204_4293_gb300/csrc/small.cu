// small.cu -- Kaiser-Squires and the starlet of small fp32 maps (n = 64, 128, 256)
// in one kernel: a cluster of n / 16 CTAs holds a map in its shared memory.
//
// A single small map is bound by launches: eight kernels whose grids are 16 to
// 64 CTAs take 25 us on the GPU and 34 us of the host for 256^2.  Here CTA `rank`
// owns 16 rows (and, between, 16 columns), every thread 16 elements:
//   rows FFT of gamma1 + i gamma2 in the CTA
//   -- cluster barrier; columns gathered from the CTAs' shared memory --
//   column FFT, times conj(D), column inverse FFT
//   -- cluster barrier; rows gathered back --
//   row inverse FFT: kappa (and kappa_B), kept in shared memory
//   per scale: row filter of the own rows; cluster barrier; column filter on
//   rows gathered from the CTAs that own them; band out, c_j kept.
// The arithmetic is that of fft32.cu's complex form and of starlet.cu, operation
// by operation, so the results are bit-identical to theirs.  What bounds it is
// the chain of J + 2 cluster barriers (two in Kaiser-Squires, one a scale, one at
// the end; about 1 us each) with little work between: KS + starlet of one map,
// J = 5 / 6 / 6, in a queue of calls, 64^2 33 -> 13 us a call, 128^2 34 -> 16,
// 256^2 34 -> 23 (replayed from a graph, the GPU alone, 12.0, 15.5 and 21.8; with
// 32 rows a CTA the kernel took 1.1, 1.2 and 1.4 times as long).
#include <cooperative_groups.h>

#include <atomic>

#include "common.cuh"
#include "fft32_core.cuh"
#include "starlet_math.cuh"

namespace fm {
namespace cg = cooperative_groups;

template <int LOGN> struct SmallMap {
    using P = FftPlan<LOGN>;
    static constexpr int N = P::N, E = P::E, TV = P::TV;
    static constexpr int R = 16, C = N / R;  // rows (and columns) of a CTA, CTAs of a map
    static constexpr int T = R * N / E;      // threads
    static constexpr int VS = N + N / E;     // exchange buffer of a row
    // buffer A: the rows' exchange, later kappa / c_j and the first row-filtered
    // copy; buffer B: the columns' exchange, later the second
    static constexpr int A_ELEMS = R * VS, B_ELEMS = N * R + N * R / E;
    static constexpr size_t smem = (size_t)(A_ELEMS + B_ELEMS) * sizeof(float2);
    static_assert(E == 16 && 2 * R * N * sizeof(float) <= A_ELEMS * sizeof(float2), "buffers");
};

// KS: from shear (in1, in2); else in1 is kappa.  ST: the pyramid (J arrays a map)
// to out1; else kappa to out1 and, unless null, kappa_B to out2.
template <int LOGN, bool KS, bool ST>
__global__ void __launch_bounds__(SmallMap<LOGN>::T) k_small_map(const float *__restrict__ in1,
                                                                 const float *__restrict__ in2,
                                                                 float *__restrict__ out1, float *__restrict__ out2,
                                                                 const float2 *__restrict__ tw, int J, int boundary,
                                                                 float scale)
{
    pdl_entry();
    using M = SmallMap<LOGN>;
    using P = typename M::P;
    constexpr int N = M::N, E = M::E, TV = M::TV, R = M::R, T = M::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *A = reinterpret_cast<float2 *>(smem_raw), *B = A + M::A_ELEMS;
    float *c = reinterpret_cast<float *>(A);  // [R][N] kappa, then c_j
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), t = threadIdx.x;
    const long map = blockIdx.x / M::C, nn = (long)N * N;
    const int y0 = rank * R;
    if constexpr (KS) {
        const int vr = t / TV, j = t % TV;  // the thread's row and first column
        float2 *row = A + vr * M::VS;
        const long off = map * nn + (long)(y0 + vr) * N + j;
        float2 v[E];
#pragma unroll
        for (int q = 0; q < E; ++q) v[q] = make_float2(__ldcs(in1 + off + q * TV), __ldcs(in2 + off + q * TV));
        fft_vec<LOGN, 1, false>(v, row, 0, j, tw);
        __syncthreads();  // the last pass's reads
#pragma unroll
        for (int q = 0; q < E; ++q) row[j + q * TV] = v[q];
        cluster.sync();
        // columns: thread (cj, cc) takes rows cj + q TV of column R rank + cc
        const int cc = t % R, cj = t / R, x = y0 + cc;
#pragma unroll
        for (int q = 0; q < E; ++q) {
            const int y = cj + q * TV;
            v[q] = cluster.map_shared_rank(A, y / R)[(y % R) * M::VS + x];
        }
        fft_vec<LOGN, R, false>(v, B, cc, cj, tw);
        const float k1 = (float)(x < N / 2 ? x : x - N), jf = (float)cj;
#pragma unroll
        for (int q = 0; q < E; ++q) {  // conj(D), as in k_cols_ks32
            const float k2 = freq_of<LOGN>(jf, q);
            const float den = k1 * k1 + k2 * k2;
            float2 d = make_float2(0.f, 0.f);
            if (den != 0.f) {
                const float inv = __fdividef(1.f, den);
                const float im = 2.f * k1 * k2 * inv;
                d = make_float2((k1 * k1 - k2 * k2) * inv, -im);
            }
            v[q] = cmul(v[q], d);
        }
        fft_vec<LOGN, R, true>(v, B, cc, cj, tw);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < E; ++q) B[(cj + q * TV) * R + cc] = v[q];
        cluster.sync();  // also: every column gather from A is done
#pragma unroll
        for (int q = 0; q < E; ++q) {
            const int kx = j + q * TV;
            v[q] = cluster.map_shared_rank(B, kx / R)[(y0 + vr) * R + kx % R];
        }
        fft_vec<LOGN, 1, true>(v, row, 0, j, tw);
        if constexpr (ST) {
            __syncthreads();  // the last pass's reads of A
#pragma unroll
            for (int q = 0; q < E; ++q) c[vr * N + j + q * TV] = v[q].x * scale;
        } else {
#pragma unroll
            for (int q = 0; q < E; ++q) {
                out1[off + q * TV] = v[q].x * scale;
                if (out2) out2[off + q * TV] = v[q].y * scale;
            }
        }
    } else {
        const float *src = in1 + map * nn + (long)y0 * N;
        for (int e = t; e < R * N; e += T) c[e] = __ldcs(src + e);
    }
    if constexpr (ST) {
        float *wout = out1 + map * J * nn + (long)y0 * N;
        constexpr int NQ = N / 4, QPT = R * NQ / T;  // vectors of a row, of a thread
        // one reflection (or wrap) reaches every tap: 2 s < n
        auto fold = [&](int i) {
            if (boundary == FM_PERIODIC) return i & (N - 1);
            i = i < 0 ? -i : i;
            return i >= N ? 2 * (N - 1) - i : i;
        };
        for (int s = 1, jj = 1; jj < J; ++jj, s *= 2) {
            float *r = jj & 1 ? c + R * N : reinterpret_cast<float *>(B);
            __syncthreads();  // c_{j-1} complete
            {
                // rows: a thread keeps its column (folded taps once) and steps down the rows
                static_assert(T % N == 0, "whole rows a step");
                const int x = t % N;
                const float *p = c + t / N * N;
                const int m2 = fold(x - 2 * s), m1 = fold(x - s), p1 = fold(x + s), p2 = fold(x + 2 * s);
                float *o = r + t;
#pragma unroll 8
                for (int k = 0; k < R * N / T; ++k)
                    o[k * T] = tap5(p[k * T + m2], p[k * T + m1], p[k * T + x], p[k * T + p1], p[k * T + p2]);
            }
            cluster.sync();
#pragma unroll
            for (int k = 0; k < QPT; ++k) {
                const int e = t + k * T, yl = e / NQ, xx = e % NQ * 4, y = y0 + yl;
                auto at = [&](int yy) {
                    const int g = fold(yy), o = g / R;
                    const float *q = o == rank ? r : cluster.map_shared_rank(r, o);
                    return p4(q + (g % R) * N + xx);
                };
                const Pair4 f = tap5(at(y - 2 * s), at(y - s), p4(r + e * 4), at(y + s), at(y + 2 * s));
                const float2 sc = make_float2(1.f / 256.f, 1.f / 256.f), m1 = make_float2(-1.f, -1.f);
                const float2 ca = __fmul2_rn(f.a, sc), cb = __fmul2_rn(f.b, sc);
                const Pair4 prev = p4(c + e * 4);
                const float2 wa = __ffma2_rn(ca, m1, prev.a), wb = __ffma2_rn(cb, m1, prev.b);
                const float4 cj = make_float4(ca.x, ca.y, cb.x, cb.y);
                __stcs(reinterpret_cast<float4 *>(wout + (jj - 1) * nn + e * 4), make_float4(wa.x, wa.y, wb.x, wb.y));
                if (jj == J - 1)
                    __stcs(reinterpret_cast<float4 *>(wout + jj * nn + e * 4), cj);
                else
                    sf4(c + e * 4, cj);
            }
        }
    }
    cluster.sync();  // other CTAs may still read this one's shared memory
}

template <int LOGN, bool KS, bool ST>
static int small_launch_t(const float *in1, const float *in2, float *out1, float *out2, int J, int batch, int boundary,
                          const float2 *tw, cudaStream_t s)
{
    using M = SmallMap<LOGN>;
    auto k = k_small_map<LOGN, KS, ST>;
    FM_CUDA_TRY(fm::smem_attr((const void *)k, M::smem));
    if (M::C > 8) FM_CUDA_TRY(cudaFuncSetAttribute((const void *)k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(batch * M::C);
    cfg.blockDim = dim3(M::T);
    cfg.dynamicSmemBytes = M::smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = M::C;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_pdl.load(std::memory_order_relaxed) ? 2 : 1;
    const float scale = kFft32Gain / ((float)M::N * (float)M::N);
    cudaError_t e = cudaLaunchKernelEx(&cfg, k, in1, in2, out1, out2, tw, J, boundary, scale);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    if (e != cudaSuccess) return cuda_fail(e, "k_small_map");
    return FM_OK;
}

template <bool KS, bool ST>
static int small_launch(const float *in1, const float *in2, float *out1, float *out2, int n, int J, int batch,
                        int boundary, cudaStream_t s)
{
    int st = FM_OK;
    const float2 *tw = nullptr;
    if (KS && !(tw = static_cast<const float2 *>(twiddles(n, FM_F32, s, &st)))) return st;
    switch (n) {
    case 64: return small_launch_t<6, KS, ST>(in1, in2, out1, out2, J, batch, boundary, tw, s);
    case 128: return small_launch_t<7, KS, ST>(in1, in2, out1, out2, J, batch, boundary, tw, s);
    default: return small_launch_t<8, KS, ST>(in1, in2, out1, out2, J, batch, boundary, tw, s);
    }
}

// Whether this device can hold a cluster of 16 CTAs of the 256^2 kernel (above
// the portable 8; asked once a device).
static bool cluster16_ok()
{
    static std::atomic<int> known[64];  // 0 unknown, 1 yes, 2 no
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev >= 64) return false;
    int v = known[dev].load(std::memory_order_relaxed);
    if (!v) {
        using M = SmallMap<8>;
        auto k = k_small_map<8, true, true>;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(M::C);
        cfg.blockDim = dim3(M::T);
        cfg.dynamicSmemBytes = M::smem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = M::C;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int fit = 0;
        const bool ok =
            fm::smem_attr((const void *)k, M::smem) == cudaSuccess &&
            cudaFuncSetAttribute((const void *)k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&fit, k, &cfg) == cudaSuccess && fit > 0;
        if (!ok) cudaGetLastError();
        known[dev].store(v = ok ? 1 : 2, std::memory_order_relaxed);
    }
    return v == 1;
}

// Whether a call takes the one-kernel form: fp32 maps of 64^2, 128^2 or 256^2
// in batches up to where the separate kernels, which spread a batch over the
// GPU with no barriers, catch up; with nothing asked for that names another
// form (depth, large path, knobs, per-kernel timing).  An autotuned plan names
// none: it describes the separate kernels, and so governs the batches above
// these limits.  J = 0: Kaiser-Squires alone.  Measured, one kernel / separate kernels (us a call,
// host included): KS + starlet 64^2 J = 5 x 256 27 / 41, x 512 51 / 58; 128^2 J
// = 6 x 48 26 / 33, x 64 41 / 36; 256^2 J = 6 x 6 23 / 33, x 8 33 / 32; KS alone
// 64^2 x 512 24 / 25, 128^2 x 96 18 / 23, x 128 25 / 23, 256^2 x 16 18 / 23, x 24
// 24 / 23.  `aligned`: the pyramid is 16-byte aligned (its stores are vectors).
bool small_map_ok(int n, int J, int batch, const fm_config &cfg, bool aligned)
{
    if (cfg.precision != FM_F32 || !aligned || cfg.fuse_depth != 0 || cfg.large_path != 0) return false;
    const int most = J == 0 ? (n == 64 ? 512 : n == 128 ? 96 : n == 256 ? 16 : 0)
                            : (n == 64 ? 256 : n == 128 ? 48 : n == 256 ? 6 : 0);
    return batch <= most && g_prof_kid.load(std::memory_order_relaxed) == 0 &&
           g_ks_real.load(std::memory_order_relaxed) != 1 && g_tile_variant.load(std::memory_order_relaxed) < 0 &&
           g_wait_test.load(std::memory_order_relaxed) == 0 &&
           g_use_tma.load(std::memory_order_relaxed) == kDefaultTma && (n < 256 || cluster16_ok());
}

int launch_small_map(const float *g1, const float *g2, float *pyr, int n, int J, int batch, int boundary,
                     cudaStream_t s)
{
    return small_launch<true, true>(g1, g2, pyr, nullptr, n, J, batch, boundary, s);
}
int launch_small_ks(const float *g1, const float *g2, float *kE, float *kB, int n, int batch, cudaStream_t s)
{
    return small_launch<true, false>(g1, g2, kE, kB, n, 0, batch, FM_MIRROR, s);
}
int launch_small_starlet(const float *kappa, float *pyr, int n, int J, int batch, int boundary, cudaStream_t s)
{
    return small_launch<false, true>(kappa, nullptr, pyr, nullptr, n, J, batch, boundary, s);
}

}  // namespace fm

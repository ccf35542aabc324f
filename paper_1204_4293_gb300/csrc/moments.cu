// moments.cu -- statistics of the aperture-mass maps (Sec. 2.2): per map and
// per pyramid array the mean, variance <M_ap^2>, skewness and excess
// kurtosis over the pixels.
//
// Two passes over the pyramid: the first sums x per (map, array), the second
// sums (x - mean)^2, ^3, ^4.  A strand is the run of at most 16 pixels S
// apart (S = 256 ceil(nn / 4096)) whose sums are formed in fp32; strands are
// added in three floats (hi + mid + lo by error-free two-sums) over a thread
// and a block, and by one FP64 atomic per block and quantity; a last tiny
// kernel forms the moments.
//
// The work is two reads of the pyramid.  FP64 adds are the scarce resource
// otherwise (one warp instruction in 16 to 32 cycles an SM on GB300): an FP64
// shuffle tree over every thread's sums kept the second pass at 219 us for 8
// pyramids of 7 x 1024^2 (235 MB, 35 us a read).  The three floats carry 72
// bits and leave FP64 a few instructions a block; 16-byte loads, eight in
// flight a thread.  Those 8 pyramids: 293 -> 84 us for the whole call; in fp64
// 234 (two floats, 48 bits, instead of three 230).  Running both passes over 20
// .. 80 MB groups of arrays, so that the second read comes from L2, was no
// faster (154 .. 90 us against 90: shorter launches).
#include <algorithm>

#include "common.cuh"

namespace fm {

// A sum of floats as hi + mid + lo: two chained two-sums (Knuth, TAOCP 4.2.2)
// carry every rounding error down, so the sum holds up to 72 bits, more than
// an FP64 sum's 53.
struct FloatSum {  // (no initialisers: it is kept in shared memory too)
    float hi, mid, lo;
    // a += b, returning the rounding error
    __device__ __forceinline__ static float two_sum(float &a, float b)
    {
        const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
        const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
        a = s;
        return e;
    }
    __device__ __forceinline__ void add(float p) { lo = __fadd_rn(lo, two_sum(mid, two_sum(hi, p))); }
    __device__ __forceinline__ void add(const FloatSum &v)
    {
        add(v.hi);
        lo = __fadd_rn(lo, __fadd_rn(two_sum(mid, v.mid), v.lo));
    }
    __device__ __forceinline__ double value() const { return (double)hi + ((double)mid + (double)lo); }
};
// Strands of 2^100 and more (and infinities and NaN) go to the FP64 sums
// directly: a block's sums of the others stay finite (2^100 x 256 threads x
// their strands, 2^14 at 8192^2 and with eight blocks an SM at 65536^2).
constexpr float kStrandMax = 1.2676506e30f;

// the sum over the first N lanes, in lane 0
template <int N> __device__ __forceinline__ FloatSum lane_sum(FloatSum v)
{
#pragma unroll
    for (int o = N / 2; o > 0; o >>= 1)
        v.add(FloatSum{__shfl_down_sync(0xffffffffu, v.hi, o), __shfl_down_sync(0xffffffffu, v.mid, o),
                       __shfl_down_sync(0xffffffffu, v.lo, o)});
    return v;
}

// grid = (blocks per array, J, batch); sums[(b * J + j) * 4 + q].  A thread takes VW neighbouring
// strands at a time (VW > 1: nn a multiple of VW and 16-byte aligned arrays).  The bound of one block an SM
// lets the compiler keep all eight loads in flight (8 x 7 x 1024^2 89 -> 84 us, 1023^2 150 -> 111).
template <typename T, int PASS, int VW>
__global__ void __launch_bounds__(256, 1) k_moments(const T *__restrict__ pyr, long nn, long S, double inv_nn,
                                                 double *__restrict__ sums)
{
    pdl_entry();
    constexpr int NQ = PASS == 0 ? 1 : 3;
    struct alignas(VW * sizeof(T)) Vec {
        T e[VW];
    };
    const long array = (long)blockIdx.z * gridDim.y + blockIdx.y;
    const T *x = pyr + array * nn;
    double *acc = sums + array * 4;
    __shared__ float s_mean;
    __shared__ FloatSum red[NQ][8];
    float mean = 0.f;
    if constexpr (PASS == 1) {
        if (threadIdx.x == 0) s_mean = (float)(acc[0] * inv_nn);
        __syncthreads();
        mean = s_mean;
    }
    FloatSum tot[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) tot[q] = FloatSum{0.f, 0.f, 0.f};
    for (long v0 = ((long)blockIdx.x * 256 + threadIdx.x) * VW; v0 < S; v0 += (long)gridDim.x * 256 * VW) {
        float s[VW][NQ] = {};
        auto add = [&](const Vec &v) {
#pragma unroll
            for (int u = 0; u < VW; ++u) {
                if constexpr (PASS == 0) {
                    s[u][0] += (float)v.e[u];
                } else {
                    const float d = (float)v.e[u] - mean, d2 = d * d;
                    s[u][0] += d2;
                    s[u][1] += d2 * d;
                    s[u][2] += d2 * d2;
                }
            }
        };
        long i = v0;
        for (; i + 7 * S < nn; i += 8 * S) {  // eight loads in flight
            Vec v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = *reinterpret_cast<const Vec *>(x + i + k * S);
#pragma unroll
            for (int k = 0; k < 8; ++k) add(v[k]);
        }
        for (; i < nn; i += S) add(*reinterpret_cast<const Vec *>(x + i));
        float big = 0.f;
#pragma unroll
        for (int u = 0; u < VW; ++u)
#pragma unroll
            for (int q = 0; q < NQ; ++q) big += fabsf(s[u][q]);
        // one test for all, so that the quantities' chains of adds run beside each other
        if (big < kStrandMax) {
#pragma unroll
            for (int u = 0; u < VW; ++u)
#pragma unroll
                for (int q = 0; q < NQ; ++q) tot[q].add(s[u][q]);
        } else {
#pragma unroll
            for (int u = 0; u < VW; ++u)
#pragma unroll
                for (int q = 0; q < NQ; ++q) atomicAdd(acc + PASS + q, (double)s[u][q]);
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const FloatSum r = lane_sum<32>(tot[q]);
        if (lane == 0) red[q][warp] = r;
    }
    __syncthreads();
    if (warp < NQ) {  // one quantity a warp
        const FloatSum r = lane_sum<8>(lane < 8 ? red[warp][lane] : FloatSum{0.f, 0.f, 0.f});
        if (lane == 0) atomicAdd(acc + PASS + warp, r.value());
    }
}

// moments[(b * J + j) * 4 + {0,1,2,3}] = mean, variance, skewness, excess kurtosis
__global__ void k_moments_final(const double *__restrict__ sums, double *__restrict__ out, long nn, int count)
{
    pdl_entry();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const double *s = sums + 4 * (long)i;
    const double m2 = s[1] / (double)nn, m3 = s[2] / (double)nn, m4 = s[3] / (double)nn;
    double *o = out + 4 * (long)i;
    o[0] = s[0] / (double)nn;
    o[1] = m2;
    o[2] = m2 > 0 ? m3 / (m2 * sqrt(m2)) : 0.0;
    o[3] = m2 > 0 ? m4 / (m2 * m2) - 3.0 : 0.0;
}

template <typename T, int VW>
static int moments_impl(const T *pyr, double *sums, int J, int batch, long nn, cudaStream_t s)
{
    const long S = (nn + 256 * 16 - 1) / (256 * 16) * 256;  // strands of at most 16 pixels (fp32 partial sums)
    // about eight blocks an SM over all arrays (4 / 8: 93 / 88 us for 8
    // pyramids of 7 x 1024^2), at least one an array
    const long count = (long)J * batch;
    const long bx = std::min<long>((S / VW + 255) / 256, std::max<long>(1, (152 * 8 + count - 1) / count));
    const dim3 grid((unsigned)bx, J, batch);
    const double inv_nn = 1.0 / (double)nn;
    FM_LAUNCH(0, (k_moments<T, 0, VW>), grid, 256, 0, s, pyr, nn, S, inv_nn, sums);
    FM_LAUNCH(0, (k_moments<T, 1, VW>), grid, 256, 0, s, pyr, nn, S, inv_nn, sums);
    return FM_OK;
}

int launch_band_moments(const void *pyr, double *moments, int n, int J, int batch, int precision, void *scratch,
                        cudaStream_t s)
{
    const long nn = (long)n * n;
    double *sums = static_cast<double *>(scratch);
    const int count = batch * J;
    FM_CUDA_TRY(cudaMemsetAsync(sums, 0, sizeof(double) * 4 * (size_t)count, s));
    const bool al = (reinterpret_cast<uintptr_t>(pyr) & 15) == 0;
    int st;
    if (precision == FM_F64)
        st = al && nn % 2 == 0 ? moments_impl<double, 2>((const double *)pyr, sums, J, batch, nn, s)
                               : moments_impl<double, 1>((const double *)pyr, sums, J, batch, nn, s);
    else
        st = al && nn % 4 == 0 ? moments_impl<float, 4>((const float *)pyr, sums, J, batch, nn, s)
                               : moments_impl<float, 1>((const float *)pyr, sums, J, batch, nn, s);
    if (st != FM_OK) return st;
    FM_LAUNCH(0, k_moments_final, (unsigned)((count + 127) / 128), 128, 0, s, sums, moments, nn, count);
    return FM_OK;
}

}  // namespace fm

// fft64.cu -- fp64 Kaiser-Squires FFT (Sec. 4.5) with register-resident radix-8
// sub-transforms, n = 64 .. 2048.
//
// The same three passes as fft32.cu (row FFT, column FFT with the spectral
// operation and the inverse column FFT, row inverse), with 8 elements a
// thread, plain loads and no bulk copies.  What bounds them is the FP64 pipe
// (one warp instruction in about 16 cycles an SM), so they save operations
// rather than bytes: kappa_E alone goes through the half spectrum (the split
// row FFT, a column pass with one inverse for two forward transforms, a
// half-length complex-to-real row pass: three quarters of the butterflies,
// see fft32.cu for the identities), the split's factors of 1/2 are left to the
// last scaling, and 1 / |k|^2 is an fp32 reciprocal with two Newton steps
// instead of a division.  One 1024^2 map: row pass 86 -> 73 us, columns 201 ->
// 140, inverse rows 87 -> 49 (the shared-memory passes of fft.cu before).
// Against extended precision kappa_E of 64^2 / 256^2 / 1024^2 is off by 3.3 / 4.0 /
// 4.8e-16 (rms), the complex form by 3.3 / 3.9 / 4.7e-16: the split and the
// half-length inverse add roundings, the reciprocal none that shows.
#include "common.cuh"
#include "dft.cuh"
#include "fft32_tables.cuh"
#include "rng.cuh"

namespace fm {

template <int LOGN> struct Plan64 {
    static constexpr int N = 1 << LOGN, LOGE = kFft64LogE, E = 1 << LOGE, TV = N / E;
    static constexpr int NPASS = (LOGN + LOGE - 1) / LOGE, LOGRL = LOGN - LOGE * (NPASS - 1);
    static constexpr int RL = 1 << LOGRL, ML = E / RL, NSL = N / RL;
    __host__ __device__ static constexpr int pass_off(int p) { return (1 << (LOGE * p)) - E; }
    static constexpr int RPC = TV >= 128 ? 1 : 128 / TV, ROW_T = RPC * TV;  // rows and threads of a row-pass CTA
    static constexpr int VS = N + N / E;                                    // exchange buffer of a vector
    static constexpr int W = N <= 512 ? 8 : 4096 / N;      // columns of a strip (complex form)
    static constexpr int WS = N <= 256 ? 8 : 2048 / N;                      // slots of a strip (real-output form)
    static constexpr int NH = WS * TV, NT = 2 * NH;
    static constexpr int RSZ = N * WS + N * WS / E + 1;
    static_assert(WS == 1 || RSZ >= 2 * N, "corner exchange");
};

__device__ __forceinline__ constexpr int padded8(int a) { return a + (a >> kFft64LogE); }

template <int NB> __device__ __forceinline__ void sync_part()
{
    if constexpr (NB == 0)
        __syncthreads();
    else
        asm volatile("bar.sync 1, %0;" ::"n"(NB) : "memory");
}

template <bool INV> __device__ __forceinline__ double2 mul_tw(double2 a, const double2 *__restrict__ tw)
{
    double2 w = __ldg(tw);
    if (INV) w.y = -w.y;
    return cmul(a, w);
}

// v[q] = x[j + q TV] -> X[j + q TV]; exchanges at sm[padded8(i W + c)]
template <int LOGN, int W, bool INV, int NB = 0>
__device__ __forceinline__ void fft_vec(double2 (&v)[8], double2 *sm, int c, int j, const double2 *__restrict__ tw)
{
    using P = Plan64<LOGN>;
    constexpr int E = P::E;
    static_assert(W <= E, "padding");
    double2 *rd = sm + padded8(j * W + c);
    auto load = [&](int q) { return rd[padded8(q * P::TV * W)]; };
    Dft<8, INV, double2>::run(v);
    sync_part<NB>();
    {
        double2 *wr = sm + j * (E * W + W) + c;
#pragma unroll
        for (int r = 0; r < E; ++r) wr[padded8(r * W)] = v[r];
    }
    sync_part<NB>();
#pragma unroll
    for (int p = 1; p + 1 < P::NPASS; ++p) {
        const int NS = 1 << (P::LOGE * p);
#pragma unroll
        for (int r = 0; r < E; ++r) v[r] = load(r);
        const int k = j & (NS - 1);
        const double2 *t = tw + P::N + P::pass_off(p) + k;
#pragma unroll
        for (int r = 1; r < E; ++r) v[r] = mul_tw<INV>(v[r], t + (r - 1) * NS);
        Dft<8, INV, double2>::run(v);
        sync_part<NB>();
        double2 *wr = sm + padded8(((j - k) * E + k) * W + c);
#pragma unroll
        for (int r = 0; r < E; ++r) wr[padded8(r * NS * W)] = v[r];
        sync_part<NB>();
    }
    const double2 *t = tw + P::N + P::pass_off(P::NPASS - 1) + j;
#pragma unroll
    for (int m = 0; m < P::ML; ++m) {
        double2 x[P::RL];
#pragma unroll
        for (int r = 0; r < P::RL; ++r) {
            x[r] = load(m + r * P::ML);
            if (r > 0) x[r] = mul_tw<INV>(x[r], t + (r - 1) * P::NSL + m * P::TV);
        }
        Dft<P::RL, INV, double2>::run(x);
#pragma unroll
        for (int r = 0; r < P::RL; ++r) v[m + r * P::ML] = x[r];
    }
}

// signed integer frequency of index j + q TV
template <int LOGN> __device__ __forceinline__ int freq_of(int j, int q)
{
    using P = Plan64<LOGN>;
    return j + q * P::TV - (q >= P::E / 2 ? P::N : 0);
}
// conj(D) = (dr, -di), D = (k1 + i k2)^2 / |k|^2 (D(0) = 0); the squares are
// exact integers below 2^25
__device__ __forceinline__ void ks_factor(int k1, int k2, double &dr, double &di)
{
    const int den = k1 * k1 + k2 * k2;
    const double d = (double)den;
    double r = (double)__frcp_rn((float)(den ? den : 1));
    r = fma(r, fma(-d, r, 1.0), r);
    r = fma(r, fma(-d, r, 1.0), r);
    if (den == 0) r = 0.0;
    dr = (double)(k1 * k1 - k2 * k2) * r;
    di = (double)(2 * k1 * k2) * r;
}

// SPLIT: each row's spectrum Z as n / 2 slots (2 Gamma1(kx), 2 Gamma2(kx)),
// slot 0 packing the real pairs at kx = 0 and n / 2
template <int LOGN, bool SPLIT, bool ROT>
__global__ void __launch_bounds__(Plan64<LOGN>::ROW_T)
    k_rows_fwd64(const double *__restrict__ in1, const double *__restrict__ in2, long in_bs, double2 *__restrict__ work,
                 long total_rows, const double2 *__restrict__ tw, const uint64_t *__restrict__ seed, int r0)
{
    pdl_wait();
    using P = Plan64<LOGN>;
    extern __shared__ __align__(16) double2 smd[];
    const int vr = threadIdx.x / P::TV, j = threadIdx.x % P::TV;
    const long row = (long)blockIdx.x * P::RPC + vr;
    double2 *sm = smd + vr * P::VS;
    const bool live = row < total_rows;
    double2 v[8];
    if (live) {
        const long b = row >> LOGN;
        const int y = (int)(row & (P::N - 1));
        const long off = b * in_bs + (long)y * P::N;
        uint64_t sd = 0;
        if constexpr (ROT) sd = *seed;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int x = j + r * P::TV;
            double a = __ldcs(in1 + off + x), c = in2 ? __ldcs(in2 + off + x) : 0.0;
            if constexpr (ROT) rotate_shear(a, c, sd, r0 + b, y, x, P::N);
            v[r] = make_double2(a, c);
        }
    } else {
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = make_double2(0.0, 0.0);
    }
    fft_vec<LOGN, 1, false>(v, sm, 0, j, tw);
    double2 *dst = work + row * P::N;
    if constexpr (SPLIT) {
        __syncthreads();  // the last pass's reads of the buffer
#pragma unroll
        for (int q = 0; q < 8; ++q) sm[padded8(j + q * P::TV)] = v[q];
        __syncthreads();
        if (!live) return;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int kx = j + q * P::TV;
            const double2 a = v[q];  // Z(kx)
            if (kx == 0) {
                const double2 h = sm[padded8(P::N / 2)];
                dst[0] = make_double2(a.x + a.x, h.x + h.x);
                dst[1] = make_double2(a.y + a.y, h.y + h.y);
            } else {
                const double2 m = sm[padded8(P::N - kx)];  // Z(n - kx)
                dst[2 * kx] = make_double2(a.x + m.x, a.y - m.y);
                dst[2 * kx + 1] = make_double2(a.y + m.y, m.x - a.x);
            }
        }
    } else if (live) {
#pragma unroll
        for (int q = 0; q < 8; ++q) dst[j + q * P::TV] = v[q];
    }
}

template <int LOGN, bool WITH_B>
__global__ void __launch_bounds__(Plan64<LOGN>::ROW_T)
    k_rows_inv64(const double2 *__restrict__ work, double *__restrict__ out1, double *__restrict__ out2,
                 long total_rows, const double2 *__restrict__ tw, double scale, double im_scale,
                 double im_scale0)
{
    pdl_wait();
    using P = Plan64<LOGN>;
    extern __shared__ __align__(16) double2 smd[];
    const int vr = threadIdx.x / P::TV, j = threadIdx.x % P::TV;
    const long row = (long)blockIdx.x * P::RPC + vr;
    const bool live = row < total_rows;
    double2 v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = live ? work[row * P::N + j + r * P::TV] : make_double2(0.0, 0.0);
    fft_vec<LOGN, 1, true>(v, smd + vr * P::VS, 0, j, tw);
    if (!live) return;
    [[maybe_unused]] const double ims = row < P::N ? im_scale0 : im_scale;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const long pos = row * P::N + j + q * P::TV;
        out1[pos] = v[q].x * scale;
        if constexpr (WITH_B) out2[pos] = v[q].y * ims;
    }
}

template <int LOGN>
__global__ void __launch_bounds__(Plan64<LOGN>::W *Plan64<LOGN>::TV)
    k_cols64(double2 *__restrict__ work, const double2 *__restrict__ tw, int op, const double2 *__restrict__ filt)
{
    pdl_wait();
    using P = Plan64<LOGN>;
    constexpr int W = P::W, N = P::N, STRIPS = N / W;
    extern __shared__ __align__(16) double2 smd[];
    const long b = blockIdx.x / STRIPS;
    const int x0 = (blockIdx.x % STRIPS) * W;
    const int c = threadIdx.x % W, j = threadIdx.x / W;
    double2 *base = work + b * (long)N * N + x0 + c;
    double2 v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = base[(long)(j + r * P::TV) * N];
    fft_vec<LOGN, W, false>(v, smd, c, j, tw);
    if (op != FFT_OP_SPECTRUM) {
        const int xi = x0 + c, k1 = xi < N / 2 ? xi : xi - N;
        const double2 *fb = filt ? filt + xi : nullptr;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            double2 d;
            if (op == FFT_OP_FILTER) {
                d = fb[(long)(j + q * P::TV) * N];
            } else {
                ks_factor(k1, freq_of<LOGN>(j, q), d.x, d.y);
                if (op == FFT_OP_KS_INV) d.y = -d.y;
            }
            v[q] = cmul(v[q], d);
        }
        fft_vec<LOGN, W, true>(v, smd, c, j, tw);
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) base[(long)(j + q * P::TV) * N] = v[q];
}

// real-output column pass: the first half of the CTA transforms the strip's
// Gamma1 columns, the second the Gamma2 columns and hands them over; the first
// half forms kappa_E_hat and runs the inverse (k_cols_ks32_e of fft32.cu)
template <int LOGN>
__global__ void __launch_bounds__(Plan64<LOGN>::NT)
    k_cols64_e(const double2 *__restrict__ work, double2 *__restrict__ half, const double2 *__restrict__ tw)
{
    pdl_wait();
    using P = Plan64<LOGN>;
    constexpr int N = P::N, WS = P::WS, NH = P::NH, STRIPS = N / 2 / WS;
    extern __shared__ __align__(16) double2 smd[];
    double2 *R1 = smd, *R2 = R1 + P::RSZ;
    double2 *U1 = R1, *U2 = WS == 1 ? R2 : R1 + N;  // corner exchange
    const long b = blockIdx.x / STRIPS;
    const int s0 = (blockIdx.x % STRIPS) * WS;
    const int hf = threadIdx.x / NH, t = threadIdx.x % NH, c = t % WS, j = t / WS;
    const double2 *src = work + b * (long)N * N + 2 * (s0 + c) + hf;
    double2 v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = src[(long)(j + r * P::TV) * N];
    fft_vec<LOGN, WS, false>(v, hf ? R2 : R1, c, j, tw);
    __syncthreads();  // the last passes' reads of R1 and R2
    if (hf) {
        if (WS == 1 && s0 == 0) {  // the corner slot: in row order
#pragma unroll
            for (int q = 0; q < 8; ++q) U2[j + q * P::TV] = v[q];
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) R2[q * NH + t] = v[q];  // for the thread t of the first half
        }
    }
    __syncthreads();
    if (hf) return;  // the rest runs on named barrier 1 of the first NH threads
    if (!(s0 == 0 && c == 0)) {
        const int k1 = s0 + c;  // 1 .. n/2 - 1
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            double dr, di;
            ks_factor(k1, freq_of<LOGN>(j, q), dr, di);
            const double2 a = v[q], g = R2[q * NH + t];
            // ky = n/2: conj(D) Gamma1
            v[q] = q == P::E / 2 && j == 0 ? make_double2(dr * a.x + di * a.y, dr * a.y - di * a.x)
                                           : make_double2(dr * a.x + di * g.x, dr * a.y + di * g.y);
        }
    }
    if (s0 == 0) {  // CTA-uniform: slot 0 packs kx = 0 and n/2 and needs ky and -ky together
        if (c == 0) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                U1[j + q * P::TV] = v[q];
                if (WS > 1) U2[j + q * P::TV] = R2[q * NH + t];
            }
        }
        sync_part<NH>();
        if (c == 0) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int yi = j + q * P::TV, yp = (N - yi) & (N - 1);
                const double2 p1 = U1[yi], q1 = U1[yp], p2 = U2[yi], q2 = U2[yp];
                const double2 a1 = make_double2(0.5 * (p1.x + q1.x), 0.5 * (p1.y - q1.y));
                const double2 b1 = make_double2(0.5 * (p1.y + q1.y), -0.5 * (p1.x - q1.x));
                const double2 b2 = make_double2(0.5 * (p2.y + q2.y), -0.5 * (p2.x - q2.x));
                // kx = 0: D = -1 (0 at k = 0); kx = n/2: k1 = -n/2
                const double2 kz = yi == 0 ? make_double2(0.0, 0.0) : make_double2(-a1.x, -a1.y);
                double dr, di;
                ks_factor(-N / 2, freq_of<LOGN>(j, q), dr, di);
                const double2 kh = (yi == 0 || yi == N / 2)
                                       ? make_double2(dr * b1.x + di * b2.x, dr * b1.y + di * b2.y)
                                       : make_double2(dr * b1.x + di * b1.y, dr * b1.y - di * b1.x);
                v[q] = make_double2(kz.x - kh.y, kz.y + kh.x);  // packed kz + i kh
            }
        }
    }
    fft_vec<LOGN, WS, true, NH>(v, R1, c, j, tw);
    double2 *dst = half + b * (long)N * (N / 2) + s0 + c;
#pragma unroll
    for (int q = 0; q < 8; ++q) dst[(long)(j + q * P::TV) * (N / 2)] = v[q];
}

// in place: a row of the half spectrum -> kappa_E's row (k_rows_inv32_c2r)
template <int LOGN>
__global__ void __launch_bounds__(Plan64<LOGN - 1>::ROW_T)
    k_rows_inv64_c2r(double *kap, long total_rows, const double2 *__restrict__ tw, const double2 *__restrict__ tw2,
                     double scale)
{
    pdl_wait();
    using P = Plan64<LOGN - 1>;
    constexpr int N2 = P::N;
    extern __shared__ __align__(16) double2 smd[];
    const int vr = threadIdx.x / P::TV, j = threadIdx.x % P::TV;
    const long row = (long)blockIdx.x * P::RPC + vr;
    const bool live = row < total_rows;
    double2 *h = reinterpret_cast<double2 *>(kap) + row * N2;
    double2 v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int k = j + r * P::TV;
        double2 z = make_double2(0.0, 0.0);
        if (live) {
            const double2 hk = h[k];
            if (k == 0) {
                z = make_double2(hk.x + hk.y, hk.x - hk.y);
            } else {
                const double2 hm = h[N2 - k];
                double2 od = make_double2(hk.x - hm.x, hk.y + hm.y);  // H(k) - conj H(n/2 - k)
                od = mul_tw<true>(od, tw + k);                        // times exp(+2 pi i k / n)
                z = make_double2(hk.x + hm.x - od.y, hk.y - hm.y + od.x);
            }
        }
        v[r] = z;
    }
    fft_vec<LOGN - 1, 1, true>(v, smd + vr * P::VS, 0, j, tw2);
    if (!live) return;
#pragma unroll
    for (int q = 0; q < 8; ++q) h[j + q * P::TV] = make_double2(v[q].x * scale, v[q].y * scale);
}

template <int LOGN>
static int impl64(const double *in1, const double *in2, long in_bs, double *out1, double *out2, double2 *work, int batch,
           int op, const double2 *filt, double out_scale, const uint64_t *seed, int r0, bool rotate, const double2 *tw,
           const double2 *tw2, cudaStream_t s, double im_scale, double im_scale0)
{
    using P = Plan64<LOGN>;
    using P2 = Plan64<LOGN - 1>;
    const long rows = (long)batch * P::N;
    const unsigned row_grid = (unsigned)((rows + P::RPC - 1) / P::RPC);
    const size_t row_smem = (size_t)P::RPC * P::VS * sizeof(double2);
    const double scale = out_scale / ((double)P::N * P::N);
    if (tw2 && (reinterpret_cast<uintptr_t>(out1) & 15) == 0) {  // inverse KS of kappa_E alone
        auto kr = rotate ? k_rows_fwd64<LOGN, true, true> : k_rows_fwd64<LOGN, true, false>;
        auto kc = k_cols64_e<LOGN>;
        auto ki = k_rows_inv64_c2r<LOGN>;
        const size_t col_smem = 2 * (size_t)P::RSZ * sizeof(double2);
        const size_t inv_smem = (size_t)P2::RPC * P2::VS * sizeof(double2);
        FM_CUDA_TRY(fm::smem_attr((const void *)kr, row_smem));
        FM_CUDA_TRY(fm::smem_attr((const void *)kc, col_smem));
        FM_CUDA_TRY(fm::smem_attr((const void *)ki, inv_smem));
        FM_LAUNCH(FM_K_FFT_ROWS_FWD, kr, row_grid, P::ROW_T, row_smem, s, in1, in2, in_bs, work, rows, tw, seed, r0);
        FM_LAUNCH(FM_K_FFT_COLS_KS, kc, (unsigned)((long)batch * (P::N / 2 / P::WS)), P::NT, col_smem, s,
                  (const double2 *)work, reinterpret_cast<double2 *>(out1), tw);
        FM_LAUNCH(FM_K_FFT_ROWS_INV, ki, (unsigned)((rows + P2::RPC - 1) / P2::RPC), P2::ROW_T, inv_smem, s, out1,
                  rows, tw, tw2, 0.5 * scale);
        return FM_OK;
    }
    auto kr = rotate ? k_rows_fwd64<LOGN, false, true> : k_rows_fwd64<LOGN, false, false>;
    auto kc = k_cols64<LOGN>;
    auto ki = out2 ? k_rows_inv64<LOGN, true> : k_rows_inv64<LOGN, false>;
    const size_t col_smem = ((size_t)P::N * P::W + P::N * P::W / P::E + 1) * sizeof(double2);
    FM_CUDA_TRY(fm::smem_attr((const void *)kr, row_smem));
    FM_CUDA_TRY(fm::smem_attr((const void *)kc, col_smem));
    FM_CUDA_TRY(fm::smem_attr((const void *)ki, row_smem));
    FM_LAUNCH(FM_K_FFT_ROWS_FWD, kr, row_grid, P::ROW_T, row_smem, s, in1, in2, in_bs, work, rows, tw, seed, r0);
    FM_LAUNCH(FM_K_FFT_COLS_KS, kc, (unsigned)((long)batch * (P::N / P::W)), P::W * P::TV, col_smem, s, work, tw, op,
              filt);
    if (op == FFT_OP_SPECTRUM) return FM_OK;
    FM_LAUNCH(FM_K_FFT_ROWS_INV, ki, row_grid, P::ROW_T, row_smem, s, (const double2 *)work, out1, out2, rows, tw,
              scale, scale * im_scale, scale * im_scale0);
    return FM_OK;
}

int launch_fft64(const double *in1, const double *in2, long in_bs, double *out1, double *out2, double2 *work, int n,
                 int batch, int op, const double2 *filt, double out_scale, const uint64_t *seed, int r0, bool rotate,
                 const double2 *tw, const double2 *tw2, cudaStream_t s, double im_scale, double im_scale0)
{
#define FM_FFT64(L) impl64<L>(in1, in2, in_bs, out1, out2, work, batch, op, filt, out_scale, seed, r0, rotate, tw, tw2, s, im_scale, im_scale0)
    switch (n) {
    case 64: return FM_FFT64(6);
    case 128: return FM_FFT64(7);
    case 256: return FM_FFT64(8);
    case 512: return FM_FFT64(9);
    case 1024: return FM_FFT64(10);
    case 2048: return FM_FFT64(11);
    }
#undef FM_FFT64
    return FM_EINVAL;
}

}  // namespace fm

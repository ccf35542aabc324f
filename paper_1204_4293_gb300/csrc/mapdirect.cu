// mapdirect.cu -- brute-force aperture mass from tangential shear,
// eq. shearmap (Sec. 2.1) evaluated as in Sec. 5.1: the comparison path whose
// O(n^2 R^2) cost the starlet removes.
//
// M(x) = sum_{0 < |d| <= R} Q(|d|) gamma_t(x + d; x),
// gamma_t = -(gamma1 cos 2 phi_d + gamma2 sin 2 phi_d), so with per-offset
// weights A(d) = -Q cos 2 phi = -Q (dx^2 - dy^2) / |d|^2 and
// B(d) = -Q sin 2 phi = -Q 2 dx dy / |d|^2 (FP64, rounded once) the map is the
// 2-D correlation M = A * gamma1 + B * gamma2, zero outside the field.
//
// A(dx, -dy) = A(dx, dy) and B(dx, -dy) = -B(dx, dy), so the rows y + dy and
// y - dy enter together: with s = gamma1(y + dy) + gamma1(y - dy) and
// d = gamma2(y + dy) - gamma2(y - dy),
//   M(x, y) = sum_{dy >= 0} sum_dx A(dx, dy) s(x + dx) + B(dx, dy) d(x + dx),
// half the multiplications of the plain sum (a pair's sum has to stay in the
// type's range: pixels below half its largest value).
//
// Kernel layout: one warp owns one output row of 32 CX columns (CX adjacent
// ones a lane) and shares nothing with the others.  For each dy it forms the
// folded row (s, d) in its own piece of shared memory, as blocks of CX
// columns padded by 16 bytes (the lanes' 16-byte loads of CX neighbouring
// blocks then hit distinct banks), and walks dx in groups of CX taps: a lane
// keeps two blocks in registers, loads one more per group and spends CX^2
// packed two-lane FMAs (fma.rn.f32x2: A s and B d in one instruction) on it.
// The groups at the rim of the disc skip the taps outside it, so a pixel
// beyond the radius never meets a weight.  Sums are two-level (a dy's taps,
// then the total).  With few rows the dy are dealt out to P warps (dy = p,
// p + P, ...: equal shares) whose sums k_direct_sum adds in order.
//
// What bounds it: the FP32 pipe and the shared-memory loads together (1024^2,
// R = 32: 52.7 M warp FMAs of two lanes, 84 us at two a cycle and SM; ncu: FMA
// pipe 58 %, shared-memory and L1 data path 77 %, 19 warps an SM).  One 1024^2
// map, starlet Q theta = 16 (R = 32): 372 -> 199 us; S98 theta = 64 1246 ->
// 618, masked 3050 -> 825; masked 2 x 1000^2 S98 theta = 16 445 -> 236; fp64
// 512^2 S98 theta = 16 3079 -> 472 (the plain sum over all rows, with a CTA's
// warps sharing each staged row behind a barrier).  16 columns a lane halve
// the window loads but need 116 to 142 registers: 225 us; groups of four taps
// instead of eight 260 us.
//
// Missing data (Sec. 4.3, Sec. 4.5): with pixel weights w >= 0 (0 = masked)
// the folded row is that of w gamma, and the same pass forms D(x) = sum
// w(x+d) over the in-field offsets 0 < |d| <= R.  D needs no multiplication:
// a lane's CX windows of one dy share all but CX - 1 columns at each end, so
// it adds the common part once (whole blocks from their sums) and the ends as
// running sums; additions of weights only, no differences.  The result is
// M = N_R S / D (0 where D <= 0), optionally coverage = D / N_R, N_R the
// aperture's pixel count.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace fm {

// ---- filters (Sec. 4), FP64 ----------------------------------------------------
__device__ static double cube(double v) { return v * v * v; }

// starlet Q(eta) printed in Sec. 4.2; the direct sum never evaluates eta = 0.
__device__ static double q_starlet(double e)
{
    const double e2 = e * e;
    double s = -279.0 * e2 * cube(fabs(e));
    s += 8.0 * (1.0 + 6.0 * e + 24.0 * e2) * cube(fabs(0.5 - e));
    s += 8.0 * (1.0 - 6.0 * e + 24.0 * e2) * cube(fabs(0.5 + e));
    s -= 9.0 * (1.0 + 3.0 * e + 6.0 * e2) * cube(fabs(1.0 - e));
    s -= 9.0 * (1.0 - 3.0 * e + 6.0 * e2) * cube(fabs(1.0 + e));
    s += (1.0 + 1.5 * e + 1.5 * e2) * cube(fabs(2.0 - e));
    s += (1.0 - 1.5 * e + 1.5 * e2) * cube(fabs(2.0 + e));
    return s / (45.0 * e2);
}

__device__ static double q_of(int filter, double v, double theta, int ell)
{
    const double t2 = theta * theta;
    switch (filter) {
    case FM_FILTER_STARLET: return q_starlet(v / theta) / t2;  // U, Q scale as 1/theta^2
    case FM_FILTER_S98: {  // eq. sch
        if (v > theta) return 0.0;
        const double x2 = v * v / t2;
        double pw = 1.0, base = 1.0 - x2;
        for (int k = ell; k > 0; k >>= 1, base *= base)
            if (k & 1) pw *= base;
        return (1.0 + ell) * (2.0 + ell) / (M_PI * t2) * x2 * pw;
    }
    case FM_FILTER_JBJ04:
    case FM_FILTER_VW98: {  // eq. mexhat with A = 1
        const double b = filter == FM_FILTER_JBJ04 ? 0.5 : 4.0;
        const double x = b * v * v / t2;
        return x * exp(-x) / t2;
    }
    }
    return 0.0;
}

static double default_cut(int filter) { return filter == FM_FILTER_STARLET ? 2.0 : filter == FM_FILTER_S98 ? 1.0 : 5.0; }

// largest dx with dx^2 + dy^2 <= R^2 (dy <= R)
__host__ __device__ static int disc_half_width(int dy, double R2)
{
    int dx = (int)sqrt(R2 - (double)dy * dy > 0 ? R2 - (double)dy * dy : 0.0);
    while (((double)(dx + 1) * (dx + 1)) + (double)dy * dy <= R2) ++dx;
    while (dx > 0 && (double)dx * dx + (double)dy * dy > R2) --dx;
    return dx;
}

// columns a lane owns, and the folded row's layout in shared memory
template <typename T> struct DirectRow {
    using V = cplx_t<T>;
    static constexpr int CX = sizeof(T) == 4 ? 8 : 4;
    static constexpr int TX = 32 * CX;
    static constexpr int BS = CX + 16 / (int)sizeof(V);  // elements of a padded block: 80 bytes
    // radius rounded up to whole blocks, blocks of a row, taps of a table row
    static int rp(int Ri) { return (Ri + CX - 1) / CX * CX; }
    static int blocks(int Ri) { return 32 + 2 * rp(Ri) / CX + 1; }
    static int tap_width(int Ri) { return 2 * rp(Ri) + CX; }
    // shared memory of a warp: (s, d); weights: w folded (blocks of CX + 1) and its block sums
    static size_t bytes(int Ri, bool mask)
    {
        const size_t nb = blocks(Ri);
        const size_t b = nb * BS * sizeof(V) + (mask ? nb * (CX + 2) * sizeof(T) : 0);
        return (b + 15) / 16 * 16;
    }
};

// Weights (A, B) of the rows dy = 0 .. Ri (the others follow by symmetry),
// dx = -rp .. rp + CX - 1, zero outside 0 < |d| <= R; and each row's half width.
// On the device: no copy from host memory, so a call can be captured, and the
// host's share of a call no longer grows with R^2 (0.1 ms at R = 32).
template <typename T>
__global__ void __launch_bounds__(64) k_direct_taps(cplx_t<T> *__restrict__ taps, int *__restrict__ dxmax, int Ri,
                                                    int rp, int tw, double R2, int filter, double theta, int ell)
{
    pdl_entry();
    const int dy = blockIdx.y, dx = blockIdx.x * blockDim.x + threadIdx.x;
    cplx_t<T> *row = taps + (long)dy * tw + rp;
    if (dx == 0) dxmax[dy] = disc_half_width(dy, R2);
    if (dx >= tw - rp) return;
    const double r2 = (double)dx * dx + (double)dy * dy;
    double a = 0, b = 0;
    if (r2 > 0 && r2 <= R2) {
        const double q = q_of(filter, sqrt(r2), theta, ell);
        a = -q * ((double)dx * dx - (double)dy * dy) / r2;
        b = -q * 2.0 * dx * dy / r2;
    }
    row[dx] = cmake<cplx_t<T>>((T)a, (T)b);
    if (dx > 0 && dx <= rp) row[-dx] = cmake<cplx_t<T>>((T)a, (T)-b);
}

__device__ __forceinline__ void tap_fma(float2 &acc, float2 ab, float2 w) { acc = __ffma2_rn(ab, w, acc); }
__device__ __forceinline__ void tap_fma(double2 &acc, double2 ab, double2 w)
{
    acc.x = fma(ab.x, w.x, acc.x);
    acc.y = fma(ab.y, w.y, acc.y);
}
// a block of CX columns of the folded row (16-byte loads)
template <typename V, int CX> __device__ __forceinline__ void load_block(V (&w)[CX], const V *p)
{
#pragma unroll
    for (int k = 0; k < CX; k += 16 / (int)sizeof(V)) {
        if constexpr (sizeof(V) == 8) {
            const float4 q = *reinterpret_cast<const float4 *>(p + k);
            w[k] = make_float2(q.x, q.y);
            w[k + 1] = make_float2(q.z, q.w);
        } else {
            w[k] = p[k];
        }
    }
}

// CX taps of a table row (16-byte aligned: rows hold 2 rp + CX taps)
template <typename V, int CX> __device__ __forceinline__ void load_taps(V (&ab)[CX], const V *p)
{
    if constexpr (sizeof(V) == 8) {
#pragma unroll
        for (int k = 0; k < CX; k += 2) {
            const float4 q = __ldg(reinterpret_cast<const float4 *>(p + k));
            ab[k] = make_float2(q.x, q.y);
            ab[k + 1] = make_float2(q.z, q.w);
        }
    } else {
#pragma unroll
        for (int k = 0; k < CX; ++k) ab[k] = __ldg(p + k);
    }
}

// grid = (ceil(n / warps), ceil(n / TX), maps * P), one output row a warp.
// P = 1: writes out (and cov); P > 1: the part's sums to parts[p][map] and,
// MASK, partw[p][map].
template <typename T, bool MASK>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 5 : 3)
    k_map_direct(const T *__restrict__ g1, const T *__restrict__ g2, const T *__restrict__ wgt, long w_bs,
                 const cplx_t<T> *__restrict__ taps, const int *__restrict__ dxmax, T *__restrict__ out,
                 T *__restrict__ cov, T *__restrict__ parts, T *__restrict__ partw, int n, int Ri, int rp, int nblocks,
                 int warp_bytes, int P, int maps, T n_r)
{
    pdl_entry();
    using V = cplx_t<T>;
    using D = DirectRow<T>;
    constexpr int CX = D::CX, BS = D::BS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int y = blockIdx.x * (blockDim.x >> 5) + warp;
    if (y >= n) return;  // warps share nothing
    V *buf = reinterpret_cast<V *>(smem_raw + (size_t)warp * warp_bytes);
    T *sw = reinterpret_cast<T *>(buf + nblocks * BS);  // folded weights, CX + 1 a block
    T *sb = sw + nblocks * (CX + 1);                    // their block sums
    const int x0 = blockIdx.y * D::TX;
    const long nn = (long)n * n, b = blockIdx.z / P;
    const int p = blockIdx.z % P;
    g1 += b * nn;
    g2 += b * nn;
    if (MASK) wgt += b * w_bs;
    const int tw = 2 * rp + CX;

    T acc[CX], accw[MASK ? CX : 1];
#pragma unroll
    for (int o = 0; o < CX; ++o) {
        acc[o] = (T)0;
        if (MASK) accw[o] = (T)0;
    }
    for (int dy = p; dy <= Ri; dy += P) {
        const bool up = y + dy < n, dn = dy > 0 && y - dy >= 0;
        if (!up && !dn) break;  // larger dy leave the field too
        const int dxm = __ldg(dxmax + dy);
        const int glo = (rp - dxm) / CX, ghi = (rp + dxm) / CX;  // groups of taps that meet the disc
        // the folded row, columns of the blocks glo .. 32 + ghi: rows and
        // addresses are fixed before the loop, whose body is loads, the fold
        // and stores at compile-time offsets
        const int c0 = glo * CX + lane, c_end = (33 + ghi) * CX;
        const int gx0 = x0 - rp + c0;
        __syncwarp();  // the last dy's reads
        auto fold = [&](auto up_, auto dn_, auto edge_) {
            constexpr bool UP = decltype(up_)::value, DN = decltype(dn_)::value, EDGE = decltype(edge_)::value;
            const long iu = (long)(y + dy) * n + gx0, id = (long)(y - dy) * n + gx0;
            const T *u1 = g1 + iu, *u2 = g2 + iu, *d1 = g1 + id, *d2 = g2 + id;
            [[maybe_unused]] const T *uw = MASK ? wgt + iu : nullptr, *dw = MASK ? wgt + id : nullptr;
            V *dst = buf + c0 / CX * BS + c0 % CX;
            [[maybe_unused]] T *dsw = sw + c0 / CX * (CX + 1) + c0 % CX, *dsb = sb + c0 / CX;
            int gx = gx0, left = c_end - c0;
#pragma unroll 4
            for (int t = (c_end - glo * CX + 31) / 32; t > 0; --t) {
                T a = (T)0, d = (T)0;
                [[maybe_unused]] T w = (T)0;
                if (!EDGE || (unsigned)gx < (unsigned)n) {
                    if constexpr (UP) {
                        a = __ldg(u1);
                        d = __ldg(u2);
                        if constexpr (MASK) {
                            w = __ldg(uw);
                            a *= w;
                            d *= w;
                        }
                    }
                    if constexpr (DN) {
                        T a2 = __ldg(d1), e2 = __ldg(d2);
                        if constexpr (MASK) {
                            const T w2 = __ldg(dw);
                            a2 *= w2;
                            e2 *= w2;
                            w += w2;
                        }
                        a += a2;
                        d -= e2;
                    }
                }
                if (left > 0) *dst = cmake<V>(a, d);
                if constexpr (MASK) {
                    if (left > 0) *dsw = w;
#pragma unroll
                    for (int o = 1; o < CX; o *= 2) w += __shfl_xor_sync(0xffffffffu, w, o);
                    if (lane % CX == 0 && left > 0) *dsb = w;
                    uw += 32;
                    dw += 32;
                    dsw += 32 / CX * (CX + 1);
                    dsb += 32 / CX;
                }
                u1 += 32;
                u2 += 32;
                d1 += 32;
                d2 += 32;
                dst += 32 / CX * BS;
                gx += 32;
                left -= 32;
            }
        };
        // columns past c_end (the last 32 of a row may overhang it) are loaded
        // but not stored: they count for the field's edge as well
        const int cl = (c_end - glo * CX + 31) / 32 * 32;
        const bool edge = x0 - rp + glo * CX < 0 || x0 - rp + glo * CX + cl > n;
        using Yes = std::true_type;
        using No = std::false_type;
        if (up && dn) {
            if (edge)
                fold(Yes(), Yes(), Yes());
            else
                fold(Yes(), Yes(), No());
        } else if (up) {
            fold(Yes(), No(), Yes());
        } else {
            fold(No(), Yes(), Yes());
        }
        __syncwarp();
        V part[CX];
#pragma unroll
        for (int o = 0; o < CX; ++o) part[o] = cmake<V>((T)0, (T)0);
        const V *trow = taps + (long)dy * tw, *src = buf + lane * BS;
        // taps g CX .. g CX + CX - 1 over the columns in a (block lane + g) and b (the next):
        // all of them, or at the rim those of the disc
        auto full = [&](int g, const V (&a)[CX], const V (&b)[CX]) {
            V ab[CX];
            load_taps<V, CX>(ab, trow + g * CX);
#pragma unroll
            for (int k = 0; k < CX; ++k)
#pragma unroll
                for (int o = 0; o < CX; ++o) tap_fma(part[o], ab[k], o + k < CX ? a[o + k] : b[o + k - CX]);
        };
        auto rim = [&](int g, const V (&a)[CX], const V (&b)[CX]) {
            const int lo = rp - dxm - g * CX, hi = rp + dxm - g * CX;
            V ab[CX];
            load_taps<V, CX>(ab, trow + g * CX);
#pragma unroll
            for (int k = 0; k < CX; ++k)
                if (k >= lo && k <= hi) {
#pragma unroll
                    for (int o = 0; o < CX; ++o) tap_fma(part[o], ab[k], o + k < CX ? a[o + k] : b[o + k - CX]);
                }
        };
        V wa[CX], wb[CX];
        load_block<V, CX>(wa, src + glo * BS);
        load_block<V, CX>(wb, src + (glo + 1) * BS);
        rim(glo, wa, wb);
        int g = glo + 1;  // wb holds block lane + g
        for (; g + 1 < ghi; g += 2) {
            load_block<V, CX>(wa, src + (g + 1) * BS);
            full(g, wb, wa);
            load_block<V, CX>(wb, src + (g + 2) * BS);
            full(g + 1, wa, wb);
        }
        if (g < ghi) {
            load_block<V, CX>(wa, src + (g + 1) * BS);
            full(g, wb, wa);
#pragma unroll
            for (int k = 0; k < CX; ++k) wb[k] = wa[k];
        }
        if (ghi > glo) {
            load_block<V, CX>(wa, src + (ghi + 1) * BS);
            rim(ghi, wb, wa);
        }
#pragma unroll
        for (int o = 0; o < CX; ++o) acc[o] += part[o].x + part[o].y;
        if constexpr (MASK) {
            // this dy's weights within |dx| <= dxm of each of the lane's columns
            // (dx = 0 left out at dy = 0); column c from the lane's first one
            const T *ws = sw + lane * (CX + 1);
            auto at = [&](int c) { return ws[rp + c + (rp + c) / CX]; };
            if (dxm < CX - 1) {
#pragma unroll
                for (int o = 0; o < CX; ++o) {
                    T t = (T)0;
                    for (int dx = -dxm; dx <= dxm; ++dx)
                        if (dx != 0 || dy != 0) t += at(o + dx);
                    accw[o] += t;
                }
            } else {
                // columns lo .. hi, whole blocks by their sums
                auto span = [&](int lo, int hi) {
                    T t = (T)0;
                    int u = rp + lo;
                    const int e = rp + hi + 1;  // blocks count from -rp
                    for (; u < e && u % CX != 0; ++u) t += ws[u + u / CX];
                    for (; u + CX <= e; u += CX) t += sb[lane + u / CX];
                    for (; u < e; ++u) t += ws[u + u / CX];
                    return t;
                };
                T mid[CX];
                if (dy == 0) {
                    const T common = span(CX - 1 - dxm, -1) + span(CX, dxm);
                    T run = (T)0;
#pragma unroll
                    for (int o = 0; o < CX; ++o) {  // own column left out: those before it, then those after it
                        mid[o] = common + run;
                        run += at(o);
                    }
                    run = (T)0;
#pragma unroll
                    for (int o = CX - 1; o >= 0; --o) {
                        mid[o] += run;
                        run += at(o);
                    }
                } else {
                    const T common = span(CX - 1 - dxm, dxm);
#pragma unroll
                    for (int o = 0; o < CX; ++o) mid[o] = common;
                }
                T left = (T)0, right = (T)0;
#pragma unroll
                for (int o = CX - 2; o >= 0; --o) {
                    left += at(o - dxm);
                    mid[o] += left;
                }
#pragma unroll
                for (int o = 1; o < CX; ++o) {
                    right += at(o + dxm);
                    mid[o] += right;
                }
#pragma unroll
                for (int o = 0; o < CX; ++o) accw[o] += mid[o];
            }
        }
    }
    const long row = (P > 1 ? (long)p * maps + b : b) * nn + (long)y * n;
#pragma unroll
    for (int o = 0; o < CX; ++o) {
        const int x = x0 + lane * CX + o;
        if (x >= n) continue;
        if (P > 1) {
            parts[row + x] = acc[o];
            if (MASK) partw[row + x] = accw[o];
        } else if constexpr (MASK) {
            const T d = accw[o];
            out[row + x] = d > (T)0 ? n_r * acc[o] / d : (T)0;
            if (cov) cov[row + x] = d / n_r;
        } else {
            out[row + x] = acc[o];
        }
    }
}

// the parts' sums in order, p = 0 .. P - 1, over `total` pixels
template <typename T, bool MASK>
__global__ void __launch_bounds__(256) k_direct_sum(const T *__restrict__ parts, const T *__restrict__ partw,
                                                    T *__restrict__ out, T *__restrict__ cov, long total, int P,
                                                    T n_r)
{
    pdl_entry();
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
        T a = (T)0, d = (T)0;
        for (int q = 0; q < P; ++q) {
            a += parts[(long)q * total + i];
            if (MASK) d += partw[(long)q * total + i];
        }
        if (MASK) {
            out[i] = d > (T)0 ? n_r * a / d : (T)0;
            if (cov) cov[i] = d / n_r;
        } else {
            out[i] = a;
        }
    }
}

// Parts of the dy: a function of n and the radius only, so that a map's
// result does not depend on the maps beside it.  Eight full loads of the GPU
// (152 SMs x 20 warps), so that the last warps to finish are short ones (one
// 1024^2 map, S98 theta = 64, two / four / eight loads 658 / 644 / 618 us), with
// at least four dy a part, eight with weights (2 x 1000^2 theta = 16 with four
// 235 -> 249 us), at most 16.
static int direct_parts(int n, int Ri, int TX, bool mask)
{
    const long warps = (long)n * ((n + TX - 1) / TX);
    long P = (8 * 152 * 20 + warps - 1) / warps;
    P = std::min<long>({P, 16, (Ri + 1) / (mask ? 8 : 4)});
    return P < 1 ? 1 : (int)P;
}
// maps per launch pair when the parts go through scratch: at most 256 MiB of
// partial sums (the order of the sums is per map, so the slicing of a batch
// does not change any result)
static int direct_slice(int P, int n, int batch, size_t es)
{
    // the grid's third dimension holds maps x parts
    const int most = std::min(batch, 65535 / P);
    if (P <= 1) return most;
    const long m = (256L << 20) / ((long)P * n * n * (long)es);
    return (int)std::max<long>(1, std::min<long>(m, most));
}

template <typename T, bool MASK>
static int map_direct_impl(const T *g1, const T *g2, const T *wgt, long w_bs, T *map, T *cov, int n, int batch,
                           int filter, double theta, int ell, double cut, cudaStream_t s)
{
    using V = cplx_t<T>;
    using D = DirectRow<T>;
    const double R = (cut > 0 ? cut : default_cut(filter)) * theta, R2 = R * R;
    const int Ri = (int)floor(R), rp = D::rp(Ri), tw = D::tap_width(Ri);
    long n_r = 0;  // lattice offsets 0 < |d| <= R
    if (MASK) {
        for (int dy = 0; dy <= Ri; ++dy) n_r += (dy ? 2 : 1) * (2L * disc_half_width(dy, R2) + 1);
        n_r -= 1;
    }
    const int P = direct_parts(n, Ri, D::TX, MASK), slice = direct_slice(P, n, batch, sizeof(T));
    auto up = [](size_t b) { return ((b + 255) / 256) * 256; };
    const size_t tap_b = up((size_t)(Ri + 1) * tw * sizeof(V)), dx_b = up((size_t)(Ri + 1) * sizeof(int));
    const long nn = (long)n * n;
    const size_t part_b = P > 1 ? up((size_t)P * slice * nn * sizeof(T)) : 0;
    Scratch sc;
    int st = scratch_alloc(sc, tap_b + dx_b + (MASK ? 2 : 1) * part_b, s);
    if (st != FM_OK) return st;
    char *base = static_cast<char *>(sc.p);
    V *taps = reinterpret_cast<V *>(base);
    int *dxmax = reinterpret_cast<int *>(base + tap_b);
    T *parts = reinterpret_cast<T *>(base + tap_b + dx_b);
    T *partw = reinterpret_cast<T *>(base + tap_b + dx_b + part_b);
    FM_LAUNCH(FM_K_MAP_DIRECT, k_direct_taps<T>, dim3((unsigned)((tw - rp + 63) / 64), (unsigned)(Ri + 1)), 64, 0, s,
              taps, dxmax, Ri, rp, tw, R2, filter, theta, ell);
    // four warps a CTA, fewer where their rows would leave the SM with few CTAs
    const size_t wb = D::bytes(Ri, MASK);
    const int nw = 4 * wb <= 56 * 1024 ? 4 : 2 * wb <= 110 * 1024 ? 2 : 1;
    auto k = k_map_direct<T, MASK>;
    FM_CUDA_TRY(fm::smem_attr((const void *)k, nw * wb));
    for (int b0 = 0; b0 < batch; b0 += slice) {
        const int bs = batch - b0 < slice ? batch - b0 : slice;
        const dim3 grid((n + nw - 1) / nw, (n + D::TX - 1) / D::TX, bs * P);
        T *o = map + b0 * nn, *oc = cov ? cov + b0 * nn : nullptr;
        FM_LAUNCH(FM_K_MAP_DIRECT, k, grid, nw * 32, nw * wb, s, g1 + b0 * nn, g2 + b0 * nn,
                  MASK ? wgt + b0 * w_bs : nullptr, w_bs, (const V *)taps, (const int *)dxmax, o, oc, parts, partw, n,
                  Ri, rp, D::blocks(Ri), (int)wb, P, bs, (T)n_r);
        if (P > 1) {
            const long total = (long)bs * nn;
            const unsigned g = (unsigned)std::min<long>((total + 255) / 256, 152L * 32);
            FM_LAUNCH(FM_K_MAP_DIRECT, (k_direct_sum<T, MASK>), g, 256, 0, s, (const T *)parts, (const T *)partw, o, oc,
                      total, P, (T)n_r);
        }
    }
    return FM_OK;
}

template <typename T>
static int map_direct_typed(const void *g1, const void *g2, const void *weight, long w_bs, void *map, void *coverage,
                            int n, int batch, int filter, double theta, int ell, double cut, cudaStream_t s)
{
    const T *a = static_cast<const T *>(g1), *b = static_cast<const T *>(g2), *w = static_cast<const T *>(weight);
    T *m = static_cast<T *>(map), *c = static_cast<T *>(coverage);
    return w ? map_direct_impl<T, true>(a, b, w, w_bs, m, c, n, batch, filter, theta, ell, cut, s)
             : map_direct_impl<T, false>(a, b, w, w_bs, m, c, n, batch, filter, theta, ell, cut, s);
}

int launch_map_direct(const void *g1, const void *g2, const void *weight, long w_bs, void *map, void *coverage, int n,
                      int batch, int filter, double theta, int ell, double cut, int precision, cudaStream_t s)
{
    return precision == FM_F64 ? map_direct_typed<double>(g1, g2, weight, w_bs, map, coverage, n, batch, filter, theta,
                                                          ell, cut, s)
                               : map_direct_typed<float>(g1, g2, weight, w_bs, map, coverage, n, batch, filter, theta,
                                                         ell, cut, s);
}

}  // namespace fm

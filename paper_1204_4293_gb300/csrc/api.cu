// api.cu -- the compute entry points of libfastmap's C ABI (declared in
// include/fastmap.h): argument validation, scratch sizing and dispatch to
// the kernels and to the batched pipeline.
#include <math.h>
#include <string.h>

#include <string>

#include "common.cuh"

namespace fm {

static fm_config cfg_or_default(const fm_config *c)
{
    fm_config d;
    memset(&d, 0, sizeof(d));
    if (c) d = *c;
    return d;
}

int check_config(const fm_config &c)
{
    if (c.precision != FM_F32 && c.precision != FM_F64) return einval("precision must be FM_F32 or FM_F64");
    if (c.boundary != FM_MIRROR && c.boundary != FM_PERIODIC) return einval("boundary must be FM_MIRROR or FM_PERIODIC");
    if (c.accum != 0 && c.accum != 1) return einval("accum must be 0 (FP64 sums) or 1 (Kahan fp32 sums)");
    if (c.accum == 1 && c.precision != FM_F32) return einval("accum = 1 (Kahan fp32 sums) needs FM_F32 maps");
    if (c.fuse_depth < -1 || c.fuse_depth > 8) return einval("fuse_depth out of range [-1, 8]");
    if (c.large_path < 0 || c.large_path > 4) return einval("large_path must be 0, 1, 2, 3 or 4");
    return FM_OK;
}

static size_t esize(const fm_config &c) { return c.precision == FM_F64 ? 8 : 4; }

static int check_fft_n(int n)
{
    if (n < 4 || n > 8192 || !is_pow2(n)) return einval("n must be a power of two in [4, 8192]");
    return FM_OK;
}

static int check_J(int n, int J)
{
    if (J < 2 || J > 20) return einval("J must be in [2, 20]");
    if ((long)n < (1L << J)) return einval("n must be >= 2^J (N >= 2^J)");
    return FM_OK;
}


size_t map_starlet_scratch_bytes(int n, int J, int batch, const fm_config &cfg)
{
    // the FFT work buffer (2 n^2 a map) and kappa (n^2); the starlet's
    // scratch maps live in the work buffer when they fit there (the chunk
    // plan's rule), else in their own buffer
    const size_t es = esize(cfg), nn = (size_t)n * n;
    const size_t st = starlet_scratch_elems(n, J, 1, cfg) <= 2 * nn ? 0 : starlet_scratch_elems(n, J, batch, cfg) * es;
    return (size_t)batch * nn * 3 * es + st + 3 * 256;
}

}  // namespace fm

using namespace fm;

extern "C" {

int fm_ks_invert(const void *g1, const void *g2, void *kappa_E, void *kappa_B, int n, int batch, const fm_config *cfgp,
                 void *stream)
{
    fm_config cfg = cfg_or_default(cfgp);
    int st = check_config(cfg);
    if (st) return st;
    if ((st = check_fft_n(n))) return st;
    if (batch < 1) return einval("batch must be >= 1");
    if (!g1 || !g2 || !kappa_E) return einval("null pointer");
    cudaStream_t s = (cudaStream_t)stream;
    // kappa laid over the shear of other maps (not in place): the separate kernels read all of it first
    const size_t map_b = (size_t)batch * n * n * esize(cfg);
    auto apart = [&](const void *out, const void *in) { return out == in || !overlap(out, map_b, in, map_b); };
    const bool one = batch == 1 || (apart(kappa_E, g1) && apart(kappa_E, g2) && apart(kappa_B, g1) && apart(kappa_B, g2));
    if (one && small_map_ok(n, 0, batch, cfg, true))
        return launch_small_ks((const float *)g1, (const float *)g2, (float *)kappa_E, (float *)kappa_B, n, batch, s);
    Scratch work;
    const size_t bytes = (size_t)batch * n * n * 2 * esize(cfg);
    if ((st = scratch_alloc(work, bytes, s))) return st;
    return launch_ks(g1, g2, (long)n * n, kappa_E, kappa_B, work.p, n, batch, cfg.precision, false, 0, 0, false, s);
}

int fm_ks_forward(const void *kappa, void *g1, void *g2, int n, int batch, const fm_config *cfgp, void *stream)
{
    fm_config cfg = cfg_or_default(cfgp);
    int st = check_config(cfg);
    if (st) return st;
    if ((st = check_fft_n(n))) return st;
    if (batch < 1) return einval("batch must be >= 1");
    if (!kappa || !g1 || !g2) return einval("null pointer");
    cudaStream_t s = (cudaStream_t)stream;
    Scratch work;
    if ((st = scratch_alloc(work, (size_t)batch * n * n * 2 * esize(cfg), s))) return st;
    return launch_ks(kappa, nullptr, (long)n * n, g1, g2, work.p, n, batch, cfg.precision, true, 0, 0, false, s);
}

int fm_starlet_forward(const void *kappa, void *pyramid, int n, int J, int batch, const fm_config *cfgp, void *stream)
{
    fm_config cfg = cfg_or_default(cfgp);
    int st = check_config(cfg);
    if (st) return st;
    if (n < 1) return einval("n must be >= 1");
    if ((st = check_J(n, J))) return st;
    if (batch < 1) return einval("batch must be >= 1");
    if (!kappa || !pyramid) return einval("null pointer");
    cudaStream_t s = (cudaStream_t)stream;
    if (small_map_ok(n, J, batch, cfg, (reinterpret_cast<uintptr_t>(pyramid) & 15) == 0))
        return launch_small_starlet((const float *)kappa, (float *)pyramid, n, J, batch, cfg.boundary, s);
    Scratch sc;
    if ((st = scratch_alloc(sc, starlet_scratch_elems(n, J, batch, cfg) * esize(cfg), s))) return st;
    return launch_starlet(kappa, pyramid, (long)J * n * n, n, J, batch, cfg, sc.p, s);
}

int fm_starlet_fuse_depth(int n, int J, const fm_config *cfgp)
{
    fm_config cfg = cfg_or_default(cfgp);
    int st = check_config(cfg);
    if (st) return st;
    if (n < 1) return einval("n must be >= 1");
    if ((st = check_J(n, J))) return st;
    return starlet_fuse_depth(n, J, cfg);
}

int fm_map_starlet(const void *g1, const void *g2, void *pyramid, int n, int J, int batch, const fm_config *cfgp,
                   void *stream)
{
    fm_config cfg = cfg_or_default(cfgp);
    int st = check_config(cfg);
    if (st) return st;
    if ((st = check_fft_n(n))) return st;
    if ((st = check_J(n, J))) return st;
    if (batch < 1) return einval("batch must be >= 1");
    if (!g1 || !g2 || !pyramid) return einval("null pointer");
    return map_starlet_run(g1, g2, pyramid, n, J, batch, cfg, (cudaStream_t)stream);
}

int fm_map_starlet_host(const void *g1_host, const void *g2_host, void *pyramid_host, int n, int J, int batch,
                        const fm_config *cfgp, void *stream)
{
    fm_config cfg = cfg_or_default(cfgp);
    int st = check_config(cfg);
    if (st) return st;
    if ((st = check_fft_n(n))) return st;
    if ((st = check_J(n, J))) return st;
    if (batch < 1) return einval("batch must be >= 1");
    if (!g1_host || !g2_host || !pyramid_host) return einval("null pointer");
    return map_starlet_host_run(static_cast<const char *>(g1_host), static_cast<const char *>(g2_host),
                                static_cast<char *>(pyramid_host), n, J, batch, cfg, (cudaStream_t)stream);
}

int fm_map_direct(const void *g1, const void *g2, void *map, int n, int filter, double theta_px, int ell,
                  double cut_over_theta, const fm_config *cfgp, void *stream)
{
    fm_config cfg = cfg_or_default(cfgp);
    int st = check_config(cfg);
    if (st) return st;
    if (n < 1 || n > 65536) return einval("n must be in [1, 65536]");
    if (filter < FM_FILTER_STARLET || filter > FM_FILTER_VW98) return einval("unknown filter");
    if (!(theta_px > 0) || theta_px > 4096) return einval("theta_px must be in (0, 4096]");
    if (filter == FM_FILTER_S98 && (ell < 0 || ell > 64)) return einval("ell must be in [0, 64]");
    const double cut = cut_over_theta > 0 ? cut_over_theta : 0.0;
    const double R = (cut > 0 ? cut : (filter == FM_FILTER_STARLET ? 2.0 : filter == FM_FILTER_S98 ? 1.0 : 5.0)) *
                     theta_px;
    if (R > 2048) return einval("cut radius above 2048 px");
    if (!g1 || !g2 || !map) return einval("null pointer");
    return launch_map_direct(g1, g2, nullptr, 0, map, nullptr, n, 1, filter, theta_px, ell, cut, cfg.precision,
                             (cudaStream_t)stream);
}

int fm_map_direct_batch(const void *g1, const void *g2, void *map, int n, int batch, int filter, double theta_px,
                        int ell, double cut_over_theta, const fm_config *cfgp, void *stream)
{
    fm_config cfg = cfg_or_default(cfgp);
    int st = check_config(cfg);
    if (st) return st;
    if (n < 1 || n > 65536) return einval("n must be in [1, 65536]");
    if (batch < 1 || batch > 65535) return einval("batch must be in [1, 65535]");
    if (filter < FM_FILTER_STARLET || filter > FM_FILTER_VW98) return einval("unknown filter");
    if (!(theta_px > 0) || theta_px > 4096) return einval("theta_px must be in (0, 4096]");
    if (filter == FM_FILTER_S98 && (ell < 0 || ell > 64)) return einval("ell must be in [0, 64]");
    const double cut = cut_over_theta > 0 ? cut_over_theta : 0.0;
    const double R = (cut > 0 ? cut : (filter == FM_FILTER_STARLET ? 2.0 : filter == FM_FILTER_S98 ? 1.0 : 5.0)) *
                     theta_px;
    if (R > 2048) return einval("cut radius above 2048 px");
    if (!g1 || !g2 || !map) return einval("null pointer");
    return launch_map_direct(g1, g2, nullptr, 0, map, nullptr, n, batch, filter, theta_px, ell, cut, cfg.precision,
                             (cudaStream_t)stream);
}

int fm_map_direct_masked(const void *g1, const void *g2, const void *weight, long weight_bstride, void *map,
                         void *coverage, int n, int batch, int filter, double theta_px, int ell,
                         double cut_over_theta, const fm_config *cfgp, void *stream)
{
    fm_config cfg = cfg_or_default(cfgp);
    int st = check_config(cfg);
    if (st) return st;
    if (n < 1 || n > 65536) return einval("n must be in [1, 65536]");
    if (batch < 1 || batch > 65535) return einval("batch must be in [1, 65535]");
    if (weight_bstride < 0) return einval("weight_bstride must be >= 0");
    if (filter < FM_FILTER_STARLET || filter > FM_FILTER_VW98) return einval("unknown filter");
    if (!(theta_px > 0) || theta_px > 4096) return einval("theta_px must be in (0, 4096]");
    if (filter == FM_FILTER_S98 && (ell < 0 || ell > 64)) return einval("ell must be in [0, 64]");
    const double cut = cut_over_theta > 0 ? cut_over_theta : 0.0;
    const double R = (cut > 0 ? cut : (filter == FM_FILTER_STARLET ? 2.0 : filter == FM_FILTER_S98 ? 1.0 : 5.0)) *
                     theta_px;
    if (R > 2048) return einval("cut radius above 2048 px");
    if (R < 1) return einval("cut radius below one pixel: the aperture holds no pixel");
    if (!g1 || !g2 || !weight || !map) return einval("null pointer");
    return launch_map_direct(g1, g2, weight, weight_bstride, map, coverage, n, batch, filter, theta_px, ell, cut,
                             cfg.precision, (cudaStream_t)stream);
}

// Noise maps (Sec. 1): one unrotated pass for w_j(data), then R rotated
// realisations in chunks, each chunk a batch through KS and the starlet with
// the bands accumulated into FP64 S1, S2; then the finalize kernel.
int fm_map_noise(const void *g1, const void *g2, double *var_out, void *snr_out, int n, int J, int R, uint64_t seed,
                 const fm_config *cfgp, void *stream)
{
    fm_config cfg = cfg_or_default(cfgp);
    int st = check_config(cfg);
    if (st) return st;
    if ((st = check_fft_n(n))) return st;
    if ((st = check_J(n, J))) return st;
    if (R < 2) return einval("R must be >= 2");
    if (!g1 || !g2 || !var_out) return einval("null pointer");
    return map_noise_run(g1, g2, var_out, snr_out, n, J, R, seed, cfg, (cudaStream_t)stream, true);
}

// Noise maps in parts (checkpoint and resume, or realisations split over
// GPUs): realisations r0 .. r0 + R - 1 added to the caller's FP64 sums, and
// the variance (and S/N) from sums of R_total realisations.
int fm_map_noise_accumulate(const void *g1, const void *g2, double *sums, int n, int J, int r0, int R, uint64_t seed,
                            const fm_config *cfgp, void *stream)
{
    fm_config cfg = cfg_or_default(cfgp);
    int st = check_config(cfg);
    if (st) return st;
    if (cfg.accum != 0) return einval("fm_map_noise_accumulate keeps FP64 sums (accum = 0)");
    if ((st = check_fft_n(n))) return st;
    if ((st = check_J(n, J))) return st;
    if (R < 1 || r0 < 0 || (long)r0 + R > 2147483647L) return einval("need R >= 1, r0 >= 0, r0 + R < 2^31");
    if (!g1 || !g2 || !sums) return einval("null pointer");
    return map_noise_accumulate_run(g1, g2, sums, n, J, r0, R, seed, cfg, (cudaStream_t)stream);
}

int fm_noise_finalize(const double *sums, const void *pyramid, double *var_out, void *snr_out, int n, int J,
                      int R_total, const fm_config *cfgp, void *stream)
{
    fm_config cfg = cfg_or_default(cfgp);
    int st = check_config(cfg);
    if (st) return st;
    if (cfg.accum != 0) return einval("fm_noise_finalize reads FP64 sums (accum = 0)");
    if ((st = check_fft_n(n))) return st;  // the sizes fm_map_noise_accumulate produces sums for
    if ((st = check_J(n, J))) return st;
    if (R_total < 2) return einval("R_total must be >= 2");
    if (!sums || !var_out) return einval("null pointer");
    if (snr_out && !pyramid) return einval("S/N needs the data's pyramid");
    return launch_noise_finalize(sums, snr_out ? pyramid : nullptr, var_out, snr_out, (long)(J - 1) * n * n,
                                 R_total, cfg.precision, 0, (cudaStream_t)stream);
}

// Exact expected noise variance (Sec. 1), periodic boundary:
// Var_j = 1/2 |K_j|^2 (*) |gamma|^2 (circular convolution).  K_j is the
// pipeline's response to unit shears at pixel 0 (Re K_j from gamma1, -Im K_j
// from gamma2); the convolutions run through the FFT pipeline, two bands at a
// time: the spectrum of |gamma|^2 once, then rows FFT of |K_j|^2 + i |K_j+p|^2
// (p = pairs, half the bands rounded up) -> columns FFT -> times that spectrum
// -> inverse, whose real and imaginary parts are the bands j and j + p
// (|gamma|^2 is real).  Band j + p enters times a power of two that brings it to
// band j's magnitude, so that its rounding is relative to itself: 4^p, as a
// band's response power falls by 4.0 to 5.5 a scale, and for band 0's partner,
// as band 0 has 20 times the power of band 1, that times 8 (4 for p = 1).  With
// 4^p alone the partner's error was 2.5 times the other bands' (rms of its
// mean, 256^2 .. 2048^2 3.3 .. 4.0e-7, now 1.3 .. 1.8e-7).  One spectrum and
// (J - 1) / 2 filter passes instead of J - 1 of each: 1024^2, J = 7 214 -> 158 us
// (145 with the later steps).
int fm_map_noise_expected(const void *g1, const void *g2, void *var_out, int n, int J, const fm_config *cfgp,
                          void *stream)
{
    fm_config cfg = cfg_or_default(cfgp);
    int st = check_config(cfg);
    if (st) return st;
    if ((st = check_fft_n(n))) return st;
    if ((st = check_J(n, J))) return st;
    if (cfg.boundary != FM_PERIODIC)
        return einval("fm_map_noise_expected needs cfg->boundary = FM_PERIODIC: with mirror edges KS + starlet is "
                      "not a convolution");
    if (!g1 || !g2 || !var_out) return einval("null pointer");
    cudaStream_t s = (cudaStream_t)stream;
    const int prec = cfg.precision;
    const size_t es = prec == FM_F64 ? 8 : 4;
    const long nn = (long)n * n;
    const int nb = J - 1;
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    const int h = nb / 2, pairs = nb - h;  // bands 0 .. h - 1 with pairs .. nb - 1; band h alone where nb is odd
    const size_t b_delta = up(2 * nn * es), b_pyr = up((size_t)2 * J * nn * es), b_q = up((size_t)nb * nn * es),
                 b_p = up(nn * es), b_spec = up((size_t)nn * 2 * es), b_work = up((size_t)pairs * nn * 2 * es);
    Scratch sc;
    if ((st = scratch_alloc(sc, 2 * b_delta + b_pyr + b_q + b_p + b_spec + b_work, s))) return st;
    char *base = static_cast<char *>(sc.p);
    char *g1d = base, *g2d = g1d + b_delta, *pyr = g2d + b_delta, *q = pyr + b_pyr, *p = q + b_q, *spec = p + b_p,
         *work = spec + b_spec;
    if ((st = launch_unit_shears(g1d, g2d, nn, prec, s))) return st;
    if ((st = map_starlet_run(g1d, g2d, pyr, n, J, 2, cfg, s))) return st;
    // |K_j|^2 = (Re K_j)^2 + (Im K_j)^2 from the two responses [2][J][n][n]
    const double up4 = ldexp(1.0, 2 * pairs), lead = up4 * (pairs > 1 ? 8 : 4);  // 4^pairs; band 0's partner
    if ((st = launch_modulus2(pyr, nn, pyr + (size_t)J * nn * es, nn, q, nn, nb, pairs, lead, up4, prec, s))) return st;
    if ((st = launch_modulus2(g1, 0, g2, 0, p, nn, 1, 1, 1.0, 1.0, prec, s))) return st;
    if ((st = launch_fft_op(p, nullptr, nn, nullptr, nullptr, spec, n, 1, prec, FFT_OP_SPECTRUM, nullptr, 1.0, 0, 0,
                            false, s)))
        return st;
    // The responses are scaled for two transforms there and back, but a unit
    // shear's transform there is exact: half of that gain is too much in K_j, the
    // whole of it once in |K_j|^2 (bias of the bands' |K_j|^2, n = 32 .. 2048: as
    // scaled 0.5 .. 1.8e-7, unscaled -0.5 .. -1.6e-7, so -0.7 .. 0.6e-7).
    const double half = prec == FM_F32 && n >= 32 ? 0.5 / kFft32Gain : 0.5;
    char *var = static_cast<char *>(var_out), *q2 = q + (size_t)pairs * nn * es;
    if (h > 0 && (st = launch_fft_op(q, q2, nn, var, var + (size_t)pairs * nn * es, work, n, h, prec, FFT_OP_FILTER,
                                     spec, half, 0, 0, false, s, false, 1.0 / up4, 1.0 / lead)))
        return st;
    if (h == pairs) return FM_OK;
    return launch_fft_op(q + (size_t)h * nn * es, nullptr, nn, var + (size_t)h * nn * es, nullptr, work, n, 1, prec,
                         FFT_OP_FILTER, spec, half, 0, 0, false, s);
}

int fm_band_moments(const void *pyramid, double *moments, int n, int J, int batch, const fm_config *cfgp,
                    void *stream)
{
    fm_config cfg = cfg_or_default(cfgp);
    int st = check_config(cfg);
    if (st) return st;
    if (n < 1 || n > 65536) return einval("n must be in [1, 65536]");
    if (J < 1 || J > 20) return einval("J must be in [1, 20]");
    if (batch < 1 || batch > 65535) return einval("batch must be in [1, 65535]");
    if (!pyramid || !moments) return einval("null pointer");
    cudaStream_t s = (cudaStream_t)stream;
    Scratch sc;
    if ((st = scratch_alloc(sc, sizeof(double) * 4 * (size_t)batch * J, s))) return st;
    return launch_band_moments(pyramid, moments, n, J, batch, cfg.precision, sc.p, s);
}

}  // extern "C"

// Random soil fields by FFT moving average (arXiv 1903.08741, Appendix A):
// white noise y on a periodic px x pz torus, z = F^-1( sqrt(F c) . F y ), keep
// the physical window, then ln Ks = z_0 and alpha = lo + span * Phi(z_1 / sigma).
//
// GPU design: the two real fields of a sample are packed into one complex
// transform (re = y_0, im = y_1); sqrt(F c) is real and even, so the filter maps
// real inputs to real outputs and the two fields come back in re / im.  Three
// kernels, one pass over the torus each, in 64-bit integers (fixed.cuh has why
// and how precise): white noise and row transforms; column transforms, filter
// and inverse column transforms; inverse row transforms and the marginal
// transforms.  The second keeps the rows of the physical window only, so the
// third runs half of them.  Within the transforms frequencies stay in
// bit-reversed order; the filter is laid out in it.  In FP64, one kernel a pass
// (noise, row and column transforms both ways, filter, window), 512 draws of a
// 128^2 pair took 63.1 ms, now 8.7; 64 of a 32^2 pair 477 us, now 94; 512
// couples of five 64^2 fields 13.1 ms, now 2.0.  What is left is the 32-bit multiply
// and add pipes (the first kernel issues on 67 % of its cycles).
// White noise: Philox4x32-10 (Salmon et al., SC'11) implemented from its
// definition, key = (seed low word, seed high word ^ level), counter = (cell
// pair, field, sample low, sample high), two uniforms -> Box-Muller.
#include "rich_internal.cuh"
#include "fixed.cuh"
#include <cmath>
#include <vector>
#include <algorithm>

namespace {
using namespace rich_fx;

struct cplx { double re, im; };

__device__ __forceinline__ void philox10(uint32_t c[4], uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        const uint64_t p0 = (uint64_t)0xD2511F53u * c[0], p1 = (uint64_t)0xCD9E8D57u * c[2];
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c[1] ^ k0, n2 = (uint32_t)(p0 >> 32) ^ c[3] ^ k1;
        c[0] = n0; c[1] = (uint32_t)p1; c[2] = n2; c[3] = (uint32_t)p0;
    }
}

// FP64 twiddles w_k = exp(-2 pi i k / n), k < n/2, of the spectrum's transform
__global__ void k_twiddles(int n, cplx* tw) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n / 2) return;
    double s, c;
    sincospi(-2.0 * (double)k / (double)n, &s, &c);
    tw[k] = cplx{c, s};
}

// Batched radix-2 FP64 FFT of lines of length n (power of two) held in shared
// memory: the covariance spectrum's, once per model and grid (its values span
// more than one fixed-point scale holds).  A block handles LPB lines; line l of sample b starts at
// b*sample_stride + l*line_stride, its elements are elem_stride apart.
// Bit-reversed load, log2(n) butterfly stages.
template <int LPB>
__global__ void k_fft_lines(cplx* data, int n, int logn, int lines, long long sample_stride,
                            int line_stride, int elem_stride, const cplx* __restrict__ tw) {
    // contiguous lines: consecutive threads take consecutive elements; strided
    // lines (columns): consecutive threads take adjacent lines
    const bool contig = elem_stride == 1;
    extern __shared__ cplx sh[];
    const int groups = lines / LPB;
    const int b = blockIdx.x / groups, g = blockIdx.x - b * groups;
    cplx* base = data + (size_t)b * sample_stride + (size_t)g * LPB * line_stride;
    const int tid = threadIdx.x, nt = blockDim.x;
    // load: element e of line l -> shared [l][rev(e)]; consecutive threads read
    // consecutive lines first so that column groups coalesce
    for (int t = tid; t < n * LPB; t += nt) {
        int l = contig ? t / n : t % LPB, e = contig ? t - (t / n) * n : t / LPB;
        int r = logn ? (int)(__brev((unsigned)e) >> (32 - logn)) : 0;
        sh[l * n + r] = base[(size_t)l * line_stride + (size_t)e * elem_stride];
    }
    __syncthreads();
    for (int m = 1, st = n >> 1; m < n; m <<= 1, st >>= 1) {
        for (int t = tid; t < (n >> 1) * LPB; t += nt) {
            int l = t / (n >> 1), bf = t - l * (n >> 1);
            int grp = bf / m, k = bf - grp * m;
            int a = grp * 2 * m + k, c = a + m;
            cplx w = tw[k * st];
            double wi = w.im;
            cplx x = sh[l * n + c], y = sh[l * n + a];
            double xr = x.re * w.re - x.im * wi;
            double xi = x.re * wi + x.im * w.re;
            sh[l * n + c] = cplx{y.re - xr, y.im - xi};
            sh[l * n + a] = cplx{y.re + xr, y.im + xi};
        }
        __syncthreads();
    }
    for (int t = tid; t < n * LPB; t += nt) {
        int l = contig ? t / n : t % LPB, e = contig ? t - (t / n) * n : t / LPB;
        base[(size_t)l * line_stride + (size_t)e * elem_stride] = sh[l * n + e];
    }
}

// covariance model of one spectrum: nu = 0 exponential sigma2 exp(-r);
// nu > 0 the Matern function of Eq. nonIsotropic, norm = sigma2 2^(1-nu)/Gamma(nu)
struct CovModel {
    double sigma2, lx, lz, nu, norm;
};

// K_nu(x) for x > 0 from K_nu(x) = int_0^inf exp(-x cosh t) cosh(nu t) dt
// (DLMF 10.32.9): trapezoidal sum, geometrically convergent for this
// analytic, doubly exponentially decaying integrand; the step resolves the
// exp(-x t^2/2) peak at large x (min(1/16, 1/(2 sqrt x))), the sum ends past
// the integrand's maximum once a term adds less than 1e-18 (at most 4095 terms)
__device__ double bessel_k(double nu, double x) {
    const double dt = x > 64.0 ? 0.5 / sqrt(x) : 0.0625;
    double acc = 0.5 * exp(-x);
    for (int k = 1; k < 4096; ++k) {
        const double t = k * dt;
        const double f = exp(-x * cosh(t)) * cosh(nu * t);
        acc += f;
        if (f <= 1e-18 * acc && x * sinh(t) > nu) break;
    }
    return dt * acc;
}

// covariance on the torus at the periodic offset of point (a, b)
__global__ void k_cov(int px, int pz, double h, CovModel cm, cplx* c) {
    int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= px * pz) return;
    int b = g / px, a = g - b * px;
    int ia = min(a, px - a), ib = min(b, pz - b);
    double dx = ia * h, dz = ib * h;
    const double r = cm.lz == cm.lx ? sqrt(dx * dx + dz * dz) / cm.lx
                                    : sqrt((dx / cm.lx) * (dx / cm.lx) + (dz / cm.lz) * (dz / cm.lz));
    double v;
    if (cm.nu == 0.0) v = cm.sigma2 * exp(-r);
    else if (r == 0.0) v = cm.sigma2;
    else {
        const double x = 2.0 * sqrt(cm.nu) * r;
        v = cm.norm * pow(x, cm.nu) * bessel_k(cm.nu, x);
    }
    c[g] = cplx{v, 0.0};
}

__device__ __forceinline__ int brev(int p, int logn) { return logn ? (int)(__brev((unsigned)p) >> (32 - logn)) : 0; }

// the filter sqrt(max(F c, 0)) in Q62 of each column's scale 2^ecol, both
// indices bit-reversed
__global__ void k_filter_table(int logpx, int logpz, const cplx* __restrict__ lam, const int* __restrict__ ecol,
                               wq* out) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >> (logpx + logpz)) return;
    const int kx = brev(g & ((1 << logpx) - 1), logpx), kz = brev(g >> logpx, logpz);
    const double v = lam[(kz << logpx) + kx].re;
    out[g] = split_w(v > 0.0 ? __double2ll_rn(ldexp(sqrt(v), 62 - ecol[kx])) : 0);
}

// marginal transforms of a packed pair: the re lane is Gaussian (shift + z,
// ln Ks) or uniform, the im lane uniform: lo + span Phi(z / sigma) with
// Phi(x) = erfc(-x/sqrt 2)/2 (Y = F_Y^-1(F_Z(Z)), Sec. 3.1)
struct PackTr {
    int re_uniform;
    double re_a, re_b;      // Gaussian: shift re_a; uniform: lo re_a, span re_b
    double im_lo, im_span;
};

__device__ __forceinline__ double uniform_of(double z, double inv_sigma, double lo, double span,
                                             const PhiEntry* __restrict__ tab) {
    return lo + span * normal_cdf(z * inv_sigma, tab);
}

// ---------------------------------------------------------------- transforms
// One radix-R pass over the block's lines in shared memory, from bit b0 of the
// n = 2^logn transform on.  Rows (COLS false) lie one after the other, an element
// of padding after every eight: the last passes' strides of 4 and 8 elements then
// meet no bank twice.  Columns lie side by side, LPB = 2^loglpb to a torus row.
// With FILT (the last pass) each value is multiplied by its filter entry and the
// first inverse pass follows in registers.
template <bool COLS>
__device__ __forceinline__ int at(int l, int p, int logn, int loglpb) {
    return COLS ? (p << loglpb) + l : l * ((1 << logn) + ((1 << logn) >> 3)) + p + (p >> 3);
}

template <int R, bool COLS, bool INV, bool FILT>
__device__ __forceinline__ void pass(fx2* sm, int logn, int loglpb, int b0, const cw* __restrict__ tw,
                                     const wq* __restrict__ filt, int fstride) {
    constexpr int RB = R == 8 ? 3 : R == 4 ? 2 : 1;
    const int lq = logn - b0 - RB;                    // log2 of the stride between a butterfly's elements
    const int sh = ((b0 + RB) >> 1) - (b0 >> 1);
    for (int it = threadIdx.x; it < 1 << (logn - RB + loglpb); it += blockDim.x) {
        const int l = COLS ? it & ((1 << loglpb) - 1) : it >> (logn - RB);
        const int g = COLS ? it >> loglpb : it & ((1 << (logn - RB)) - 1);
        const int k = g & ((1 << lq) - 1), base = ((g >> lq) << (lq + RB)) + k;
        fx2 a[R];
#pragma unroll
        for (int j = 0; j < R; ++j) a[j] = sm[at<COLS>(l, base + (j << lq), logn, loglpb)];
        if (FILT) {
            dft_fwd<R>(a);
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const wq f = filt[(size_t)(base + j) * fstride + l];
                a[j] = fx2{rmul(rshift(a[j].re, sh), f), rmul(rshift(a[j].im, sh), f)};
            }
            dft_inv<R>(a);
        } else if (!INV) {
            dft_fwd<R>(a);
            a[0] = fx2{rshift(a[0].re, sh), rshift(a[0].im, sh)};
#pragma unroll
            for (int j = 1; j < R; ++j) a[j] = cmul(a[j], tw[(k * revr<R>(j)) << b0], sh);
        } else {
            if (lq > 0) {
#pragma unroll
                for (int j = 1; j < R; ++j) {
                    cw w = tw[(k * revr<R>(j)) << b0];
                    w.im = neg(w.im);
                    a[j] = cmul(a[j], w, 0);
                }
            }
            dft_inv<R>(a);
        }
#pragma unroll
        for (int j = 0; j < R; ++j) sm[at<COLS>(l, base + (j << lq), logn, loglpb)] = a[j];
    }
    __syncthreads();
}

template <bool COLS, bool INV, bool FILT>
__device__ __forceinline__ void any_pass(int bits, fx2* sm, int logn, int loglpb, int b0, const cw* tw,
                                         const wq* filt = nullptr, int fstride = 0) {
    if (bits == 3) pass<8, COLS, INV, FILT>(sm, logn, loglpb, b0, tw, filt, fstride);
    else if (bits == 2) pass<4, COLS, INV, FILT>(sm, logn, loglpb, b0, tw, filt, fstride);
    else pass<2, COLS, INV, FILT>(sm, logn, loglpb, b0, tw, filt, fstride);
}

// inverse passes below bit `top` (the passes of the forward order, last first)
template <bool COLS>
__device__ __forceinline__ void inverse_passes(fx2* sm, int logn, int loglpb, int top, const cw* tw) {
    int b0s[8], np = 0;
    for (int b = 0; b < top; b += pass_bits(logn, b)) b0s[np++] = b;
    while (np-- > 0) any_pass<COLS, true, false>(pass_bits(logn, b0s[np]), sm, logn, loglpb, b0s[np], tw);
}

constexpr int FT = 256;                     // threads of the transform kernels

// the noise of the torus and its row transforms, frequencies bit-reversed;
// 2^loglpb rows a block.  The coarse member's noise is half the 2x2 sums of the
// torus of twice the sides (it stays standard normal: Appendix A, Eq. averaging):
// a block of two rows or more leaves it in `coarse` for the LOADED launch (drawing
// it again there: 512 couples of five 64^2 fields 3.7 ms, so 2.0); where only one
// row of 8192 fits, the COARSE launch does draw it again.
// (first sample = *first_dev + first when first_dev is given: a captured CUDA
// graph can advance the sample range between replays)
struct RowArgs {
    long long lines;
    int logpx, logpz, loglpb;
    uint64_t seed;
    uint32_t level, fld0;
    int im;                                 // 0: the im lane's field is not wanted
    int64_t first;
    const int64_t* first_dev;
    const NormTab* norm;
    const cw* tw;
    fx2* out;
    fx2* coarse;
};
enum { FINE, COARSE, LOADED };

template <int SRC>
__global__ void __launch_bounds__(FT, 3) k_noise_rows(const RowArgs A) {
    extern __shared__ fx2 sm[];
    const int logn = A.logpx, n = 1 << logn, lpb = 1 << A.loglpb;
    const long long line0 = (long long)blockIdx.x << A.loglpb;
    const int64_t first = (A.first_dev ? *A.first_dev : 0) + A.first;
    const uint32_t k0 = (uint32_t)A.seed, k1 = (uint32_t)(A.seed >> 32) ^ A.level;
    auto draw = [&](uint32_t q, int fld, uint64_t sample, long long& y0, long long& y1) {
        uint32_t c[4] = {q, A.fld0 + (uint32_t)fld, (uint32_t)sample, (uint32_t)(sample >> 32)};
        philox10(c, k0, k1);
        normal_pair(c[0], c[1], c[2], c[3], A.norm, y0, y1);
    };
    const int lw = SRC == FINE ? logn - 1 : logn;     // a thread's unit: two neighbours; a point
    for (int it = threadIdx.x; it < lpb << lw; it += FT) {
        const int l = it >> lw, x = it & ((1 << lw) - 1);
        const long long line = line0 + l;
        if (line >= A.lines) break;
        if (SRC == LOADED) {
            sm[at<false>(l, x, logn, 0)] = A.coarse[(line << logn) + x];
            continue;
        }
        const uint64_t sample = (uint64_t)(first + (line >> A.logpz));
        const uint32_t row = (uint32_t)(line & ((1ll << A.logpz) - 1));
        long long y[2][2] = {};
#pragma unroll 1
        for (int f = 0; f < (A.im ? 2 : 1); ++f) {
            long long a, b;
            if (SRC == COARSE) {
                long long c, d;
                draw(((2 * row) << logn) + x, f, sample, a, b);
                draw(((2 * row + 1) << logn) + x, f, sample, c, d);
                a = (a + b + c + d + 1) >> 1;
            } else {
                draw((row << lw) + x, f, sample, a, b);
            }
            if (f) { y[1][0] = a; y[1][1] = b; } else { y[0][0] = a; y[0][1] = b; }
        }
        if (SRC == COARSE) {
            sm[at<false>(l, x, logn, 0)] = fx2{y[0][0], y[1][0]};
        } else {
            sm[at<false>(l, 2 * x, logn, 0)] = fx2{y[0][0], y[1][0]};
            sm[at<false>(l, 2 * x + 1, logn, 0)] = fx2{y[0][1], y[1][1]};
        }
    }
    __syncthreads();
    if (SRC == FINE && A.coarse) {
        for (int t = threadIdx.x; t < n << A.loglpb >> 2; t += FT) {
            const int l = 2 * (t >> (logn - 1)), x = 2 * (t & ((n >> 1) - 1));
            if (line0 + l >= A.lines) break;
            const fx2 v = sm[at<false>(l, x, logn, 0)] + sm[at<false>(l, x + 1, logn, 0)] +
                          sm[at<false>(l + 1, x, logn, 0)] + sm[at<false>(l + 1, x + 1, logn, 0)];
            A.coarse[(((line0 + l) >> 1) << (logn - 1)) + (x >> 1)] = fx2{(v.re + 1) >> 1, (v.im + 1) >> 1};
        }
        __syncthreads();
    }
    for (int b = 0; b < logn;) {
        const int w = pass_bits(logn, b);
        any_pass<false, false, false>(w, sm, logn, A.loglpb, b, A.tw);
        b += w;
    }
    for (int t = threadIdx.x; t < n << A.loglpb; t += FT) {
        const int l = t >> logn, p = t & (n - 1);
        if (line0 + l < A.lines) A.out[((line0 + l) << logn) + p] = sm[at<false>(l, p, logn, 0)];
    }
}

// column transforms, filter and inverse column transforms of 2^loglpb columns a
// block, in place; only the window's rows (the first nz) are written
__global__ void __launch_bounds__(FT, 3)
k_columns(int logpx, int logpz, int loglpb, int nz, const cw* __restrict__ tw, const wq* __restrict__ filt, fx2* data) {
    extern __shared__ fx2 sm[];
    const int c0 = (blockIdx.x & ((1 << (logpx - loglpb)) - 1)) << loglpb, lpb = 1 << loglpb;
    fx2* d = data + ((size_t)(blockIdx.x >> (logpx - loglpb)) << (logpx + logpz)) + c0;
    for (int t = threadIdx.x; t < lpb << logpz; t += FT)
        sm[t] = d[((size_t)(t >> loglpb) << logpx) + (t & (lpb - 1))];
    __syncthreads();
    int b = 0, w = pass_bits(logpz, 0);
    for (; b + w < logpz; w = pass_bits(logpz, b)) {
        any_pass<true, false, false>(w, sm, logpz, loglpb, b, tw);
        b += w;
    }
    any_pass<true, false, true>(w, sm, logpz, loglpb, b, tw, filt + c0, 1 << logpx);
    inverse_passes<true>(sm, logpz, loglpb, b, tw);
    for (int t = threadIdx.x; t < nz << loglpb; t += FT)
        d[((size_t)(t >> loglpb) << logpx) + (t & (lpb - 1))] = sm[t];
}

// inverse row transforms of the window's rows (their columns brought to one
// scale first) -> the pair's two fields, compact [S][nz][nx] real arrays (al
// may be null: the im lane is unused); nx and nz are powers of two
__global__ void __launch_bounds__(FT, 3)
k_rows_window(long long lines, int logpx, int logpz, int loglpb, int lognx, int lognz, const cw* __restrict__ tw,
              const int* __restrict__ colsh, double scale, const fx2* __restrict__ data, double inv_sigma, PackTr tr,
              const PhiEntry* __restrict__ tab, double* lk, double* al) {
    extern __shared__ fx2 sm[];
    const int n = 1 << logpx;
    const long long line0 = (long long)blockIdx.x << loglpb;
    for (int t = threadIdx.x; t < n << loglpb; t += FT) {
        const int l = t >> logpx, p = t & (n - 1);
        const long long line = line0 + l;
        fx2 v{0, 0};
        const int sh = colsh[p];
        if (line < lines && sh < 62) {
            v = data[((line >> lognz) << (logpx + logpz)) + ((line & ((1ll << lognz) - 1)) << logpx) + p];
            v = fx2{rshift(v.re, sh), rshift(v.im, sh)};
        }
        sm[at<false>(l, p, logpx, 0)] = v;
    }
    __syncthreads();
    inverse_passes<false>(sm, logpx, loglpb, logpx, tw);
    for (int t = threadIdx.x; t < 1 << (lognx + loglpb); t += FT) {
        const int l = t >> lognx, i = t & ((1 << lognx) - 1);
        if (line0 + l >= lines) break;
        const long long g = ((line0 + l) << lognx) + i;
        const fx2 v = sm[at<false>(l, i, logpx, 0)];
        const double re = (double)v.re * scale;
        lk[g] = tr.re_uniform ? uniform_of(re, inv_sigma, tr.re_a, tr.re_b, tab) : re + tr.re_a;
        if (al) al[g] = uniform_of((double)v.im * scale, inv_sigma, tr.im_lo, tr.im_span, tab);
    }
}

// one 2x2 averaging step of both fields
__global__ void k_avg2(int S, int nxc, int nzc, const double* __restrict__ lf,
                       const double* __restrict__ af, double* lc, double* ac) {
    long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int nc = nxc * nzc, fx = 2 * nxc;
    if (g >= (long long)S * nc) return;
    int s = (int)(g / nc), q = (int)(g - (long long)s * nc);
    int J = q / nxc, I = q - J * nxc;
    size_t f00 = (size_t)s * 4 * nc + (size_t)(2 * J) * fx + 2 * I, f01 = f00 + fx;
    lc[g] = 0.25 * (lf[f00] + lf[f00 + 1] + lf[f01] + lf[f01 + 1]);
    if (ac) ac[g] = 0.25 * (af[f00] + af[f00 + 1] + af[f01] + af[f01 + 1]);
}

inline unsigned nb(long long w, int t = 256) { return (unsigned)((w + t - 1) / t); }
inline int ilog2(int n) { int l = 0; while ((1 << l) < n) ++l; return l; }
inline bool pow2(int n) { return n > 0 && (n & (n - 1)) == 0; }

template <int L>
int fft_pass(cplx* d, int S, int n, int lines, long long sstride, int lstride, int estride,
             const cplx* tw, cudaStream_t st) {
    size_t sm = (size_t)L * n * sizeof(cplx);
    RICH_CUDA(cudaFuncSetAttribute(k_fft_lines<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    rich_count_launch();
    k_fft_lines<L><<<(unsigned)S * (lines / L), 256, sm, st>>>(d, n, ilog2(n), lines, sstride, lstride, estride,
                                                               tw);
    return 0;
}

// lines per block: the largest of 8, 4, 2, 1 that divides the line count and
// keeps the block's lines within 128 KB of shared memory
int fft_dispatch(cplx* d, int S, int n, int lines, long long sstride, int lstride, int estride,
                 const cplx* tw, cudaStream_t st) {
    for (int L = 8; L >= 1; L >>= 1) {
        if (lines % L || (size_t)L * n * sizeof(cplx) > (128u << 10)) continue;
        switch (L) {
            case 8: return fft_pass<8>(d, S, n, lines, sstride, lstride, estride, tw, st);
            case 4: return fft_pass<4>(d, S, n, lines, sstride, lstride, estride, tw, st);
            case 2: return fft_pass<2>(d, S, n, lines, sstride, lstride, estride, tw, st);
            default: return fft_pass<1>(d, S, n, lines, sstride, lstride, estride, tw, st);
        }
    }
    return RICH_ERR_INVALID;
}

int fft2(cplx* d, int S, int px, int pz, const cplx* twx, const cplx* twz, cudaStream_t st) {
    const long long ss = (long long)px * pz;
    if (int e = fft_dispatch(d, S, px, pz, ss, px, 1, twx, st)) return e;   // rows (x)
    if (int e = fft_dispatch(d, S, pz, px, ss, 1, px, twz, st)) return e;   // columns (z)
    RICH_CUDA(cudaGetLastError());
    return 0;
}

}  // namespace

// ---------------------------------------------------------------- host side
// a field model outside the supported range: sigma2, corr_len > 0,
// corr_len_z >= 0 (0: isotropic), 0 <= nu <= 16
bool bad_field(const rich_field_t* fd) {
    return !(fd->sigma2 > 0) || !(fd->corr_len > 0) || !(fd->corr_len_z >= 0) || !(fd->nu >= 0) ||
           !(fd->nu <= 16);
}

// exp(-2 pi i k / n), k < n: a quarter turn from the host's functions, the rest
// by symmetry
static void make_twiddles(int n, cw* w) {
    for (int k = 0; k < n; ++k) {
        if (n < 4 || k < n / 4) {
            w[k] = circle_point(-k, n);
        } else {
            const cw v = w[k - n / 4];
            w[k] = cw{v.im, neg(v.re)};                       // times -i
        }
    }
}

static const NormTab& norm_tab() {
    static const NormTab t = [] { NormTab v; make_norm_tab(v); return v; }();
    return t;
}

// The filter sqrt(F c) on a px x pz torus of spacing h, with what the transforms
// read, cached in the context.  Scales: column kx of the filter is in units of
// 2^e, the power of two above its Euclidean norm (so that its unnormalised
// inverse transform of unit values stays one); the rows' transforms take the
// power above the whole filter's norm.
static int spectrum_on(rich_ctx* ctx, int px, int pz, double h, const rich_field_t* fd,
                       cudaStream_t st, const rich_spectrum** out, double* min_ratio) {
    const double sigma2 = fd->sigma2, corr_len = fd->corr_len, nu = fd->nu;
    const double lz = fd->corr_len_z > 0 ? fd->corr_len_z : fd->corr_len;
    for (const rich_spectrum& e : ctx->spectra)
        if (e.px == px && e.pz == pz && e.h == h && e.sigma2 == sigma2 && e.corr_len == corr_len &&
            e.corr_len_z == lz && e.nu == nu) {
            *out = &e;
            if (min_ratio) *min_ratio = e.min_ratio;
            return 0;
        }
    const int npts = px * pz;
    rich_spectrum e{};
    e.px = px; e.pz = pz; e.h = h; e.sigma2 = sigma2; e.corr_len = corr_len; e.corr_len_z = lz; e.nu = nu;
    const CovModel cm{sigma2, corr_len, lz, nu, nu > 0 ? sigma2 * pow(2.0, 1.0 - nu) / tgamma(nu) : 0.0};
    struct Bufs { void *a = nullptr, *b = nullptr, *t = nullptr; ~Bufs() { cudaFree(a); cudaFree(b); cudaFree(t); } } tmp;
    RICH_CUDA(cudaMalloc(&tmp.a, sizeof(cplx) * npts));
    RICH_CUDA(cudaMalloc(&tmp.b, sizeof(cplx) * (px / 2 + pz / 2 + 2)));
    cplx *c = (cplx*)tmp.a, *tw = (cplx*)tmp.b;
    rich_count_launch(); k_twiddles<<<nb(px / 2), 256, 0, st>>>(px, tw);
    rich_count_launch(); k_twiddles<<<nb(pz / 2), 256, 0, st>>>(pz, tw + px / 2 + 1);
    rich_count_launch(); k_cov<<<nb(npts), 256, 0, st>>>(px, pz, h, cm, c);
    if (int r = fft2(c, 1, px, pz, tw, tw + px / 2 + 1, st)) return r;
    std::vector<cplx> hl(npts);
    RICH_CUDA(cudaMemcpyAsync(hl.data(), c, sizeof(cplx) * npts, cudaMemcpyDeviceToHost, st));
    RICH_CUDA(cudaStreamSynchronize(st));
    double lmin = hl[0].re, lmax = hl[0].re, sum = 0.0, total = 0.0;
    for (const cplx& v : hl) { lmin = std::min(lmin, v.re); lmax = std::max(lmax, v.re); }
    // sums in units of 4^eu, about the largest eigenvalue: they do not overflow
    // before the eigenvalues do
    int eu = 0;
    if (std::isfinite(lmax)) frexp(lmax, &eu);
    eu = std::max(-500, std::min(500, eu / 2));
    const double unit = ldexp(1.0, -2 * eu);
    std::vector<double> col(px, 0.0);
    for (int g = 0; g < npts; ++g) {
        const double v = hl[g].re * unit;
        sum += v;
        if (v > 0.0) { col[g & (px - 1)] += v; total += v; }
    }
    e.min_ratio = lmin / lmax;
    // tables: Q62 twiddles of rows and columns, the normals', the columns'
    // exponents (natural order) and their distance to the rows' (bit-reversed)
    const size_t n_tw = sizeof(cw) * (px + pz), o_norm = n_tw, o_e = o_norm + sizeof(NormTab),
                 o_sh = o_e + sizeof(int) * px, o_f = (o_sh + sizeof(int) * px + 255) & ~(size_t)255;
    std::vector<char> hb(o_f);
    cw* htw = (cw*)hb.data();
    make_twiddles(px, htw);
    if (pz == px) std::copy(htw, htw + px, htw + px);
    else make_twiddles(pz, htw + px);
    *(NormTab*)(hb.data() + o_norm) = norm_tab();
    const bool finite = std::isfinite(sum);               // (an infinite variance: the fields are NaN)
    int etot = 0;
    if (finite) frexp(sqrt(total), &etot);
    etot += eu;
    int* he = (int*)(hb.data() + o_e);
    int* hsh = (int*)(hb.data() + o_sh);
    const int lx = ilog2(px), lzz = ilog2(pz);
    for (int k = 0; k < px; ++k) {
        he[k] = etot - 62;
        if (finite && col[k] > 0.0) { frexp(sqrt(col[k]), &he[k]); he[k] += eu; }
        he[k] = std::max(he[k], etot - 62);               // below: nothing of it is left in a row
    }
    for (int p = 0; p < px; ++p) {
        int k = 0;
        for (int b = 0; b < lx; ++b) k |= ((p >> b) & 1) << (lx - 1 - b);
        hsh[p] = std::max(0, etot - he[k]);
    }
    e.scale = finite ? ldexp(1.0, etot - FX_BITS + lx / 2 + lzz / 2 - lx - lzz) : NAN;
    RICH_CUDA(cudaMalloc(&tmp.t, o_f + sizeof(wq) * (size_t)npts));
    char* d = (char*)tmp.t;
    RICH_CUDA(cudaMemcpyAsync(d, hb.data(), o_f, cudaMemcpyHostToDevice, st));
    e.twx = d; e.twz = (cw*)d + px; e.norm = d + o_norm; e.colsh = (int*)(d + o_sh); e.filt = d + o_f;
    rich_count_launch(); k_filter_table<<<nb(npts), 256, 0, st>>>(lx, lzz, c, (int*)(d + o_e), (wq*)e.filt);
    RICH_CUDA(cudaGetLastError());
    RICH_CUDA(cudaStreamSynchronize(st));
    e.tab = tmp.t; tmp.t = nullptr;
    if (ctx->spectra.size() >= 16) {               // bounded cache: drop the oldest
        cudaFree(ctx->spectra.front().tab);
        ctx->spectra.erase(ctx->spectra.begin());
    }
    ctx->spectra.push_back(e);
    *out = &ctx->spectra.back();
    if (min_ratio) *min_ratio = e.min_ratio;
    return 0;
}

// smallest power-of-two torus of at least twice the grid per side whose
// circulant spectrum has no eigenvalue below -1e-12 max (doubled up to 3 times)
static int choose_torus(rich_ctx* ctx, int nx, int nz, const rich_field_t* fd, cudaStream_t st,
                        int* px, int* pz) {
    const double h = 1.0 / nz;
    int a = 1, b = 1;
    while (a < 2 * nx) a <<= 1;
    while (b < 2 * nz) b <<= 1;
    for (int tries = 0; tries < 4; ++tries) {
        const rich_spectrum* e = nullptr;
        double ratio = 0;
        if (int r = spectrum_on(ctx, a, b, h, fd, st, &e, &ratio)) return r;
        if (ratio >= -1e-12 || tries == 3) { *px = a; *pz = b; return 0; }
        a *= 2; b *= 2;
    }
    return RICH_ERR_INVALID;
}

static int ensure_work(rich_ctx* ctx, size_t bytes) {
    if (ctx->field_work && ctx->field_work_bytes >= bytes) return 0;
    if (ctx->field_work) cudaFree(ctx->field_work);
    ctx->field_work = nullptr; ctx->field_work_bytes = 0;
    cudaError_t e = cudaMalloc(&ctx->field_work, bytes);
    if (e != cudaSuccess) { cudaGetLastError(); return RICH_ERR_OOM; }
    ctx->field_work_bytes = bytes;
    return 0;
}

constexpr int PAIR_LOG = 12;                // two rows of 4096 points fit a block, two of 8192 do not

// log2 of the lines of n points a block takes: 2048 points (8 a thread, 36 KB of
// shared memory), fewer while that leaves SMs without a block; at least `least`
// where `bytes` hold them, and no more than `most`
static int log_lines(const rich_ctx* ctx, int logn, long long lines, int least, int most, long long bytes) {
    int l = std::max(11 - logn, least);
    while (l > 0 && (16ll << (logn + l)) > bytes) --l;
    while (l > least && logn + l > 8 && (lines >> l) < ctx->sm_count) --l;
    return std::min(l, most);
}

static size_t row_smem(int logn, int loglpb) {
    return sizeof(fx2) * ((size_t)((1 << logn) + ((1 << logn) >> 3)) << loglpb);
}

template <typename K>
static int allow_smem(K kernel, size_t bytes) {
    if (bytes > (48u << 10))
        RICH_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    return 0;
}

// FFT-MA of one packed pair of fields for cs samples in `work` ([cs][pz][px]):
// the window's nx x nz cells to re and im (im null: that lane is not wanted).
// A pair's first member leaves the second one's noise in `noise` (PAIR_FINE; see
// k_noise_rows).
enum { SINGLE, PAIR_FINE, PAIR_COARSE };
static int fftma(rich_ctx* ctx, const rich_spectrum* sp, fx2* work, int cs, uint64_t seed, uint32_t level,
                 int64_t first, const int64_t* first_dev, uint32_t fld0, int role, fx2* noise, int nx, int nz,
                 double inv_sigma, const PackTr& tr, double* re, double* im, cudaStream_t st) {
    const int lx = ilog2(sp->px), lz = ilog2(sp->pz), lnx = ilog2(nx), lnz = ilog2(nz);
    RowArgs A{};
    A.lines = (long long)cs << lz;
    A.logpx = lx; A.logpz = lz; A.loglpb = log_lines(ctx, lx, A.lines, role == PAIR_FINE ? 1 : 0, 11, 128 << 10);
    A.seed = seed; A.level = level; A.fld0 = fld0; A.im = im != nullptr; A.first = first; A.first_dev = first_dev;
    A.norm = (const NormTab*)sp->norm; A.tw = (const cw*)sp->twx; A.out = work;
    // (the finer torus has rows of twice this one's length)
    const bool shared = role == PAIR_FINE ? A.loglpb > 0 : role == PAIR_COARSE && lx + 1 <= PAIR_LOG;
    A.coarse = shared ? noise : nullptr;
    size_t smem = row_smem(lx, A.loglpb);
    auto* rows = role != PAIR_COARSE ? k_noise_rows<FINE> : shared ? k_noise_rows<LOADED> : k_noise_rows<COARSE>;
    if (int e = allow_smem(rows, smem)) return e;
    rich_count_launch();
    rows<<<(unsigned)((A.lines + (1ll << A.loglpb) - 1) >> A.loglpb), FT, smem, st>>>(A);
    // columns: eight side by side fill a 128-byte line
    const int lc = log_lines(ctx, lz, (long long)cs << lx, std::min(3, lx), lx, 64 << 10);
    smem = sizeof(fx2) << (lz + lc);
    if (int e = allow_smem(k_columns, smem)) return e;
    rich_count_launch();
    k_columns<<<(unsigned)((long long)cs << (lx - lc)), FT, smem, st>>>(lx, lz, lc, nz, (const cw*)sp->twz,
                                                                       (const wq*)sp->filt, work);
    const long long wl = (long long)cs << lnz;
    const int lw = log_lines(ctx, lx, wl, 0, 11, 128 << 10);
    smem = row_smem(lx, lw);
    if (int e = allow_smem(k_rows_window, smem)) return e;
    rich_count_launch();
    k_rows_window<<<(unsigned)((wl + (1ll << lw) - 1) >> lw), FT, smem, st>>>(
        wl, lx, lz, lw, lnx, lnz, (const cw*)sp->twx, sp->colsh, sp->scale, work, inv_sigma, tr,
        ((const NormTab*)sp->norm)->phi, re, im);
    RICH_CUDA(cudaGetLastError());
    return 0;
}

constexpr size_t CHUNK_BYTES = 512ull << 20;

// one packed pair of fields: noise streams fld0, fld0 + 1, their marginal
// transforms and [S][nz>>c][nx>>c] outputs (out_im null: im lane unused)
struct Pack {
    uint32_t fld0;
    PackTr tr;
    double* out_re;
    double* out_im;
};

// FFT-MA draws of npk packed pairs per sample, chunked over samples so the
// complex work buffer stays within CHUNK_BYTES
static int packs_device(rich_ctx* ctx, const rich_field_t* fd, int nx, int nz, uint32_t level,
                        int64_t first, int S, int coarsen, int npk, const Pack* pk, cudaStream_t st,
                        const int64_t* first_dev) {
    if (!pow2(nx) || !pow2(nz) || coarsen < 0 || (nx >> coarsen) < 1 || (nz >> coarsen) < 1 ||
        bad_field(fd))
        return RICH_ERR_INVALID;
    if (S == 0) return 0;
    int px = 0, pz = 0;
    if (int e = choose_torus(ctx, nx, nz, fd, st, &px, &pz)) return e;
    const rich_spectrum* sp = nullptr;
    if (int e = spectrum_on(ctx, px, pz, 1.0 / nz, fd, st, &sp, nullptr)) return e;
    const int npts = px * pz;
    const size_t per = (size_t)npts * sizeof(fx2) + (coarsen ? 32 * (size_t)nx * nz : 0);
    const int chunk = (int)std::max<size_t>(1, CHUNK_BYTES / per);
    if (int e = ensure_work(ctx, per * std::min(chunk, S))) return e;
    fx2* work = (fx2*)ctx->field_work;
    const int cap = std::min(chunk, S);
    double* tmp = (double*)(work + (size_t)npts * cap);   // [cap][4][nz][nx] real scratch
    const int nxo = nx >> coarsen, nzo = nz >> coarsen;
    const double inv_sigma = 1.0 / sqrt(fd->sigma2);
    for (int s0 = 0; s0 < S; s0 += cap) {
        int cs = std::min(cap, S - s0);
        for (int k = 0; k < npk; ++k) {
            const Pack& P = pk[k];
            // real scratch: two ping-pong pairs of [cs][nz][nx] arrays
            const size_t blk = (size_t)cs * nx * nz;
            double* bl[2] = {tmp, tmp + 2 * blk};
            double* ba[2] = {tmp + blk, tmp + 3 * blk};
            const bool im = P.out_im != nullptr;
            double* wl = coarsen ? bl[0] : P.out_re + (size_t)s0 * nx * nz;
            double* wa = !im ? nullptr : coarsen ? ba[0] : P.out_im + (size_t)s0 * nx * nz;
            if (int e = fftma(ctx, sp, work, cs, fd->seed, level, first + s0, first_dev, P.fld0, SINGLE, nullptr, nx,
                              nz, inv_sigma, P.tr, wl, wa, st))
                return e;
            int cx = nx, cz = nz, cur = 0;
            for (int c = 0; c < coarsen; ++c) {
                int ncx = cx / 2, ncz = cz / 2;
                bool last = c == coarsen - 1;
                double* ol = last ? P.out_re + (size_t)s0 * nxo * nzo : bl[1 - cur];
                double* oa = !im ? nullptr : last ? P.out_im + (size_t)s0 * nxo * nzo : ba[1 - cur];
                rich_count_launch();
                k_avg2<<<nb((long long)cs * ncx * ncz), 256, 0, st>>>(cs, ncx, ncz, bl[cur], im ? ba[cur] : nullptr,
                                                                       ol, oa);
                cur = 1 - cur;
                cx = ncx; cz = ncz;
            }
        }
    }
    RICH_CUDA(cudaGetLastError());
    return 0;
}

int rich_fields_device(rich_ctx* ctx, const rich_field_t* fd, int nx, int nz, uint32_t level,
                       int64_t first, int S, int coarsen, double* lnKs, double* alpha,
                       cudaStream_t st, const int64_t* first_dev) {
    const Pack pk{0u, PackTr{0, 0.0, 0.0, fd->alpha_lo, fd->alpha_span}, lnKs, alpha};
    return packs_device(ctx, fd, nx, nz, level, first, S, coarsen, 1, &pk, st, first_dev);
}

// The five soil fields (Table soilparams): streams 0/1 ln Ks (lnks_mean + Z)
// and alpha, 2/3 n and theta_s, 4 theta_r (the im lane of the last pack
// unused); theta fields are skipped when their outputs are null
int rich_soil_device(rich_ctx* ctx, const rich_field_t* fd, const rich_soil_model_t* sm, int nx, int nz,
                     uint32_t level, int64_t first, int S, int coarsen, const rich_soil_t* out,
                     cudaStream_t st) {
    if (!(sm->n_span >= 0) || !(sm->theta_s_span >= 0) || !(sm->theta_r_span >= 0) ||
        !(sm->lnks_mean > -700 && sm->lnks_mean < 700))
        return RICH_ERR_INVALID;
    Pack pk[3];
    int npk = 0;
    pk[npk++] = Pack{0u, PackTr{0, sm->lnks_mean, 0.0, fd->alpha_lo, fd->alpha_span}, out->lnKs, out->alpha};
    if (out->theta_s)
        pk[npk++] = Pack{2u, PackTr{1, sm->n_lo, sm->n_span, sm->theta_s_lo, sm->theta_s_span}, out->n, out->theta_s};
    else
        pk[npk++] = Pack{2u, PackTr{1, sm->n_lo, sm->n_span, 0.0, 0.0}, out->n, nullptr};
    if (out->theta_r)
        pk[npk++] = Pack{4u, PackTr{1, sm->theta_r_lo, sm->theta_r_span, 0.0, 0.0}, out->theta_r, nullptr};
    return packs_device(ctx, fd, nx, nz, level, first, S, coarsen, npk, pk, st, nullptr);
}

// one packed pair of fields drawn as a fine/coarse couple: outputs on the
// fine grid (f_*) and on the half grid (c_*); im outputs null: lane unused
struct PairPack {
    uint32_t fld0;
    PackTr tr;
    double *f_re, *f_im, *c_re, *c_im;
};

// Fine fields on nx x nz and coarse fields on (nx/2) x (nz/2) from one draw by
// covariance upscaling (Appendix A, Eqs. averaging, cov_upscale): the coarse
// white noise is half the 2x2 sums of the fine noise on the torus, filtered
// with the coarse grid's own spectrum on the half-size torus.
static int pair_packs_device(rich_ctx* ctx, const rich_field_t* fd, int nx, int nz, uint32_t level,
                             int64_t first, int S, int npk, const PairPack* pk, cudaStream_t st) {
    if (!pow2(nx) || !pow2(nz) || nx < 2 || nz < 2 || bad_field(fd))
        return RICH_ERR_INVALID;
    if (S == 0) return 0;
    int px = 0, pz = 0;
    if (int e = choose_torus(ctx, nx, nz, fd, st, &px, &pz)) return e;
    const rich_spectrum *spf = nullptr, *spc = nullptr;
    if (int e = spectrum_on(ctx, px, pz, 1.0 / nz, fd, st, &spf, nullptr)) return e;
    if (int e = spectrum_on(ctx, px / 2, pz / 2, 2.0 / nz, fd, st, &spc, nullptr)) return e;
    // spectrum_on may reallocate the cache vector: look both up again
    spectrum_on(ctx, px, pz, 1.0 / nz, fd, st, &spf, nullptr);
    spectrum_on(ctx, px / 2, pz / 2, 2.0 / nz, fd, st, &spc, nullptr);
    const int npf = px * pz;
    const size_t per = (size_t)(npf + npf / 4) * sizeof(fx2);
    const int cap = (int)std::min<size_t>((size_t)S, std::max<size_t>(1, CHUNK_BYTES / per));
    if (int e = ensure_work(ctx, per * cap)) return e;
    fx2* work = (fx2*)ctx->field_work;         // the two members take turns
    fx2* noise = work + (size_t)npf * cap;
    const double inv_sigma = 1.0 / sqrt(fd->sigma2);
    const int ncx = nx / 2, ncz = nz / 2;
    for (int s0 = 0; s0 < S; s0 += cap) {
        int cs = std::min(cap, S - s0);
        for (int k = 0; k < npk; ++k) {
            const PairPack& P = pk[k];
            const size_t of = (size_t)s0 * nx * nz, oc = (size_t)s0 * ncx * ncz;
            if (int e = fftma(ctx, spf, work, cs, fd->seed, level, first + s0, nullptr, P.fld0, PAIR_FINE, noise,
                              nx, nz, inv_sigma, P.tr, P.f_re + of, P.f_im ? P.f_im + of : nullptr, st))
                return e;
            if (int e = fftma(ctx, spc, work, cs, fd->seed, level, first + s0, nullptr, P.fld0, PAIR_COARSE, noise,
                              ncx, ncz, inv_sigma, P.tr, P.c_re + oc, P.c_im ? P.c_im + oc : nullptr, st))
                return e;
        }
    }
    RICH_CUDA(cudaGetLastError());
    return 0;
}

int rich_fields_pair_device(rich_ctx* ctx, const rich_field_t* fd, int nx, int nz, uint32_t level,
                            int64_t first, int S, double* lk_f, double* al_f, double* lk_c,
                            double* al_c, cudaStream_t st) {
    const PairPack pk{0u, PackTr{0, 0.0, 0.0, fd->alpha_lo, fd->alpha_span}, lk_f, al_f, lk_c, al_c};
    return pair_packs_device(ctx, fd, nx, nz, level, first, S, 1, &pk, st);
}

// the five soil fields as covariance-upscaled fine/coarse couples (theta
// outputs may be null: not drawn)
int rich_soil_pair_device(rich_ctx* ctx, const rich_field_t* fd, const rich_soil_model_t* sm, int nx, int nz,
                          uint32_t level, int64_t first, int S, const rich_soil_t* fine,
                          const rich_soil_t* coarse, cudaStream_t st) {
    PairPack pk[3];
    int npk = 0;
    pk[npk++] = PairPack{0u, PackTr{0, sm->lnks_mean, 0.0, fd->alpha_lo, fd->alpha_span}, fine->lnKs, fine->alpha,
                         coarse->lnKs, coarse->alpha};
    const bool ts = fine->theta_s && coarse->theta_s;
    pk[npk++] = PairPack{2u, PackTr{1, sm->n_lo, sm->n_span, ts ? sm->theta_s_lo : 0.0, ts ? sm->theta_s_span : 0.0},
                         fine->n, ts ? fine->theta_s : nullptr, coarse->n, ts ? coarse->theta_s : nullptr};
    if (fine->theta_r && coarse->theta_r)
        pk[npk++] = PairPack{4u, PackTr{1, sm->theta_r_lo, sm->theta_r_span, 0.0, 0.0}, fine->theta_r, nullptr,
                             coarse->theta_r, nullptr};
    return pair_packs_device(ctx, fd, nx, nz, level, first, S, npk, pk, st);
}

// 2x2 block means of both fields (the coarse member of an MLMC pair; al and
// alc may be null)
int rich_fields_average(rich_ctx* ctx, int S, int nx, int nz, const double* lk, const double* al,
                        double* lkc, double* alc, cudaStream_t st) {
    (void)ctx;
    if (nx % 2 || nz % 2) return RICH_ERR_INVALID;
    if (S == 0) return 0;
    const int ncx = nx / 2, ncz = nz / 2;
    rich_count_launch();
    k_avg2<<<nb((long long)S * ncx * ncz), 256, 0, st>>>(S, ncx, ncz, lk, al, lkc, alc);
    RICH_CUDA(cudaGetLastError());
    return 0;
}

// Randomized fit of the inverse-Hessian symbol expansion and its application
// as a preconditioner (sm_103a, FP64).
//
// probe_fit (Sec. 1.4): with x_j = H y_j, the columns of the least-squares
// problem are (B_i x_j)(x) = alpha_lam(x) * IFFT[beta_m(k) FFT(x_j)](x),
// i = (lam, m), m = (angular a, radial q).  One batched D2Z transform of the
// p zero-padded trials, one multiply + batched Z2D transform per distinct k
// multiplier beta_m; then the least-squares problem min ||A c - y|| over the
// rows of all trials is solved through a QR factorisation of A in FP64 by
// CholeskyQR2 (Cholesky QR with one reorthogonalisation):
//     pass 1:  A^T A = R1^T R1                       (Cholesky)
//     pass 2:  Q1 = A R1^{-1} row by row, Q1^T Q1 = R2^T R2, z = Q1^T y
//     A = Q R with Q = Q1 R2^{-1}, R = R2 R1:  c = R^{-1} Q^T y = R1^{-1} R2^{-1} R2^{-T} z.
// Up to 64 terms and cond(A) of about 1e5 (1e4 for targets far outside the range of A), pass 2 is replaced by one
// step of iterative refinement with R1 (fit_refine), a pass over the data at a twentieth of its cost: 128^3, 60 terms, 4 pairs 93 -> 39.8 ms.
// The Gram matrix of the reorthogonalised Q1 is within a few units of round-off
// of the identity whenever cond(A) is below about 1e7, so the solution has the
// accuracy of a Householder QR (error ~ cond(A) eps) instead of the
// cond(A)^2 eps of the normal equations M c = A^T y that Sec. 1.4 writes; the
// first Cholesky factorisation fails (PROBE_ERR_STATE) only when A is
// numerically rank deficient.  Gram matrices: P <= 64 -- pass 1 from the sums over the trials at each
// point (k_fit_gram_s), pass 2 (above those conditions) with the columns formed and solved against R1 in shared memory, one row
// per thread (k_fit_gram<true>); P up to 1024 -- [A | y] formed in column-major chunks
// of about 256 MB, R1^{-1} applied row by row, and a tiled FP64 Gram kernel.
// A second pass forms ||y - sum_i c_i B_i x|| / ||y||.
//
// probe_apply_precond (end of Sec. 1.5): one D2Z transform of the image, the spectrum times the
// combined multiplier sum_m c_(lam,m) beta_m(k) of each spatial mode (k_precond_spectra), a batched
// Z2D transform, and out = sum_lam alpha_lam * w_lam.
//
// cuFFT provides the plain FFTs; every other step is a kernel of this file.
#include <cufft.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <tuple>

#include "common.cuh"
#include "handle.h"
#include "internal.h"

namespace probe {

constexpr int kMaxTerms = 1024;   // P = nspatial x nangular x nradial
constexpr int kMaxSmall = 64;     // P <= 64: Gram pairs accumulated in one CTA's registers
constexpr int kMaxSpatial = 32;
constexpr int kMaxAngular = 16;
constexpr int kMaxRadial = 16;
constexpr int kMaxMult = 32;      // nangular * nradial
constexpr int kGramRows = 32;     // rows staged per Gram iteration
constexpr int kGramBlocks = 608;  // 4 CTAs per SM
constexpr int kGqBlocks = 304;    // 2 CTAs of 128 staged rows (100 KB) per SM
constexpr int kRefBlocks = 608;   // k_fit_refine: 4 CTAs per SM
constexpr size_t kGramSmemMax = 100 << 10;  // staged factors of k_fit_gram_s: at least 2 CTAs per SM
constexpr long long kChunkBytes = 256ll << 20;  // large-P path: [A | y] chunk size

struct BasisDev {
    int ndim;
    int n[3];          // interior sizes (z, y, x); 2D uses n[1] = 1
    int Nf[3];         // FFT sizes
    int fp;            // fft pad (y axis unpadded in 2D)
    double h[3];
    int nspatial, nangular, nradial, NM, P;
    int spatial[kMaxSpatial][3];
    int angular[kMaxAngular];
    double L, order;
    long long Nreal, Ncplx, npts;
};

struct FitCache {
    std::map<std::tuple<int, int, int, int, int>, cufftHandle> plans;  // (ndim, Nz, Ny, Nx, kind*batch)
    DevBuf xr, Xc, Wc, w, beta, alpha, part, coef, misc;
    DevBuf gram, L1, L2, chunk;  // CholeskyQR2: Gram matrix, the two Cholesky factors, [A | y] chunk
};

void fit_cache_destroy(probe_t h) {
    if (!h || !h->fit) return;
    for (auto& kv : h->fit->plans) cufftDestroy(kv.second);
    DevBuf* bufs[] = {&h->fit->xr, &h->fit->Xc, &h->fit->Wc, &h->fit->w,  &h->fit->beta, &h->fit->alpha,
                      &h->fit->part, &h->fit->coef, &h->fit->misc, &h->fit->gram, &h->fit->L1, &h->fit->L2,
                      &h->fit->chunk};
    for (DevBuf* b : bufs)
        if (b->p) cudaFree(b->p);
    delete h->fit;
    h->fit = nullptr;
}

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------
__device__ __forceinline__ void unravel(long long i, const BasisDev& B, int& iz, int& iy, int& ix) {
    ix = (int)(i % B.n[2]);
    const long long r = i / B.n[2];
    iy = (int)(r % B.n[1]);
    iz = (int)(r / B.n[1]);
}

__device__ __forceinline__ long long fft_index(const BasisDev& B, int iz, int iy, int ix) {
    const int fpy = (B.ndim == 3) ? B.fp : 0;
    return ((long long)(iz + B.fp) * B.Nf[1] + (iy + fpy)) * B.Nf[2] + (ix + B.fp);
}

// zero-padded FP64 copies of `cnt` interior FP32 fields
__global__ void k_fit_pad(const float* __restrict__ src, double* __restrict__ dst, int cnt, BasisDev B) {
    const long long tot = (long long)cnt * B.npts;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < tot;
         i += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(i / B.npts);
        int iz, iy, ix;
        unravel(i - (long long)j * B.npts, B, iz, iy, ix);
        dst[(long long)j * B.Nreal + fft_index(B, iz, iy, ix)] = (double)src[i];
    }
}

// The k-space factors of one bin of the half (real-FFT) grid: t, the argument of the Chebyshev
// polynomials, |k|^order (0 on the bins that every term maps to zero) and the unit wave vector.
struct KBin {
    double t, kpow, uz, uy, ux;
};

__device__ __forceinline__ KBin kbin(const BasisDev& B, long long r) {
    const int hx = B.Nf[2] / 2 + 1;
    const int jx = (int)(r % hx);
    r /= hx;
    const int jy = (int)(r % B.Nf[1]);
    const int jz = (int)(r / B.Nf[1]);
    auto freq = [](int j, int N) { return (j <= (N - 1) / 2) ? j : j - N; };
    const double two_pi = 6.283185307179586476925286766559;
    const double kz = two_pi * freq(jz, B.Nf[0]) / (B.Nf[0] * B.h[0]);
    const double ky = (B.ndim == 3) ? two_pi * freq(jy, B.Nf[1]) / (B.Nf[1] * B.h[1]) : 0.0;
    const double kx = two_pi * jx / (B.Nf[2] * B.h[2]);
    bool nyq = ((B.Nf[0] % 2) == 0 && jz == B.Nf[0] / 2) || ((B.Nf[2] % 2) == 0 && jx == B.Nf[2] / 2);
    if (B.ndim == 3) nyq = nyq || ((B.Nf[1] % 2) == 0 && jy == B.Nf[1] / 2);
    const double kn = sqrt(kz * kz + ky * ky + kx * kx);
    KBin k = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (kn > 0.0 && !nyq) {
        const double inv = 1.0 / kn;
        k.uz = kz * inv;
        k.uy = ky * inv;
        k.ux = kx * inv;
        k.t = (kn - B.L) / (kn + B.L);
        k.kpow = (B.order == -1.0) ? inv : (B.order == 0.0 ? 1.0 : pow(kn, B.order));
    }
    return k;
}

// Angular factor.  2D: cos(q theta), sin(|q| theta) with e^{i theta} = ux + i uz, as the |q|-th
// power of that unit number by repeated squaring (no inverse or direct trigonometric function).  |q| as an
// unsigned number: every index is accepted, and the magnitude of the lowest is no int (as a negative
// one, shifted right, it would never reach zero).
__device__ __forceinline__ double angular_factor(const BasisDev& B, const KBin& k, int ang) {
    if (B.ndim == 2) {
        double c = 1.0, s = 0.0, bc = k.ux, bs = k.uz;
        for (unsigned e = ang < 0 ? 0u - (unsigned)ang : (unsigned)ang; e; e >>= 1) {
            if (e & 1) {
                const double t = c * bc - s * bs;
                s = c * bs + s * bc;
                c = t;
            }
            const double t = bc * bc - bs * bs;
            bs = 2.0 * bc * bs;
            bc = t;
        }
        return ang >= 0 ? c : s;
    }
    switch (ang) {
        case 0: return 1.0;
        case 1: return k.ux * k.uy;
        case 2: return k.uy * k.uz;
        case 3: return k.ux * k.uz;
        case 4: return k.ux * k.ux - k.uy * k.uy;
        default: return 3.0 * k.uz * k.uz - 1.0;
    }
}

// beta_m(k) for every multiplier m = a * nradial + q on the half (real-FFT) grid.
// Bound by FP64 arithmetic (two FP64 lanes per SM and clock).  One thread forms all multipliers of
// a bin: the geometry once per bin, the radial functions by the Chebyshev recurrence
// T_{q+1} = 2 t T_q - T_{q-1}, the angular ones by products.  12 multipliers of a 160^3 transform:
// 0.40 ms (the 200 MB written are 0.03 ms of it); cos(q acos t), atan2 and pow evaluated for every
// multiplier took 10.4 ms.
__global__ void k_fit_beta(double* __restrict__ beta, BasisDev B) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < B.Ncplx;
         i += (long long)gridDim.x * blockDim.x) {
        const KBin k = kbin(B, i);
        for (int a = 0; a < B.nangular; ++a) {
            const double A = angular_factor(B, k, B.angular[a]) * k.kpow;
            double t0 = 1.0, t1 = k.t;
            for (int q = 0; q < B.nradial; ++q) {
                beta[(long long)(a * B.nradial + q) * B.Ncplx + i] = A * t0;
                const double t2 = fma(2.0 * k.t, t1, -t0);
                t0 = t1;
                t1 = t2;
            }
        }
    }
}

// Preconditioner spectra: out[lam][k] = X[k] / N * sum_m c[lam * NM + m] beta_m(k), the multipliers
// formed in registers from the bin's geometry (no beta or gamma table in memory).  c holds the
// coefficients with nradial padded to NQ by zeros, [lam][a][NQ].  Bound by FP64 arithmetic; one
// pass over X and the output.  60 terms (5 modes x 12) of a 288^3 transform: 3.2 ms; with a table of
// the 12 multipliers (58 ms), a table of the 5 combinations (1.3 ms) and a product pass, 60 ms.
constexpr int kLamBlock = 4;  // spatial modes summed per walk over the angular factors
template <int NQ>
__global__ void __launch_bounds__(256) k_precond_spectra(const double2* __restrict__ X, const double* __restrict__ c,
                                                         double2* __restrict__ out, BasisDev B, double invN) {
    extern __shared__ double cs[];  // [nspatial rounded up to kLamBlock][nangular][NQ]
    const int nl = (B.nspatial + kLamBlock - 1) / kLamBlock * kLamBlock;
    for (int i = threadIdx.x; i < nl * B.nangular * NQ; i += blockDim.x) {
        const int q = i % NQ, la = i / NQ;
        cs[i] = (q < B.nradial && la < B.nspatial * B.nangular) ? c[la * B.nradial + q] : 0.0;
    }
    __syncthreads();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < B.Ncplx;
         i += (long long)gridDim.x * blockDim.x) {
        const KBin k = kbin(B, i);
        double T[NQ];
        T[0] = 1.0;
        if (NQ > 1) T[1] = k.t;
#pragma unroll
        for (int q = 2; q < NQ; ++q) T[q] = fma(2.0 * k.t, T[q - 1], -T[q - 2]);
        const double sc = k.kpow * invN;
        const double2 x = X[i];
        for (int l0 = 0; l0 < B.nspatial; l0 += kLamBlock) {
            double g[kLamBlock] = {0.0, 0.0, 0.0, 0.0};
            for (int a = 0; a < B.nangular; ++a) {
                const double A = angular_factor(B, k, B.angular[a]);
#pragma unroll
                for (int l = 0; l < kLamBlock; ++l) {
                    if (l0 + l >= B.nspatial) break;
                    const double* cl = cs + ((l0 + l) * B.nangular + a) * NQ;
                    double s = cl[0];
#pragma unroll
                    for (int q = 1; q < NQ; ++q) s = fma(cl[q], T[q], s);
                    g[l] = fma(A, s, g[l]);
                }
            }
#pragma unroll
            for (int l = 0; l < kLamBlock; ++l)
                if (l0 + l < B.nspatial) {
                    const double v = g[l] * sc;
                    out[(long long)(l0 + l) * B.Ncplx + i] = make_double2(v * x.x, v * x.y);
                }
        }
    }
}

// alpha tables: alpha[lam][axis][i] (axis order z, y, x; unused axes hold 1)
__global__ void k_fit_alpha(double* __restrict__ alpha, BasisDev B, int nmax) {
    const long long tot = (long long)B.nspatial * 3 * nmax;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < tot;
         i += (long long)gridDim.x * blockDim.x) {
        const int lam = (int)(i / (3 * nmax));
        const int rem = (int)(i - (long long)lam * 3 * nmax);
        const int ax = rem / nmax, idx = rem % nmax;
        const int n = B.n[ax];
        const int k = (B.ndim == 2) ? (ax == 0 ? B.spatial[lam][0] : (ax == 2 ? B.spatial[lam][1] : 0))
                                    : B.spatial[lam][ax];
        const double two_pi = 6.283185307179586476925286766559;
        double v = 1.0;
        if (idx < n && k != 0)
            v = (k > 0) ? cos(two_pi * k * idx / n) : sin(two_pi * (-k) * idx / n);
        alpha[i] = v;
    }
}

// out[c][j][k] = mult[c or 0][k] * X[j][k] / N  for the spectra of cnt fields
__global__ void k_fit_mult(const double2* __restrict__ X, const double* __restrict__ mult, double2* __restrict__ out,
                           int nmult, int cnt, long long Ncplx, double invN) {
    const long long tot = (long long)nmult * cnt * Ncplx;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < tot;
         i += (long long)gridDim.x * blockDim.x) {
        const long long k = i % Ncplx;
        const long long mj = i / Ncplx;
        const int j = (int)(mj % cnt);
        const int m = (int)(mj / cnt);
        const double b = mult[(long long)m * Ncplx + k] * invN;
        const double2 x = X[(long long)j * Ncplx + k];
        out[i] = make_double2(b * x.x, b * x.y);
    }
}

__device__ __forceinline__ double alpha_at(const double* __restrict__ alpha, int nmax, int lam, int iz, int iy, int ix) {
    const double* a = alpha + (long long)lam * 3 * nmax;
    return a[iz] * a[nmax + iy] * a[2 * nmax + ix];
}

// Small-P path (P <= 64), pass 1 of CholeskyQR2.  Column i = (lam, m) of A is alpha_lam(x) w_m(j, x),
// so  (A^T A)_{(l,m),(l',m')} = sum_x alpha_l alpha_l' S_mm'(x),  S_mm'(x) = sum_j w_m(j,x) w_m'(j,x),
// and (A^T y)_{(l,m)} = sum_x alpha_l sum_j w_m y.  Forming the trial sums S once per point and then
// the (spatial pair) x (multiplier pair) sums needs about P^2/4 + p NM^2/2 multiply-adds per point
// instead of p P^2/2.  Bound by FP64 arithmetic (two lanes per SM and clock).  128^3 points,
// P = 60 (5 x 12), p = 4: 6.9 ms; 28.6 ms with every pair of columns summed over every row.
// Taken with two or more spatial modes (with one, nothing is shared) and while the staged factors
// leave two CTAs per SM.
// "left" factors of a point: the ns (ns + 1) / 2 products alpha_l alpha_l' (l <= l'), the ns
// alphas, and 1; "right" factors: S_mm' (m <= m'), sum_j w_m y, sum_j y^2.  Outputs: pairs x pairs,
// then alphas x (w y), then y^2.  partial[CTA][output].
struct GramPlan {
    int na2, ns2, nl, nr, nout;  // pair counts, left and right factors, outputs
};
__host__ __device__ inline GramPlan gram_plan(const BasisDev& B) {
    GramPlan g;
    g.na2 = B.nspatial * (B.nspatial + 1) / 2;
    g.ns2 = B.NM * (B.NM + 1) / 2;
    g.nl = g.na2 + B.nspatial + 1;
    g.nr = g.ns2 + B.NM + 1;
    g.nout = g.na2 * g.ns2 + B.P + 1;
    return g;
}
// e-th pair (a, b), a <= b < n, in row order
__host__ __device__ inline void pair_of(int e, int n, int& a, int& b) {
    a = 0;
    while (e >= n - a) e -= n - a, ++a;
    b = a + e;
}
constexpr int kGramOut = 7;  // outputs per thread: nout <= 7 * 256 for every P <= 64

size_t gram_s_smem(const BasisDev& B) {
    const GramPlan g = gram_plan(B);
    return (size_t)kGramRows * (g.nl + g.nr + B.NM + 1) * 8;
}

__global__ void __launch_bounds__(256) k_fit_gram_s(const double* __restrict__ w, const float* __restrict__ y,
                                                    const double* __restrict__ alpha, int nmax, int p, BasisDev B,
                                                    double* __restrict__ partial) {
    extern __shared__ double sm[];
    const GramPlan g = gram_plan(B);
    double* left = sm;                                   // [nl][kGramRows]
    double* right = left + g.nl * kGramRows;             // [nr][kGramRows]
    double* wv = right + g.nr * kGramRows;               // [NM + 1][kGramRows]: w_m(j, .), y_j
    __shared__ long long fidx[kGramRows];
    __shared__ unsigned char pa[kMaxSpatial * (kMaxSpatial + 1) / 2][2], pm[(kMaxMult + 1) * (kMaxMult + 2) / 2][2];
    const int tid = threadIdx.x;
    for (int e = tid; e < g.na2; e += 256) {
        int a, b;
        pair_of(e, B.nspatial, a, b);
        pa[e][0] = (unsigned char)a, pa[e][1] = (unsigned char)b;
    }
    for (int e = tid; e < g.nr; e += 256) {  // right factor e: staged rows whose product it sums
        int a, b;
        if (e < g.ns2)
            pair_of(e, B.NM, a, b);
        else
            a = (e < g.ns2 + B.NM) ? e - g.ns2 : B.NM, b = B.NM;
        pm[e][0] = (unsigned char)a, pm[e][1] = (unsigned char)b;
    }
    int lo[kGramOut], ro[kGramOut];
    double acc[kGramOut];
#pragma unroll
    for (int k = 0; k < kGramOut; ++k) {
        const int t = tid + 256 * k;
        int a = g.nl - 1, r = g.nr - 1;  // y^2 (also the idle slots: in bounds, not written)
        if (t < g.na2 * g.ns2)
            a = t / g.ns2, r = t % g.ns2;
        else if (t < g.na2 * g.ns2 + B.P)
            a = g.na2 + (t - g.na2 * g.ns2) / B.NM, r = g.ns2 + (t - g.na2 * g.ns2) % B.NM;
        lo[k] = a * kGramRows;
        ro[k] = r * kGramRows;
        acc[k] = 0.0;
    }
    const long long wstride = (long long)p * B.Nreal;
    const int lane = tid & (kGramRows - 1), grp = tid / kGramRows;
    for (long long x0 = (long long)blockIdx.x * kGramRows; x0 < B.npts; x0 += (long long)gridDim.x * kGramRows) {
        __syncthreads();
        const bool in = x0 + lane < B.npts;
        int iz = 0, iy = 0, ix = 0;
        if (in) unravel(x0 + lane, B, iz, iy, ix);
        if (grp == 0) fidx[lane] = in ? fft_index(B, iz, iy, ix) : -1;
        for (int l = grp; l < B.nspatial; l += 256 / kGramRows)
            left[(g.na2 + l) * kGramRows + lane] = in ? alpha_at(alpha, nmax, l, iz, iy, ix) : 0.0;
        if (grp == 1) left[(g.nl - 1) * kGramRows + lane] = 1.0;
        __syncthreads();
        for (int e = grp; e < g.na2; e += 256 / kGramRows)
            left[e * kGramRows + lane] =
                left[(g.na2 + pa[e][0]) * kGramRows + lane] * left[(g.na2 + pa[e][1]) * kGramRows + lane];
        for (int j = 0; j < p; ++j) {
            const long long q = fidx[lane];
            for (int m = grp; m <= B.NM; m += 256 / kGramRows)
                wv[m * kGramRows + lane] =
                    q < 0 ? 0.0
                          : (m < B.NM ? w[(long long)m * wstride + (long long)j * B.Nreal + q]
                                      : (double)y[(long long)j * B.npts + x0 + lane]);
            __syncthreads();
            for (int e = grp; e < g.nr; e += 256 / kGramRows) {
                const double v = wv[pm[e][0] * kGramRows + lane], u = wv[pm[e][1] * kGramRows + lane];
                double* s = right + e * kGramRows + lane;
                *s = (j == 0) ? v * u : fma(v, u, *s);
            }
            __syncthreads();
        }
        // left and right factors of 32 points are staged: their outer product, summed.  The point
        // index is skewed by the lane so that a warp's lanes read different banks.
#pragma unroll
        for (int k = 0; k < kGramOut; ++k) {
            if (tid + 256 * k >= g.nout) break;
            double a = acc[k];
#pragma unroll 8
            for (int r = 0; r < kGramRows; ++r) {
                const int x = (r + tid) & (kGramRows - 1);
                a = fma(left[lo[k] + x], right[ro[k] + x], a);
            }
            acc[k] = a;
        }
    }
#pragma unroll
    for (int k = 0; k < kGramOut; ++k)
        if (tid + 256 * k < g.nout) partial[(long long)blockIdx.x * g.nout + tid + 256 * k] = acc[k];
}

// The sum of one value over nblocks partials (stride apart) by a warp, in a fixed order.
__device__ __forceinline__ double warp_sum_partials(const double* part, int nblocks, long long stride) {
    double s = 0.0;
    for (int b = threadIdx.x & 31; b < nblocks; b += 32) s += part[(long long)b * stride];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// k_fit_gram_s's outputs summed over the CTAs into the dense lower triangle of C (n x n, n = P + 1).
__global__ void k_fit_out_to_C(const double* __restrict__ partial, int nblocks, BasisDev B, double* __restrict__ C) {
    const GramPlan g = gram_plan(B);
    const int n = B.P + 1;
    for (int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < g.nout; t += (gridDim.x * blockDim.x) >> 5) {
        const double s = warp_sum_partials(partial + t, nblocks, g.nout);
        if (threadIdx.x & 31) continue;
        if (t < g.na2 * g.ns2) {
            int l, l2, m, m2;
            pair_of(t / g.ns2, B.nspatial, l, l2);
            pair_of(t % g.ns2, B.NM, m, m2);
            const int i = l * B.NM + m, k = l2 * B.NM + m2, i2 = l * B.NM + m2, k2 = l2 * B.NM + m;
            C[(long long)max(i, k) * n + min(i, k)] = s;
            C[(long long)max(i2, k2) * n + min(i2, k2)] = s;
        } else {
            C[(long long)B.P * n + (t - g.na2 * g.ns2)] = s;  // A^T y, then y^T y on the diagonal
        }
    }
}

// Small-P path, all column pairs over all rows: per-CTA partial sums of the upper triangle of
// [A y]^T [A y] (pairs (i, k), i <= k <= P) or, with QPASS (pass 2 of CholeskyQR2), of [Q1 y]^T [Q1 y]
// with Q1 = A R1^{-1} = A L1^{-T}.  Bound by FP64 arithmetic: P^2/2 multiply-adds per row for the
// sums and as many again for the triangular solve.  A CTA stages 128 rows, one per thread; each
// thread forms its row's columns and solves its own row (eight columns at a time in registers, the
// factor broadcast from shared memory, the diagonal as reciprocals), so the solve needs no
// communication; then each thread sums up to 17 pairs over the 128 rows.  Pass 1 uses this kernel
// where the staged factors of k_fit_gram_s would not fit (few spatial modes, many multipliers).
// Pass 2 of the fit above: 55.4 ms, 0.96 of the FP64 rate of the sums (28.6 ms) and as many
// multiply-adds again; 149 ms when eight threads shared a row's solve through shuffles.
constexpr int kGqRows = 128, kGqPitch = kMaxSmall + 1;
constexpr int kGqPairs = ((kMaxSmall + 1) * (kMaxSmall + 2) / 2 + kGqRows - 1) / kGqRows;
constexpr size_t kGqSmem = (size_t)(kGqRows * kGqPitch + kMaxSmall * kMaxSmall + kMaxSmall) * 8;
template <bool QPASS>
__global__ void __launch_bounds__(kGqRows) k_fit_gram(const double* __restrict__ w, const float* __restrict__ y,
                                                      const double* __restrict__ alpha, int nmax, int p, BasisDev B,
                                                      const double* __restrict__ L1, double* __restrict__ partial) {
    extern __shared__ double sm[];
    double* cols = sm;                           // [kGqRows][kGqPitch], y in column kMaxSmall
    double* LT = cols + kGqRows * kGqPitch;      // [i][j] = L1[j][i], zero outside P x P
    double* rinv = LT + kMaxSmall * kMaxSmall;   // 1 / L1[j][j], zero past P
    const int P = B.P, PC = P + 1, tid = threadIdx.x;
    const int npairs = PC * (PC + 1) / 2;
    int ii[kGqPairs], kk[kGqPairs];
    double acc[kGqPairs];
#pragma unroll
    for (int s = 0; s < kGqPairs; ++s) {
        acc[s] = 0.0;
        int a = 0, b = 0;
        if (tid + s * kGqRows < npairs) pair_of(tid + s * kGqRows, PC, a, b);
        ii[s] = (a == P) ? kMaxSmall : a;
        kk[s] = (b == P) ? kMaxSmall : b;
    }
    if (QPASS) {
        for (int t = tid; t < kMaxSmall * kMaxSmall; t += kGqRows) {
            const int i = t / kMaxSmall, j = t % kMaxSmall;
            LT[t] = (i < P && j < P && i <= j) ? L1[(long long)j * P + i] : 0.0;
        }
        if (tid < kMaxSmall) rinv[tid] = tid < P ? 1.0 / L1[(long long)tid * P + tid] : 0.0;
    }
    const long long rows = (long long)p * B.npts;
    const long long wstride = (long long)p * B.Nreal;  // between multipliers
    double* my = cols + tid * kGqPitch;
    for (int c = P; c < kMaxSmall; ++c) my[c] = 0.0;
    __syncthreads();
    for (long long r0 = (long long)blockIdx.x * kGqRows; r0 < rows; r0 += (long long)gridDim.x * kGqRows) {
        const long long row = r0 + tid;
        if (row < rows) {
            const int j = (int)(row / B.npts);
            int iz, iy, ix;
            unravel(row - (long long)j * B.npts, B, iz, iy, ix);
            const double* wp = w + (long long)j * B.Nreal + fft_index(B, iz, iy, ix);
            for (int l = 0; l < B.nspatial; ++l) {
                const double al = alpha_at(alpha, nmax, l, iz, iy, ix);
                for (int m = 0; m < B.NM; ++m) my[l * B.NM + m] = al * wp[(long long)m * wstride];
            }
            my[kMaxSmall] = (double)y[row];
        } else {
            for (int c = 0; c < P; ++c) my[c] = 0.0;
            my[kMaxSmall] = 0.0;
        }
        if (QPASS) {
            for (int jb = 0; jb < P; jb += 8) {
                double q[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) q[c] = my[jb + c];
                for (int i = 0; i < jb; ++i) {
                    const double v = -my[i];
                    const double* l = LT + i * kMaxSmall + jb;
#pragma unroll
                    for (int c = 0; c < 8; ++c) q[c] = fma(v, l[c], q[c]);
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    q[c] *= rinv[jb + c];
                    const double* l = LT + (jb + c) * kMaxSmall + jb;
#pragma unroll
                    for (int d = c + 1; d < 8; ++d) q[d] = fma(-q[c], l[d], q[d]);
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) my[jb + c] = q[c];
            }
        }
        __syncthreads();
#pragma unroll
        for (int s = 0; s < kGqPairs; ++s) {
            if (tid + s * kGqRows >= npairs) break;
            const double *ci = cols + ii[s], *ck = cols + kk[s];
            double a = acc[s];
#pragma unroll 8
            for (int r = 0; r < kGqRows; ++r) a = fma(ci[r * kGqPitch], ck[r * kGqPitch], a);
            acc[s] = a;
        }
        __syncthreads();
    }
#pragma unroll
    for (int s = 0; s < kGqPairs; ++s)
        if (tid + s * kGqRows < npairs) partial[(long long)blockIdx.x * npairs + tid + s * kGqRows] = acc[s];
}

// k_fit_gram's per-CTA pair sums reduced in a fixed order into the dense lower triangle of
// C (n x n, n = P + 1, row-major): C[k][i] = sum (i <= k).
__global__ void k_fit_pairs_to_C(const double* __restrict__ partial, int nblocks, int n, double* __restrict__ C) {
    const int npairs = n * (n + 1) / 2;
    for (int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < npairs; t += (gridDim.x * blockDim.x) >> 5) {
        const double s = warp_sum_partials(partial + t, nblocks, npairs);
        int i, k;
        pair_of(t, n, i, k);
        if ((threadIdx.x & 31) == 0) C[(long long)k * n + i] = s;
    }
}

// [A | y] for stacked rows r0 .. r0 + rc - 1 (row = j * npts + pt) as a column-major FP64 block
// with leading dimension rc: column i < P is (B_i x_j)(pt) = alpha_lam(pt) w_m(j, pt) with
// i = lam * NM + m, column P is y_j(pt).  Rows past the end are zero (they add nothing).
__global__ void k_fit_cols(const double* __restrict__ w, const float* __restrict__ y,
                           const double* __restrict__ alpha, int nmax, int p, BasisDev B, long long r0, int rc,
                           double* __restrict__ A) {
    const long long rows = (long long)p * B.npts;
    const long long wstride = (long long)p * B.Nreal;
    const long long tot = (long long)rc * (B.P + 1);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < tot;
         i += (long long)gridDim.x * blockDim.x) {
        const int col = (int)(i / rc);
        const int r = (int)(i - (long long)col * rc);
        const long long row = r0 + r;
        double v = 0.0;
        if (row < rows) {
            const int j = (int)(row / B.npts);
            int iz, iy, ix;
            unravel(row - (long long)j * B.npts, B, iz, iy, ix);
            if (col < B.P) {
                const int lam = col / B.NM, m = col - lam * B.NM;
                v = alpha_at(alpha, nmax, lam, iz, iy, ix) *
                    w[(long long)m * wstride + (long long)j * B.Nreal + fft_index(B, iz, iy, ix)];
            } else {
                v = (double)y[row];
            }
        }
        A[i] = v;
    }
}

// Gram matrix of a column-major block A (rc rows, n columns, ld rc): tile (ti, tk), ti >= tk, of
// 64 x 64 entries over the rows of slice blockIdx.y; part[slice][i * n + k] for every (i, k) of
// the tile (the diagonal tiles hold both triangles).  256 threads, 4 x 4 entries each.
constexpr int kSyT = 64, kSyR = 32;
__global__ void __launch_bounds__(256) k_fit_syrk(const double* __restrict__ A, int rc, int n, int rows_per_slice,
                                                  double* __restrict__ part) {
    __shared__ double As[kSyR][kSyT + 1], Bs[kSyR][kSyT + 1];
    int t = blockIdx.x, ti = 0;
    while (t > ti) {  // lower tiles in row order: (0,0), (1,0), (1,1), (2,0), ...
        t -= ti + 1;
        ++ti;
    }
    const int tk = t;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int r_beg = blockIdx.y * rows_per_slice, r_end = min(rc, r_beg + rows_per_slice);
    double acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
    for (int r0 = r_beg; r0 < r_end; r0 += kSyR) {
        for (int q = threadIdx.x; q < kSyR * kSyT; q += 256) {
            const int r = q & (kSyR - 1), c = q / kSyR;
            const int row = r0 + r;
            const int ci = ti * kSyT + c, ck = tk * kSyT + c;
            As[r][c] = (row < r_end && ci < n) ? A[(long long)ci * rc + row] : 0.0;
            Bs[r][c] = (row < r_end && ck < n) ? A[(long long)ck * rc + row] : 0.0;
        }
        __syncthreads();
#pragma unroll 4
        for (int r = 0; r < kSyR; ++r) {
            double av[4], bv[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) av[a] = As[r][ty * 4 + a];
#pragma unroll
            for (int b = 0; b < 4; ++b) bv[b] = Bs[r][tx * 4 + b];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = fma(av[a], bv[b], acc[a][b]);
        }
        __syncthreads();
    }
    double* out = part + (long long)blockIdx.y * n * n;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int i = ti * kSyT + ty * 4 + a;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int k = tk * kSyT + tx * 4 + b;
            if (i < n && k < n) out[(long long)i * n + k] = acc[a][b];
        }
    }
}

// C[e] (+)= sum over slices of part[s][e] for the lower triangle, in slice order.
__global__ void k_fit_reduce(const double* __restrict__ part, int nslices, int n, int accumulate,
                             double* __restrict__ C) {
    const long long tot = (long long)n * n;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
         e += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(e / n), k = (int)(e - (long long)i * n);
        if (k > i) continue;
        double s = accumulate ? C[e] : 0.0;
        for (int q = 0; q < nslices; ++q) s += part[(long long)q * tot + e];
        C[e] = s;
    }
}

// Largest diagonal entry of the leading P x P block of S (ld = ld) -> *dmax.
__global__ void k_fit_dmax(const double* __restrict__ S, int ld, int P, double* dmax) {
    double m = 0.0;
    for (int i = threadIdx.x; i < P; i += blockDim.x) m = fmax(m, S[(long long)i * ld + i]);
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    __shared__ double red[8];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmax(m, red[w]);
        *dmax = m;
    }
}

// Step k of the right-looking Cholesky factorisation S = L L^T of the leading P x P block of S
// (lower triangle, ld = ld): CTA 0 writes column k of L (ld P); every CTA applies the rank-one
// update S_ij -= l_ik l_jk to its share of k < j <= i < P.  Column k of S is only read.  A pivot
// below 1e-13 of the largest diagonal entry marks S as not numerically positive definite.
__global__ void k_fit_chol_step(double* __restrict__ S, int ld, int P, int k, const double* __restrict__ dmax,
                                double* __restrict__ L, int* status) {
    const double d = S[(long long)k * ld + k];
    const bool bad = !(d > 1e-13 * (*dmax));
    const double lkk = bad ? 1.0 : sqrt(d);
    const double inv = 1.0 / lkk;
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) {
            L[(long long)k * P + k] = lkk;
            if (bad) *status = 1;
        }
        for (int i = k + 1 + threadIdx.x; i < P; i += blockDim.x) L[(long long)i * P + k] = S[(long long)i * ld + k] * inv;
    }
    const int m = P - k - 1;
    const long long tot = (long long)m * m;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x) {
        const int i = k + 1 + (int)(t / m), j = k + 1 + (int)(t % m);
        if (j > i) continue;
        S[(long long)i * ld + j] -= (S[(long long)i * ld + k] * inv) * (S[(long long)j * ld + k] * inv);
    }
}

// Rows of a column-major block A (rc rows, first P columns) times R^{-1} = L^{-T}, in place:
// q_j = (a_j - sum_{i<j} q_i L_ji) / L_jj, one thread per row.
__global__ void k_fit_trsm_rows(double* __restrict__ A, int rc, int P, const double* __restrict__ L) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= rc) return;
    for (int j = 0; j < P; ++j) {
        const double* Lj = L + (long long)j * P;
        double s = A[(long long)j * rc + r];
        for (int i = 0; i < j; ++i) s = fma(-A[(long long)i * rc + r], Lj[i], s);
        A[(long long)j * rc + r] = s / Lj[j];
    }
}

// One CTA: x = L^{-1} b (trans = 0) or x = L^{-T} b (trans = 1), L lower with ld P; x may alias b.
__global__ void __launch_bounds__(256) k_fit_trsv(const double* __restrict__ L, int P, int trans,
                                                  const double* b, double* x) {
    __shared__ double xs[kMaxTerms];
    __shared__ double red[8];
    for (int i = threadIdx.x; i < P; i += blockDim.x) xs[i] = b[i];
    __syncthreads();
    for (int s = 0; s < P; ++s) {
        const int i = trans ? P - 1 - s : s;
        double part = 0.0;
        if (!trans) {
            for (int j = threadIdx.x; j < i; j += blockDim.x) part = fma(L[(long long)i * P + j], xs[j], part);
        } else {
            for (int j = i + 1 + threadIdx.x; j < P; j += blockDim.x) part = fma(L[(long long)j * P + i], xs[j], part);
        }
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
            xs[i] = (xs[i] - t) / L[(long long)i * P + i];
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < P; i += blockDim.x) x[i] = xs[i];
}

// The refinement step's pass over the data (P <= 64): per-CTA partial sums of g = A^T (y - A c).  At a point x
// the coefficients of the multipliers, d_m = sum_l alpha_l c_lm, serve all its trials, and
// h_m = sum_j w_m(j) r_j is summed before it meets the spatial modes:  g_lm = sum_x alpha_l h_m.  So a
// point costs 2 P + 2 p NM multiply-adds where the reorthogonalising pass (k_fit_gram<true>) needs
// p P^2.  Eight groups of 32 threads take 32 points, a group every eighth multiplier; then thread
// (l, m) sums its output over the points of its quarter.  Bound by FP64 arithmetic and the
// barrier per trial; 128^3 points, P = 60 (5 x 12), p = 4: 2.6 ms against 55.4 ms of the pass it stands
// for (the bytes alone, 0.84 GB of interior columns, would take 0.13 ms).
__global__ void __launch_bounds__(256) k_fit_refine(const double* __restrict__ w, const float* __restrict__ y,
                                                    const double* __restrict__ alpha, int nmax, int p, BasisDev B,
                                                    const double* __restrict__ coef, double* __restrict__ partial) {
    constexpr int NX = 32, PT = NX + 1, MG = kMaxMult / 8;
    __shared__ double cs[kMaxSmall], al[kMaxSpatial][PT], hs[kMaxMult][PT], red[2][8][PT], sums[4][kMaxSmall];
    const int tid = threadIdx.x, lane = tid & (NX - 1), grp = tid / NX;
    const int t = tid & (kMaxSmall - 1), quarter = tid / kMaxSmall;
    const int tl = t / B.NM, tm = t - tl * B.NM;
    const long long wstride = (long long)p * B.Nreal;
    if (tid < B.P) cs[tid] = coef[tid];
    double acc = 0.0;
    for (long long x0 = (long long)blockIdx.x * NX; x0 < B.npts; x0 += (long long)gridDim.x * NX) {
        const bool in = x0 + lane < B.npts;
        int iz = 0, iy = 0, ix = 0;
        if (in) unravel(x0 + lane, B, iz, iy, ix);
        const double* wq = w + fft_index(B, iz, iy, ix);
        double wn[MG];
        float yn = 0.f;
        auto fetch = [&](int j) {
#pragma unroll
            for (int k = 0; k < MG; ++k) {
                const int m = grp + 8 * k;
                wn[k] = (in && m < B.NM) ? wq[(long long)m * wstride + (long long)j * B.Nreal] : 0.0;
            }
            yn = in ? y[(long long)j * B.npts + x0 + lane] : 0.f;
        };
        fetch(0);
        __syncthreads();  // the sums over the last points are done with al and hs
        for (int l = grp; l < B.nspatial; l += 8) al[l][lane] = in ? alpha_at(alpha, nmax, l, iz, iy, ix) : 0.0;
        __syncthreads();
        double d[MG], hm[MG];
#pragma unroll
        for (int k = 0; k < MG; ++k) {
            const int m = grp + 8 * k;
            d[k] = hm[k] = 0.0;
            if (m < B.NM)
                for (int l = 0; l < B.nspatial; ++l) d[k] = fma(al[l][lane], cs[l * B.NM + m], d[k]);
        }
        for (int j = 0; j < p; ++j) {
            double wv[MG], s = 0.0;
            const double yv = (double)yn;
#pragma unroll
            for (int k = 0; k < MG; ++k) {
                wv[k] = wn[k];
                s = fma(d[k], wv[k], s);
            }
            red[j & 1][grp][lane] = s;
            if (j + 1 < p) fetch(j + 1);
            __syncthreads();
            double r = yv;
#pragma unroll
            for (int q = 0; q < 8; ++q) r -= red[j & 1][q][lane];
#pragma unroll
            for (int k = 0; k < MG; ++k) hm[k] = fma(wv[k], r, hm[k]);
        }
#pragma unroll
        for (int k = 0; k < MG; ++k)
            if (grp + 8 * k < B.NM) hs[grp + 8 * k][lane] = hm[k];
        __syncthreads();
        if (t < B.P) {
#pragma unroll
            for (int q = 0; q < NX / 4; ++q) acc = fma(al[tl][quarter * (NX / 4) + q], hs[tm][quarter * (NX / 4) + q], acc);
        }
    }
    sums[quarter][t] = acc;
    __syncthreads();
    if (tid < B.P)
        partial[(long long)blockIdx.x * B.P + tid] = (sums[0][tid] + sums[1][tid]) + (sums[2][tid] + sums[3][tid]);
}

// One CTA: g = the sum of nblocks partials (P <= 64 each), v = L^{-1} g, coef += L^{-T} v, *norm2 = |v|^2.
// Each substitution is one warp's, the unknowns in its registers.  With inv2, warps 2 and 3 meanwhile invert
// L by columns, a column per thread, into the unused half of the staged factor (128^3, P = 60, 4 pairs: no
// difference in the call's 39.8 ms), and inv2[0] + inv2[1] = |L^{-1} D|_F^2, D = diag of L's row norms (the norms of A's columns).
__global__ void __launch_bounds__(256) k_fit_refine_step(const double* __restrict__ partial, int nblocks, int P,
                                                         const double* __restrict__ L, double* __restrict__ coef,
                                                         double* __restrict__ norm2, double* __restrict__ inv2) {
    __shared__ double Ls[kMaxSmall][kMaxSmall + 1], sums[4][kMaxSmall];
    const int tid = threadIdx.x, lane = tid & 31;
    for (int i = tid; i < P * P; i += 256) Ls[i / P][i % P] = L[i];
    const int t = tid & (kMaxSmall - 1), quarter = tid / kMaxSmall;
    double s = 0.0;
    if (t < P)
        for (int b = quarter; b < nblocks; b += 4) s += partial[(long long)b * P + t];
    sums[quarter][t] = s;
    __syncthreads();
    if (inv2 && tid >= 64 && tid < 128) {  // entry (r, t) of the inverse, r >= t, at Ls[t][r + 1]
        double d2 = 0.0, x2 = 0.0;
        if (t < P) {
            for (int k = 0; k <= t; ++k) d2 = fma(Ls[t][k], Ls[t][k], d2);
            for (int r = t; r < P; ++r) {
                double v0 = r == t ? 1.0 : 0.0, v1 = 0.0;
                int k = t;
                for (; k + 1 < r; k += 2) {
                    v0 = fma(-Ls[r][k], Ls[t][k + 1], v0);
                    v1 = fma(-Ls[r][k + 1], Ls[t][k + 2], v1);
                }
                if (k < r) v0 = fma(-Ls[r][k], Ls[t][k + 1], v0);
                const double x = (v0 + v1) / Ls[r][r];
                Ls[t][r + 1] = x;
                x2 = fma(x, x, x2);
            }
        }
        double v = d2 * x2;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) inv2[(tid >> 5) - 2] = v;
    }
    if (tid >= 32) return;
    const int t1 = lane + 32;
    double x0 = (sums[0][lane] + sums[1][lane]) + (sums[2][lane] + sums[3][lane]);
    double x1 = (sums[0][t1] + sums[1][t1]) + (sums[2][t1] + sums[3][t1]);
    for (int i = 0; i < P; ++i) {
        const double xi = __shfl_sync(0xffffffffu, i < 32 ? x0 : x1, i & 31) / Ls[i][i];
        if (lane == i) x0 = xi;
        if (t1 == i) x1 = xi;
        if (lane > i && lane < P) x0 = fma(-Ls[lane][i], xi, x0);
        if (t1 > i && t1 < P) x1 = fma(-Ls[t1][i], xi, x1);
    }
    double v = (lane < P ? x0 * x0 : 0.0) + (t1 < P ? x1 * x1 : 0.0);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) *norm2 = v;
    for (int i = P - 1; i >= 0; --i) {
        const double xi = __shfl_sync(0xffffffffu, i < 32 ? x0 : x1, i & 31) / Ls[i][i];
        if (lane == i) x0 = xi;
        if (t1 == i) x1 = xi;
        if (lane < i) x0 = fma(-Ls[i][lane], xi, x0);
        if (t1 < i) x1 = fma(-Ls[i][t1], xi, x1);
    }
    if (lane < P) coef[lane] += x0;
    if (t1 < P) coef[t1] += x1;
}

// Per-CTA sums of (y - sum_i c_i col_i)^2 and y^2.
__global__ void __launch_bounds__(256) k_fit_resid(const double* __restrict__ w, const float* __restrict__ y,
                                                   const double* __restrict__ alpha, int nmax, int p, BasisDev B,
                                                   const double* __restrict__ coef, double* __restrict__ partial) {
    const long long rows = (long long)p * B.npts;
    const long long wstride = (long long)p * B.Nreal;
    double rr = 0.0, yy = 0.0;
    for (long long row = blockIdx.x * (long long)blockDim.x + threadIdx.x; row < rows;
         row += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(row / B.npts);
        int iz, iy, ix;
        unravel(row - (long long)j * B.npts, B, iz, iy, ix);
        const long long q = (long long)j * B.Nreal + fft_index(B, iz, iy, ix);
        double s = 0.0;
        for (int lam = 0; lam < B.nspatial; ++lam) {
            double t = 0.0;
            for (int m = 0; m < B.NM; ++m) t += coef[lam * B.NM + m] * w[(long long)m * wstride + q];
            s += alpha_at(alpha, nmax, lam, iz, iy, ix) * t;
        }
        const double yv = (double)y[row];
        rr += (yv - s) * (yv - s);
        yy += yv * yv;
    }
    for (int o = 16; o > 0; o >>= 1) {
        rr += __shfl_xor_sync(0xffffffffu, rr, o);
        yy += __shfl_xor_sync(0xffffffffu, yy, o);
    }
    __shared__ double red[2][8];
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = rr;
        red[1][threadIdx.x >> 5] = yy;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, c = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
            a += red[0][i];
            c += red[1][i];
        }
        partial[2 * blockIdx.x] = a;
        partial[2 * blockIdx.x + 1] = c;
    }
}

__global__ void k_fit_resid_final(const double* __restrict__ partial, int nblocks, double* out) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double a = 0.0, c = 0.0;
        for (int i = 0; i < nblocks; ++i) {
            a += partial[2 * i];
            c += partial[2 * i + 1];
        }
        out[0] = c > 0.0 ? sqrt(a / c) : 0.0;
    }
}

// out(x) = sum_lam alpha_lam(x) w_lam(x) on the interior (FP32 result)
__global__ void k_precond_combine(const double* __restrict__ w, const double* __restrict__ alpha, int nmax, BasisDev B,
                                  float* __restrict__ out) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < B.npts;
         i += (long long)gridDim.x * blockDim.x) {
        int iz, iy, ix;
        unravel(i, B, iz, iy, ix);
        const long long q = fft_index(B, iz, iy, ix);
        double s = 0.0;
        for (int lam = 0; lam < B.nspatial; ++lam)
            s += alpha_at(alpha, nmax, lam, iz, iy, ix) * w[(long long)lam * B.Nreal + q];
        out[i] = (float)s;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {

int grid_of(long long n, int cap = 152 * 16) {
    long long b = (n + 255) / 256;
    return (int)std::max(1LL, std::min<long long>(b, cap));
}

probe_status make_basis(probe_t h, const probe_basis* bs, BasisDev& B) {
    if (!bs) return fail(h, PROBE_ERR_ARG, "basis is NULL");
    if (bs->ndim != h->ndim) return fail(h, PROBE_ERR_ARG, "basis ndim differs from the grid's");
    if (bs->nspatial < 1 || bs->nspatial > kMaxSpatial || !bs->spatial)
        return fail(h, PROBE_ERR_ARG, "nspatial must be in [1, 32] with a spatial table");
    if (bs->nangular < 1 || bs->nangular > kMaxAngular || !bs->angular)
        return fail(h, PROBE_ERR_ARG, "nangular must be in [1, 16] with an angular table");
    if (bs->nradial < 1 || bs->nradial > kMaxRadial) return fail(h, PROBE_ERR_ARG, "nradial must be in [1, 16]");
    if (!(bs->L > 0) || !std::isfinite(bs->L)) return fail(h, PROBE_ERR_ARG, "L must be > 0");
    if (!std::isfinite(bs->order)) return fail(h, PROBE_ERR_ARG, "order must be finite");
    if (bs->fft_pad < 0 || bs->fft_pad > 4096) return fail(h, PROBE_ERR_ARG, "fft_pad out of range");
    memset(&B, 0, sizeof(B));
    B.ndim = h->ndim;
    B.n[0] = h->nz;
    B.n[1] = h->ndim == 3 ? h->ny : 1;
    B.n[2] = h->nx;
    B.h[0] = h->hz;
    B.h[1] = h->ndim == 3 ? h->hy : 1.0;
    B.h[2] = h->hx;
    B.fp = bs->fft_pad;
    B.Nf[0] = B.n[0] + 2 * B.fp;
    B.Nf[1] = h->ndim == 3 ? B.n[1] + 2 * B.fp : 1;
    B.Nf[2] = B.n[2] + 2 * B.fp;
    B.nspatial = bs->nspatial;
    B.nangular = bs->nangular;
    B.nradial = bs->nradial;
    B.NM = bs->nangular * bs->nradial;
    B.P = B.nspatial * B.NM;
    if (B.NM > kMaxMult) return fail(h, PROBE_ERR_ARG, "nangular * nradial must be <= 32");
    if (B.P > kMaxTerms) return fail(h, PROBE_ERR_ARG, "the number of terms P must be <= 1024");
    for (int l = 0; l < B.nspatial; ++l)
        for (int a = 0; a < bs->ndim; ++a) B.spatial[l][a] = bs->spatial[l * bs->ndim + a];
    for (int a = 0; a < B.nangular; ++a) {
        B.angular[a] = bs->angular[a];
        if (B.ndim == 3 && (B.angular[a] < 0 || B.angular[a] > 5))
            return fail(h, PROBE_ERR_ARG, "3D angular indices must be in [0, 5]");
    }
    B.L = bs->L;
    B.order = bs->order;
    B.Nreal = (long long)B.Nf[0] * B.Nf[1] * B.Nf[2];
    B.Ncplx = (long long)B.Nf[0] * B.Nf[1] * (B.Nf[2] / 2 + 1);
    B.npts = (long long)B.n[0] * B.n[1] * B.n[2];
    return PROBE_OK;
}

probe_status get_plan(probe_t h, const BasisDev& B, cufftType type, int batch, cudaStream_t st, cufftHandle* out) {
    if (!h->fit) h->fit = new FitCache();
    auto key = std::make_tuple(B.ndim, B.Nf[0], B.Nf[1], B.Nf[2], (type == CUFFT_D2Z ? 1 : 2) * 100000 + batch);
    auto it = h->fit->plans.find(key);
    cufftHandle plan;
    if (it == h->fit->plans.end()) {
        int n2[2] = {B.Nf[0], B.Nf[2]};
        int n3[3] = {B.Nf[0], B.Nf[1], B.Nf[2]};
        const int idist = (int)(type == CUFFT_D2Z ? B.Nreal : B.Ncplx);
        const int odist = (int)(type == CUFFT_D2Z ? B.Ncplx : B.Nreal);
        cufftResult r = cufftPlanMany(&plan, B.ndim, B.ndim == 2 ? n2 : n3, nullptr, 1, idist, nullptr, 1, odist,
                                      type, batch);
        if (r != CUFFT_SUCCESS) return fail(h, PROBE_ERR_CUDA, "cufftPlanMany failed (" + std::to_string((int)r) + ")");
        h->fit->plans[key] = plan;
    } else {
        plan = it->second;
    }
    if (cufftSetStream(plan, st) != CUFFT_SUCCESS) return fail(h, PROBE_ERR_CUDA, "cufftSetStream failed");
    *out = plan;
    return PROBE_OK;
}

probe_status fft_check(probe_t h, cufftResult r, const char* what) {
    if (r != CUFFT_SUCCESS) return fail(h, PROBE_ERR_CUDA, std::string(what) + " failed (" + std::to_string((int)r) + ")");
    return PROBE_OK;
}

// Stage an FP32 array of n elements on the device; returns the device pointer.
probe_status stage_f32(probe_t h, const float* p, size_t n, DevBuf& buf, const float** out, cudaStream_t st) {
    if (is_device_ptr(p)) {
        *out = p;
        return PROBE_OK;
    }
    PROBE_TRY(ensure_buf(h, buf, n * 4));
    PROBE_CK(h, cudaMemcpyAsync(buf.p, p, n * 4, cudaMemcpyHostToDevice, st));
    *out = (const float*)buf.p;
    return PROBE_OK;
}

// alpha tables of a basis and (beta non-null) its multiplier tables into the cache; returns pointers
// and nmax.
probe_status tables(probe_t h, const BasisDev& B, cudaStream_t st, double** beta, double** alpha, int* nmax) {
    FitCache& c = *h->fit;
    *nmax = std::max(B.n[0], std::max(B.n[1], B.n[2]));
    if (beta) {
        PROBE_TRY(ensure_buf(h, c.beta, (size_t)B.NM * B.Ncplx * 8));
        k_fit_beta<<<grid_of(B.Ncplx), 256, 0, st>>>((double*)c.beta.p, B);
        *beta = (double*)c.beta.p;
    }
    PROBE_TRY(ensure_buf(h, c.alpha, (size_t)B.nspatial * 3 * (*nmax) * 8));
    k_fit_alpha<<<grid_of((long long)B.nspatial * 3 * (*nmax)), 256, 0, st>>>((double*)c.alpha.p, B, *nmax);
    PROBE_CK(h, cudaGetLastError());
    *alpha = (double*)c.alpha.p;
    return PROBE_OK;
}

// Gram matrix [A | y]^T [A | y] (pass 1) or [Q1 | y]^T [Q1 | y] with Q1 = A R1^{-1} (pass 2, L1 =
// R1^T given) into the dense lower triangle of C (n x n, n = P + 1).
probe_status fit_gram(probe_t h, const BasisDev& B, const double* w, const float* yd, const double* alpha, int nmax,
                      int p, const double* L1, double* C, cudaStream_t st) {
    FitCache& c = *h->fit;
    const int P = B.P, n = P + 1;
    const long long rows = (long long)p * B.npts;
    if (P <= kMaxSmall) {
        const size_t sm = gram_s_smem(B);
        if (!L1 && B.nspatial > 1 && sm <= kGramSmemMax) {
            const int nout = gram_plan(B).nout;
            PROBE_TRY(ensure_buf(h, c.part, (size_t)kGramBlocks * nout * 8));
            // the most that any basis takes, not this one's: another thread's call may set it before the launch
            PROBE_CK(h, cudaFuncSetAttribute(k_fit_gram_s, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kGramSmemMax));
            k_fit_gram_s<<<kGramBlocks, 256, sm, st>>>(w, yd, alpha, nmax, p, B, (double*)c.part.p);
            k_fit_out_to_C<<<grid_of(32ll * nout), 256, 0, st>>>((const double*)c.part.p, kGramBlocks, B, C);
            PROBE_CK(h, cudaGetLastError());
            return PROBE_OK;
        }
        const int npairs = n * (n + 1) / 2;
        PROBE_TRY(ensure_buf(h, c.part, (size_t)kGqBlocks * npairs * 8));
        auto kernel = L1 ? k_fit_gram<true> : k_fit_gram<false>;
        PROBE_CK(h, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGqSmem));
        kernel<<<kGqBlocks, kGqRows, kGqSmem, st>>>(w, yd, alpha, nmax, p, B, L1, (double*)c.part.p);
        k_fit_pairs_to_C<<<grid_of(32ll * npairs), 256, 0, st>>>((const double*)c.part.p, kGqBlocks, n, C);
        PROBE_CK(h, cudaGetLastError());
        return PROBE_OK;
    }
    long long rcl = std::max<long long>(1024, kChunkBytes / (8ll * n));
    rcl = std::min(rcl, (rows + 31) / 32 * 32);
    const int rc = (int)((rcl + 31) / 32 * 32);
    const int T = (n + kSyT - 1) / kSyT, tiles = T * (T + 1) / 2;
    const int nslices = std::max(1, std::min(kGramBlocks / tiles, (rc + 255) / 256));
    const int rps = ((rc + nslices - 1) / nslices + kSyR - 1) / kSyR * kSyR;
    PROBE_TRY(ensure_buf(h, c.chunk, (size_t)rc * n * 8));
    PROBE_TRY(ensure_buf(h, c.part, (size_t)nslices * n * n * 8));
    double* A = (double*)c.chunk.p;
    for (long long r0 = 0; r0 < rows; r0 += rc) {
        k_fit_cols<<<grid_of((long long)rc * n), 256, 0, st>>>(w, yd, alpha, nmax, p, B, r0, rc, A);
        if (L1) k_fit_trsm_rows<<<(rc + 127) / 128, 128, 0, st>>>(A, rc, P, L1);
        k_fit_syrk<<<dim3(tiles, nslices), 256, 0, st>>>(A, rc, n, rps, (double*)c.part.p);
        k_fit_reduce<<<grid_of((long long)n * n), 256, 0, st>>>((const double*)c.part.p, nslices, n, r0 > 0 ? 1 : 0,
                                                               C);
        PROBE_CK(h, cudaGetLastError());
    }
    return PROBE_OK;
}

// Cholesky factor L (P x P, lower, ld P) of the leading block of C (ld n), destroying that block.
probe_status fit_cholesky(probe_t h, double* C, int n, int P, double* L, double* dmax, int* status,
                          cudaStream_t st) {
    PROBE_CK(h, cudaMemsetAsync(L, 0, (size_t)P * P * 8, st));
    k_fit_dmax<<<1, 256, 0, st>>>(C, n, P, dmax);
    for (int k = 0; k < P; ++k) {
        const long long m = (long long)(P - k - 1) * (P - k - 1);
        k_fit_chol_step<<<(int)std::max<long long>(1, std::min<long long>((m + 255) / 256, 1024)), 256, 0, st>>>(
            C, n, P, k, dmax, L, status);
    }
    PROBE_CK(h, cudaGetLastError());
    return PROBE_OK;
}

// Least squares with the factor of the first pass alone (P <= 64): c = (L1 L1^T)^{-1} A^T y, then
// one step of iterative refinement with the corrected seminormal equations (Bjorck, Linear Algebra
// Appl. 88/89, 1987): r = y - A c, c += (L1 L1^T)^{-1} A^T r.  A step shrinks the error by about
// cond(A)^2 eps.  Taken while two things are small; else *done = false and the reorthogonalising pass
// follows, whose error is the smaller one there.
// (1) The condition of A with its columns scaled to unit norm, from the factor's inverse in the Frobenius
//     norm (1.3 to 13 times that of the 2-norm on the bases measured, 1.3 to 5 above 1e4): up to 2e5.
// (2) The first solution's own misfit eta = |A dc| / |A c|, up to 1e-9, which is also large where the
//     residual is and the rounding of A^T r then limits the step (cond(A) above about 1e4).  Alone it does not see the
//     condition: a target in the dominant directions of A has a small eta at any, and errors of 1.3e-7
//     (cond 4e6) and 1.6e-5 (2e7) passed where the other pass gives 1e-9 and 3.5e-9.
// Error of the coefficients against extended precision as a multiple of the reorthogonalising pass's
// (geometric means over 276 fits of 8 to 60 terms; targets fitted, dominant, noisy and white): bound (1) at
// 2e4 to 6e4 0.70, 0.43, 0.51 and 1.6; at 6e4 to 2e5 0.48, 0.84, 1.28 (white: by (2) never refined); at 6e5 to 2e6 about
// 1, with single fits three times as far off; beyond, up to five orders.
// z = A^T y; *status is the factorisation's.
constexpr double kRefineMax = 1e-9, kRefineCond = 2e5;
probe_status fit_refine(probe_t h, const BasisDev& B, const double* w, const float* yd, const double* alpha, int nmax,
                        int p, const double* L1, const double* z, double* coef, int* status, bool* done,
                        cudaStream_t st) {
    FitCache& c = *h->fit;
    PROBE_TRY(ensure_buf(h, c.part, (size_t)kRefBlocks * B.P * 8));
    double* part = (double*)c.part.p;
    double* norms = (double*)c.misc.p + 3;  // |A c|^2, |A dc|^2, |L^{-1} D|_F^2 in two parts
    PROBE_CK(h, cudaMemsetAsync(coef, 0, (size_t)B.P * 8, st));
    k_fit_refine_step<<<1, 256, 0, st>>>(z, 1, B.P, L1, coef, norms, nullptr);
    k_fit_refine<<<kRefBlocks, 256, 0, st>>>(w, yd, alpha, nmax, p, B, coef, part);
    k_fit_refine_step<<<1, 256, 0, st>>>(part, kRefBlocks, B.P, L1, coef, norms + 1, norms + 2);
    PROBE_CK(h, cudaGetLastError());
    int bad = 0;
    double n2[4];
    PROBE_CK(h, cudaMemcpyAsync(&bad, status, sizeof(int), cudaMemcpyDeviceToHost, st));
    PROBE_CK(h, cudaMemcpyAsync(n2, norms, sizeof(n2), cudaMemcpyDeviceToHost, st));
    PROBE_CK(h, cudaStreamSynchronize(st));
    // rank deficient (reported by the caller), or refined; a NaN is not
    *done = bad || (n2[1] <= kRefineMax * kRefineMax * n2[0] && B.P * (n2[2] + n2[3]) <= kRefineCond * kRefineCond);
    return PROBE_OK;
}

// Least squares of the fit, refined or by CholeskyQR2: coefficients into coef (device, P);
// status[0] = 1 when A^T A (or Q1^T Q1) is not numerically positive definite.
probe_status fit_solve(probe_t h, const BasisDev& B, const double* w, const float* yd, const double* alpha,
                            int nmax, int p, double* coef, int* status, cudaStream_t st) {
    FitCache& c = *h->fit;
    const int P = B.P, n = P + 1;
    PROBE_TRY(ensure_buf(h, c.gram, (size_t)n * n * 8));
    PROBE_TRY(ensure_buf(h, c.L1, (size_t)P * P * 8));
    PROBE_TRY(ensure_buf(h, c.L2, (size_t)P * P * 8));
    double* C = (double*)c.gram.p;
    double* L1 = (double*)c.L1.p;
    double* L2 = (double*)c.L2.p;
    double* dmax = (double*)c.misc.p + 2;
    double* v = coef + P;  // scratch of P doubles after the coefficients
    PROBE_CK(h, cudaMemsetAsync(status, 0, sizeof(int), st));
    PROBE_TRY(fit_gram(h, B, w, yd, alpha, nmax, p, nullptr, C, st));   // [A y]^T [A y]
    PROBE_TRY(fit_cholesky(h, C, n, P, L1, dmax, status, st));         // R1 = L1^T
    if (P <= kMaxSmall) {
        bool done = false;
        PROBE_TRY(fit_refine(h, B, w, yd, alpha, nmax, p, L1, C + (long long)P * n, coef, status, &done, st));
        if (done) return PROBE_OK;
    }
    PROBE_TRY(fit_gram(h, B, w, yd, alpha, nmax, p, L1, C, st));        // [Q1 y]^T [Q1 y]
    PROBE_TRY(fit_cholesky(h, C, n, P, L2, dmax, status, st));         // R2 = L2^T
    const double* z = C + (long long)P * n;                             // Q1^T y (row P of C)
    k_fit_trsv<<<1, 256, 0, st>>>(L2, P, 0, z, v);                      // R2^{-T} z
    k_fit_trsv<<<1, 256, 0, st>>>(L2, P, 1, v, v);                      // R2^{-1} R2^{-T} z
    k_fit_trsv<<<1, 256, 0, st>>>(L1, P, 1, v, coef);                   // c = R1^{-1} (...)
    PROBE_CK(h, cudaGetLastError());
    return PROBE_OK;
}

}  // namespace
}  // namespace probe

using namespace probe;

extern "C" probe_status probe_fit(probe_t h, const probe_basis* basis, const float* y, const float* Hy, int p,
                                  double* coeffs, double* resid_rel, probe_stream_t stream) {
    if (!h) return PROBE_ERR_ARG;
    if (p < 1) return fail(h, PROBE_ERR_ARG, "need at least one trial function");
    if (!y || !Hy || !coeffs) return fail(h, PROBE_ERR_ARG, "NULL array");
    BasisDev B;
    PROBE_TRY(make_basis(h, basis, B));
    cudaStream_t st = (cudaStream_t)stream;
    if (!h->fit) h->fit = new FitCache();
    FitCache& c = *h->fit;
    DevBuf ystage, xstage;
    const float *yd = nullptr, *xd = nullptr;
    probe_status s = PROBE_OK;
    do {
        if ((s = stage_f32(h, y, (size_t)p * B.npts, ystage, &yd, st)) != PROBE_OK) break;
        if ((s = stage_f32(h, Hy, (size_t)p * B.npts, xstage, &xd, st)) != PROBE_OK) break;
        if ((s = ensure_buf(h, c.xr, (size_t)p * B.Nreal * 8)) != PROBE_OK) break;
        if ((s = ensure_buf(h, c.Xc, (size_t)p * B.Ncplx * 16)) != PROBE_OK) break;
        if ((s = ensure_buf(h, c.Wc, (size_t)p * B.Ncplx * 16)) != PROBE_OK) break;
        if ((s = ensure_buf(h, c.w, (size_t)B.NM * p * B.Nreal * 8)) != PROBE_OK) break;
        if ((s = ensure_buf(h, c.coef, (size_t)(2 * B.P + 8) * 8)) != PROBE_OK) break;
        if ((s = ensure_buf(h, c.misc, 64)) != PROBE_OK) break;
        double *beta, *alpha;
        int nmax;
        if ((s = tables(h, B, st, &beta, &alpha, &nmax)) != PROBE_OK) break;
        cufftHandle fwd, inv;
        if ((s = get_plan(h, B, CUFFT_D2Z, p, st, &fwd)) != PROBE_OK) break;
        if ((s = get_plan(h, B, CUFFT_Z2D, p, st, &inv)) != PROBE_OK) break;
        cudaError_t e = cudaMemsetAsync(c.xr.p, 0, (size_t)p * B.Nreal * 8, st);
        if (e != cudaSuccess) { s = cuda_fail(h, e, "memset"); break; }
        k_fit_pad<<<grid_of((long long)p * B.npts), 256, 0, st>>>(xd, (double*)c.xr.p, p, B);
        if ((s = fft_check(h, cufftExecD2Z(fwd, (double*)c.xr.p, (cufftDoubleComplex*)c.Xc.p), "D2Z")) != PROBE_OK) break;
        const double invN = 1.0 / (double)B.Nreal;
        for (int m = 0; m < B.NM && s == PROBE_OK; ++m) {
            k_fit_mult<<<grid_of((long long)p * B.Ncplx), 256, 0, st>>>(
                (const double2*)c.Xc.p, beta + (long long)m * B.Ncplx, (double2*)c.Wc.p, 1, p, B.Ncplx, invN);
            s = fft_check(h, cufftExecZ2D(inv, (cufftDoubleComplex*)c.Wc.p, (double*)c.w.p + (long long)m * p * B.Nreal),
                          "Z2D");
        }
        if (s != PROBE_OK) break;
        int* status = (int*)c.misc.p;
        double* coef = (double*)c.coef.p;
        if ((s = fit_solve(h, B, (const double*)c.w.p, yd, alpha, nmax, p, coef, status, st)) != PROBE_OK) break;
        if ((s = ensure_buf(h, c.part, (size_t)kGramBlocks * 2 * 8)) != PROBE_OK) break;
        k_fit_resid<<<kGramBlocks, 256, 0, st>>>((const double*)c.w.p, yd, alpha, nmax, p, B, coef, (double*)c.part.p);
        k_fit_resid_final<<<1, 32, 0, st>>>((const double*)c.part.p, kGramBlocks, (double*)c.misc.p + 1);
        if ((e = cudaGetLastError()) != cudaSuccess) { s = cuda_fail(h, e, "fit kernels"); break; }
        int stat_h = 0;
        double res_h = 0.0;
        if ((e = cudaMemcpyAsync(&stat_h, status, sizeof(int), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
            (e = cudaMemcpyAsync(&res_h, (double*)c.misc.p + 1, sizeof(double), cudaMemcpyDeviceToHost, st)) !=
                cudaSuccess ||
            (e = cudaMemcpyAsync(coeffs, coef, (size_t)B.P * 8, cudaMemcpyDefault, st)) != cudaSuccess ||
            (e = cudaStreamSynchronize(st)) != cudaSuccess) {
            s = cuda_fail(h, e, "fit result copy");
            break;
        }
        if (resid_rel) *resid_rel = res_h;
        if (stat_h) s = fail(h, PROBE_ERR_STATE, "the fit columns B_i x_j are numerically rank deficient");
    } while (0);
    cudaStreamSynchronize(st);
    if (ystage.p) cudaFree(ystage.p);
    if (xstage.p) cudaFree(xstage.p);
    return s;
}

extern "C" probe_status probe_apply_precond(probe_t h, const probe_basis* basis, const double* coeffs,
                                            const float* img, float* out, probe_stream_t stream) {
    if (!h) return PROBE_ERR_ARG;
    if (!coeffs || !img || !out) return fail(h, PROBE_ERR_ARG, "NULL array");
    BasisDev B;
    PROBE_TRY(make_basis(h, basis, B));
    cudaStream_t st = (cudaStream_t)stream;
    if (!h->fit) h->fit = new FitCache();
    FitCache& c = *h->fit;
    DevBuf istage, ostage;
    const float* id = nullptr;
    probe_status s = PROBE_OK;
    const bool host_out = !is_device_ptr(out);
    do {
        if ((s = stage_f32(h, img, (size_t)B.npts, istage, &id, st)) != PROBE_OK) break;
        float* od = out;
        if (host_out) {
            if ((s = ensure_buf(h, ostage, (size_t)B.npts * 4)) != PROBE_OK) break;
            od = (float*)ostage.p;
        }
        if ((s = ensure_buf(h, c.xr, (size_t)B.Nreal * 8)) != PROBE_OK) break;
        if ((s = ensure_buf(h, c.Xc, (size_t)B.Ncplx * 16)) != PROBE_OK) break;
        if ((s = ensure_buf(h, c.Wc, (size_t)B.nspatial * B.Ncplx * 16)) != PROBE_OK) break;
        if ((s = ensure_buf(h, c.w, (size_t)B.nspatial * B.Nreal * 8)) != PROBE_OK) break;
        if ((s = ensure_buf(h, c.coef, (size_t)(2 * B.P + 8) * 8)) != PROBE_OK) break;
        double* alpha;
        int nmax;
        if ((s = tables(h, B, st, nullptr, &alpha, &nmax)) != PROBE_OK) break;
        cudaError_t e = cudaMemcpyAsync(c.coef.p, coeffs, (size_t)B.P * 8, cudaMemcpyDefault, st);
        if (e != cudaSuccess) { s = cuda_fail(h, e, "coefficient copy"); break; }
        cufftHandle fwd, inv;
        if ((s = get_plan(h, B, CUFFT_D2Z, 1, st, &fwd)) != PROBE_OK) break;
        if ((s = get_plan(h, B, CUFFT_Z2D, B.nspatial, st, &inv)) != PROBE_OK) break;
        if ((e = cudaMemsetAsync(c.xr.p, 0, (size_t)B.Nreal * 8, st)) != cudaSuccess) { s = cuda_fail(h, e, "memset"); break; }
        k_fit_pad<<<grid_of(B.npts), 256, 0, st>>>(id, (double*)c.xr.p, 1, B);
        if ((s = fft_check(h, cufftExecD2Z(fwd, (double*)c.xr.p, (cufftDoubleComplex*)c.Xc.p), "D2Z")) != PROBE_OK) break;
        {
            const int NQ = B.nradial <= 4 ? 4 : (B.nradial <= 8 ? 8 : 16);
            const size_t sm = (size_t)((B.nspatial + kLamBlock - 1) / kLamBlock * kLamBlock) * B.nangular * NQ * 8;
            auto kernel = NQ == 4 ? k_precond_spectra<4> : (NQ == 8 ? k_precond_spectra<8> : k_precond_spectra<16>);
            kernel<<<grid_of(B.Ncplx), 256, sm, st>>>((const double2*)c.Xc.p, (const double*)c.coef.p,
                                                     (double2*)c.Wc.p, B, 1.0 / (double)B.Nreal);
        }
        if ((s = fft_check(h, cufftExecZ2D(inv, (cufftDoubleComplex*)c.Wc.p, (double*)c.w.p), "Z2D")) != PROBE_OK) break;
        k_precond_combine<<<grid_of(B.npts), 256, 0, st>>>((const double*)c.w.p, alpha, nmax, B, od);
        if ((e = cudaGetLastError()) != cudaSuccess) { s = cuda_fail(h, e, "precond kernels"); break; }
        if (host_out) {
            if ((e = cudaMemcpyAsync(out, od, (size_t)B.npts * 4, cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
                (e = cudaStreamSynchronize(st)) != cudaSuccess) {
                s = cuda_fail(h, e, "precond output copy");
                break;
            }
        }
    } while (0);
    if (istage.p || ostage.p) {
        cudaStreamSynchronize(st);
        if (istage.p) cudaFree(istage.p);
        if (ostage.p) cudaFree(ostage.p);
    }
    return s;
}

// sp_spectral.cu -- semi-implicit Fourier spectral step (the paper's spectral
// solver scheme, Sec. "Construction of Semi-Implicit Fourier Spectral Scheme";
// the paper runs it on the host only), with this file's own FFTs.
//
// Linear terms are integrated implicitly in Fourier space with the continuous
// symbol -|k|^2, the cubic term explicitly in real space:
//   Allen-Cahn     L(k) = c1 - |k|^2,            N^ = (-c2 phi^3)^
//   Cahn-Hilliard  L(k) = |k|^2 (c1 - kappa |k|^2), N^ = -|k|^2 (c2 phi^3)^
//   phi^' = (phi^ + dt N^) / (1 - dt L(k)),   k = 2 pi m / (n h) per axis.
//
// Transforms (sp_spectral.cuh).  The real-to-complex transform runs along x (the
// contiguous axis), then complex transforms along y (and z): the order of numpy's
// rfftn, whose inverse irfftn runs the complex axes first and takes the real part of
// the zero and Nyquist bins along x.  Two real rows are transformed as one complex row
// (real part and imaginary part) and separated afterwards.  Sides need prime factors
// 2, 3, 5, 7 and at most 4096 (FP64) or 8192 (FP32) points when all are powers of two,
// half that otherwise (a line is transformed by one CTA).
//
// Layout.  The half spectrum (nx/2+1 modes along x) is stored transposed,
// x-mode slowest: Z[kx][z][y] (y fastest), so that the y transforms read
// contiguous lines and the z transforms groups of adjacent lines.  The
// resident spectrum phi^ / N has the same layout.
//
// One step (2D; 3D adds a forward y pass before and an inverse y pass after the
// z pass, which then holds the update):
//   rows:  phi -> cube -> forward x transforms -> Z       (first step of a call)
//   lines: Z -> forward y -> phi^ update (resident) -> inverse y -> Z
//   rows:  Z -> inverse x transforms -> phi, and, when another step follows,
//          cube -> forward x transforms -> Z for it.
// The normalisation 1/N is in the resident spectrum and in the cube's coefficient, the
// 1/2 of the row separation in the coefficient of the forward x transforms.
#include <cmath>
#include <string>
#include <vector>

#include "sp_spectral.cuh"

namespace sp {

static std::string g_fft_err;
const char *spectral_last_error() { return g_fft_err.c_str(); }

// phi^ of a real phi is Hermitian.  The half spectrum holds both of a pair of conjugate modes only
// in its planes kx = 0 and, for even nx, kx = nx / 2; there rounding leaves a non-Hermitian part
// that the inverse transform drops, so the cubic term never holds it, while the linear part
// multiplies it by up to G = 1 / (1 - dt max L(k)) per step.  Left alone it reached phi through
// the rounding of the inverse transform: at dt = 0.5 Allen-Cahn (G = 2) was lost after 60 steps in
// single and 130 in double precision, Cahn-Hilliard (G = 8/7) after 300 and 600.  So each pair
// (u, v) of these planes is set to ((u + conj v) / 2, its conjugate) before the noise has grown by
// 2^20, that is after 20 / log2 G steps: what enters phi stays 2^20 u of a rounding, 1/16 of one in
// single precision.  (A launch takes 4 to 5 us: every 10 steps at G = 2 it cost 45 x 128 x 128 FP32
// Allen-Cahn 1.3 %.)
template <typename C>
__global__ void __launch_bounds__(256) hermitian_kernel(C *uh, int ny, int nz, size_t nyquist) {
    pdl_enter();
    const size_t n = (size_t)ny * nz, i = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const int z = (int)(i / ny), y = (int)(i - (size_t)z * ny);
    const size_t j = (size_t)(z ? nz - z : 0) * ny + (y ? ny - y : 0);
    if (j < i) return;  // the partner's thread does both
    C *p = uh + (blockIdx.y ? nyquist * n : 0);
    const C u = p[i], v = p[j];
    const C m{(u.x + v.x) / 2, (u.y - v.y) / 2};
    p[i] = m;
    if (j != i) p[j] = C{m.x, -m.y};
}

template <typename C> static cudaError_t make_hermitian(const SpectralPlan *P, C *uh, cudaStream_t s) {
    const size_t n = (size_t)P->ny * P->nz;
    return launch_pdl(hermitian_kernel<C>, dim3((unsigned)((n + 255) / 256), P->nx % 2 ? 1 : 2), dim3(256), 0, s, uh, P->ny,
                      P->nz, (size_t)P->nx / 2);
}

static bool is_pow2(int n) { return (n & (n - 1)) == 0; }

// The stages of an n-point transform, `lines` of which make a pass; false if n has another
// prime factor than 2, 3, 5, 7.  4 points per thread where 16 would leave an SM fewer than
// four warps (256^2 FP64 75 -> 22 us per step, FP32 20 -> 8).
static bool factor_len(int n, long long lines, int n_sm, FftLen *L) {
    L->n = n;
    L->lgn = 0;
    while ((1 << L->lgn) < n) ++L->lgn;
    L->nst = L->V = 0;
    if (is_pow2(n) && n >= 32) {
        L->V = n <= 1024 && lines * (n / 16) < 4LL * 32 * n_sm ? 4 : 16;
        FftStages &S = L->reg;  // radix V, then as few stages as possible, of even radices
        const int lgv = L->V == 16 ? 4 : 2;
        S.nst = 0;
        S.lgr[S.nst++] = lgv;
        for (int rest = L->lgn - lgv; rest > 0; rest -= S.lgr[S.nst - 1]) {
            const int left = (rest + lgv - 1) / lgv;
            S.lgr[S.nst++] = (rest + left - 1) / left;
        }
        return true;
    }
    int m = n;
    for (int r : {8, 4, 2, 3, 5, 7})
        while (m % r == 0) {
            if (L->nst == kFftMaxStages) return false;
            L->rad[L->nst++] = r;
            m /= r;
        }
    return m == 1;
}

int spectral_create(int dtype, int dims, int nx, int ny, int nz, double h, double growth, SpectralPlan **out) {
    *out = nullptr;
    SpectralPlan *P = new (std::nothrow) SpectralPlan();
    if (!P) return SP_ENOMEM;
    P->dtype = dtype;
    P->dims = dims;
    P->nx = nx;
    P->ny = ny;
    P->nz = nz;
    P->nxh = nx / 2 + 1;
    P->N = (size_t)nx * ny * nz;
    P->Nc = (size_t)P->nxh * ny * nz;
    const int sides[3] = {nx, ny, nz};
    FftLen *ls[3] = {&P->lx, &P->ly, &P->lz};
    const bool f64 = dtype == SP_F64, pow2 = is_pow2(nx) && is_pow2(ny) && is_pow2(nz);
    const int longest = (f64 ? 4096 : 8192) / (pow2 ? 1 : 2);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&P->n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        g_fft_err = "device look-up failed";
        delete P;
        return SP_ECUDA;
    }
    const long long lines[3] = {((long long)ny * nz + 1) / 2, (long long)P->nxh * nz, (long long)P->nxh * ny};
    for (int a = 0; a < 3; ++a)
        if (sides[a] > longest || !factor_len(sides[a], lines[a], P->n_sm, ls[a])) {
            g_fft_err = std::string("the spectral scheme needs sides with prime factors 2, 3, 5, 7 of at most ") +
                        (f64 ? "4096 (FP64, powers of two; 2048 otherwise)" : "8192 (FP32, powers of two; 4096 otherwise)") +
                        " points (got " + std::to_string(sides[a]) + ")";
            delete P;
            return SP_EINVAL;
        }
    P->h = h;
    const double lg = growth > 1.0 ? std::log2(growth) : 0.0;
    P->every = lg > 1e-8 ? std::max(1LL, (long long)(20.0 / lg)) : 1LL << 40;
    // FP32 with G = 1 / (1 - dt max L(k)) > 4/3: the staged implementation (see its file)
    if (!f64 && growth > 4.0 / 3.0) {
        P->first = (long long)(50.0 / lg);
        const int rc = staged::create(dims, nx, ny, nz, &P->stg);
        if (rc != SP_OK) {
            g_fft_err = "device allocation for the spectral plan failed";
            delete P;
            return rc;
        }
        *out = P;
        return SP_OK;
    }
    // twiddles of each distinct side (see FftStages, FftLen), in long double on the host,
    // rounded once to the working precision; squared wavenumbers of each axis in FP64,
    // rounded once
    std::vector<long double> re, im;
    std::vector<double> k2;
    const long double two_pi = 6.283185307179586476925286766559005768L;
    auto root = [&](long long t, int n) {
        const long double ang = two_pi * (long double)t / (long double)n;
        re.push_back(cosl(ang));
        im.push_back(-sinl(ang));
    };
    for (int a = 0; a < 3; ++a) {
        FftLen &L = *ls[a];
        L.k2_off = (int)k2.size();
        for (int m = 0; m < L.n; ++m) {  // numpy's fftfreq order
            const double k = (double)(two_pi / ((long double)L.n * (long double)h)) * (m < (L.n + 1) / 2 ? m : m - L.n);
            k2.push_back(k * k);
        }
        int same = -1;
        for (int b = 0; b < a; ++b)
            if (sides[b] == sides[a] && ls[b]->V == L.V) same = b;
        if (same >= 0) {
            L.tw_off = ls[same]->tw_off;
            L.reg.tw_off = ls[same]->reg.tw_off;
            continue;
        }
        L.tw_off = L.reg.tw_off = (int)re.size();
        if (!L.V)
            for (int t = 0; t < L.n; ++t) root(t, L.n);
        else
            for (int i = 1, lgp = L.reg.lgr[0]; i < L.reg.nst; lgp += L.reg.lgr[i++]) {
                const int lgr = L.reg.lgr[i];
                for (int l = 1; l <= lgr; ++l)  // w^(R >> l) exp(-2 pi i m / 2^l)
                    for (int m = 0; m < std::max(1, 1 << l >> 2); ++m)
                        for (int k = 0; k < (1 << lgp); ++k)
                            root(((long long)k << (lgr - l)) + ((long long)m << (lgp + lgr - l)), 1 << (lgp + lgr));
            }
    }
    const size_t rb = f64 ? sizeof(double) : sizeof(float), cb = 2 * rb;
    std::vector<unsigned char> host(re.size() * cb), host2(k2.size() * rb);
    for (size_t i = 0; i < re.size(); ++i) {
        if (f64) reinterpret_cast<double2 *>(host.data())[i] = double2{(double)re[i], (double)im[i]};
        else reinterpret_cast<float2 *>(host.data())[i] = float2{(float)re[i], (float)im[i]};
    }
    for (size_t i = 0; i < k2.size(); ++i) {
        if (f64) reinterpret_cast<double *>(host2.data())[i] = k2[i];
        else reinterpret_cast<float *>(host2.data())[i] = (float)k2[i];
    }
    if (cudaMalloc(&P->uh, P->Nc * cb) != cudaSuccess || cudaMalloc(&P->z, P->Nc * cb) != cudaSuccess ||
        cudaMalloc(&P->tw, host.size()) != cudaSuccess || cudaMalloc(&P->k2, host2.size()) != cudaSuccess ||
        cudaMemcpy(P->tw, host.data(), host.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(P->k2, host2.data(), host2.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaGetLastError();
        spectral_destroy(P);
        g_fft_err = "device allocation for the spectral plan failed";
        return SP_ENOMEM;
    }
    *out = P;
    return SP_OK;
}

void spectral_destroy(SpectralPlan *P) {
    if (!P) return;
    staged::destroy(P->stg);
    if (P->uh) cudaFree(P->uh);
    if (P->z) cudaFree(P->z);
    if (P->tw) cudaFree(P->tw);
    if (P->k2) cudaFree(P->k2);
    delete P;
}

// phi^ / N = forward transform of phi / N (after the initial condition or a write)
template <typename R> static int spectral_load_t(SpectralPlan *P, const R *phi, cudaStream_t s) {
    typedef typename Cplx<R>::type C;
    C *uh = static_cast<C *>(P->uh);
    const SpecCoef<R> c{};
    cudaError_t e = run_rows<R>(P, kRowLoad, const_cast<R *>(phi), uh, (R)(0.5 / (double)P->N), s);
    if (e == cudaSuccess && P->ny > 1) e = run_lines<R>(P, 1, kLineForward, AC, c, uh, s);
    if (e == cudaSuccess && P->nz > 1) e = run_lines<R>(P, 2, kLineForward, AC, c, uh, s);
    P->nh_valid = false;
    if (e != cudaSuccess) {
        g_fft_err = std::string("forward transform: ") + cudaGetErrorString(e);
        return SP_ECUDA;
    }
    return SP_OK;
}

int spectral_load(SpectralPlan *P, const void *phi, cudaStream_t s) {
    P->done = P->since = 0;
    if (P->stg) {
        const cudaError_t e = staged::load(P->stg, static_cast<const float *>(phi), s);
        if (e == cudaSuccess) return SP_OK;
        g_fft_err = std::string("forward transform: ") + cudaGetErrorString(e);
        return SP_ECUDA;
    }
    if (P->dtype == SP_F64) return spectral_load_t<double>(P, static_cast<const double *>(phi), s);
    return spectral_load_t<float>(P, static_cast<const float *>(phi), s);
}

template <typename R>
static cudaError_t spectral_step_t(SpectralPlan *P, int model, R *phi, double dt, double c1, double c2, double kappa,
                                   bool more, cudaStream_t s) {
    typedef typename Cplx<R>::type C;
    C *Z = static_cast<C *>(P->z);
    const R coef = (R)((model == AC ? -c2 : c2) * 0.5 / (double)P->N);
    const SpecCoef<R> c{(R)c1, (R)kappa, (R)dt};
    cudaError_t e = cudaSuccess;
    if (!P->nh_valid) e = run_rows<R>(P, kRowCube, phi, Z, coef, s);
    if (P->dims == 2) {
        if (e == cudaSuccess) e = run_lines<R>(P, 1, kLineUpdate, model, c, Z, s);
    } else {
        if (e == cudaSuccess) e = run_lines<R>(P, 1, kLineForward, model, c, Z, s);
        if (e == cudaSuccess) e = run_lines<R>(P, 2, kLineUpdate, model, c, Z, s);
        if (e == cudaSuccess) e = run_lines<R>(P, 1, kLineInverse, model, c, Z, s);
    }
    if (e == cudaSuccess) e = run_rows<R>(P, more ? kRowInverseNext : kRowInverse, phi, Z, coef, s);
    P->nh_valid = more && e == cudaSuccess;
    return e;
}

int spectral_step(SpectralPlan *P, int model, void *phi, double dt, double c1, double c2, double kappa, cudaStream_t s,
                  bool more) {
    cudaError_t e = cudaSuccess;
    if (P->since >= P->every && P->done >= P->first) {
        e = P->stg ? make_hermitian(P, staged::spectrum(P->stg), s)
            : P->dtype == SP_F64 ? make_hermitian(P, static_cast<double2 *>(P->uh), s)
                                 : make_hermitian(P, static_cast<float2 *>(P->uh), s);
        P->since = 0;
    }
    ++P->done;
    ++P->since;
    if (e == cudaSuccess)
        e = P->stg ? staged::step(P->stg, model, (float *)phi, P->h, dt, c1, c2, kappa, s, more)
            : P->dtype == SP_F64
                ? spectral_step_t<double>(P, model, (double *)phi, dt, c1, c2, kappa, more, s)
                : spectral_step_t<float>(P, model, (float *)phi, dt, c1, c2, kappa, more, s);
    if (e != cudaSuccess) {
        g_fft_err = std::string("spectral step: ") + cudaGetErrorString(e);
        return SP_ECUDA;
    }
    return SP_OK;
}

}  // namespace sp

// sp_spectral.cuh -- transforms of the semi-implicit Fourier spectral step: the plan,
// the kernels and their launch.  Included by one translation unit per precision
// (sp_spectral_f32.cu, sp_spectral_f64.cu) and by the host side (sp_spectral.cu).
#pragma once

#include "sp_internal.h"

namespace sp {

constexpr int kFftMaxStages = 16;

// The stages of a register transform with V points per thread: radices 2^lgr[s], the
// first one V.  tw_off: complex offset of the stages' twiddles in the plan's table, for
// every later stage (radix R after radices of product p) R/2 rows of p entries:
// w^(R >> l) exp(-2 pi i m / 2^l), w = exp(-2 pi i k / (R p)), k < p, for the levels l = 1 ..
// log2 R and m < max(1, 2^(l-2)).
struct FftStages {
    int nst, lgr[8], tw_off;
};

// One transform length.  A power of two from 32 on is transformed in registers
// (fft_regs), other lengths by mixed-radix stages in shared memory (fft_lines).
struct FftLen {
    int n, lgn;
    int V;                 // points per thread of the register transform, 16 or 4; 0: mixed radices
    FftStages reg;
    int nst, rad[kFftMaxStages];
    int tw_off;            // mixed: complex offset of exp(-2 pi i t / n), t < n, in the plan's table
    int k2_off;            // real offset of (2 pi freq(m) / (n h))^2, m < n, in the plan's wavenumber table
};

template <typename R> struct Cplx;
template <> struct Cplx<double> { typedef double2 type; };
template <> struct Cplx<float> { typedef float2 type; };

// The staged single-precision implementation (sp_spectral_staged.cu).
namespace staged {
struct Plan;
int create(int dims, int nx, int ny, int nz, Plan **out);
void destroy(Plan *P);
cudaError_t load(Plan *P, const float *phi, cudaStream_t s);
cudaError_t step(Plan *P, int model, float *phi, double h, double dt, double c1, double c2, double kappa, cudaStream_t s,
                 bool more);
float2 *spectrum(Plan *P);  // resident, Z[kx][z][y]
}  // namespace staged

struct SpectralPlan {
    staged::Plan *stg;            // FP32 with strong linear growth: everything below but h is unused
    double h;
    int dtype, dims, nx, ny, nz, nxh, n_sm;
    size_t N, Nc;                 // real points, half-spectrum modes
    FftLen lx, ly, lz;
    void *uh, *z;                 // resident spectrum (scaled by 1/N) and the transform buffer (Nc complex each)
    void *tw;                     // twiddles of every axis length
    void *k2;                     // squared wavenumbers of every axis
    bool nh_valid;                // z holds the transformed cubic term of the current phi
    // see make_hermitian (sp_spectral.cu)
    long long done, since;        // steps since the spectrum was computed from phi; since it was made Hermitian
    long long every, first;       // made Hermitian after `every` steps, from step `first` on
};

// coefficients of the Fourier update
template <typename R> struct SpecCoef {
    R c1, kappa, dt;
};

enum RowMode { kRowLoad = 0, kRowCube = 1, kRowInverse = 2, kRowInverseNext = 3 };
enum LineMode { kLineForward = 0, kLineInverse = 1, kLineUpdate = 2 };

// x pass over all rows.  kRowLoad / kRowCube: coef f (resp. coef f^3) forward into Z;
// kRowInverse: Z into phi; kRowInverseNext: the same, then coef phi^3 forward into Z.
// coef holds the factor 1/2 of the row separation.
template <typename R>
cudaError_t run_rows(const SpectralPlan *P, RowMode mode, R *f, typename Cplx<R>::type *Z, R coef, cudaStream_t s);
// y (axis 1) or z (axis 2) lines of Z; kLineUpdate holds the Fourier update of P->uh.
template <typename R>
cudaError_t run_lines(const SpectralPlan *P, int axis, LineMode mode, int model, const SpecCoef<R> &c,
                      typename Cplx<R>::type *Z, cudaStream_t s);

#ifdef SP_SPECTRAL_KERNELS

// ------------------------------------------------------- complex helpers --

template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return C{a.x + b.x, a.y + b.y}; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return C{a.x - b.x, a.y - b.y}; }
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
    return C{FMA(a.x, b.x, -(a.y * b.y)), FMA(a.x, b.y, a.y * b.x)};
}
template <typename C> __device__ __forceinline__ C swapped(C a) { return C{a.y, a.x}; }

// p = a + t b, m = a - t b: six multiply-adds (m = 2a - p)
template <typename C> __device__ __forceinline__ void butterfly(C &a, C &b, C t) {
    const C p{FMA(-t.y, b.y, FMA(t.x, b.x, a.x)), FMA(t.y, b.x, FMA(t.x, b.y, a.y))};
    typedef decltype(a.x) R;
    b = C{FMA(R(2), a.x, -p.x), FMA(R(2), a.y, -p.y)};
    a = p;
}

// ============================================ powers of two, in registers ==
//
// A line of n points is held by T = n / V threads, V values each: thread t has points
// t + j T, before and after a transform, so the loads and stores of lines are
// coalesced, the Fourier update and the cube run on registers, and a forward
// transform is followed by an inverse one without a pass through memory.  The stages
// are those of a Stockham transform, the first of radix V; between two stages the
// values change threads through one shared-memory buffer.
// Radix-R butterflies are decimation in time with the stage's twiddles merged into
// every level as multiply-adds (after Goedecker, SIAM J. Sci. Comput. 18, 1997: six
// per two points and level): 192 operations and 8 distinct twiddles for 16 points
// where separate twiddles take 228 and 15; the first stage, whose twiddles are
// constants, takes 148.  The twiddles come from tables in the order in which the
// threads need them, through L1 (computing them from a two-level table in shared
// memory took a quarter of the FP32 instructions).
// The inverse is the forward transform of values with real and imaginary part
// exchanged.  Every transform here therefore runs the same code.
// V = 16 for throughput.  V = 4 where V = 16 would leave fewer than four warps per SM
// (a single FP64 warp gets a quarter of the SM's FP64 rate, and short code matters when
// every instruction is fetched for one warp).

__host__ __device__ constexpr int bit_reverse(int m, int lg) {
    int r = 0;
    for (int b = 0; b < lg; ++b)
        if (m >> b & 1) r |= 1 << (lg - 1 - b);
    return r;
}

// exp(-2 pi i m / 16), m < 4
template <typename C> __device__ __forceinline__ C root16(int m) {
    typedef decltype(C{}.x) R;
    constexpr double c1 = 0.92387953251128675613, s1 = 0.38268343236508977173, h = 0.70710678118654752440;
    return m == 0 ? C{R(1), R(0)} : m == 1 ? C{R(c1), R(-s1)} : m == 2 ? C{R(h), R(-h)} : C{R(s1), R(-c1)};
}

// R-point butterflies of the values u[q + j Q] (Q = V / R), q < Q; output m of
// butterfly q is left at u[q + bit_reverse(m) Q].  TW: with twiddles, tw(q, row) the
// factor of level s and m in row (s < 3 ? s - 1 : 2^(s-2) + m) of the stage's table (m <
// max(1, 2^(s-2)); the other half of a level is those times -i).
template <int LGR, bool TW, int V, typename C, typename TwF>
__device__ __forceinline__ void dit(C (&u)[V], const TwF &tw) {
    constexpr int R = 1 << LGR, Q = V / R;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
#pragma unroll
        for (int s = 1; s <= LGR; ++s) {
            const int half = R >> s, nm = 1 << (s - 1), nt = nm < 2 ? 1 : nm / 2;
#pragma unroll
            for (int mt = 0; mt < nt; ++mt) {
                C t{1, 0};
                if constexpr (TW) t = tw(q, s < 3 ? s - 1 : nt + mt);
                else t = root16<C>(mt << (4 - s > 0 ? 4 - s : 0));
#pragma unroll
                for (int rot = 0; rot < (nm < 2 ? 1 : 2); ++rot) {
                    const int m = mt + rot * nt;
#pragma unroll
                    for (int j = 0; j < half; ++j) {
                        const int ia = j + bit_reverse(m, s - 1) * (R >> (s - 1)), ib = ia + half;
                        C &a = u[q + ia * Q], &b = u[q + ib * Q];
                        if (!TW && mt == 0) {
                            const C x = a, y = rot ? C{b.y, -b.x} : b;
                            a = cadd(x, y);
                            b = csub(x, y);
                        } else {
                            butterfly(a, b, rot ? C{t.y, -t.x} : t);
                        }
                    }
                }
            }
        }
    }
}

// Shared-memory slot of point i of a line: for 256 points and more (V = 16) one empty
// slot after every 16 (the first stage's stores, 16 points apart, and all loads are then
// free of bank conflicts).  sh is 4 or 31; slot(a + b) = slot(a) + slot(b) for b a
// multiple of 16 or sh = 31.
__device__ __forceinline__ int slot_of(int i, int sh) { return i + (i >> sh); }
template <int V> __host__ __device__ __forceinline__ int pad_shift(int n) { return V == 16 && n >= 256 ? 4 : 31; }

// the position of this thread in its line and the synchronisation of a line's threads
struct LineThread {
    int t, lgT;
    bool warp_local;  // a line's threads are in one warp
    __device__ __forceinline__ void sync() const {
        if (warp_local) __syncwarp();
        else __syncthreads();
    }
};

// twiddled stage of radix 2^LGR after radices of product 2^lgp; tw: the stage's table
template <int LGR, int V, typename C>
__device__ __forceinline__ void twiddled_stage(C (&u)[V], const C *tw, int t, int lgT, int lgp) {
    dit<LGR, true>(u, [&](int q, int row) -> C {
        const int k = (t + (q << lgT)) & ((1 << lgp) - 1);
        return __ldg(tw + k + (row << lgp));
    });
}

// outputs of a radix-2^LGR stage to their sorted places in buf
template <int LGR, int V, typename C>
__device__ __forceinline__ void scatter(const C (&u)[V], C *buf, int t, int lgT, int lgp, int sh) {
    constexpr int R = 1 << LGR, Q = V / R;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int b = t + (q << lgT), k = b & ((1 << lgp) - 1);
        const int base = slot_of(((b - k) << LGR) + k, sh), inc = slot_of(1 << lgp, sh);
#pragma unroll
        for (int m = 0; m < R; ++m) buf[base + m * inc] = u[q + bit_reverse(m, LGR) * Q];
    }
}

// natural order of the last stage's outputs (registers renamed)
template <int LGR, int V, typename C> __device__ __forceinline__ void unscramble(C (&u)[V]) {
    constexpr int R = 1 << LGR, Q = V / R;
    C v[V];
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int m = 0; m < R; ++m) v[q + m * Q] = u[q + bit_reverse(m, LGR) * Q];
#pragma unroll
    for (int j = 0; j < V; ++j) u[j] = v[j];
}

// Forward transform (unnormalised) of the line whose points t + j T this thread holds.
// buf: the line's buffer, free for use once the line's threads have synchronised.
template <int V, typename C>
__device__ __forceinline__ void fft_regs(C (&u)[V], C *buf, const FftLen &L, const C *tw_all, const LineThread &lt) {
    constexpr int LGV = V == 16 ? 4 : 2;
    const FftStages &S = L.reg;
    const int t = lt.t, lgT = lt.lgT, sh = pad_shift<V>(L.n);
    const int rd = slot_of(t, sh), rinc = slot_of(1 << lgT, sh);
    const C *tw = tw_all + S.tw_off;
    dit<LGV, false>(u, [](int, int) { return C{1, 0}; });
    lt.sync();
#pragma unroll
    for (int m = 0; m < V; ++m) buf[slot_of(t << LGV, sh) + m] = u[bit_reverse(m, LGV)];
    int lgp = LGV;
#pragma unroll 1
    for (int s = 1; s < S.nst; ++s) {
        lt.sync();
#pragma unroll
        for (int j = 0; j < V; ++j) u[j] = buf[rd + j * rinc];
        const bool last = s + 1 == S.nst;
        const int lgr = S.lgr[s];
        switch (lgr) {
#define SP_STAGE(LG)                                    \
    case LG:                                            \
        if constexpr (LG <= LGV) {                      \
            twiddled_stage<LG>(u, tw, t, lgT, lgp);     \
            if (!last) {                                \
                lt.sync();                              \
                scatter<LG>(u, buf, t, lgT, lgp, sh);   \
            } else {                                    \
                unscramble<LG>(u);                      \
            }                                           \
        }                                               \
        break;
            SP_STAGE(4)
            SP_STAGE(3)
            SP_STAGE(2)
            SP_STAGE(1)
#undef SP_STAGE
        }
        tw += (size_t)1 << (lgp + lgr - 1);
        lgp += lgr;
    }
}

// Fourier update of one mode: *uh (the resident mode over N) advances, its new value
// is returned.  k2 = |k|^2.
template <typename R, int MODEL>
__device__ __forceinline__ typename Cplx<R>::type update_mode(typename Cplx<R>::type *uh, typename Cplx<R>::type nh,
                                                              R k2, const SpecCoef<R> &c) {
    typedef typename Cplx<R>::type C;
    const R L = (MODEL == AC) ? c.c1 - k2 : k2 * FMA(-c.kappa, k2, c.c1);
    const R w = (MODEL == AC) ? c.dt : -(c.dt * k2);
    const R denom = FMA(-c.dt, L, R(1));
    R rd;
    if constexpr (sizeof(R) == 8) rd = __drcp_rn(denom);
    else rd = __frcp_rn(denom);
    const C a = *uh;
    const C v{FMA(w, nh.x, a.x) * rd, FMA(w, nh.y, a.y) * rd};
    *uh = v;
    return v;
}

// Geometry of a pass: lines of a CTA, their threads and their addresses.
struct PassGeom {
    int G, lgI;            // lines per CTA; adjacent threads take 2^lgI adjacent lines
    int LS;                // complex slots between the lines' buffers
    int per_kx;            // strided lines (axis 2): groups per x mode; 0: contiguous lines
    int nlines;            // contiguous lines or row pairs in all
    int ny, nz, nxh, nrows;
    int ahead;             // contiguous lines: CTAs resident at once, the distance of the L2 prefetch
};

// n bytes at p (16-byte aligned, n a multiple of 16) into L2
__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t n) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "r"(n) : "memory");
}

// this thread's line within the CTA and its place in it (V points per thread)
template <int V> __device__ __forceinline__ int line_thread(const FftLen &L, const PassGeom &g, LineThread &lt) {
    lt.lgT = L.lgn - (V == 16 ? 4 : 2);
    const int I = 1 << g.lgI, lo = threadIdx.x & (I - 1), r = threadIdx.x >> g.lgI;
    lt.t = r & ((1 << lt.lgT) - 1);
    lt.warp_local = lt.lgT + g.lgI <= 5;
    return ((r >> lt.lgT) << g.lgI) + lo;
}

// Registers: 64 per thread (FP32) keep two CTAs of 512 threads on an SM, 128 (FP64)
// two of 256.
template <typename R> struct FftBounds {
    static constexpr int NT = sizeof(R) == 8 ? 256 : 512, MINB = 2;
};

template <typename R, int MODE, int V>
__global__ void __launch_bounds__(FftBounds<R>::NT, FftBounds<R>::MINB)
    rows_regs_kernel(R *f, typename Cplx<R>::type *Z, const __grid_constant__ PassGeom g, R coef,
                     const __grid_constant__ FftLen L, const typename Cplx<R>::type *tw) {
    typedef typename Cplx<R>::type C;
    constexpr int H = V / 2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_enter();
    LineThread lt;
    const int l = line_thread<V>(L, g, lt);
    C *buf = reinterpret_cast<C *>(smem_raw) + l * g.LS;
    const int n = L.n, sh = pad_shift<V>(n), T = 1 << lt.lgT, t = lt.t;
    const int pair = blockIdx.x * g.G + l;
    const bool on = pair < g.nlines;
    const int ra = 2 * pair;
    const bool has_b = ra + 1 < g.nrows, vec = (g.nrows & 1) == 0;
    const size_t ro = (size_t)ra * n;
    C u[V];
    auto read_pair = [&](const C *p, C &A, C &B) {  // a mode of the two rows
        if (sizeof(R) == 4 && vec) {
            const float4 q = *reinterpret_cast<const float4 *>(p);
            A = C{(R)q.x, (R)q.y};
            B = C{(R)q.z, (R)q.w};
        } else {
            A = p[0];
            B = has_b ? p[1] : C{0, 0};
        }
    };
    if constexpr (MODE == kRowInverse || MODE == kRowInverseNext) {
        // Hermitian extension: this thread reads the modes t + j T below n/2 once; the
        // conjugate half goes to its owners through the buffer.  The zero and Nyquist
        // bins are real.  Values are held with real and imaginary part exchanged.
        if (on) {
            C A, B;
            const C *p = Z + ((uint64_t)(uint32_t)t * (uint32_t)g.nrows + (uint32_t)ra);
            const size_t step = (size_t)T * g.nrows;
#pragma unroll
            for (int j = 0; j < H; ++j, p += step) {
                const int i = t + j * T;
                read_pair(p, A, B);
                if (i == 0) A.y = B.y = R(0);
                u[j] = C{A.y + B.x, A.x - B.y};
                if (i > 0) buf[slot_of(n - i, sh)] = C{B.x - A.y, A.x + B.y};
            }
            if (t == 0) {
                read_pair(p, A, B);  // mode n/2
                buf[slot_of(n / 2, sh)] = C{B.x, A.x};
            }
        }
        lt.sync();
#pragma unroll
        for (int j = H; j < V; ++j) u[j] = buf[slot_of(t + j * T, sh)];
    } else {
        if (on) {
#pragma unroll
            for (int j = 0; j < V; ++j) {
                const int i = t + j * T;
                R a = f[ro + i], b = has_b ? f[ro + n + i] : R(0);
                if (MODE == kRowCube) a = (a * a) * a, b = (b * b) * b;
                u[j] = C{coef * a, coef * b};
            }
        }
    }
#pragma unroll 1
    for (int pass = 0; pass < (MODE == kRowInverseNext ? 2 : 1); ++pass) {
        fft_regs(u, buf, L, tw, lt);
        if ((MODE == kRowInverse || MODE == kRowInverseNext) && pass == 0) {
            if (on) {
#pragma unroll
                for (int j = 0; j < V; ++j) {
                    const int i = t + j * T;
                    const R a = u[j].y, b = u[j].x;
                    f[ro + i] = a;
                    if (has_b) f[ro + n + i] = b;
                    if (MODE == kRowInverseNext) u[j] = C{coef * ((a * a) * a), coef * ((b * b) * b)};
                }
            }
        }
    }
    if constexpr (MODE != kRowInverse) {
        // separate the two rows: A = z_k + conj z_(n-k), B = -i (z_k - conj z_(n-k))
        // (coef holds the 1/2); the upper half reaches its partners through the buffer
        lt.sync();
#pragma unroll
        for (int j = H; j < V; ++j) buf[slot_of(t + j * T, sh)] = u[j];
        lt.sync();
        if (on) {
            auto put = [&](C *p, C zk, C zc) {
                const C A{zk.x + zc.x, zk.y - zc.y}, B{zk.y + zc.y, zc.x - zk.x};
                if (sizeof(R) == 4 && vec) {
                    *reinterpret_cast<float4 *>(p) = make_float4((float)A.x, (float)A.y, (float)B.x, (float)B.y);
                } else {
                    p[0] = A;
                    if (has_b) p[1] = B;
                }
            };
            // from the highest mode down (see lines_regs_kernel)
            const size_t step = (size_t)T * g.nrows;
            C *p = Z + ((uint64_t)(uint32_t)(t + H * T) * (uint32_t)g.nrows + (uint32_t)ra);
            if (t == 0) put(p, u[H], u[H]);
#pragma unroll
            for (int j = H - 1; j >= 0; --j) {
                const int k = t + j * T;
                p -= step;
                put(p, u[j], k == 0 ? u[j] : buf[slot_of(n - k, sh)]);
            }
        }
    }
}

// What a CTA will want from HBM and would otherwise wait for: its lines of the resident
// spectrum, needed only after the forward transform, and the lines of Z of the CTA that
// runs `ahead` CTAs later.
template <typename C>
__device__ __forceinline__ void prefetch_lines(const C *Z, const C *uh, const PassGeom &g, int n, bool update, size_t base,
                                               int l, int t, int T) {
    if (g.per_kx == 0) {
        if (threadIdx.x != 0) return;
        const long long first = (long long)blockIdx.x * g.G, next = first + (long long)g.ahead * g.G;
        if (update) prefetch_l2(uh + first * n, (uint32_t)(min((long long)g.G, g.nlines - first) * n * sizeof(C)));
        if (g.ahead && next < g.nlines)
            prefetch_l2(Z + next * n, (uint32_t)(min((long long)g.G, g.nlines - next) * n * sizeof(C)));
    } else if (update && l == 0) {
        for (int i = t; i < n; i += T)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(__cvta_generic_to_global(uh + base + (uint64_t)(uint32_t)i * g.ny)) : "memory");
    }
}

template <typename R, int MODE, int MODEL, int V>
__global__ void __launch_bounds__(FftBounds<R>::NT, FftBounds<R>::MINB)
    lines_regs_kernel(typename Cplx<R>::type *Z, typename Cplx<R>::type *uh, const __grid_constant__ PassGeom g, const __grid_constant__ FftLen L,
                      const typename Cplx<R>::type *tw, const R *kx2, const R *ky2, const R *kz2, SpecCoef<R> c) {
    typedef typename Cplx<R>::type C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_enter();
    LineThread lt;
    const int l = line_thread<V>(L, g, lt);
    C *buf = reinterpret_cast<C *>(smem_raw) + l * g.LS;
    const int T = 1 << lt.lgT, t = lt.t;
    size_t base;       // first point of the line
    uint32_t es;       // elements between its points (a line spans less than 2^31)
    R kb = 0;          // the squared wavenumber of the other axes
    const R *kl;       // and along the line
    bool on;
    if (g.per_kx == 0) {  // y lines: line = kx * nz + z
        const int line = blockIdx.x * g.G + l;
        on = line < g.nlines;
        base = (size_t)line * L.n;
        es = 1;
        kl = ky2;
        if (MODE == kLineUpdate && on) kb = kx2[line];  // 2D only: nz == 1
    } else {              // z lines: adjacent y within one kx
        const int kx = blockIdx.x / g.per_kx, y = (blockIdx.x - kx * g.per_kx) * g.G + l;
        on = y < g.ny;
        base = (size_t)kx * g.nz * g.ny + y;
        es = g.ny;
        kl = kz2;
        if (MODE == kLineUpdate && on) kb = kx2[kx] + ky2[y];
    }
    if (MODE == kLineUpdate || g.ahead) prefetch_lines(Z, uh, g, L.n, MODE == kLineUpdate, base, l, t, T);
    // Addresses advance by `step`; the stores at the end run backwards, so that the compiler
    // does not keep the loads' 16 addresses for them (it spilled 430 bytes per thread).
    const size_t step = (size_t)T * es, own = base + (uint64_t)(uint32_t)t * es;
    C u[V];
    if (on) {
        const C *p = Z + own;
#pragma unroll
        for (int j = 0; j < V; ++j, p += step) u[j] = MODE == kLineInverse ? swapped(*p) : *p;
    }
#pragma unroll 1
    for (int pass = 0; pass < (MODE == kLineUpdate ? 2 : 1); ++pass) {
        fft_regs(u, buf, L, tw, lt);
        if (MODE == kLineUpdate && pass == 0 && on) {
            C *p = uh + own;
            const R *k = kl + t;
#pragma unroll
            for (int j = 0; j < V; ++j, p += step, k += T) u[j] = swapped(update_mode<R, MODEL>(p, u[j], kb + *k, c));
        }
    }
    if (on) {
        C *p = Z + own + (V - 1) * step;
#pragma unroll
        for (int j = V - 1; j >= 0; --j, p -= step) *p = MODE == kLineForward ? u[j] : swapped(u[j]);
    }
}

// ============================================ other lengths, shared memory ==
//
// A mixed-radix Stockham transform (radices 8, 4, 2, 3, 5, 7) of G lines in shared
// memory: at each stage every thread reads its butterflies' inputs, applies the
// twiddles, takes the radix-R transform and stores the outputs at their sorted
// positions in a second buffer (the two alternate, one barrier per stage).

constexpr int kMixV = 8;  // points of a line per thread

// 2, 4 and 8 points
template <typename C> __device__ __forceinline__ void dft(C (&u)[2]) {
    const C t = u[0];
    u[0] = cadd(t, u[1]);
    u[1] = csub(t, u[1]);
}
template <typename C> __device__ __forceinline__ void dft4(C &u0, C &u1, C &u2, C &u3) {
    const C t0 = cadd(u0, u2), t1 = csub(u0, u2), t2 = cadd(u1, u3), d = csub(u1, u3);
    const C t3{d.y, -d.x};
    u0 = cadd(t0, t2);
    u2 = csub(t0, t2);
    u1 = cadd(t1, t3);
    u3 = csub(t1, t3);
}
template <typename C> __device__ __forceinline__ void dft(C (&u)[4]) { dft4(u[0], u[1], u[2], u[3]); }
template <typename C> __device__ __forceinline__ void dft(C (&u)[8]) {
    C e0 = u[0], e1 = u[2], e2 = u[4], e3 = u[6], o0 = u[1], o1 = u[3], o2 = u[5], o3 = u[7];
    dft4(e0, e1, e2, e3);
    dft4(o0, o1, o2, o3);
    u[0] = cadd(e0, o0);
    u[4] = csub(e0, o0);
    u[2] = C{e2.x + o2.y, e2.y - o2.x};
    u[6] = C{e2.x - o2.y, e2.y + o2.x};
    u[1] = e1, u[5] = o1;
    butterfly(u[1], u[5], root16<C>(2));
    u[3] = e3, u[7] = o3;
    const C w3{root16<C>(2).y, -root16<C>(2).x};  // exp(-2 pi i 3/8)
    butterfly(u[3], u[7], w3);
}

// Odd radices from the sums and differences of the conjugate pairs u_l, u_(R-l):
// X_m = u_0 + sum_l c_lm (u_l + u_(R-l)) -+ i sum_l s_lm (u_l - u_(R-l)), the cosine and
// sine parts shared by outputs m and R - m (radix 3: 16 operations, 5: 40, 7: 84).
template <int RAD, typename C> __device__ __forceinline__ void dft_odd(C (&u)[RAD]) {
    typedef decltype(u[0].x) R;
    constexpr int H = (RAD - 1) / 2;
    constexpr double cs[3][4] = {{1.0, -0.5, 0, 0},
                                 {1.0, 0.30901699437494742410, -0.80901699437494742410, 0},
                                 {1.0, 0.62348980185873353053, -0.22252093395631440429, -0.90096886790241912624}};
    constexpr double sn[3][4] = {{0.0, 0.86602540378443864676, 0, 0},
                                 {0.0, 0.95105651629515357212, 0.58778525229247312917, 0},
                                 {0.0, 0.78183148246802980871, 0.97492791218182360702, 0.43388373911755812048}};
    constexpr int row = RAD == 3 ? 0 : RAD == 5 ? 1 : 2;
    C a[H], d[H];
#pragma unroll
    for (int l = 0; l < H; ++l) a[l] = cadd(u[l + 1], u[RAD - 1 - l]), d[l] = csub(u[l + 1], u[RAD - 1 - l]);
    const C u0 = u[0];
    C s0 = u0;
#pragma unroll
    for (int l = 0; l < H; ++l) s0 = cadd(s0, a[l]);
    u[0] = s0;
#pragma unroll
    for (int m = 1; m <= H; ++m) {
        C re = u0, im{0, 0};
#pragma unroll
        for (int l = 1; l <= H; ++l) {
            const int e = (m * l) % RAD, f = e <= H ? e : RAD - e;  // cos even, sin odd in e
            const R cc = (R)cs[row][f], ss = (R)(e <= H ? sn[row][f] : -sn[row][f]);
            re = C{FMA(cc, a[l - 1].x, re.x), FMA(cc, a[l - 1].y, re.y)};
            im = l == 1 ? C{ss * d[0].x, ss * d[0].y} : C{FMA(ss, d[l - 1].x, im.x), FMA(ss, d[l - 1].y, im.y)};
        }
        u[m] = C{re.x + im.y, re.y - im.x};
        u[RAD - m] = C{re.x - im.y, re.y + im.x};
    }
}
template <typename C> __device__ __forceinline__ void dft(C (&u)[3]) { dft_odd<3>(u); }
template <typename C> __device__ __forceinline__ void dft(C (&u)[5]) { dft_odd<5>(u); }
template <typename C> __device__ __forceinline__ void dft(C (&u)[7]) { dft_odd<7>(u); }

// One radix-RAD stage on G lines of n points from buf into out (line l at offset l n of
// each; p is the product of the radices of the earlier stages).  Butterfly b of a line
// reads its inputs at stride n/RAD and writes them at stride p from (b - k) RAD + k,
// k = b mod p.  FP64 reads every twiddle power from the table, FP32 one and multiplies.
template <int RAD, typename C>
__device__ __forceinline__ void mixed_stage(const C *buf, C *out, int n, int G, int p, const C *tw) {
    constexpr int QMAX = (kMixV + RAD - 1) / RAD;
    const int m = n / RAD, step = m / p, total = G * m;
#pragma unroll
    for (int q = 0; q < QMAX; ++q) {
        const int b = threadIdx.x + q * blockDim.x;
        if (b >= total) break;
        const int line = b / m, i = b - line * m, k = p == 1 ? 0 : i % p, src = line * n + i;
        C u[RAD];
#pragma unroll
        for (int j = 0; j < RAD; ++j) u[j] = buf[src + j * m];
        if (p > 1) {
            const C w1 = __ldg(tw + k * step);
            C w = w1;
#pragma unroll
            for (int j = 1; j < RAD; ++j) {
                if (j > 1) w = sizeof(C) == 16 ? __ldg(tw + j * k * step) : cmul(w, w1);
                u[j] = cmul(u[j], w);
            }
        }
        dft(u);
        const int ob = line * n + (i - k) * RAD + k;
#pragma unroll
        for (int j = 0; j < RAD; ++j) out[ob + j * p] = u[j];
    }
    __syncthreads();
}

// Forward transform of G lines in buf (alt: the second buffer); returns the buffer that
// holds the result.  After a barrier, with at least G n / kMixV threads.
template <typename C>
__device__ __forceinline__ C *fft_lines(C *buf, C *alt, const FftLen &L, int G, const C *tw_all) {
    const C *tw = tw_all + L.tw_off;
    int p = 1;
#pragma unroll 1
    for (int s = 0; s < L.nst; ++s) {
        switch (L.rad[s]) {
        case 8: mixed_stage<8>(buf, alt, L.n, G, p, tw); break;
        case 4: mixed_stage<4>(buf, alt, L.n, G, p, tw); break;
        case 2: mixed_stage<2>(buf, alt, L.n, G, p, tw); break;
        case 3: mixed_stage<3>(buf, alt, L.n, G, p, tw); break;
        case 5: mixed_stage<5>(buf, alt, L.n, G, p, tw); break;
        default: mixed_stage<7>(buf, alt, L.n, G, p, tw); break;
        }
        p *= L.rad[s];
        C *t = buf;
        buf = alt;
        alt = t;
    }
    return buf;
}

template <typename R, int MODE>
__global__ void __launch_bounds__(512)
    rows_mixed_kernel(R *f, typename Cplx<R>::type *Z, const __grid_constant__ PassGeom g, R coef,
                      const __grid_constant__ FftLen L, const typename Cplx<R>::type *tw) {
    typedef typename Cplx<R>::type C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *buf = reinterpret_cast<C *>(smem_raw), *alt = buf + g.G * L.n;
    pdl_enter();
    const int n = L.n, half = n / 2, pair0 = blockIdx.x * g.G, nl = min(g.G, g.nlines - pair0);
    if constexpr (MODE == kRowInverse || MODE == kRowInverseNext) {
        // both halves of the Hermitian extension from one read (parts exchanged)
        for (int e = threadIdx.x; e < nl * (half + 1); e += blockDim.x) {
            const int k = e / nl, l = e - k * nl, ra = 2 * (pair0 + l);
            const C *p = Z + (size_t)k * g.nrows + ra;
            C A = p[0], B = ra + 1 < g.nrows ? p[1] : C{0, 0};
            if (k == 0 || 2 * k == n) A.y = B.y = R(0);
            buf[l * n + k] = C{A.y + B.x, A.x - B.y};
            if (k > 0 && 2 * k < n) buf[l * n + n - k] = C{B.x - A.y, A.x + B.y};
        }
    } else {
        for (int e = threadIdx.x; e < nl * n; e += blockDim.x) {
            const int l = e / n, i = e - l * n, ra = 2 * (pair0 + l);
            R a = f[(size_t)ra * n + i], b = ra + 1 < g.nrows ? f[(size_t)(ra + 1) * n + i] : R(0);
            if (MODE == kRowCube) a = (a * a) * a, b = (b * b) * b;
            buf[e] = C{coef * a, coef * b};
        }
    }
    __syncthreads();
    C *res = fft_lines(buf, alt, L, nl, tw);
    if constexpr (MODE == kRowInverse || MODE == kRowInverseNext) {
        for (int e = threadIdx.x; e < nl * n; e += blockDim.x) {
            const int l = e / n, i = e - l * n, ra = 2 * (pair0 + l);
            const R a = res[e].y, b = res[e].x;
            f[(size_t)ra * n + i] = a;
            if (ra + 1 < g.nrows) f[(size_t)(ra + 1) * n + i] = b;
            if (MODE == kRowInverseNext) res[e] = C{coef * ((a * a) * a), coef * ((b * b) * b)};
        }
        if (MODE == kRowInverse) return;
        __syncthreads();
        res = fft_lines(res, res == buf ? alt : buf, L, nl, tw);
    }
    for (int e = threadIdx.x; e < nl * (half + 1); e += blockDim.x) {
        const int k = e / nl, l = e - k * nl, ra = 2 * (pair0 + l);
        const C zk = res[l * n + k], zc = res[l * n + (k == 0 ? 0 : n - k)];
        C *p = Z + (size_t)k * g.nrows + ra;
        p[0] = C{zk.x + zc.x, zk.y - zc.y};
        if (ra + 1 < g.nrows) p[1] = C{zk.y + zc.y, zc.x - zk.x};
    }
}

template <typename R, int MODE, int MODEL>
__global__ void __launch_bounds__(512)
    lines_mixed_kernel(typename Cplx<R>::type *Z, typename Cplx<R>::type *uh, const __grid_constant__ PassGeom g, const __grid_constant__ FftLen L,
                       const typename Cplx<R>::type *tw, const R *kx2, const R *ky2, const R *kz2, SpecCoef<R> c) {
    typedef typename Cplx<R>::type C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *buf = reinterpret_cast<C *>(smem_raw), *alt = buf + g.G * L.n;
    pdl_enter();
    const int n = L.n;
    int nl, first, kx = 0;  // lines of this CTA; first line (contiguous) or first y (strided)
    size_t base;
    const bool contig = g.per_kx == 0;
    if (contig) {
        first = blockIdx.x * g.G;
        nl = min(g.G, g.nlines - first);
        base = (size_t)first * n;
    } else {
        kx = blockIdx.x / g.per_kx;
        first = (blockIdx.x - kx * g.per_kx) * g.G;
        nl = min(g.G, g.ny - first);
        base = (size_t)kx * g.nz * g.ny + first;
    }
    // element e of the group: global offset and (line, point); coalesced either way
    auto place = [&](int e, int &l, int &i) -> size_t {
        if (contig) {
            l = e / n, i = e - l * n;
            return base + e;
        }
        i = e / nl, l = e - i * nl;
        return base + l + (size_t)i * g.ny;
    };
    for (int e = threadIdx.x; e < nl * n; e += blockDim.x) {
        int l, i;
        const C v = Z[place(e, l, i)];
        buf[l * n + i] = MODE == kLineInverse ? swapped(v) : v;
    }
    __syncthreads();
    C *res = fft_lines(buf, alt, L, nl, tw);
    if constexpr (MODE == kLineUpdate) {
        for (int e = threadIdx.x; e < nl * n; e += blockDim.x) {
            int l, i;
            const size_t at = place(e, l, i);
            const R k2 = contig ? kx2[first + l] + ky2[i] : kx2[kx] + ky2[first + l] + kz2[i];
            res[l * n + i] = swapped(update_mode<R, MODEL>(uh + at, res[l * n + i], k2, c));
        }
        __syncthreads();
        res = fft_lines(res, res == buf ? alt : buf, L, nl, tw);
    }
    for (int e = threadIdx.x; e < nl * n; e += blockDim.x) {
        int l, i;
        const size_t at = place(e, l, i);
        const C v = res[l * n + i];
        Z[at] = MODE == kLineForward ? v : swapped(v);
    }
}

// ----------------------------------------------------------------- launch --

// Lines per CTA: as many as `most` threads hold, but no more than leaves every SM two
// CTAs (a small grid is bound by the SMs at work, not by full CTAs); at least `least`.
inline int lines_per_cta(int most, int least, long long lines, int n_sm) {
    int G = most;
    while (G > least && (lines + G - 1) / G < 2LL * n_sm) G /= 2;
    return std::max(G, least);
}

// geometry, threads and shared memory of a pass; a CTA interleaves up to 2^lgI_max lines
template <typename R>
void pass_shape(const SpectralPlan *P, const FftLen &L, long long lines, int lgI_max, PassGeom &g, int &threads,
                size_t &smem) {
    constexpr size_t cb = 2 * sizeof(R);
    g.ny = P->ny;
    g.nz = P->nz;
    g.nxh = P->nxh;
    g.nrows = P->ny * P->nz;
    if (L.V) {
        const int T = L.n / L.V, most = std::max(1, (L.n >= 4096 ? FftBounds<R>::NT : 256) / T);
        g.G = lines_per_cta(most, std::max(1, 32 / T), lines, P->n_sm);
        g.lgI = 0;
        while (g.lgI < lgI_max && (2 << g.lgI) <= g.G) ++g.lgI;
        // lines of adjacent threads start in different banks
        const int phase = sizeof(R) == 8 ? 8 : 16, want = g.lgI ? std::max(1, phase >> g.lgI) : 0;
        g.LS = L.n + (L.n >> (L.V == 16 ? pad_shift<16>(L.n) : pad_shift<4>(L.n)));
        while (g.lgI && g.LS % phase != want % phase) ++g.LS;
        threads = g.G * T;
        smem = cb * (size_t)g.G * g.LS;
    } else {
        const int T = (L.n + kMixV - 1) / kMixV;
        int most = std::max(1, 256 / T);
        while (most > 1 && 2 * cb * most * L.n > 48 * 1024) --most;
        g.G = lines_per_cta(most, 1, lines, P->n_sm);
        g.lgI = g.LS = 0;
        // few lines: fewer points per thread, down to 2, while an SM has under 8 warps
        int t = T;
        while (g.G * t * 2 <= 256 && 2 * t * 2 <= L.n && lines * t < 8LL * 32 * P->n_sm) t *= 2;
        threads = std::max(32, (g.G * t + 31) / 32 * 32);
        smem = 2 * cb * (size_t)g.G * L.n;
    }
}

template <typename K> cudaError_t allow_smem(K kern, size_t bytes) {
    if (bytes > 48 * 1024) return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    return cudaSuccess;
}

template <typename R, int MODE>
static cudaError_t rows_mode(const SpectralPlan *P, R *f, typename Cplx<R>::type *Z, R coef, cudaStream_t s) {
    typedef typename Cplx<R>::type C;
    PassGeom g{};
    int threads;
    size_t smem;
    g.nlines = (P->ny * P->nz + 1) / 2;
    // FP32: adjacent threads take up to four row pairs, 64 bytes of every mode (one pair
    // is half a sector: 128^3 47.1 us per step with one, 40.2 with two, 37.3 with four)
    pass_shape<R>(P, P->lx, g.nlines, sizeof(R) == 4 ? 2 : 0, g, threads, smem);
    const unsigned blocks = (unsigned)((g.nlines + g.G - 1) / g.G);
    auto kern = P->lx.V == 16  ? rows_regs_kernel<R, MODE, 16>
                : P->lx.V == 4 ? rows_regs_kernel<R, MODE, 4>
                               : rows_mixed_kernel<R, MODE>;
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(kern, dim3(blocks), dim3(threads), smem, s, f, Z, g, coef, P->lx, static_cast<const C *>(P->tw));
}

template <typename R>
cudaError_t run_rows(const SpectralPlan *P, RowMode mode, R *f, typename Cplx<R>::type *Z, R coef, cudaStream_t s) {
    switch (mode) {
    case kRowLoad: return rows_mode<R, kRowLoad>(P, f, Z, coef, s);
    case kRowCube: return rows_mode<R, kRowCube>(P, f, Z, coef, s);
    case kRowInverse: return rows_mode<R, kRowInverse>(P, f, Z, coef, s);
    default: return rows_mode<R, kRowInverseNext>(P, f, Z, coef, s);
    }
}

template <typename R, int MODE, int MODEL>
static cudaError_t lines_mode(const SpectralPlan *P, int axis, const SpecCoef<R> &c, typename Cplx<R>::type *Z,
                              cudaStream_t s) {
    typedef typename Cplx<R>::type C;
    const FftLen &L = axis == 1 ? P->ly : P->lz;
    PassGeom g{};
    int threads;
    size_t smem;
    const long long lines = (long long)P->nxh * (axis == 1 ? P->nz : P->ny);
    g.nlines = (int)lines;
    pass_shape<R>(P, L, lines, axis == 1 ? 0 : 4, g, threads, smem);
    unsigned blocks = (unsigned)((lines + g.G - 1) / g.G);
    if (axis == 2) {
        g.per_kx = (P->ny + g.G - 1) / g.G;
        blocks = (unsigned)(P->nxh * g.per_kx);
    }
    g.ahead = axis == 1 && lines * L.n * 2 * sizeof(R) > (32u << 20) ? 2 * P->n_sm : 0;
    auto kern = L.V == 16  ? lines_regs_kernel<R, MODE, MODEL, 16>
                : L.V == 4 ? lines_regs_kernel<R, MODE, MODEL, 4>
                           : lines_mixed_kernel<R, MODE, MODEL>;
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    const R *k2 = static_cast<const R *>(P->k2);
    return launch_pdl(kern, dim3(blocks), dim3(threads), smem, s, Z, static_cast<C *>(P->uh), g, L,
                      static_cast<const C *>(P->tw), k2 + P->lx.k2_off, k2 + P->ly.k2_off, k2 + P->lz.k2_off, c);
}

template <typename R>
cudaError_t run_lines(const SpectralPlan *P, int axis, LineMode mode, int model, const SpecCoef<R> &c,
                      typename Cplx<R>::type *Z, cudaStream_t s) {
    switch (mode) {
    case kLineForward: return lines_mode<R, kLineForward, AC>(P, axis, c, Z, s);
    case kLineInverse: return lines_mode<R, kLineInverse, AC>(P, axis, c, Z, s);
    default:
        return model == AC ? lines_mode<R, kLineUpdate, AC>(P, axis, c, Z, s)
                           : lines_mode<R, kLineUpdate, CH>(P, axis, c, Z, s);
    }
}

#endif  // SP_SPECTRAL_KERNELS

}  // namespace sp

// sp_reduce.cu -- FP64 reductions over a resident field: mass, discrete Landau
// free energy, sums, sum of squares, min and max.
//
// Mass M = h^d sum phi (conserved by Model B, Eq. (model-b)); free energy
// F_h = h^d sum [1/2 sum_axes ((phi_{i+e} - phi_i)/h)^2 - c1/2 phi^2 + c2/4 phi^4],
// the Landau density whose functional derivative (Eq. (2) of the paper, first-
// order case) gives Models A and B, with forward differences.
//
// Two passes, deterministic for a fixed grid size: every thread keeps a
// Neumaier-compensated (sum, correction) pair over a grid-stride range (fed
// with FP64 sums of 16-value blocks); warps combine pairs with shuffles,
// blocks through shared memory, and each block writes its pair to a scratch
// array; a single block then combines the block pairs in index order and
// writes the scaled result.
#include <cmath>
#include <type_traits>

#include "sp_internal.h"

namespace sp {

__device__ __forceinline__ void neu_add(double &s, double &c, double x) {
    const double t = s + x;
    c += (fabs(s) >= fabs(x)) ? ((s - t) + x) : ((x - t) + s);
    s = t;
}

__device__ __forceinline__ void neu_merge(double &s, double &c, double s2, double c2) {
    neu_add(s, c, s2);
    c += c2;
}

template <int WHAT>
__device__ __forceinline__ void combine(double &s, double &c, double s2, double c2) {
    if constexpr (WHAT == SP_MIN_U) s = fmin(s, s2);
    else if constexpr (WHAT == SP_MAX_U) s = fmax(s, s2);
    else neu_merge(s, c, s2, c2);
}

template <int WHAT>
__device__ __forceinline__ void block_combine(double &s, double &c) {
    __shared__ double ws[32], wc[32];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const double s2 = __shfl_down_sync(0xffffffffu, s, off);
        const double c2 = __shfl_down_sync(0xffffffffu, c, off);
        combine<WHAT>(s, c, s2, c2);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) { ws[warp] = s; wc[warp] = c; }
    __syncthreads();
    if (warp == 0) {
        s = lane < nw ? ws[lane] : ((WHAT == SP_MIN_U) ? INFINITY : (WHAT == SP_MAX_U ? -INFINITY : 0.0));
        c = lane < nw ? wc[lane] : 0.0;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const double s2 = __shfl_down_sync(0xffffffffu, s, off);
            const double c2 = __shfl_down_sync(0xffffffffu, c, off);
            combine<WHAT>(s, c, s2, c2);
        }
    }
}

// Point value of a plain reduction (sum, mass, sum of squares) in FP64.
template <int WHAT> __device__ __forceinline__ double point_value(double p) {
    if constexpr (WHAT == SP_SUMSQ_U) return p * p;
    else return p;
}

// Exact widening to FP64 with integer instructions.  A conversion instruction runs at
// the rate of the FP64 pipe (about 2 per clock per SM here; one that is predicated off
// still takes its slot), integer instructions at 32 times that: the exponent is moved,
// a denormal first scaled by 2^64, zeros, infinities and NaN by their own offsets.
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) {
    const bool small = fabsf(x) < 0x1p-126f;
    const uint32_t b = __float_as_uint(small ? x * 0x1p64f : x), mag = b & 0x7fffffffu;
    const uint32_t off = mag >= 0x7f800000u ? 0x70000000u : mag == 0u ? 0u : small ? 0x34000000u : 0x38000000u;
    return __hiloint2double((int)((b & 0x80000000u) | ((mag >> 3) + off)), (int)(b << 29));
}

// The same of normal values alone.
__device__ __forceinline__ double widen_normal(double x) { return x; }
__device__ __forceinline__ double widen_normal(float x) {
    const int b = __float_as_int(x);
    return __hiloint2double(((b >> 3) & (int)0x8fffffff) + 0x38000000, b << 29);
}

// Sum of a block of 32 FP32 values (BF16 values widen to FP32 exactly) in
// fixed point, with integer arithmetic only.  A value with biased exponent e
// and 24-bit significand m is m * 2^(max(e,1) - 150).  With E the largest
// exponent of the block, every value is expressed in units of 2^(E - 150 - K),
// K = 33: v = floor(m * 2^(K - (E - max(e,1)))), so the block's largest values
// keep every bit and values more than 2^33 times smaller lose the bits below
// the unit (an error below 2^-56 max|x| each, at most 2^-51 max|x| per block).
// 32 values of at most 24 + 33 bits sum exactly in 62 bits.  The integer sum is
// converted to FP64 once (one rounding) and scaled by the exact power of two.
// A block holding an infinity or a NaN (E = 255) is summed in FP64 instead, so
// that those propagate as in plain summation.
__device__ __forceinline__ double fixed_block_sum32(const float *x) {
    constexpr int K = 33;
    uint32_t b[32];
    int emax = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        b[j] = __float_as_uint(x[j]);
        emax = max(emax, (int)((b[j] >> 23) & 0xffu));
    }
    if (emax == 255) {
        double s = 0.0;
#pragma unroll
        for (int j = 0; j < 32; ++j) s += (double)x[j];
        return s;
    }
    const int em = max(emax, 1);
    long long acc = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const int e = (int)((b[j] >> 23) & 0xffu);
        const unsigned long long m = (unsigned long long)((b[j] & 0x7fffffu) | (e ? 0x800000u : 0u));
        const int sh = min(em - max(e, 1), 63);
        const long long v = (long long)((m << K) >> sh);
        const long long sgn = -(long long)(b[j] >> 31);  // 0 or -1
        acc += (v ^ sgn) - sgn;
    }
    // 2^(em - 150 - K) as an FP64 power of two (em - 183 >= -182: a normal number)
    const double unit = __longlong_as_double((long long)(em - 150 - K + 1023) << 52);
    return __ll2double_rn(acc) * unit;
}

// Block partials.  Sums: each thread reads 16-byte vectors in a grid-stride
// loop.  FP32 / BF16 mass and plain sums: the vectors are taken in groups of
// 32 values per thread (a warp's group interleaves its lanes, so every load
// instruction is coalesced), each group is summed exactly in fixed point
// (fixed_block_sum32) and folded into the thread's Neumaier pair, so the FP64
// pipe (slow on this part) sees ~0.3 operations per value; error bound u|S| +
// 5u sum|x| per thread (truncation 4u, conversion u).  FP64 fields and sums of
// squares: plain FP64 additions over blocks of 16 values folded into the
// Neumaier pair, ~2 FP64 operations per value, bound u|S| + 15u sum|x|.  The
// remaining vectors and the scalar tail take the FP64 block path.  Min / max run
// in the compute type.  The free energy has its own kernel below.
template <typename T, int WHAT>
__global__ void __launch_bounds__(kReduceThreads)
reduce_partial_kernel(const T *__restrict__ f, uint64_t N, double *__restrict__ partials) {
    typedef typename Cmp<T>::type C;
    constexpr int VE = 16 / sizeof(T);       // values per vector
    constexpr int kBlockVecs = (16 + VE - 1) / VE;
    double s = (WHAT == SP_MIN_U) ? INFINITY : (WHAT == SP_MAX_U ? -INFINITY : 0.0), c = 0.0;
    const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    {
        // vector part when the base is 16-byte aligned (library buffers always are;
        // a caller's pointer may not be), then the scalar tail
        const bool aligned = (reinterpret_cast<uintptr_t>(f) & 15u) == 0;
        const uint64_t NV = aligned ? N / VE : 0;
        C mn = C(INFINITY), mx = C(-INFINITY);
        double blk = 0.0;
        int nb = 0;
        uint64_t v0 = 0;  // first vector of the FP64 block path
        if constexpr (!std::is_same<T, double>::value && (WHAT == SP_MASS || WHAT == SP_SUM_U)) {
            constexpr int G = 32 / VE;  // vectors per thread per group
            const uint64_t lane = threadIdx.x & 31u, warp = tid >> 5;
            const uint64_t nwarps = stride >> 5;
            const uint64_t ngroups = NV / (32u * G);
            for (uint64_t gi = warp; gi < ngroups; gi += nwarps) {
                float x[32];
#pragma unroll
                for (int j = 0; j < G; ++j) {
                    C xv[VE];
                    load_vec<T, VE>(f + ((gi * G + j) * 32u + lane) * VE, xv);
#pragma unroll
                    for (int q = 0; q < VE; ++q) x[j * VE + q] = xv[q];
                }
                neu_add(s, c, fixed_block_sum32(x));
            }
            v0 = ngroups * 32u * G;
        }
        for (uint64_t v = v0 + tid; v < NV; v += stride) {
            C x[VE];
            load_vec<T, VE>(f + v * VE, x);
            if constexpr (WHAT == SP_MIN_U) {
#pragma unroll
                for (int j = 0; j < VE; ++j) mn = fmin(mn, x[j]);
            } else if constexpr (WHAT == SP_MAX_U) {
#pragma unroll
                for (int j = 0; j < VE; ++j) mx = fmax(mx, x[j]);
            } else {
#pragma unroll
                for (int j = 0; j < VE; ++j) blk += point_value<WHAT>(widen(x[j]));
                if (++nb == kBlockVecs) {
                    neu_add(s, c, blk);
                    blk = 0.0;
                    nb = 0;
                }
            }
        }
        for (uint64_t i = NV * VE + tid; i < N; i += stride) {
            const C x = to_c(f[i]);
            if constexpr (WHAT == SP_MIN_U) mn = fmin(mn, x);
            else if constexpr (WHAT == SP_MAX_U) mx = fmax(mx, x);
            else blk += point_value<WHAT>((double)x);
        }
        if constexpr (WHAT == SP_MIN_U) s = (double)mn;
        else if constexpr (WHAT == SP_MAX_U) s = (double)mx;
        else neu_add(s, c, blk);
    }
    block_combine<WHAT>(s, c);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = s;
        partials[2 * blockIdx.x + 1] = c;
    }
}

// Energy density of one point, term by term (the definition): for values that the sums below
// are not made for.
__device__ __noinline__ double energy_density(int dims, int extra, const double *p, double h, double c1, double c2, double c3) {
    const double gx = (p[1] - p[0]) / h, gy = (p[2] - p[0]) / h;
    double g2 = gx * gx + gy * gy;
    if (dims == 3) {
        const double gz = (p[3] - p[0]) / h;
        g2 = g2 + gz * gz;
    }
    const double p2 = p[0] * p[0], r = p[4];
    if (extra == 1) return 0.5 * g2 - 0.5 * c1 * p2 + 0.25 * c2 * p2 * p2 + 0.5 * r * r - c3 * p2 * r;
    double q = r * r + p[5] * p[5];
    if (dims == 3) q = q + p[6] * p[6];
    const double d = 0.5 * g2 - 0.5 * c1 * p2 + 0.25 * c2 * p2 * p2;
    return extra == 2 ? d + 0.5 * q : d;
}

// The bits of |x| (FP64: the upper half) and the first value that the energy's sums leave to
// energy_density: infinities and NaN, in FP64 from 2^200 on, whose fourth power may overflow.
__device__ __forceinline__ uint32_t size_bits(float x) { return __float_as_uint(x) & 0x7fffffffu; }
__device__ __forceinline__ uint32_t size_bits(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }
template <typename C> constexpr uint32_t kSizeLimit = sizeof(C) == 8 ? 0x4c700000u : 0x7f800000u;
// below kUsualLimit: values that widen_normal takes, below the limit above
__device__ __forceinline__ uint32_t usual_bits(float x) { return size_bits(x) - 0x00800000u; }
__device__ __forceinline__ uint32_t usual_bits(double x) { return size_bits(x); }
template <typename C> constexpr uint32_t kUsualLimit = sizeof(C) == 8 ? 0x4c700000u : 0x7f000000u;

// a 2^k as an unevaluated sum (x + y)
__device__ __noinline__ double2 fixed_value(__int128 a, int k) {
    const bool neg = a < 0;
    const unsigned __int128 m = neg ? -(unsigned __int128)a : (unsigned __int128)a;
    auto part = [&](int at) {  // 43 bits from `at` on: below the 2^52 that the upper half adds
        const uint64_t b = (uint64_t)(m >> at) & ((1ull << 43) - 1);
        return __hiloint2double((int)(0x43300000u | (uint32_t)(b >> 32)), (int)(uint32_t)b) - 0x1p52;
    };
    const double c0 = part(0), c1 = part(43) * 0x1p43, c2 = part(86) * 0x1p86;
    const double hi = c2 + c1, lo = (c1 - (hi - c2)) + c0;
    double x, y;
    if (k > -900 && k < 900) {
        const double p = __hiloint2double((k + 1023) << 20, 0);
        x = hi * p, y = lo * p;
    } else {
        x = scalbn(hi, k), y = scalbn(lo, k);
    }
    return neg ? double2{-x, -y} : double2{x, y};
}

// A sum of finite doubles in fixed point, with integer instructions only: 96 bits of units of
// 2^(top - 1097), top the largest biased exponent that they hold (68 at least, so that zeros and
// denormals count as nothing).  A value keeps its bits down to 2^-74 of 2^(top - 1023), and a million
// of them fit.  Negative values are added as complements, the ones that these lack in `lack`.
struct FixedSum {
    uint32_t w0 = 0, w1 = 0, w2 = 0, lack = 0;
    int top = 68;
    double s = 0.0, c = 0.0;  // what was summed in smaller units, a Neumaier pair
    __device__ __forceinline__ __int128 bits() const {
        return ((__int128)(int)w2 << 64 | (unsigned __int128)((uint64_t)w1 << 32 | w0)) + lack;
    }
    __device__ __forceinline__ int unit() const { return top - 1097; }
    // before values with the biased exponent e (and some of 2^12 times theirs, so that it happens seldom)
    __device__ __forceinline__ void hold(int e) {
        if (e <= top) return;
        if ((w0 | w1 | w2 | lack) != 0) {
            const double2 v = fixed_value(bits(), unit());
            neu_add(s, c, v.x);
            c += v.y;
            w0 = w1 = w2 = lack = 0;
        }
        top = e + 12;
    }
    // adds x (SIGNED false: of at least 0), whose exponent is held: its 53 bits from bit 74 on,
    // `sh` lower where x is smaller, without branches (the FP64 work of other points goes on beside it)
    template <bool SIGNED> __device__ __forceinline__ void add(double x) {
        const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
        const int sh = top + 10 - (int)(SIGNED ? (hi << 1) >> 21 : hi >> 20);
        const uint32_t m = (hi & 0xfffffu) | 0x100000u;
        const bool in = sh < 64, low = sh >= 32;
        const uint32_t x2 = low ? 0u : m, x1 = low ? (in ? m : 0u) : lo, x0 = low && in ? lo : 0u;
        uint32_t v0 = __funnelshift_r(x0, x1, sh), v1 = __funnelshift_r(x1, x2, sh), v2 = __funnelshift_r(x2, 0u, sh);
        if constexpr (SIGNED) {
            const uint32_t neg = (uint32_t)((int)hi >> 31);
            v0 ^= neg, v1 ^= neg, v2 ^= neg;
            lack -= neg;
        }
        asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
            : "+r"(w0), "+r"(w1), "+r"(w2) : "r"(v0), "r"(v1), "r"(v2));
    }
};

// Sum over a warp, in lane 0, of a 2^k, in the largest of the lanes' units.
__device__ __forceinline__ void warp_sum(__int128 &a, int &k) {
    const int km = __reduce_max_sync(0xffffffffu, k);
    a >>= min(km - k, 127);
    k = km;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const uint64_t lo = __shfl_down_sync(0xffffffffu, (uint64_t)a, off);
        const long long hi = __shfl_down_sync(0xffffffffu, (long long)(a >> 64), off);
        a += (__int128)hi << 64 | lo;
    }
}

// The values of NS FixedSums over a block, one in each of its first NS threads.
template <int NS> __device__ __forceinline__ double2 block_sums(const FixedSum (&f)[NS]) {
    constexpr int NW = kReduceThreads / 32;
    __shared__ uint64_t lo[NS * NW];
    __shared__ long long hi[NS * NW];
    __shared__ int ks[NS * NW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        __int128 a = f[i].bits();
        int k = f[i].unit();
        warp_sum(a, k);
        if (lane == 0) lo[i * NW + warp] = (uint64_t)a, hi[i * NW + warp] = (long long)(a >> 64), ks[i * NW + warp] = k;
    }
    __syncthreads();
    if (threadIdx.x >= NS) return double2{0.0, 0.0};
    const int first = threadIdx.x * NW;
    int k = ks[first];
#pragma unroll 1
    for (int w = 1; w < NW; ++w) k = max(k, ks[first + w]);
    __int128 a = 0;
#pragma unroll 1
    for (int w = 0; w < NW; ++w) {
        const __int128 part = (__int128)hi[first + w] << 64 | lo[first + w];  // (signed: the shift keeps the sign)
        a += part >> min(k - ks[first + w], 127);
    }
    return fixed_value(a, k);
}

// Free energy: block partials of sum [1/2 sum_axes ((f_{i+e} - f_i)/h)^2 - c1/2 f^2
// + c2/4 f^4] (forward differences, periodic).  EXTRA 1 (Model C) adds rho^2/2 -
// c3 f^2 rho, EXTRA 2 (Model H) the currents' |j|^2/2.
//
// The FP64 pipe bounds it (2 operations per clock per SM), so the work per point is
// 8 FP64 operations in 3D: three differences, the sum of their squares by a product and two
// multiply-adds, f^2 and f^4.  Each of the three (and what the extra fields give) is summed over all
// points for itself, exactly, in fixed point (FixedSum: the integer units are idle otherwise), and the
// coefficients, 1/(2h^2) as a sum of two doubles, are applied to the block's sums.  So nothing but a
// point's own roundings enters the sum, as with one compensated addition per point, which takes 6
// FP64 operations.  (Plain FP64 sums of 8 points before the compensated one, a rounded 1/(2h^2) and
// local densities formed per point took 9.6; their error, relative to the sum of 16^3 points of FP32
// noise at h = 1, was 1.1e-16, now 1.1e-17.)
// Every thread takes chunks of V consecutive points of a row (16-byte loads of the chunk and of
// its y and z neighbours where alignment allows; the neighbour plane comes from L2), so
// the index arithmetic is per chunk.  512^3: FP32 14.0 ms and FP64 12.7 ms with a division per
// difference, one point per thread and a Neumaier update per point; 2.38 and 2.39 ms with the
// blocks of 8; now 2.01 and 2.10, 8 operations per point at 535 Gop/s.  Chunks with infinities, NaN or
// huge values, and coefficients or steps beyond 2^+-100 (wild), take energy_density point by point.
template <typename T, int DIMS, int EXTRA>
__global__ void __launch_bounds__(kReduceThreads, kReduceBlocksPerSM)
reduce_energy_kernel(const T *__restrict__ f, const T *__restrict__ rho, const T *__restrict__ j0,
                     const T *__restrict__ j1, const T *__restrict__ j2, int nx, int ny, int nz, double2 half_inv_h2,
                     double c1, double c2, double c3, double h, int wild, double *__restrict__ partials) {
    typedef typename Cmp<T>::type C;
    constexpr int V = 16 / sizeof(T);
    const bool vec = nx % V == 0 && ((reinterpret_cast<uintptr_t>(f) | reinterpret_cast<uintptr_t>(rho) | reinterpret_cast<uintptr_t>(j0) |
                                      reinterpret_cast<uintptr_t>(j1) | reinterpret_cast<uintptr_t>(j2)) & 15u) == 0;
    const uint64_t cpr = (uint64_t)(nx + V - 1) / V, rows = (uint64_t)ny * nz, chunks = cpr * rows;
    const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    double s = 0.0, c = 0.0;
    // sums of the squared differences, of f^2, of f^4, and of rho^2 - 2 c3 f^2 rho or |j|^2
    constexpr int NS = EXTRA ? 4 : 3;
    FixedSum sum[NS];
    const double twice_c3 = 2.0 * c3;
    (void)twice_c3;
    const uint32_t limit = wild ? 0u : kUsualLimit<C>;
    for (uint64_t u = tid; u < chunks; u += stride) {
        uint64_t row;
        int x0;
        if (chunks >> 32) {
            row = u / cpr;
            x0 = (int)(u - row * cpr) * V;
        } else {
            const uint32_t r = (uint32_t)u / (uint32_t)cpr;
            x0 = (int)((uint32_t)u - r * (uint32_t)cpr) * V;
            row = r;
        }
        int y, z = 0;
        if constexpr (DIMS == 3) {
            if (rows >> 32) {
                z = (int)(row / (uint64_t)ny);
                y = (int)(row - (uint64_t)z * ny);
            } else {
                z = (int)((uint32_t)row / (uint32_t)ny);
                y = (int)((uint32_t)row - (uint32_t)z * (uint32_t)ny);
            }
        } else {
            y = (int)row;
        }
        const T *p0 = f + row * (uint64_t)nx + x0;
        const T *py = y + 1 == ny ? p0 - (uint64_t)(ny - 1) * nx : p0 + nx;
        const uint64_t plane = (uint64_t)nx * ny;
        const T *pz = z + 1 == nz ? p0 - (uint64_t)(nz - 1) * plane : p0 + plane;
        const int n = vec ? V : min(V, nx - x0);  // points of this chunk
        // the order parameter here, in y and in z; the density or the currents
        constexpr int NE = EXTRA == 1 ? 1 : EXTRA == 2 ? DIMS : 0, NX = DIMS + NE;
        C x[NX][V];
#pragma unroll
        for (int a = 0; a < NX; ++a) {
            const int k = a - DIMS;
            const T *p = a == 0   ? p0
                         : a == 1 ? py
                         : k < 0  ? pz
                                  : (EXTRA == 1 ? rho : k == 0 ? j0 : k == 1 ? j1 : j2) + row * (uint64_t)nx + x0;
            if (vec) {
                load_vec<T, V>(p, x[a]);
            } else {
#pragma unroll
                for (int j = 0; j < V; ++j) x[a][j] = j < n ? load_one(p + j) : C(1);
            }
        }
        const C last = load_one(x0 + n == nx ? p0 - x0 : p0 + n);
        uint32_t usual = usual_bits(last);
#pragma unroll
        for (int a = 0; a < NX; ++a)
#pragma unroll
            for (int j = 0; j < V; ++j) usual = max(usual, usual_bits(x[a][j]));
        double w[NX][V], wl;
        if (usual < limit) {
            wl = widen_normal(last);
#pragma unroll
            for (int a = 0; a < NX; ++a)
#pragma unroll
                for (int j = 0; j < V; ++j) w[a][j] = widen_normal(x[a][j]);
        } else {
            uint32_t size = size_bits(last);
            wl = widen(last);
#pragma unroll
            for (int a = 0; a < NX; ++a)
#pragma unroll
                for (int j = 0; j < V; ++j) {
                    w[a][j] = widen(x[a][j]);
                    size = max(size, size_bits(x[a][j]));
                }
            if (wild || size >= kSizeLimit<C>) {
                for (int j = 0; j < n; ++j) {
                    double q[7] = {};
#pragma unroll
                    for (int i = 0; i < V; ++i)
                        if (i == j) {
                            q[0] = w[0][i];
                            q[1] = i + 1 < n ? w[0][i + 1 < V ? i + 1 : 0] : wl;
                            q[2] = w[1][i];
                            if constexpr (DIMS == 3) q[3] = w[2][i];
#pragma unroll
                            for (int a = 0; a < NE; ++a) q[4 + a] = w[DIMS + a][i];
                        }
                    neu_add(s, c, energy_density(DIMS, EXTRA, q, h, c1, c2, c3));
                }
                continue;
            }
        }
        double t[NS][V];
#pragma unroll
        for (int j = 0; j < V; ++j) {
            const double p = w[0][j], dx = (j + 1 < n ? w[0][j + 1 < V ? j + 1 : 0] : wl) - p, dy = w[1][j] - p;
            double g = FMA(dy, dy, dx * dx);
            if constexpr (DIMS == 3) {
                const double dz = w[2][j] - p;
                g = FMA(dz, dz, g);
            }
            const double p2 = p * p;
            t[0][j] = g, t[1][j] = p2, t[2][j] = p2 * p2;
            if constexpr (EXTRA == 1) {
                const double r = w[DIMS][j];
                t[NS - 1][j] = FMA(-(twice_c3 * p2), r, r * r);
            }
            if constexpr (EXTRA == 2) {
                double q = w[DIMS][j] * w[DIMS][j];
#pragma unroll
                for (int a = 1; a < NE; ++a) q = FMA(w[DIMS + a][j], w[DIMS + a][j], q);
                t[NS - 1][j] = q;
            }
            if (j >= n)
#pragma unroll
                for (int i = 0; i < NS; ++i) t[i][j] = 0.0;
        }
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            uint32_t m = 0;
#pragma unroll
            for (int j = 0; j < V; ++j) m = max(m, size_bits(t[i][j]));
            sum[i].hold((int)(m >> 20));
#pragma unroll
            for (int j = 0; j < V; ++j) {
                if (EXTRA == 1 && i == 3) sum[i].template add<true>(t[i][j]);
                else sum[i].template add<false>(t[i][j]);
            }
        }
    }
    // k (x + y) of sum i, whose coefficient is k, into the pair
    const double2 coef[4] = {half_inv_h2, {-0.5 * c1, 0.0}, {0.25 * c2, 0.0}, {0.5, 0.0}};
    auto fold = [&](int i, double x, double y) {
        const double2 k = coef[i];
        const double v = k.x * x;
        neu_add(s, c, v);
        c += FMA(k.x, x, -v) + FMA(k.x, y, k.y * x);
    };
    // (the pairs are in use only after larger units or a chunk summed point by point)
    bool used = s != 0.0 || c != 0.0;
#pragma unroll
    for (int i = 0; i < NS; ++i) used |= sum[i].s != 0.0;
    if (__syncthreads_or(used)) {
#pragma unroll
        for (int i = 0; i < NS; ++i) fold(i, sum[i].s, sum[i].c);
        block_combine<SP_SUM_U>(s, c);
    }
    const double2 mine = block_sums(sum);
    if (threadIdx.x < 32) {
#pragma unroll
        for (int i = 0; i < NS; ++i) fold(i, __shfl_sync(0xffffffffu, mine.x, i), __shfl_sync(0xffffffffu, mine.y, i));
    }
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = s;
        partials[2 * blockIdx.x + 1] = c;
    }
}

template <int WHAT>
__global__ void __launch_bounds__(kReduceThreads)
reduce_final_kernel(const double *__restrict__ partials, int nblocks, double scale, double *__restrict__ out) {
    double s = (WHAT == SP_MIN_U) ? INFINITY : (WHAT == SP_MAX_U ? -INFINITY : 0.0), c = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) combine<WHAT>(s, c, partials[2 * b], partials[2 * b + 1]);
    block_combine<WHAT>(s, c);
    if (threadIdx.x == 0) {
        if constexpr (WHAT == SP_MIN_U || WHAT == SP_MAX_U) out[0] = s;
        else out[0] = scale * (isfinite(s) ? s + c : s);  // an infinite sum keeps its sign (c is NaN then)
    }
}

template <typename T, int DIMS>
static void launch_energy(const T *f, const ReduceGeom &g, double *partials, int nblocks, cudaStream_t s) {
    const T *rho = static_cast<const T *>(g.rho);
    const T *j[3] = {static_cast<const T *>(g.jq[0]), static_cast<const T *>(g.jq[1]), static_cast<const T *>(g.jq[2])};
    auto tame = [](double x) { return std::fabs(x) <= 0x1p100; };
    const int wild = !(g.h >= 0x1p-100 && tame(g.h) && tame(g.c1) && tame(g.c2) && tame(g.c3));
    // 1/(2 h^2) as a sum of two doubles (0 where no sum takes it)
    const double hh = g.h * g.h, rest = std::fma(g.h, g.h, -hh), k = wild ? 0.0 : 0.5 / hh;
    const double k2 = wild ? 0.0 : (std::fma(-k, hh, 0.5) - k * rest) / hh;
    auto kern = g.nq > 0 ? reduce_energy_kernel<T, DIMS, 2> : g.rho ? reduce_energy_kernel<T, DIMS, 1> : reduce_energy_kernel<T, DIMS, 0>;
    kern<<<nblocks, kReduceThreads, 0, s>>>(f, rho, j[0], j[1], j[2], g.nx, g.ny, g.nz, double2{k, k2}, g.c1, g.c2, g.c3,
                                            g.h, wild, partials);
}

template <typename T, int WHAT>
static cudaError_t launch_reduce_t(const void *f, const ReduceGeom &g, double *partials, int nblocks,
                                   double *out, cudaStream_t s) {
    const double scale = (WHAT == SP_MASS || WHAT == SP_FREE_ENERGY) ? g.cell_volume : 1.0;
    const T *field = static_cast<const T *>(f);
    if constexpr (WHAT == SP_FREE_ENERGY) {
        if (g.dims == 3) launch_energy<T, 3>(field, g, partials, nblocks, s);
        else launch_energy<T, 2>(field, g, partials, nblocks, s);
    } else {
        reduce_partial_kernel<T, WHAT><<<nblocks, kReduceThreads, 0, s>>>(field, (uint64_t)g.nx * g.ny * g.nz, partials);
    }
    reduce_final_kernel<WHAT><<<1, kReduceThreads, 0, s>>>(partials, nblocks, scale, out);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_reduce_dt(int what, const void *f, const ReduceGeom &g, double *partials, int nblocks,
                                    double *out, cudaStream_t s) {
    switch (what) {
    case SP_MASS: return launch_reduce_t<T, SP_MASS>(f, g, partials, nblocks, out, s);
    case SP_FREE_ENERGY: return launch_reduce_t<T, SP_FREE_ENERGY>(f, g, partials, nblocks, out, s);
    case SP_SUM_U:
    case SP_SUM_V: return launch_reduce_t<T, SP_SUM_U>(f, g, partials, nblocks, out, s);
    case SP_MIN_U: return launch_reduce_t<T, SP_MIN_U>(f, g, partials, nblocks, out, s);
    case SP_MAX_U: return launch_reduce_t<T, SP_MAX_U>(f, g, partials, nblocks, out, s);
    case SP_SUMSQ_U: return launch_reduce_t<T, SP_SUMSQ_U>(f, g, partials, nblocks, out, s);
    }
    return cudaErrorInvalidValue;
}

int reduce_blocks(uint64_t N, int n_sm) {
    const uint64_t want = (N + kReduceThreads - 1) / kReduceThreads;
    const uint64_t cap = (uint64_t)n_sm * kReduceBlocksPerSM;
    const uint64_t b = want < cap ? want : cap;
    return (int)(b > 0 ? b : 1);
}

cudaError_t launch_reduce(int dtype, int what, const void *f, const ReduceGeom &g, double *partials,
                          int nblocks, double *out, cudaStream_t s) {
    switch (dtype) {
    case SP_F64: return launch_reduce_dt<double>(what, f, g, partials, nblocks, out, s);
    case SP_F32: return launch_reduce_dt<float>(what, f, g, partials, nblocks, out, s);
    default: return launch_reduce_dt<bf16>(what, f, g, partials, nblocks, out, s);
    }
}

}  // namespace sp

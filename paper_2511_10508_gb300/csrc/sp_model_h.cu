// sp_model_h.cu -- Model H (Sec. "Model H", transverse projector at unity), a
// conserved scalar m and a d-vector current j, signs of the paper's listing:
//   mu    = -kappa lap m - c1 m + c2 m^3
//   dm/dt = lap mu - c3 div(m j)
//   dj/dt = lap j - c3 m grad mu
// grad and div are central differences of the Laplacian stencil's order.
//
// Like the paper's solver (one temporary for Model H, Table 2), the per-point
// kernels take two passes: mu for every point into a compute-precision buffer,
// then the update of m and of each component of j, which reads mu, m and j
// through periodic taps (the flux m j_a is formed at each tap, with the
// rounding of the product m * j_a).  2D FP32 / BF16 grids instead use one
// shared-memory tile pass with mu kept on chip (FP64 is bound by the FP64
// pipe, where the halo mu of a tile costs more than the buffer).  Fixed order per point (FP64 results equal the oracle's bit for bit):
//   mu  = fma(m, fma(c2, m*m, -c1), -((kappa/q_h2) * S(m)))
//   div = (D_x(m j_x) + D_y(m j_y)) [+ D_z(m j_z)]
//   m'  = fma(dt, fma(1/q_h2, S(mu), -(c3g * div)), m)
//   j_a' = fma(dt, fma(1/q_h2, S(j_a), -(c3g * (m * D_a mu))), j_a)
// with D f = f(+1) - f(-1) (radius-1 stencils) or fma(8, f(+1) - f(-1),
// -(f(+2) - f(-2))) (radius 2) and c3g = c3 / (2h) or c3 / (12h).
#include <type_traits>

#include "sp_internal.h"
#include "sp_step.cuh"

namespace sp {

// Wrapped offsets of the planes and rows within the stencil radius around a
// 256-point row segment (computed once per segment).
template <int R>
struct TapRows {
    size_t zb[2 * R + 1], yb[2 * R + 1];
    __device__ __forceinline__ TapRows(int y, int z, int nx, int ny, int nz) {
#pragma unroll
        for (int d = -R; d <= R; ++d) {
            zb[d + R] = (size_t)wrap_idx(z + d, nz) * ny * nx;
            yb[d + R] = (size_t)wrap_idx(y + d, ny) * nx;
        }
    }
    __device__ __forceinline__ size_t at(int x, int nx, int dx, int dy, int dz) const {
        return zb[dz + R] + yb[dy + R] + wrap_idx(x + dx, nx);
    }
};

struct MhArgs {
    const void *m, *j[3];
    void *mo, *jo[3];
    void *mu;
    int nx, ny, nz;
    StepConsts k;
    StepConstsF kf;
};

__device__ __forceinline__ void mh_seg(long long u, int segs, const MhArgs &a, int &x, int &y, int &z, size_t &row) {
    const long long r = u / segs;
    x = (int)(u - r * segs) * 256 + (int)threadIdx.x;
    y = (int)(r % a.ny);
    z = (int)(r / a.ny);
    row = (size_t)r * a.nx;
}

// central difference along axis A of f at the tap origin
template <int R, int A, typename Fn>
__device__ __forceinline__ auto central(const Fn &f) -> decltype(f(0, 0, 0)) {
    constexpr int ex = (A == 0), ey = (A == 1), ez = (A == 2);
    const auto d1 = f(ex, ey, ez) - f(-ex, -ey, -ez);
    if constexpr (R == 1) {
        return d1;
    } else {
        const auto d2 = f(2 * ex, 2 * ey, 2 * ez) - f(-2 * ex, -2 * ey, -2 * ez);
        return FMA(decltype(d1)(8), d1, -d2);
    }
}

template <int ST, typename T>
__global__ void __launch_bounds__(256) mh_mu_kernel(MhArgs a, int segs) {
    pdl_enter();
    typedef typename Cmp<T>::type C;
    constexpr int R = StencilInfo<ST>::r;
    const ConstsC<C> k(a.k, a.kf);
    const T *m = static_cast<const T *>(a.m);
    C *mu = static_cast<C *>(a.mu);
    const long long units = (long long)a.ny * a.nz * segs;
    for (long long u = blockIdx.x; u < units; u += gridDim.x) {
        int x, y, z;
        size_t row;
        mh_seg(u, segs, a, x, y, z, row);
        const TapRows<R> tp(y, z, a.nx, a.ny, a.nz);
        if (x >= a.nx) continue;
        auto P = [&](int dx, int dy, int dz) -> C { return to_c(m[tp.at(x, a.nx, dx, dy, dz)]); };
        mu[row + x] = ch_mu<C>(to_c(m[row + x]), stencil_sum<ST, C>(P), k);
    }
}

template <int ST, typename T, int DIMS>
__global__ void __launch_bounds__(256) mh_update_kernel(MhArgs a, int segs, typename Cmp<T>::type c3g) {
    pdl_enter();
    typedef typename Cmp<T>::type C;
    constexpr int R = StencilInfo<ST>::r;
    const ConstsC<C> k(a.k, a.kf);
    const T *m = static_cast<const T *>(a.m);
    const C *mu = static_cast<const C *>(a.mu);
    const T *j[3] = {static_cast<const T *>(a.j[0]), static_cast<const T *>(a.j[1]), static_cast<const T *>(a.j[2])};
    T *jo[3] = {static_cast<T *>(a.jo[0]), static_cast<T *>(a.jo[1]), static_cast<T *>(a.jo[2])};
    const long long units = (long long)a.ny * a.nz * segs;
    for (long long u = blockIdx.x; u < units; u += gridDim.x) {
        int x, y, z;
        size_t row;
        mh_seg(u, segs, a, x, y, z, row);
        const TapRows<R> tp(y, z, a.nx, a.ny, a.nz);
        if (x >= a.nx) continue;
        const size_t i = row + x;
        auto Pmu = [&](int dx, int dy, int dz) -> C { return mu[tp.at(x, a.nx, dx, dy, dz)]; };
        auto flux = [&](int ax) {
            return [&, ax](int dx, int dy, int dz) -> C {
                const size_t t = tp.at(x, a.nx, dx, dy, dz);
                return to_c(m[t]) * to_c(j[ax][t]);
            };
        };
        C div = central<R, 0>(flux(0)) + central<R, 1>(flux(1));
        if constexpr (DIMS == 3) div = div + central<R, 2>(flux(2));
        const C mi = to_c(m[i]);
        static_cast<T *>(a.mo)[i] = from_c<T>(FMA(k.dt, FMA(k.sAC, stencil_sum<ST, C>(Pmu), -(c3g * div)), mi));
#pragma unroll
        for (int ax = 0; ax < DIMS; ++ax) {
            C gm;
            if (ax == 0) gm = central<R, 0>(Pmu);
            else if (ax == 1) gm = central<R, 1>(Pmu);
            else gm = central<R, 2>(Pmu);
            auto Pj = [&](int dx, int dy, int dz) -> C { return to_c(j[ax][tp.at(x, a.nx, dx, dy, dz)]); };
            jo[ax][i] = from_c<T>(FMA(k.dt, FMA(k.sAC, stencil_sum<ST, C>(Pj), -(c3g * (mi * gm))), to_c(j[ax][i])));
        }
    }
}

// 2D tiles (FP32 / BF16 storage): one BX x BY output tile per CTA.  m and the
// components of j are fetched once with a 2R halo (x padded to whole 16-byte
// chunks), mu is evaluated on the tile grown by R into shared memory, and the
// update reads everything from shared memory: one pass over HBM instead of two
// plus the mu buffer.  The same expressions as the per-point kernels, so the
// results are identical to theirs.
template <int ST, typename T, int BX, int BY>
struct MhTile2dShape {
    typedef typename Cmp<T>::type C;
    static constexpr int R = StencilInfo<ST>::r;
    static constexpr int RIN = 2 * R;
    static constexpr int CK = 16 / sizeof(T);
    static constexpr int HC = (RIN + CK - 1) / CK;
    static constexpr int NCK = BX / CK + 2 * HC;
    static constexpr int SW = NCK * CK, X0 = HC * CK;
    static constexpr int HIN = BY + 2 * RIN;
    static constexpr int NF = 3;  // m, j_x, j_y
    static constexpr int WMU = BX + 2 * R, HMU = BY + 2 * R;
    static constexpr size_t bytes_in = sizeof(T) * (size_t)NF * HIN * SW;
    static constexpr size_t smem_bytes = bytes_in + sizeof(C) * (size_t)WMU * HMU;
    static_assert(bytes_in % 16 == 0, "mu array alignment");
};

template <int ST, typename T, int BX, int BY, int NT>
__global__ void __launch_bounds__(NT) mh_tile2d_kernel(MhArgs a, typename Cmp<T>::type c3g) {
    pdl_enter();
    typedef MhTile2dShape<ST, T, BX, BY> Sh;
    typedef typename Sh::C C;
    constexpr int R = Sh::R, RIN = Sh::RIN, CK = Sh::CK, NCK = Sh::NCK, SW = Sh::SW, X0 = Sh::X0;
    constexpr int HIN = Sh::HIN, NF = Sh::NF, WMU = Sh::WMU, HMU = Sh::HMU;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *s_in = reinterpret_cast<T *>(smem_raw);                 // [NF][HIN][SW]: m, j_x, j_y
    C *s_mu = reinterpret_cast<C *>(smem_raw + Sh::bytes_in);  // [HMU][WMU]
    const ConstsC<C> k(a.k, a.kf);
    const int nx = a.nx, ny = a.ny, t = threadIdx.x;
    const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY;
    const bool vec_ok = (nx % CK) == 0;
    const T *in[NF] = {static_cast<const T *>(a.m), static_cast<const T *>(a.j[0]), static_cast<const T *>(a.j[1])};
    T *out[NF] = {static_cast<T *>(a.mo), static_cast<T *>(a.jo[0]), static_cast<T *>(a.jo[1])};

    // chunk c of shared row i holds columns x0 - X0 + c*CK .. +CK-1 of grid row y0 - RIN + i
    for (int q = t; q < HIN * NCK; q += NT) {
        const int i = q / NCK, c = q - i * NCK;
        const int y = wrap_idx(y0 - RIN + i, ny);
        const int x = x0 - X0 + c * CK;
        const size_t row = (size_t)y * (size_t)nx;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            T *dst = s_in + ((size_t)f * HIN + i) * SW + c * CK;
            if (vec_ok) {  // a chunk wraps as a whole
                cp_async16(dst, in[f] + row + wrap_idx(x, nx));
            } else {
#pragma unroll
                for (int jj = 0; jj < CK; ++jj) cp_async_elem(dst + jj, in[f] + row + wrap_idx(x + jj, nx));
            }
        }
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();

    // field f at tile coordinates (i, j), -RIN <= i < BY + RIN, -X0 <= j < BX + X0
    auto fld = [&](int f, int i, int j) -> C { return to_c(s_in[((size_t)f * HIN + i + RIN) * SW + j + X0]); };
    for (int q = t; q < HMU * WMU; q += NT) {
        const int i = q / WMU - R, j = q % WMU - R;
        auto P = [&](int dx, int dy, int) -> C { return fld(0, i + dy, j + dx); };
        s_mu[q] = ch_mu<C>(fld(0, i, j), stencil_sum<ST, C>(P), k);
    }
    __syncthreads();
    for (int q = t; q < BY * BX; q += NT) {
        const int i = q / BX, j = q - i * BX;
        const int y = y0 + i, x = x0 + j;
        if (y >= ny || x >= nx) continue;
        const size_t o = (size_t)y * (size_t)nx + x;
        auto Pmu = [&](int dx, int dy, int) -> C { return s_mu[(i + R + dy) * WMU + (j + R + dx)]; };
        auto flux = [&](int ax) {
            return [&, ax](int dx, int dy, int) -> C { return fld(0, i + dy, j + dx) * fld(1 + ax, i + dy, j + dx); };
        };
        const C div = central<R, 0>(flux(0)) + central<R, 1>(flux(1));
        const C mi = fld(0, i, j);
        out[0][o] = from_c<T>(FMA(k.dt, FMA(k.sAC, stencil_sum<ST, C>(Pmu), -(c3g * div)), mi));
#pragma unroll
        for (int ax = 0; ax < 2; ++ax) {
            const C gm = (ax == 0) ? central<R, 0>(Pmu) : central<R, 1>(Pmu);
            auto Pj = [&](int dx, int dy, int) -> C { return fld(1 + ax, i + dy, j + dx); };
            out[1 + ax][o] = from_c<T>(FMA(k.dt, FMA(k.sAC, stencil_sum<ST, C>(Pj), -(c3g * (mi * gm))), fld(1 + ax, i, j)));
        }
    }
}

// 3D FP32 / BF16: xy tiles streamed along z.  Each loaded plane (tile plus a 2R
// halo, all four fields, widened to FP32) enters a ring of D = 3R + 2 planes in
// shared memory; mu of plane i - R (tile grown by R) goes to a ring of 2R + 1
// planes; the update of plane i - 2R then reads m and j on planes i - 3R .. i - R
// and mu from the rings.  The ring depth keeps the plane committed at iteration i
// clear of every plane a thread still in iteration i - 1 may read.  Work items
// are (z segment, tile) pairs handed out round by round, segment-major, so the
// resident CTAs stream the same z range together and the halo rows and columns
// that neighbouring tiles share are still in L2 when the second tile reads them.
// The same expressions as the per-point kernels, so the results are identical.
template <int ST, typename T, int TX, int TY>
struct MhRing3dShape {
    static constexpr int R = StencilInfo<ST>::r;
    static constexpr int RIN = 2 * R;
    static constexpr int WIN = TX + 2 * RIN, HIN = TY + 2 * RIN, AIN = WIN * HIN;
    static constexpr int D = 3 * R + 2;
    static constexpr int NF = 4;  // m, j_x, j_y, j_z
    static constexpr int WMU = TX + 2 * R, HMU = TY + 2 * R, AMU = WMU * HMU, DMU = 2 * R + 1;
    static constexpr size_t smem_bytes = sizeof(float) * ((size_t)NF * D * AIN + (size_t)DMU * AMU);
};

template <int ST, typename T, int TX, int TY, int NT>
__global__ void __launch_bounds__(NT) mh_ring3d_kernel(MhArgs a, float c3g, int tiles_x, int tiles_y, int segs) {
    pdl_enter();
    typedef float C;
    typedef MhRing3dShape<ST, T, TX, TY> Sh;
    constexpr int R = Sh::R, RIN = Sh::RIN, WIN = Sh::WIN, AIN = Sh::AIN, D = Sh::D, NF = Sh::NF;
    constexpr int WMU = Sh::WMU, AMU = Sh::AMU, DMU = Sh::DMU;
    constexpr int EPT = (AIN + NT - 1) / NT;  // loaded cells per thread per field
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *s_in = reinterpret_cast<C *>(smem_raw);  // [NF][D][AIN]
    C *s_mu = s_in + (size_t)NF * D * AIN;      // [DMU][AMU]
    const ConstsC<C> k(a.k, a.kf);
    const int nx = a.nx, ny = a.ny, nz = a.nz, t = threadIdx.x;
    const size_t plane = (size_t)nx * (size_t)ny;
    const T *in[NF] = {static_cast<const T *>(a.m), static_cast<const T *>(a.j[0]), static_cast<const T *>(a.j[1]),
                       static_cast<const T *>(a.j[2])};
    T *out[NF] = {static_cast<T *>(a.mo), static_cast<T *>(a.jo[0]), static_cast<T *>(a.jo[1]),
                  static_cast<T *>(a.jo[2])};
    auto S_in = [&](int f, int i) -> const C * { return s_in + ((size_t)f * D + (i % D)) * AIN; };

    const int tiles = tiles_x * tiles_y;
    for (long long it = blockIdx.x; it < (long long)tiles * segs; it += gridDim.x) {
        const int seg = (int)(it / tiles), tile = (int)(it - (long long)seg * tiles);
        const int z0 = (int)((long long)seg * nz / segs), z1 = (int)((long long)(seg + 1) * nz / segs);
        const int x0 = (tile % tiles_x) * TX, y0 = (tile / tiles_x) * TY;
        const int nplanes = (z1 - z0) + 2 * RIN;  // loaded plane i is z = z0 - RIN + i

        int loff[EPT];
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            const int c = t + e * NT;
            if (c < AIN) {
                const int yi = c / WIN, xi = c - yi * WIN;
                loff[e] = wrap_idx(y0 - RIN + yi, ny) * nx + wrap_idx(x0 - RIN + xi, nx);
            } else {
                loff[e] = -1;
            }
        }
        C pf[NF][EPT];
        auto fetch = [&](int i) {
            const size_t zoff = (size_t)wrap_idx(z0 - RIN + i, nz) * plane;
#pragma unroll
            for (int f = 0; f < NF; ++f)
#pragma unroll
                for (int e = 0; e < EPT; ++e)
                    if (loff[e] >= 0) pf[f][e] = to_c(in[f][zoff + loff[e]]);
        };
        auto commit = [&](int i) {
#pragma unroll
            for (int f = 0; f < NF; ++f)
#pragma unroll
                for (int e = 0; e < EPT; ++e)
                    if (loff[e] >= 0) s_in[((size_t)f * D + (i % D)) * AIN + t + e * NT] = pf[f][e];
        };

        fetch(0);
        for (int i = 0; i < nplanes; ++i) {
            commit(i);
            if (i + 1 < nplanes) fetch(i + 1);
            __syncthreads();
            if (i >= 2 * R) {
                // mu of plane i - R over the tile grown by R
                C *mu = s_mu + (size_t)((i - R) % DMU) * AMU;
                for (int c = t; c < AMU; c += NT) {
                    const int ym = c / WMU, xm = c - ym * WMU;
                    const int base = (ym + R) * WIN + (xm + R);
                    auto P = [&](int dx, int dy, int dz) -> C { return S_in(0, i - R + dz)[base + dy * WIN + dx]; };
                    mu[c] = ch_mu<C>(S_in(0, i - R)[base], stencil_sum<ST, C>(P), k);
                }
            }
            __syncthreads();
            if (i >= 4 * R) {
                const int o = i - 2 * R;  // loaded index of the output plane
                const size_t zo = (size_t)(z0 + o - RIN) * plane;
                for (int c = t; c < TX * TY; c += NT) {
                    const int yy = c / TX, xx = c - yy * TX;
                    const int x = x0 + xx, y = y0 + yy;
                    if (x >= nx || y >= ny) continue;
                    const int b = (yy + RIN) * WIN + xx + RIN;
                    const int mb = (yy + R) * WMU + (xx + R);
                    auto Pmu = [&](int dx, int dy, int dz) -> C {
                        return s_mu[(size_t)((o + dz) % DMU) * AMU + mb + dy * WMU + dx];
                    };
                    auto fld = [&](int f, int dx, int dy, int dz) -> C { return S_in(f, o + dz)[b + dy * WIN + dx]; };
                    auto flux = [&](int ax) {
                        return [&, ax](int dx, int dy, int dz) -> C { return fld(0, dx, dy, dz) * fld(1 + ax, dx, dy, dz); };
                    };
                    const C div = (central<R, 0>(flux(0)) + central<R, 1>(flux(1))) + central<R, 2>(flux(2));
                    const C mi = fld(0, 0, 0, 0);
                    const size_t oi = zo + (size_t)y * nx + x;
                    out[0][oi] = from_c<T>(FMA(k.dt, FMA(k.sAC, stencil_sum<ST, C>(Pmu), -(c3g * div)), mi));
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) {
                        const C gm = (ax == 0) ? central<R, 0>(Pmu) : (ax == 1 ? central<R, 1>(Pmu) : central<R, 2>(Pmu));
                        auto Pj = [&](int dx, int dy, int dz) -> C { return fld(1 + ax, dx, dy, dz); };
                        out[1 + ax][oi] =
                            from_c<T>(FMA(k.dt, FMA(k.sAC, stencil_sum<ST, C>(Pj), -(c3g * (mi * gm))), fld(1 + ax, 0, 0, 0)));
                    }
                }
            }
        }
        __syncthreads();  // the rings are reused by the next segment
    }
}

// 3D FP32 / BF16, radius-1 stencils: rows of LN = 32 lanes or, two per warp, 16.  A row of a
// tile of 4 (LN - 2) x TY outputs (TY + 4 rows with the 2-cell halo) has the cells 4 l .. 4 l + 3 in
// lane l (the first and the last lane are halo), so every
// shared-memory access is a 16-byte chunk and the x neighbours come from the adjacent
// lanes (ring_stencil).  Planes stream along z through cp.async rings: m needs 3R + 2
// planes, the components of j, whose loads trail by R + 1 planes, 2R + 1, each plus P in
// flight; mu of plane j - R goes to a ring of 2R + 2 planes, the update runs one plane
// behind it, so one barrier per plane suffices.  The same expressions as the per-point
// kernels, so the results are identical.  (z segment, tile) items segment-major, as in
// mh_ring3d_kernel, which reads ~50 scalar shared-memory values per point and was bound by
// them: 256^3 7-point 195 us per step, 166 now; 27-point 413 -> 271.  One CTA of 448 threads fits
// an SM beside the rings, so latency between barriers bounds it now.  The radius-2 rings
// would not fit beside a useful tile; those stencils keep it.
// AL: nx a multiple of 4 and 16-byte aligned fields; otherwise (FP32) RaggedRow.
template <int ST, typename T, int TY, int LN_>
struct MhRows3dShape {
    static constexpr int R = StencilInfo<ST>::r, V = 4, CB = V * (int)sizeof(T), LN = LN_;
    static_assert(R == 1, "radius-2 rings do not fit");
    static constexpr int TX = (LN - 2) * V, HIN = TY + 4 * R, NT = LN * HIN;
    static_assert(NT % 32 == 0 && R % 2 == 1, "whole warps; the output rows of a warp are both or none");
    static constexpr int P = 2, DM = 3 * R + 2 + P, DJ = 2 * R + 1 + P, DMU = 2 * R + 2;
    static constexpr size_t plane_bytes = (size_t)HIN * LN * CB, mu_plane = (size_t)HIN * LN * V;
    static constexpr size_t in_bytes = (DM + 3 * DJ) * plane_bytes;
    static constexpr size_t smem_bytes = in_bytes + DMU * mu_plane * sizeof(float);
    static constexpr size_t stage_bytes = (size_t)HIN * LN * 16;  // not AL: an output row per row
};

template <int ST, typename T, int TY, int LN, bool AL>
__global__ void __launch_bounds__(MhRows3dShape<ST, T, TY, LN>::NT)
    mh_rows3d_kernel(MhArgs a, float c3g, int tiles_x, int tiles_y, int segs) {
    pdl_enter();
    typedef MhRows3dShape<ST, T, TY, LN> Sh;
    constexpr int R = Sh::R, V = Sh::V, CB = Sh::CB, HIN = Sh::HIN, P = Sh::P;
    constexpr unsigned FULL = 0xffffffffu;
    typedef typename VecT<CB>::type W;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const ConstsC<float> k(a.k, a.kf);
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const int lane = threadIdx.x & (LN - 1), w = LN == 32 ? __shfl_sync(0xffffffffu, threadIdx.x / 32, 0) : threadIdx.x / LN;
    const size_t plane = (size_t)nx * (size_t)ny;
    constexpr size_t PL = (size_t)HIN * LN;  // chunks of a plane
    W *const m_own = reinterpret_cast<W *>(smem_raw) + (size_t)w * LN + lane;
    W *const j_own = m_own + Sh::DM * PL;    // [3][DJ] planes
    float *const mu_own = reinterpret_cast<float *>(smem_raw + Sh::in_bytes) + ((size_t)w * LN + lane) * V;
    float *const stage = reinterpret_cast<float *>(smem_raw + Sh::smem_bytes) + w * LN * V;  // not AL
    (void)stage;
    const T *in[4] = {static_cast<const T *>(a.m), static_cast<const T *>(a.j[0]), static_cast<const T *>(a.j[1]),
                      static_cast<const T *>(a.j[2])};
    T *out[4] = {static_cast<T *>(a.mo), static_cast<T *>(a.jo[0]), static_cast<T *>(a.jo[1]), static_cast<T *>(a.jo[2])};
    auto extend = [&](float *e) {
        e[0] = __shfl_up_sync(FULL, e[V], 1, LN);
        e[V + 1] = __shfl_down_sync(FULL, e[1], 1, LN);
    };
    auto widen = [&](const W *p, float *dst) {
        union { W c; T t[V]; } u;
        u.c = *p;
#pragma unroll
        for (int i = 0; i < V; ++i) dst[i] = to_c(u.t[i]);
    };
    // chunks of m, component f of j and mu: plane q, row offset dy
    auto m_at = [&](int q, int dy, float *dst) { widen(m_own + (q % Sh::DM) * PL + dy * LN, dst); };
    auto j_at = [&](int f, int q, int dy, float *dst) { widen(j_own + (f * Sh::DJ + q % Sh::DJ) * PL + dy * LN, dst); };
    auto mu_at = [&](int q, int dy, float *dst) {
        const float4 v = *reinterpret_cast<const float4 *>(mu_own + (q % Sh::DMU) * Sh::mu_plane + dy * LN * V);
        dst[0] = v.x, dst[1] = v.y, dst[2] = v.z, dst[3] = v.w;
    };
    const bool pair = !AL && pair_rows(nx, a.m, a.j[0], a.mo, a.jo[0]) && pair_rows(nx, a.j[1], a.j[2], a.jo[1], a.jo[2]);
    const bool out_row = w >= 2 * R && w < HIN - 2 * R;  // the same for both rows of a warp
    // mu is formed by whole warps: the outermost rows, which need none, repeat their neighbour's
    const int mu_dy = w < R ? R - w : w >= HIN - R ? HIN - 1 - R - w : 0;

    const int tiles = tiles_x * tiles_y;
    for (long long it = blockIdx.x; it < (long long)tiles * segs; it += gridDim.x) {
        const int seg = (int)(it / tiles), tile = (int)(it - (long long)seg * tiles);
        const int z0 = (int)((long long)seg * nz / segs), z1 = (int)((long long)(seg + 1) * nz / segs);
        const int x0 = (tile % tiles_x) * Sh::TX, y0 = (tile / tiles_x) * TY;
        const int n = (z1 - z0) + 4 * R;  // loaded plane i is z = z0 - 2R + i
        const int col = x0 + (lane - 1) * V, yo = y0 - 2 * R + w;
        const size_t roff = (size_t)wrap_idx(yo, ny) * nx + (AL ? wrap_idx(col, nx) : 0);
        const bool store = out_row && lane >= 1 && lane <= LN - 2 && col < nx && yo < ny;
        const typename std::conditional<AL, NoRow, RaggedRow<LN>>::type rag(x0 - V, lane, nx, pair);
        size_t dst_off = (size_t)z0 * plane + (size_t)yo * nx + (AL ? col : 0);
        auto put = [&](int f, const float (&o)[V]) {
            if constexpr (AL) {
                if (store) store_vec<T, V>(out[f] + dst_off, o);
            } else {
                rag.put(out[f] + dst_off, stage, o, nx, yo < ny);
            }
        };
        auto fetch = [&](W *dst, const T *field, int i) {
            const T *src = field + (size_t)wrap_idx(z0 - 2 * R + i, nz) * plane + roff;
            if constexpr (!AL) rag.fetch(reinterpret_cast<T *>(dst - lane), src);
            else if constexpr (CB == 16) cp_async16(dst, src);
            else cp_async8(dst, src);
        };
        // group g: plane g of m, plane g - 1 - R of j (planes R .. n-1-R are read)
        auto issue = [&](int g) {
            if (g < n) fetch(m_own + (g % Sh::DM) * PL, in[0], g);
            const int i = g - 1 - R;
            if (i >= R && i < n - R)
#pragma unroll
                for (int f = 0; f < 3; ++f) fetch(j_own + (f * Sh::DJ + i % Sh::DJ) * PL, in[1 + f], i);
            cp_async_commit();
        };
#pragma unroll
        for (int g = 0; g < P; ++g) issue(g);
        for (int j = 0; j <= n; ++j) {
            cp_async_wait<P - 1>();
            __syncthreads();  // group j and mu of plane j-1-R published; slots written below are no longer read
            issue(j + P);
            const int t = j - 1 - 2 * R;  // output plane
            if (out_row && t >= 2 * R) {
                float S[V], cen[V], mu_e[V + 2], up[V], dn[V];
                float mc[V], o[V], div[V];
                m_at(t, 0, mc);
                {   // D_x(m j_x) + D_y(m j_y) + D_z(m j_z), the product formed at every tap
                    float e[V + 2], q[V];
                    j_at(0, t, 0, q);
#pragma unroll
                    for (int c = 0; c < V; ++c) e[1 + c] = mc[c] * q[c];
                    extend(e);
#pragma unroll
                    for (int c = 0; c < V; ++c) div[c] = e[c + 2] - e[c];
                    float ma[V], mb[V];
                    m_at(t, 1, ma), j_at(1, t, 1, up), m_at(t, -1, mb), j_at(1, t, -1, dn);
#pragma unroll
                    for (int c = 0; c < V; ++c) div[c] = div[c] + (ma[c] * up[c] - mb[c] * dn[c]);
                    m_at(t + 1, 0, ma), j_at(2, t + 1, 0, up), m_at(t - 1, 0, mb), j_at(2, t - 1, 0, dn);
#pragma unroll
                    for (int c = 0; c < V; ++c) div[c] = div[c] + (ma[c] * up[c] - mb[c] * dn[c]);
                }
                ring_stencil<ST>([&](int dz, int dy, float *d) { mu_at(t + dz, dy, d); }, extend, S, cen);
#pragma unroll
                for (int c = 0; c < V; ++c) o[c] = FMA(k.dt, FMA(k.sAC, S[c], -(c3g * div[c])), mc[c]);
                put(0, o);
#pragma unroll
                for (int c = 0; c < V; ++c) mu_e[1 + c] = cen[c];
                extend(mu_e);
#pragma unroll
                for (int f = 0; f < 3; ++f) {
                    if (f == 1) mu_at(t, 1, up), mu_at(t, -1, dn);
                    if (f == 2) mu_at(t + 1, 0, up), mu_at(t - 1, 0, dn);
                    ring_stencil<ST>([&](int dz, int dy, float *d) { j_at(f, t + dz, dy, d); }, extend, S, cen);
#pragma unroll
                    for (int c = 0; c < V; ++c) {
                        const float g = f == 0 ? mu_e[c + 2] - mu_e[c] : up[c] - dn[c];
                        o[c] = FMA(k.dt, FMA(k.sAC, S[c], -(c3g * (mc[c] * g))), cen[c]);
                    }
                    put(1 + f, o);
                }
                dst_off += plane;
            }
            if (j >= 2 * R && j < n) {  // mu of plane j - R
                float S[V], cen[V];
                ring_stencil<ST>([&](int dz, int dy, float *d) { m_at(j - R + dz, mu_dy + dy, d); }, extend, S, cen);
                *reinterpret_cast<float4 *>(mu_own + ((j - R) % Sh::DMU) * Sh::mu_plane) =
                    make_float4(ch_mu<float>(cen[0], S[0], k), ch_mu<float>(cen[1], S[1], k),
                                ch_mu<float>(cen[2], S[2], k), ch_mu<float>(cen[3], S[3], k));
            }
        }
        cp_async_wait<0>();
        __syncthreads();  // the rings are reused by the next item
    }
}

template <int ST, typename T, int TY, int LN, bool AL>
static cudaError_t launch_mh_rows_tile(const MhArgs &a, double c3g, cudaStream_t s, int n_sm) {
    typedef MhRows3dShape<ST, T, TY, LN> Sh;
    constexpr size_t smem = Sh::smem_bytes + (AL ? 0 : Sh::stage_bytes);
    static_assert(smem <= 227 * 1024, "shared memory per CTA");
    auto kern = mh_rows3d_kernel<ST, T, TY, LN, AL>;
    static const int occ = [&] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int o = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, Sh::NT, smem);
        return o;
    }();
    const int tx = (a.nx + Sh::TX - 1) / Sh::TX, ty = (a.ny + TY - 1) / TY;
    const long long wave = (long long)n_sm * std::max(occ, 1);
    const int segs = lockstep_segments((long long)tx * ty, a.nz, 4 * Sh::R, wave);
    return launch_pdl(kern, dim3((unsigned)std::min((long long)tx * ty * segs, wave)), dim3(Sh::NT), smem, s, a,
                      (float)c3g, tx, ty, segs);
}

// 120 x 12 tiles (32-lane rows) or 56 x 28 (16-lane rows): the one whose tiles cover the grid
// in less time, 1.2 to 1.33 (12 to 13.5 us per 1000 planes of a tile): 256^3 7-point 208 against
// 166 us per step, 360 x 300 x 400 345 / 432, 320 x 161 x 112 63 / 58.
template <int ST, typename T, bool AL>
static cudaError_t launch_mh_rows(const MhArgs &a, double c3g, cudaStream_t s, int n_sm) {
    const double wide = 1.2 * ((a.nx + 119) / 120) * ((a.ny + 11) / 12);
    const double narrow = 1.33 * ((a.nx + 55) / 56) * ((a.ny + 27) / 28);
    if (wide <= narrow) return launch_mh_rows_tile<ST, T, 12, 32, AL>(a, c3g, s, n_sm);
    return launch_mh_rows_tile<ST, T, 28, 16, AL>(a, c3g, s, n_sm);
}

template <int ST, typename T>
static cudaError_t launch_mh_t(const MhArgs &a, double c3g, cudaStream_t s, int n_sm) {
    typedef typename Cmp<T>::type C;
    if constexpr (StencilInfo<ST>::dims == 2 && !std::is_same<T, double>::value) {
        // family 0: shared-memory tiles; family 1: the two per-point passes
        if (g_step_variant != 1) {
            constexpr int BX = 128, BY = 16, NT = 256;
            typedef MhTile2dShape<ST, T, BX, BY> Sh;
            auto kern = mh_tile2d_kernel<ST, T, BX, BY, NT>;
            static const bool attr = [&] {
                cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem_bytes);
                return true;
            }();
            (void)attr;
            return launch_pdl(kern, dim3((a.nx + BX - 1) / BX, (a.ny + BY - 1) / BY), dim3(NT), Sh::smem_bytes, s, a, (C)c3g);
        }
    }
    if constexpr (StencilInfo<ST>::dims == 3 && !std::is_same<T, double>::value) {
        // family 0: warp rows (radius 1) or z-streaming tiles; family 1: the two per-point passes
        if constexpr (StencilInfo<ST>::r == 1) {
            bool al = a.nx % 4 == 0;
            for (int f = 0; f < 3; ++f) al = al && ((uintptr_t)a.j[f] | (uintptr_t)a.jo[f]) % 16 == 0;
            al = al && ((uintptr_t)a.m | (uintptr_t)a.mo) % 16 == 0;
            if (g_step_variant != 1 && al) return launch_mh_rows<ST, T, true>(a, c3g, s, n_sm);
            // unaligned rows cost the 7-point kernel more than the tile ring's scalar reads
            // (255 x 253 x 257: 254 against 207 us; 27-point 364 against 464)
            if constexpr (sizeof(T) == 4 && ST == L27) {
                if (g_step_variant != 1) return launch_mh_rows<ST, T, false>(a, c3g, s, n_sm);
            }
        }
        if (g_step_variant != 1) {
            constexpr int TX = 32, TY = 16, NT = 256;
            typedef MhRing3dShape<ST, T, TX, TY> Sh;
            auto kern = mh_ring3d_kernel<ST, T, TX, TY, NT>;
            static const int occ = [&] {
                cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem_bytes);
                int o = 1;
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, NT, Sh::smem_bytes);
                return o;
            }();
            const int tx = (a.nx + TX - 1) / TX, ty = (a.ny + TY - 1) / TY;
            const long long wave = (long long)n_sm * std::max(occ, 1);
            const int segs = lockstep_segments((long long)tx * ty, a.nz, 2 * Sh::RIN, wave);
            const long long items = (long long)tx * ty * segs;
            return launch_pdl(kern, dim3((unsigned)std::min(items, wave)), dim3(NT), Sh::smem_bytes, s, a, (C)c3g, tx, ty, segs);
        }
    }
    const int segs = (a.nx + 255) / 256;
    const long long units = (long long)a.ny * a.nz * segs;
    const unsigned blocks = (unsigned)std::min<long long>(units, (long long)n_sm * 8);
    cudaError_t e = launch_pdl(mh_mu_kernel<ST, T>, dim3(blocks), dim3(256), 0, s, a, segs);
    if (e != cudaSuccess) return e;
    if constexpr (StencilInfo<ST>::dims == 2)
        return launch_pdl(mh_update_kernel<ST, T, 2>, dim3(blocks), dim3(256), 0, s, a, segs, (C)c3g);
    else
        return launch_pdl(mh_update_kernel<ST, T, 3>, dim3(blocks), dim3(256), 0, s, a, segs, (C)c3g);
}

template <typename T>
static cudaError_t launch_mh_st(int stencil, const MhArgs &a, double c3g, cudaStream_t s, int n_sm) {
    switch (stencil) {
    case L5: return launch_mh_t<L5, T>(a, c3g, s, n_sm);
    case L9BOX: return launch_mh_t<L9BOX, T>(a, c3g, s, n_sm);
    case L9X4: return launch_mh_t<L9X4, T>(a, c3g, s, n_sm);
    case L7: return launch_mh_t<L7, T>(a, c3g, s, n_sm);
    case L27: return launch_mh_t<L27, T>(a, c3g, s, n_sm);
    default: return launch_mh_t<L13X4, T>(a, c3g, s, n_sm);
    }
}

cudaError_t launch_model_h(int dtype, int stencil, void *const in[4], void *const out[4], void *mu, int nx, int ny,
                           int nz, const StepConsts &k, double c3g, cudaStream_t s, int n_sm) {
    MhArgs a;
    a.m = in[0];
    a.mo = out[0];
    for (int c = 0; c < 3; ++c) {
        a.j[c] = in[1 + c] ? in[1 + c] : in[1];
        a.jo[c] = out[1 + c] ? out[1 + c] : out[1];
    }
    a.mu = mu;
    a.nx = nx;
    a.ny = ny;
    a.nz = nz;
    a.k = k;
    a.kf = to_float(k);
    switch (dtype) {
    case SP_F64: return launch_mh_st<double>(stencil, a, c3g, s, n_sm);
    case SP_F32: return launch_mh_st<float>(stencil, a, c3g, s, n_sm);
    default: return launch_mh_st<bf16>(stencil, a, c3g, s, n_sm);
    }
}

}  // namespace sp

// sp_gen2d.cu -- generated cross stencils (order 2R) in 2D FP32 on warp rows.
#include <algorithm>

#include "sp_gen.cuh"
#include "sp_step.cuh"

namespace sp {

// A warp per strip of 32 x 4 columns, as step2d_warp_kernel: the last 2R + 1 rows of each field
// (Model C: of the order parameter and of the density's chemical potential), and of mu for
// Cahn-Hilliard, lie in registers, own cells only; the R cells beside a lane's in the centre row
// come by shuffles when that row is used.  The first and last lane (Cahn-Hilliard of
// R > 2: two) are halo.  The tiles' gen_block_sums read 1.25 cells per cell and stencil from
// shared memory and evaluate mu on a halo of R rows and columns; here issue bounds it.  The same
// expressions, so the same results bit for bit.
// us per step on tiles and now: Cahn-Hilliard 8192^2 order 8 177 / 135, order 6 158 / 108, order 4
// 151 / 110; 4097 x 4095 order 8 68 / 51; Gray-Scott 4097 x 4095 order 2 101 / 63, order 8 117 / 67.
template <int MODEL, int R> struct Gen2dShape {
    static constexpr int V = 4, NF = num_fields<MODEL>(), RIN = MODEL == CH ? 2 * R : R, HL = (RIN + V - 1) / V;
    static constexpr int U = 2 * R + 1, OUT_COLS = (32 - 2 * HL) * V, D = 8, NT = 64;
    __host__ __device__ static constexpr size_t warp_smem(bool al) { return (size_t)(D * NF + (al ? 0 : 1)) * 32 * 16; }
};

template <int MODEL, int R, bool AL>
__global__ void __launch_bounds__(Gen2dShape<MODEL, R>::NT) gen2d_warp_kernel(GenArgs g, int strips, int groups, long long rows_per_cta) {
    pdl_enter();
    typedef Gen2dShape<MODEL, R> Sh;
    constexpr int V = Sh::V, NF = Sh::NF, U = Sh::U, D = Sh::D, RIN = Sh::RIN, HL = Sh::HL;
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const StepArgs &a = g.a;
    const int lane = threadIdx.x & 31;
    const int wpc = blockDim.x >> 5, warp = __shfl_sync(FULL, threadIdx.x >> 5, 0);
    float4 *ring = reinterpret_cast<float4 *>(smem_raw) + warp * (Sh::warp_smem(AL) / 16);  // [D][NF][32]
    float *stage = reinterpret_cast<float *>(ring + D * NF * 32);                          // [128] (not AL)
    (void)stage;
    const ConstsC<float> k(a.k, a.kf);
    const ConstsF2 k2(k);
    const int nx = a.nx, ny = a.ny;
    const float *in[2] = {static_cast<const float *>(a.in0), static_cast<const float *>(a.in1)};
    float *out[2] = {static_cast<float *>(a.out0), static_cast<float *>(a.out1)};
    const bool pair = !AL && pair_rows(nx, in[0], in[NF - 1], out[0], out[NF - 1]);

    long long g0 = (long long)blockIdx.x * rows_per_cta;
    const long long gend = min(g0 + rows_per_cta, (long long)groups * ny);
    while (g0 < gend) {
        const int group = (int)(g0 / ny);
        const int y0 = (int)(g0 - (long long)group * ny);
        const int y1 = (int)min((long long)ny, (long long)y0 + (gend - g0));
        g0 += y1 - y0;
        const int strip = group * wpc + warp;
        if (strip >= strips) continue;
        const int col = strip * Sh::OUT_COLS + (lane - HL) * V;
        const int colw = wrap_idx(col, nx);
        const bool store = lane >= HL && lane < 32 - HL && col < nx;
        const typename std::conditional<AL, NoRow, RaggedRow<32, HL>>::type rag(strip * Sh::OUT_COLS - HL * V, lane, nx, pair);
        const int jbeg = y0 - RIN;
        const int n = (y1 - y0) + 2 * RIN;

        auto issue = [&](int i) {
            if (i < n) {
                const size_t row = (size_t)wrap_idx(jbeg + i, ny) * nx;
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    float4 *dst = &ring[((i % D) * NF + f) * 32];
                    if constexpr (AL) cp_async16(dst + lane, in[f] + row + colw);
                    else rag.fetch(reinterpret_cast<float *>(dst), in[f] + row);
                }
            }
            cp_async_commit();  // empty groups keep the count uniform
        };
#pragma unroll
        for (int s = 0; s < D - 1; ++s) issue(s);

        // windows, newest row in slot u: the fields (Model C: phi and mu of rho), Cahn-Hilliard's
        // mu, and Model C's rho
        float ph[NF][U][V] = {}, mu[MODEL == CH ? U : 1][V] = {}, rho[MODEL == MC ? U : 1][V] = {};
        (void)mu;
        (void)rho;
        for (int i0 = 0; i0 < n; i0 += U) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = i0 + u;
                if (i < n) {
                    if constexpr (!AL) __syncwarp();  // every lane has read the slot that is refilled
                    issue(i + D - 1);
                    cp_async_wait<D - 1>();
                    if constexpr (!AL) __syncwarp();  // every lane's cells have landed
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        const float4 v = ring[((i % D) * NF + f) * 32 + lane];
                        ph[f][u][0] = v.x, ph[f][u][1] = v.y, ph[f][u][2] = v.z, ph[f][u][3] = v.w;
                    }
                    if constexpr (MODEL == MC) {
#pragma unroll
                        for (int c = 0; c < V; ++c) {
                            rho[u][c] = ph[NF - 1][u][c];
                            ph[NF - 1][u][c] = mc_mu<float>(ph[0][u][c], rho[u][c], k);
                        }
                    }
                    // window slot of the row `m` iterations back
#define SLOT(m) ((u - (m) + 4 * U) % U)
                    // stencil sums of the window's centre row (gen_sum's taps in its order, two
                    // cells per instruction)
                    auto sums = [&](const float (&win)[U][V], float (&S)[V]) {
                        float x[3 * V];
#pragma unroll
                        for (int c = 0; c < V; ++c) x[V + c] = win[SLOT(R)][c];
#pragma unroll
                        for (int h = 0; h < R; ++h) {
                            x[V - 1 - h] = __shfl_up_sync(FULL, x[2 * V - 1 - h], 1);
                            x[2 * V + h] = __shfl_down_sync(FULL, x[V + h], 1);
                        }
#pragma unroll
                        for (int c = 0; c < V; c += 2) {
                            const int q = V + c;
                            float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                            for (int jj = R; jj >= 1; --jj) {
                                float2 xp;
                                if (jj % 2 == 0) xp = add2(make_float2(x[q + jj], x[q + 1 + jj]), make_float2(x[q - jj], x[q + 1 - jj]));
                                else xp = make_float2(x[q + jj] + x[q - jj], x[q + 1 + jj] + x[q + 1 - jj]);
                                const float2 yp = add2(make_float2(win[SLOT(R - jj)][c], win[SLOT(R - jj)][c + 1]),
                                                       make_float2(win[SLOT(R + jj)][c], win[SLOT(R + jj)][c + 1]));
                                const float2 pj = add2(xp, yp);
                                const float2 w = splat2(g.W.wf[jj]);
                                acc = jj == R ? mul2(w, pj) : fma2(w, pj, acc);
                            }
                            const float2 s2 = fma2(splat2(g.W.wf[0]), make_float2(x[q], x[q + 1]), acc);
                            S[c] = s2.x;
                            S[c + 1] = s2.y;
                        }
                    };
                    float S[V], o[2][V];
                    sums(ph[0], S);
                    if constexpr (MODEL == CH) {
#pragma unroll
                        for (int c = 0; c < V; c += 2) {
                            const float *p = ph[0][SLOT(R)];
                            const float2 m2 = ch_mu2(make_float2(p[c], p[c + 1]), make_float2(S[c], S[c + 1]), k2);
                            mu[u][c] = m2.x;
                            mu[u][c + 1] = m2.y;
                        }
                        sums(mu, S);
#pragma unroll
                        for (int c = 0; c < V; c += 2) {
                            const float *p = ph[0][SLOT(2 * R)];
                            const float2 o2 = ch_update2(make_float2(p[c], p[c + 1]), make_float2(S[c], S[c + 1]), k2);
                            o[0][c] = o2.x;
                            o[0][c + 1] = o2.y;
                        }
                    } else if constexpr (MODEL == AC) {
#pragma unroll
                        for (int c = 0; c < V; ++c) o[0][c] = ac_update<float>(ph[0][SLOT(R)][c], S[c], k);
                    } else {
                        float S1[V];
                        sums(ph[NF - 1], S1);
                        const float *q = MODEL == MC ? rho[SLOT(R) % (MODEL == MC ? U : 1)] : ph[NF - 1][SLOT(R)];
#pragma unroll
                        for (int c = 0; c < V; ++c)
                            two_field_update<MODEL, float>(ph[0][SLOT(R)][c], q[c], S[c], S1[c], k, o[0][c], o[1][c]);
                    }
#undef SLOT
                    if (i >= 2 * RIN) {
                        const size_t row = (size_t)(jbeg + i - RIN) * nx;
#pragma unroll
                        for (int f = 0; f < NF; ++f) {
                            if constexpr (AL) {
                                if (store) store_vec<float, V>(out[f] + row + col, o[f]);
                            } else {
                                rag.put(out[f] + row, stage, o[f], nx, true);
                            }
                        }
                    }
                }
            }
        }
        cp_async_wait<0>();  // the ring is reused by the next segment
        if constexpr (!AL) __syncwarp();
    }
}

template <int MODEL, int R, bool AL> static cudaError_t launch_gen2d(const GenArgs &g, cudaStream_t s, int n_sm) {
    typedef Gen2dShape<MODEL, R> Sh;
    constexpr int WPC = Sh::NT / 32;
    auto kern = gen2d_warp_kernel<MODEL, R, AL>;
    static const auto occ = warp_occupancy<WPC>(kern, Sh::warp_smem(AL));
    const int strips = (g.a.nx + Sh::OUT_COLS - 1) / Sh::OUT_COLS;
    const int wpc = strips >= 32 ? WPC : 1, groups = (strips + wpc - 1) / wpc;
    const long long total = (long long)groups * g.a.ny;
    const long long rows = warptb_rows(total, 2 * Sh::RIN, wpc, occ[wpc], n_sm);
    return launch_pdl(kern, dim3((unsigned)((total + rows - 1) / rows)), dim3(32 * wpc), Sh::warp_smem(AL) * wpc, s, g,
                      strips, groups, rows);
}

template <int MODEL, int R> static cudaError_t launch_gen2d_any(const GenArgs &g, cudaStream_t s, int n_sm) {
    const bool al = g.a.nx % 4 == 0 &&
                    ((uintptr_t)g.a.in0 | (uintptr_t)g.a.in1 | (uintptr_t)g.a.out0 | (uintptr_t)g.a.out1) % 16 == 0;
    // Tiles where they are faster (us per step, tiles / warp rows).  Aligned: grids of middling size,
    // whose short runs of rows are mostly halo (Cahn-Hilliard order 2 256^2 3.0 / 2.2, 512^2 3.0 / 3.4, 1536^2
    // 5.6 / 5.4; order 8 2048^2 13 / 23, 4096^2 48 / 47), the smallest with a wide halo (order 8 256^2
    // 4.1 / 6.5) and large order-2 grids, bound by memory alone (Allen-Cahn 4096^2 25.9 / 24.7, 8192^2 92 / 101).
    // Other rows, which tiles copy element by element: one field and a wide halo (1503 x 1001
    // Allen-Cahn order 4 6.7 / 6.0, order 6 7.1 / 7.8, Cahn-Hilliard order 4 8.3 / 9.2; Gray-Scott order 8 17.6 / 14.5).
    typedef Gen2dShape<MODEL, R> Sh;
    const long long n = (long long)g.a.nx * g.a.ny;
    const bool rows = (n <= 1LL << 17 && Sh::RIN <= 3) || n >= 1LL << 23 || (al ? R == 1 && n >= 1LL << 21 : Sh::NF == 2 || Sh::RIN <= 2);
    if (!rows || (al && R == 1 && (MODEL == AC || MODEL == GS) && n >= 1LL << 25)) return cudaErrorNotSupported;
    return al ? launch_gen2d<MODEL, R, true>(g, s, n_sm) : launch_gen2d<MODEL, R, false>(g, s, n_sm);
}

template <int MODEL> static cudaError_t launch_gen2d_r(int r, const GenArgs &g, cudaStream_t s, int n_sm) {
    switch (r) {
    case 1: return launch_gen2d_any<MODEL, 1>(g, s, n_sm);
    case 2: return launch_gen2d_any<MODEL, 2>(g, s, n_sm);
    case 3: return launch_gen2d_any<MODEL, 3>(g, s, n_sm);
    case 4: return launch_gen2d_any<MODEL, 4>(g, s, n_sm);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_gen2d_f32(int model, int r, const GenArgs &g, cudaStream_t s, int n_sm) {
    switch (model) {
    case AC: return launch_gen2d_r<AC>(r, g, s, n_sm);
    case CH: return launch_gen2d_r<CH>(r, g, s, n_sm);
    case GS: return launch_gen2d_r<GS>(r, g, s, n_sm);
    case MC: return launch_gen2d_r<MC>(r, g, s, n_sm);
    }
    return cudaErrorInvalidValue;
}

}  // namespace sp

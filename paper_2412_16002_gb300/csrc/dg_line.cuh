// dg_line.cuh -- the split-precision step of 2D Euler by lines: N / R threads per cell, each with R node rows and R
// node columns (Q^1: two threads with one, Q^2: three with one, Q^3: two with two).
//
// The volume term, both end traces, their fluxes and lifts, and the S_K points of a line need that line
// only.  Rows live in registers; a component's values go through shared memory once to be read as columns,
// and the columns' part comes back the same way.  One thread for a whole cell would hold all of its
// deviations and G: two warps a scheduler, 31% of the issue slots, and a half or a third of the
// threads on a small mesh.  Averages of a stage are sums of two floats (an FP64 conversion takes its pipe 64
// cycles).
#pragma once

#include "dg_cell.cuh"

namespace crkdg {
namespace pc {

constexpr int LT = 128;  // threads of a block

// Lanes: whole cells per warp; the lanes past the last one (Q^2: two) shadow the last thread.
template <int N>
struct Line {
    static constexpr int R = N == 4 ? 2 : 1;      // rows (and columns) of a thread
    static constexpr int TPC = N / R;             // threads of a cell
    static constexpr int CPW = 32 / TPC;          // cells of a warp
    static constexpr int CPB = CPW * (LT / 32);   // cells of a block
    static constexpr int NV = R * N;              // values of a component in a thread
    static constexpr int LD = N == 4 ? 20 : N == 3 ? 9 : 5;  // pitch of a cell's node values
    static constexpr int LR = N == 4 ? 20 : 12;   // pitch of a cell's traces
    static constexpr int BLOCKS = N == 4 ? 3 : 5;  // resident blocks the register budget is for
};

template <int N>
struct LineSmem {
    using K = Line<N>;
    float buf[M][K::CPB][K::LD];                    // node values, then the columns' part of G
    alignas(16) float tr[M][K::CPB][K::LR];         // traces on their way out
    float dv0[M][K::NV][LT], acc[M][K::NV][LT];     // u^n's deviations at this thread's nodes; u*'s
};

// this thread's place: cell within the block, thread within the cell, the cell's first lane
template <int N>
__device__ __forceinline__ void line_place(int &cl, int &h, int &base) {
    using K = Line<N>;
    int l = threadIdx.x & 31;
    if (l >= K::CPW * K::TPC) l = K::CPW * K::TPC - 1;
    const int w = l / K::TPC;
    h = l - w * K::TPC;
    base = l - h;
    cl = (threadIdx.x >> 5) * K::CPW + w;
}
// sum and largest over the threads of a cell, the same bits in each
template <int N>
__device__ __forceinline__ float cell_sum(float x, int base) {
    if constexpr (Line<N>::TPC == 2) return x + __shfl_xor_sync(0xffffffffu, x, 1);
    return (__shfl_sync(0xffffffffu, x, base) + __shfl_sync(0xffffffffu, x, base + 1)) + __shfl_sync(0xffffffffu, x, base + 2);
}
template <int N>
__device__ __forceinline__ float cell_max(float x, int base) {
    if constexpr (Line<N>::TPC == 2) return fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 1));
    return fmaxf(fmaxf(__shfl_sync(0xffffffffu, x, base), __shfl_sync(0xffffffffu, x, base + 1)),
                 __shfl_sync(0xffffffffu, x, base + 2));
}

// One line of a cell (direction DIR): u the deviations at its nodes, thin whether a density of the warp may be
// ill-conditioned, dens the density rule of a trace; g the line's part of G (volume term and lifts), tr
// its end traces, gsum the face sums with weight wk.  A node with an ill-conditioned density takes
// no part here (ill_nodes).
template <int N, int DIR, class Density>
__device__ __forceinline__ void line_G(float rh, float gm1, const float *ubf, const float (&u)[M][N], bool thin, Density dens,
                                       float wk, float (&g)[M][N], float (&tr)[2][M], float (&gsum)[M]) {
    const NodalTables &T = c_tab[N - 2];
    float f[M][N];
#pragma unroll
    for (int a = 0; a < N; ++a) {
        const float mx = ubf[1] + u[1][a], my = ubf[2] + u[2][a], E = ubf[3] + u[3][a];
        float r = ubf[0] + u[0][a], k = rh;
        if (thin && rho_ill(r, ubf[0], u[0][a])) r = 1.0f, k = 0.0f;
        const float ri = recip_f(r), wx = mx * ri, wy = my * ri;
        const float p = gm1 * (E - 0.5f * (mx * wx + my * wy)), s = k * (DIR ? wy : wx);
        f[0][a] = k * (DIR ? my : mx);
        f[1][a] = DIR ? mx * s : fmaf(mx, s, k * p);
        f[2][a] = DIR ? fmaf(my, s, k * p) : my * s;
        f[3][a] = (E + p) * s;
    }
#pragma unroll
    for (int c = 0; c < M; ++c)
#pragma unroll
        for (int a = 0; a < N; ++a) {
            float s = 0.0f;
#pragma unroll
            for (int q = 0; q < N; ++q) s = fmaf(T.Dhatf[a][q], f[c][q], s);
            g[c][a] = s;
        }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float *l = e ? T.lpf : T.lmf;
        float d[M];
#pragma unroll
        for (int c = 0; c < M; ++c) {
            float s = 0.0f;
#pragma unroll
            for (int a = 0; a < N; ++a) s = fmaf(l[a], u[c][a], s);
            d[c] = s;
        }
        const float r = dens(d[0]), mx = ubf[1] + d[1], my = ubf[2] + d[2], E = ubf[3] + d[3];
        tr[e][0] = r, tr[e][1] = mx, tr[e][2] = my, tr[e][3] = E;
        const float ri = recip_f(r), wx = mx * ri, wy = my * ri;
        const float p = gm1 * (E - 0.5f * (mx * wx + my * wy)), s = rh * (DIR ? wy : wx);
        float fe[M];
        fe[0] = rh * (DIR ? my : mx);
        fe[1] = DIR ? mx * s : fmaf(mx, s, rh * p);
        fe[2] = DIR ? fmaf(my, s, rh * p) : my * s;
        fe[3] = (E + p) * s;
#pragma unroll
        for (int c = 0; c < M; ++c) {
            gsum[c] = fmaf(e ? -wk : wk, fe[c], gsum[c]);
#pragma unroll
            for (int a = 0; a < N; ++a)
                g[c][a] = e ? fmaf(-T.liftpf[a], fe[c], g[c][a]) : fmaf(T.liftmf[a], fe[c], g[c][a]);
        }
    }
}

// The S_K points of a line: true when the screen clears all of them (point_clear).
template <int N>
__device__ __forceinline__ bool line_clear(float eps, const float *ubf, const float *vb, const float *mean,
                                           const float (&u)[M][N]) {
    const NodalTables &T = c_tab[N - 2];
    bool ok = true;
#pragma unroll
    for (int al = 0; al < nlob(N); ++al) {
        float v[M];
#pragma unroll
        for (int c = 0; c < M; ++c) {
            float s = 0.0f;
#pragma unroll
            for (int a = 0; a < N; ++a) s = fmaf(T.Iglf[al][a], u[c][a], s);
            v[c] = ubf[c] + (s - mean[c]);
        }
        ok = ok && point_clear(eps, v, vb);
    }
    return ok;
}

// This thread's rows to a cell's part of the buffer; a column from it; the columns' part to rows.
template <int N>
__device__ __forceinline__ void put_rows(float (*buf)[Line<N>::CPB][Line<N>::LD], int cl, int h,
                                         const float (&u)[M][Line<N>::R][N]) {
#pragma unroll
    for (int c = 0; c < M; ++c)
#pragma unroll
        for (int r = 0; r < Line<N>::R; ++r) {
            float *p = &buf[c][cl][(Line<N>::R * h + r) * N];
            if constexpr (N == 4) {
                *reinterpret_cast<float4 *>(p) = make_float4(u[c][r][0], u[c][r][1], u[c][r][2], u[c][r][3]);
            } else {
#pragma unroll
                for (int a = 0; a < N; ++a) p[a] = u[c][r][a];
            }
        }
}
template <int N>
__device__ __forceinline__ void get_column(const float (*buf)[Line<N>::CPB][Line<N>::LD], int cl, int k, float (&u)[M][N]) {
#pragma unroll
    for (int c = 0; c < M; ++c)
#pragma unroll
        for (int b = 0; b < N; ++b) u[c][b] = buf[c][cl][N * b + k];
}
template <int N>
__device__ __forceinline__ void add_rows(const float (*buf)[Line<N>::CPB][Line<N>::LD], int cl, int h,
                                         float (&g)[M][Line<N>::R][N]) {
#pragma unroll
    for (int c = 0; c < M; ++c)
#pragma unroll
        for (int r = 0; r < Line<N>::R; ++r) {
            const float *p = &buf[c][cl][(Line<N>::R * h + r) * N];
            if constexpr (N == 4) {
                const float4 x = *reinterpret_cast<const float4 *>(p);
                g[c][r][0] += x.x, g[c][r][1] += x.y, g[c][r][2] += x.z, g[c][r][3] += x.w;
            } else {
#pragma unroll
                for (int a = 0; a < N; ++a) g[c][r][a] += p[a];
            }
        }
}
// The volume terms of a cell's nodes with an ill-conditioned density (rho_ill), which line_G leaves out: the flux
// in FP64 from ub + (double)d, rounded once, d the node values in the cell's part of the buffer.  The sums over
// such nodes go to out[c * stride + node], the cell's place in the array that u* is written to at the end.
// By one thread of the cell and out of line: near vacuum only.
template <int N>
__device__ __noinline__ void ill_nodes(const Params &P, const double *ub, const float *ubf,
                                       const float (*buf)[Line<N>::CPB][Line<N>::LD], int cl, float *out, size_t stride) {
    const NodalTables &T = c_tab[N - 2];
    float g[M][N * N];
    for (int c = 0; c < M; ++c)
        for (int q = 0; q < N * N; ++q) g[c][q] = 0.0f;
#pragma unroll 1
    for (int q = 0; q < N * N; ++q) {
        float x[M], fx[M], fy[M];
        for (int c = 0; c < M; ++c) x[c] = buf[c][cl][q];
        if (!rho_ill(ubf[0] + x[0], ubf[0], x[0])) continue;
        flux_xy_fallback<2>(P, ub, x, fx, fy);
        const int b = q / N, a = q - b * N;
        for (int c = 0; c < M; ++c)
            for (int j = 0; j < N; ++j) {
                g[c][N * b + j] = fmaf(T.Dhatf[j][a], P.f.rhx * fx[c], g[c][N * b + j]);
                g[c][N * j + a] = fmaf(T.Dhatf[j][b], P.f.rhy * fy[c], g[c][N * j + a]);
            }
    }
    for (int c = 0; c < M; ++c)
        for (int q = 0; q < N * N; ++q) out[c * stride + q] = g[c][q];
}
// Consecutive values in global memory (16-byte accesses where rows are whole vectors).
template <int K>
__device__ __forceinline__ void load_run(const float *p, float *v) {
    if constexpr (K % 4 == 0) {
#pragma unroll
        for (int q = 0; q < K; q += 4) {
            const float4 x = *reinterpret_cast<const float4 *>(p + q);
            v[q] = x.x, v[q + 1] = x.y, v[q + 2] = x.z, v[q + 3] = x.w;
        }
    } else if constexpr (K == 2) {
        const float2 x = *reinterpret_cast<const float2 *>(p);
        v[0] = x.x, v[1] = x.y;
    } else {
#pragma unroll
        for (int q = 0; q < K; ++q) v[q] = p[q];
    }
}
template <int K>
__device__ __forceinline__ void store_run(float *p, const float *v) {
    if constexpr (K % 4 == 0) {
#pragma unroll
        for (int q = 0; q < K; q += 4) *reinterpret_cast<float4 *>(p + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
    } else {
#pragma unroll
        for (int q = 0; q < K; ++q) p[q] = v[q];
    }
}

}  // namespace pc

// Inner stages (tableaux whose A has only a sub-diagonal).  Bound by issue (Q^2 83% of the slots, Q^3 64% at three
// blocks an SM): 2048^2 Q^3 3.08 ms a launch, 131^2 Q^3 27 us, 1024^2 Q^2 350 us (one thread per cell: 5.40 ms, 49
// and 684 us; Q^3 on the tensor cores 7.07 ms).
template <int N>
__global__ void __launch_bounds__(pc::LT, pc::Line<N>::BLOCKS) k_inner_l(const __grid_constant__ Params P, const __grid_constant__ MixBufs X) {
    using namespace pc;
    using K = Line<N>;
    constexpr int R = K::R, NV = K::NV, NTR = 4 * N;
    extern __shared__ __align__(16) unsigned char line_smem[];
    LineSmem<N> &S = *reinterpret_cast<LineSmem<N> *>(line_smem);
    const NodalTables &T = c_tab[N - 2];
    const int t = threadIdx.x;
    int cl, h, base;
    line_place<N>(cl, h, base);
    const int cell = blockIdx.x * K::CPB + cl;
    const int w0 = (t >> 5) * K::CPW, cell0 = blockIdx.x * K::CPB + w0;  // the warp's first cell
    const bool active = cell < P.ncell, own = active && h == 0 && owned(P, cell);
    const size_t cs = (size_t)P.ncell;
    Bufs B;
    B.flag = X.flag;
    B.nlim = X.nlim;
    B.thmin = X.thmin;
    const float rhx = P.f.rhx, rhy = P.f.rhy, gm1 = P.f.gm1;
    float wr[R];  // weights of this thread's rows (and columns)
#pragma unroll
    for (int r = 0; r < R; ++r) wr[r] = T.w1f[R * h + r];

    float dv[M][R][N], gb[M], uh[M], ul[M];
#pragma unroll
    for (int c = 0; c < M; ++c) {
        float v[NV];
#pragma unroll
        for (int q = 0; q < NV; ++q) v[q] = 0.0f;
        if (active) load_run<NV>(X.dv + (c * cs + cell) * (N * N) + NV * h, v);
        two_floats(active ? X.ub[c * cs + cell] : (c == 0 || c == M - 1 ? 1.0 : 0.0), uh[c], ul[c]);
        gb[c] = 0.0f;
#pragma unroll
        for (int q = 0; q < NV; ++q) S.dv0[c][q][t] = S.acc[c][q][t] = dv[c][q / N][q % N] = v[q];
    }
#pragma unroll 1
    for (int i = 0; i < P.s; ++i) {
        const float a_prev = i > 0 ? P.f.dtA[i][i - 1] : 0.0f;
        float ubf[M];
#pragma unroll
        for (int c = 0; c < M; ++c) {  // (float)(ubar + dt a G's average): two-sum, rounded once
            const float x = __fmul_rn(a_prev, gb[c]), s = __fadd_rn(uh[c], x), z = __fsub_rn(s, uh[c]);
            const float err = __fadd_rn(__fsub_rn(uh[c], __fsub_rn(s, z)), __fsub_rn(x, z));
            ubf[c] = __fadd_rn(s, __fadd_rn(err, ul[c]));
        }
        auto average = [&](double *ub) {
#pragma unroll
            for (int c = 0; c < M; ++c) {
                const double u = active ? X.ub[c * cs + cell] : (c == 0 || c == M - 1 ? 1.0 : 0.0);
                ub[c] = i > 0 ? u + (double)(a_prev * gb[c]) : u;
            }
        };
        put_rows<N>(S.buf, cl, h, dv);
        __syncwarp();
        // ---- scaling limiter of the stage value (stages 2..s)
        if (i > 0) {
            float mean[M], vb[M];
#pragma unroll
            for (int c = 0; c < M; ++c) {
                float m = 0.0f;
#pragma unroll
                for (int q = 0; q < NV; ++q) m = fmaf(wr[q / N] * T.w1f[q % N], dv[c][q / N][q % N], m);
                mean[c] = cell_sum<N>(m, base);
                vb[c] = 2.384185791015625e-07f * fabsf(ubf[c]);
            }
            const float epsf = P.f.eps * 1.0000002f;
            bool clear = true;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float u[M][N];
#pragma unroll
                for (int c = 0; c < M; ++c)
#pragma unroll
                    for (int a = 0; a < N; ++a) u[c][a] = dv[c][r][a];
                clear = line_clear<N>(epsf, ubf, vb, mean, u) && clear;
                get_column<N>(S.buf, cl, R * h + r, u);
                clear = line_clear<N>(epsf, ubf, vb, mean, u) && clear;
            }
            if (own && !point_clear(epsf, ubf, vb)) {
                double ub[M];
                average(ub);
                if (!admissible<PH_EULER, 2>(P, ub)) atomicOr(B.flag, 1);
            }
            const unsigned no = __ballot_sync(0xffffffffu, !clear);
            if (no) {
                if ((no >> base) & ((1u << K::TPC) - 1u)) {  // this cell: both threads take the same scaling
                    double ub[M];
                    float d[M][N * N], mm[M], s0, s1;
                    average(ub);
#pragma unroll
                    for (int c = 0; c < M; ++c) {
                        mm[c] = mean[c];
#pragma unroll
                        for (int q = 0; q < N * N; ++q) d[c][q] = S.buf[c][cl][q];
                    }
                    if (limit_cell<N>(P, B, ub, d, mm, own, s0, s1)) {
#pragma unroll
                        for (int c = 0; c < M; ++c)
#pragma unroll
                            for (int q = 0; q < NV; ++q)
                                dv[c][q / N][q % N] = (c == 0 ? s0 : s1) * (dv[c][q / N][q % N] - mean[c]);
                    }
                }
                __syncwarp();
                put_rows<N>(S.buf, cl, h, dv);
                __syncwarp();
            }
        }
        // near vacuum (rho_ill) a trace's density is the rounded FP64 value and a node's flux is formed in
        // FP64; a uniform branch asks first whether any density of the warp's cells is that small: sum_a |l_a(+-1)| < 3, so a trace
        // deviation is above 3 min - 3 max of the nodes'
        float dmx = 0.0f, dmn = 0.0f;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            dmx = fmaxf(dmx, dv[0][q / N][q % N]);
            dmn = fminf(dmn, dv[0][q / N][q % N]);
        }
        dmx = cell_max<N>(dmx, base);
        dmn = -cell_max<N>(-dmn, base);
        const float spread = 3.0f * (dmx - dmn);
        const bool thin = __any_sync(0xffffffffu, !(ubf[0] - spread > 9.5367431640625e-07f * (ubf[0] + spread)));
        // a trace's; an S_K point, so at least eps (a cell that the limiter left as it was has been tested
        // with its mean taken off, which these values keep)
        auto density = [&](float d) {
            float r = ubf[0] + d;
            if (thin && rho_ill(r, ubf[0], d)) {
                const double u = active ? X.ub[cell] : 1.0;
                r = fmaxf((float)((i > 0 ? u + (double)(a_prev * gb[0]) : u) + (double)d), P.scr_eps);
            }
            return r;
        };
        bool ill = false;  // a node of this cell is
        if (thin) {
#pragma unroll
            for (int q = 0; q < NV; ++q)
                ill = ill || rho_ill(ubf[0] + dv[0][q / N][q % N], ubf[0], dv[0][q / N][q % N]);
            const unsigned any = __ballot_sync(0xffffffffu, ill);
            ill = active && ((any >> base) & ((1u << K::TPC) - 1u)) != 0u;
            if (ill && h == 0) {
                double ub[M];
                float uf[M];
                average(ub);
#pragma unroll
                for (int c = 0; c < M; ++c) uf[c] = ubf[c];
                ill_nodes<N>(P, ub, uf, S.buf, cl, X.dv_s + (size_t)cell * (N * N), cs * (N * N));
            }
            __syncwarp();
        }
        // ---- lines: rows in registers, columns from (and their part of G back to) the buffer
        const int slot = P.slot[i];
        float g[M][R][N], gsum[M];
#pragma unroll
        for (int c = 0; c < M; ++c) gsum[c] = 0.0f;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float u[M][N], gl[M][N], tr[2][M];
#pragma unroll
            for (int c = 0; c < M; ++c)
#pragma unroll
                for (int a = 0; a < N; ++a) u[c][a] = dv[c][r][a];
            line_G<N, 0>(rhx, gm1, ubf, u, thin, density, 0.5f * wr[r], gl, tr, gsum);
#pragma unroll
            for (int c = 0; c < M; ++c) {
#pragma unroll
                for (int a = 0; a < N; ++a) g[c][r][a] = gl[c][a];
                S.tr[c][cl][R * h + r] = tr[0][c];
                S.tr[c][cl][N + R * h + r] = tr[1][c];
            }
        }
#pragma unroll
        for (int j = 0; j < R; ++j) {
            float u[M][N], gl[M][N], tr[2][M];
            get_column<N>(S.buf, cl, R * h + j, u);
            line_G<N, 1>(rhy, gm1, ubf, u, thin, density, 0.5f * wr[j], gl, tr, gsum);
            // a column is read by its own thread and, in Q^2, by the two lanes that shadow the last one: they have
            // read it before any of them writes
            if constexpr (K::CPW * K::TPC < 32) __syncwarp();
#pragma unroll
            for (int c = 0; c < M; ++c) {
#pragma unroll
                for (int b = 0; b < N; ++b) S.buf[c][cl][N * b + R * h + j] = gl[c][b];
                S.tr[c][cl][2 * N + R * h + j] = tr[0][c];
                S.tr[c][cl][3 * N + R * h + j] = tr[1][c];
            }
        }
        __syncwarp();
        if (ill)
#pragma unroll
            for (int c = 0; c < M; ++c)
#pragma unroll
                for (int q = 0; q < NV; ++q) g[c][q / N][q % N] += X.dv_s[(c * cs + cell) * (N * N) + NV * h + q];
        add_rows<N>(S.buf, cl, h, g);
        if (slot >= 0) {
#pragma unroll
            for (int c = 0; c < M; ++c) {
                float *dst = X.tr + ((size_t)slot * M + c) * cs * NTR;
#pragma unroll
                for (int k = 0; k < (K::CPW * N + 31) / 32; ++k) {  // whole vectors: N a cell
                    const int e = k * 32 + (t & 31), r = e / N, q = 4 * (e - r * N);
                    if (r < K::CPW && cell0 + r < P.ncell)
                        *reinterpret_cast<float4 *>(dst + (size_t)(cell0 + r) * NTR + q) =
                            *reinterpret_cast<const float4 *>(&S.tr[c][w0 + r][q]);
                }
                if (active && h == 0) X.tavg[((size_t)slot * M + c) * cs + cell] = ubf[c];
            }
        }
        // ---- G's deviations; the next stage value and u*
        const float b_i = P.f.dtb[i], a_next = i + 1 < P.s ? P.f.dtA[i + 1][i] : 0.0f;
#pragma unroll
        for (int c = 0; c < M; ++c) {
            float m = 0.0f;
#pragma unroll
            for (int q = 0; q < NV; ++q) m = fmaf(wr[q / N] * T.w1f[q % N], g[c][q / N][q % N], m);
            m = cell_sum<N>(m, base);
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                const float gd = g[c][q / N][q % N] - m;
                if (b_i != 0.0f) S.acc[c][q][t] = fmaf(b_i, gd, S.acc[c][q][t]);
                dv[c][q / N][q % N] = fmaf(a_next, gd, S.dv0[c][q][t]);
            }
            gb[c] = cell_sum<N>(gsum[c], base);
        }
        __syncwarp();  // the buffers are free
    }
    if (active)
#pragma unroll
        for (int c = 0; c < M; ++c) {
            float v[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) v[q] = S.acc[c][q][t];
            store_run<NV>(X.dv_s + (c * cs + cell) * (N * N) + NV * h, v);
        }
}

namespace pc {

// The cell's FP32 mean of its deviations in mean_of's order and roundings: the chain over the nodes passes
// from thread to thread.
template <int N>
__device__ __forceinline__ float line_mean(const float (&d)[Line<N>::R][N], int h, int base) {
    const NodalTables &T = c_tab[N - 2];
    constexpr int NV = Line<N>::NV;
    float p[NV], m = 0.0f;
#pragma unroll
    for (int q = 0; q < NV; ++q) p[q] = __fmul_rn(T.w2f[NV * h + q], d[q / N][q % N]);
#pragma unroll
    for (int k = 0; k < Line<N>::TPC; ++k) {
        float s = k == 0 ? 0.0f : m;
#pragma unroll
        for (int q = 0; q < NV; ++q) s = __fadd_rn(s, p[q]);
        m = __shfl_sync(0xffffffffu, s, base + k);
    }
    return m;
}

// Largest trial-step rate over a line's S_K points (FP32 values), and whether the screen clears them.
template <int N>
__device__ __forceinline__ bool line_rate(const Params &P, float eps, const float *ubf, const float *vb, const float *mean,
                                          const float (&u)[M][N], float &rate) {
    const NodalTables &T = c_tab[N - 2];
    const float hx = 0.5f * P.f.rhx, hy = 0.5f * P.f.rhy;
    bool ok = true;
#pragma unroll
    for (int al = 0; al < nlob(N); ++al) {
        float v[M];
#pragma unroll
        for (int c = 0; c < M; ++c) {
            float s = 0.0f;
#pragma unroll
            for (int a = 0; a < N; ++a) s = fmaf(T.Iglf[al][a], u[c][a], s);
            v[c] = ubf[c] + (s - mean[c]);
        }
        ok = ok && point_clear(eps, v, vb);
        const float ri = recip_f(v[0]), kin = fmaf(v[1], v[1], v[2] * v[2]);
        const float c = root_f(P.f.gamma * P.f.gm1 * fmaf(-0.5f * kin, ri, v[3]) * ri);
        rate = fmaxf(rate, fmaf(fabsf(v[1] * ri) + c, hx, (fabsf(v[2] * ri) + c) * hy));
    }
    return ok;
}

// The two faces of a cell across direction DIR (this thread's R points of each): the sums over the traced stages
// of b_i (fhat - f_int) (dc) and of b_i fhat (fh).  A stage's loads for both faces are issued together: the kernel
// waits on them with three to five warps a scheduler (face by face the meshes below take 3.14 ms, 26 and 370 us).
template <int N, int DIR>
__device__ __forceinline__ void face_sums(const Params &P, const MixBufs &X, int cell, bool active, int h, int base,
                                          float (&dc)[2][M][Line<N>::R], float (&fh)[2][M][Line<N>::R]) {
    constexpr int R = Line<N>::R, NTR = 4 * N;
    const size_t cs = (size_t)P.ncell, tcs = cs * NTR;
    int nb[2];
    size_t io[2], eo[2];
#pragma unroll
    for (int f = 0; f < 2; ++f) {
        const int face = 2 * DIR + f;
        nb[f] = active ? neighbour(P, cell, face) : -1;
        io[f] = (size_t)(active ? cell : 0) * NTR + face * N + R * h;
        eo[f] = (size_t)max(nb[f], 0) * NTR + (face ^ 1) * N + R * h;
#pragma unroll
        for (int c = 0; c < M; ++c)
#pragma unroll
            for (int r = 0; r < R; ++r) dc[f][c][r] = fh[f][c][r] = 0.0f;
    }
#pragma unroll 1
    for (int i = 0; i < P.s; ++i) {
        const int slot = P.slot[i];
        if (slot < 0) continue;
        const float *tr = X.tr + (size_t)slot * M * tcs;
        float ui[2][M][R], ue[2][M][R];
#pragma unroll
        for (int f = 0; f < 2; ++f)
#pragma unroll
            for (int c = 0; c < M; ++c) {
#pragma unroll
                for (int r = 0; r < R; ++r) ui[f][c][r] = ue[f][c][r] = c == 0 || c == M - 1 ? 1.0f : 0.0f;
                if (active) load_run<R>(tr + c * tcs + io[f], ui[f][c]);
                if (nb[f] >= 0) load_run<R>(tr + c * tcs + eo[f], ue[f][c]);
            }
        const float bi = P.f.b[i];
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            if (active && nb[f] < 0) {
                float av[M];
#pragma unroll
                for (int c = 0; c < M; ++c) av[c] = X.tavg[((size_t)slot * M + c) * cs + cell];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    float a[M], b[M];
#pragma unroll
                    for (int c = 0; c < M; ++c) a[c] = ui[f][c][r];
                    exterior_state_f<PH_EULER, 2>(P, 2 * DIR + f, a, av, b);
#pragma unroll
                    for (int c = 0; c < M; ++c) ue[f][c][r] = b[c];
                }
            }
            float fi[R][M], fe[R][M], alpha = 0.0f;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float a[M], b[M];
#pragma unroll
                for (int c = 0; c < M; ++c) a[c] = ui[f][c][r], b[c] = ue[f][c][r];
                alpha = fmaxf(alpha, face_flux_f<DIR>(P, a, fi[r]));
                alpha = fmaxf(alpha, face_flux_f<DIR>(P, b, fe[r]));
            }
            alpha = cell_max<N>(alpha, base);
            const float ha = -0.5f * alpha;
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < M; ++c) {
                    const float du = f ? __fsub_rn(ue[f][c][r], ui[f][c][r]) : __fsub_rn(ui[f][c][r], ue[f][c][r]);
                    const float fhat = fmaf(ha, du, __fmul_rn(0.5f, __fadd_rn(fi[r][c], fe[r][c])));
                    dc[f][c][r] = fmaf(bi, __fsub_rn(fhat, fi[r][c]), dc[f][c][r]);
                    fh[f][c][r] = fmaf(bi, fhat, fh[f][c][r]);
                }
        }
    }
}

// The cell's sum from its threads' parts.
template <int N>
__device__ __forceinline__ RunSum cell_run(const RunSum &p, int base) {
    RunSum o{0, 0};
#pragma unroll
    for (int k = 0; k < Line<N>::TPC; ++k) {
        const long long x = __shfl_sync(0xffffffffu, p.x, base + k);
        const int e = __shfl_sync(0xffffffffu, p.e, base + k), top = max(o.e, e);
        o.x = (o.x >> min(top - o.e, 63)) + (x >> min(top - e, 63));
        o.e = top;
    }
    return o;
}

}  // namespace pc

// Final stage (see k_final_x for the formulas): the fluxes of every traced stage at this thread's points of the
// four faces, their lifts along its rows and columns, and their fixed-point sums into the averages; then
// the limiter, or with the indicator the averages and the unlimited deviations for the troubled-cell
// pass.  The FP64 part of the averages is spread over the cell's threads.  Bound by the latency of the trace
// loads: 2048^2 Q^3 3.11 ms a launch, 131^2 Q^3 23 us, 1024^2 Q^2 347 us (one thread per cell: 3.53 ms, 47 and 376 us).
template <int N>
__global__ void __launch_bounds__(pc::LT, pc::Line<N>::BLOCKS) k_final_l(const __grid_constant__ Params P, const __grid_constant__ MixBufs X) {
    using namespace pc;
    using K = Line<N>;
    constexpr int R = K::R, NV = K::NV, NN = N * N;
    __shared__ __align__(16) float s_buf[M][K::CPB][K::LD];
    const NodalTables &T = c_tab[N - 2];
    int cl, h, base;
    line_place<N>(cl, h, base);
    const int cell = blockIdx.x * K::CPB + cl;
    const bool active = cell < P.ncell, own = active && owned(P, cell);
    const size_t cs = (size_t)P.ncell;
    Bufs B;
    B.flag = X.flag;
    B.nlim = X.nlim;
    B.thmin = X.thmin;
    RunSum sum[M];
    float dv[M][R][N];
#pragma unroll
    for (int c = 0; c < M; ++c) sum[c] = RunSum{0, 0};
    {
        float dc[2][M][R], fh[2][M][R];
        auto add = [&](const Fx *k) {
#pragma unroll
            for (int c = 0; c < M; ++c) {
                run_add<R>(sum[c], fh[0][c], k + R * h, false);
                run_add<R>(sum[c], fh[1][c], k + R * h, true);
            }
        };
        face_sums<N, 1>(P, X, cell, active, h, base, dc, fh);
        add(P.fx.ky);
#pragma unroll
        for (int c = 0; c < M; ++c)
#pragma unroll
            for (int j = 0; j < R; ++j)
#pragma unroll
                for (int b = 0; b < N; ++b)
                    s_buf[c][cl][N * b + R * h + j] =
                        fmaf(-T.liftpf[b], P.f.rhy * dc[1][c][j], T.liftmf[b] * (P.f.rhy * dc[0][c][j]));
        __syncwarp();
        face_sums<N, 0>(P, X, cell, active, h, base, dc, fh);
        add(P.fx.kx);
#pragma unroll
        for (int c = 0; c < M; ++c)
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int a = 0; a < N; ++a)
                    dv[c][r][a] = fmaf(-T.liftpf[a], P.f.rhx * dc[1][c][r], T.liftmf[a] * (P.f.rhx * dc[0][c][r]));
        add_rows<N>(s_buf, cl, h, dv);
        __syncwarp();
    }
    // averages: ubar - dt/|K| sum of the face fluxes; component k TPC + h in round k
    double ub[M];
#pragma unroll
    for (int c = 0; c < M; ++c) sum[c] = cell_run<N>(sum[c], base);
#pragma unroll
    for (int k = 0; k < (M + K::TPC - 1) / K::TPC; ++k) {
        RunSum s = sum[k * K::TPC];
        int c = k * K::TPC;
#pragma unroll
        for (int j = 1; j < K::TPC; ++j)
            if (k * K::TPC + j < M && h == j) s = sum[k * K::TPC + j], c = k * K::TPC + j;
        const double g = s.e == 0xff ? NAN : fx_double(s.x, 56 + s.e - 185 - P.fx.kk);
        const double u = active ? fma(P.dt, g, X.ub[c * cs + cell]) : (c == 0 || c == M - 1 ? 1.0 : 0.0);
        if (active && (h < M - k * K::TPC)) {
            X.ub_n[c * cs + cell] = u;
            if (P.defer_limit) X.aux[(size_t)cell * M + c] = u;
        }
#pragma unroll
        for (int j = 0; j < K::TPC; ++j)
            if (k * K::TPC + j < M) ub[k * K::TPC + j] = __shfl_sync(0xffffffffu, u, base + j);
    }
    // deviations: the correction without its mean
    float ubf[M], vb[M], mean[M];
    const float fdt = P.f.dt;
#pragma unroll
    for (int c = 0; c < M; ++c) {
        float m = 0.0f, d0[NV];
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            m = fmaf(T.w2f[NV * h + q], dv[c][q / N][q % N], m);
            d0[q] = 0.0f;
        }
        m = cell_sum<N>(m, base);
        if (active) load_run<NV>(X.dv_s + (c * cs + cell) * NN + NV * h, d0);
#pragma unroll
        for (int q = 0; q < NV; ++q) dv[c][q / N][q % N] = fmaf(fdt, dv[c][q / N][q % N] - m, d0[q]);
        ubf[c] = (float)ub[c];
        vb[c] = 2.384185791015625e-07f * fabsf(ubf[c]);
        mean[c] = line_mean<N>(dv[c], h, base);
    }
    const float epsf = P.f.eps * 1.0000002f;
    if (own && h == 0 && !point_clear(epsf, ubf, vb) && !admissible<PH_EULER, 2>(P, ub)) atomicOr(B.flag, 1);
    if (!P.defer_limit) {
        put_rows<N>(s_buf, cl, h, dv);
        __syncwarp();
        float rate = 0.0f;
        bool clear = true;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float u[M][N];
#pragma unroll
            for (int c = 0; c < M; ++c)
#pragma unroll
                for (int a = 0; a < N; ++a) u[c][a] = dv[c][r][a];
            clear = line_rate<N>(P, epsf, ubf, vb, mean, u, rate) && clear;
            get_column<N>(s_buf, cl, R * h + r, u);
            clear = line_rate<N>(P, epsf, ubf, vb, mean, u, rate) && clear;
        }
        const unsigned no = __ballot_sync(0xffffffffu, !clear);
        if ((no >> base) & ((1u << K::TPC) - 1u)) {  // this cell: its threads take the same scaling
            float d[M][NN];
#pragma unroll
            for (int c = 0; c < M; ++c)
#pragma unroll
                for (int q = 0; q < NN; ++q) d[c][q] = s_buf[c][cl][q];
            rate = limit_final<N>(P, B, ub, d, own && h == 0);
#pragma unroll
            for (int c = 0; c < M; ++c)
#pragma unroll
                for (int q = 0; q < NV; ++q) dv[c][q / N][q % N] = d[c][NV * h + q];
        }
        __syncwarp();
        post_rate_x(X, own ? rate : 0.0f);
    }
    if (active)
#pragma unroll
        for (int c = 0; c < M; ++c) store_run<NV>(X.dv_n + (c * cs + cell) * NN + NV * h, &dv[c][0][0]);
}

template <int N>
inline cudaError_t launch_line(int kernel, cudaStream_t st, const Params &P, const MixBufs &X) {
    const int grid = (P.ncell + pc::Line<N>::CPB - 1) / pc::Line<N>::CPB;
    if (kernel == KX_INNER) {
        const int smem = (int)sizeof(pc::LineSmem<N>);
        const cudaError_t e = cudaFuncSetAttribute(k_inner_l<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        k_inner_l<N><<<grid, pc::LT, smem, st>>>(P, X);
    } else if (kernel == KX_FINAL) {
        k_final_l<N><<<grid, pc::LT, 0, st>>>(P, X);
    } else {
        return launch_cell<N>(kernel, st, P, X);
    }
    return cudaGetLastError();
}

}  // namespace crkdg

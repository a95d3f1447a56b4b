// dg_run1d.cuh -- device-resident step loop for 1D meshes (one persistent
// cooperative launch runs many limited cRKDG steps).
//
// Small 1D problems (a few thousand cells) finish a step in a few microseconds
// of FP64 work, less than a host round trip.  Here one launch keeps the whole
// Sec. 4.1 loop on the device: every block owns chunks of NCB-2 consecutive
// cells plus one halo cell on each side, recomputes the (cell-local) inner
// stages of the halo cells itself, so the final stage's Lax--Friedrichs fluxes
// need no neighbour data from other blocks (compactness, Sec. 1), and only one
// grid barrier per attempt decides acceptance, restart (dt halved) and the next
// trial step from the global admissibility flag and wave-speed rate.
#pragma once

#include "dg_core.cuh"

namespace crkdg {

// Whole cells per warp (CfgW), so that a stage of a cell needs no block barrier, and four warps (two
// for N = 2), one for each scheduler of an SM: a mesh of this size leaves one block on an SM, and a
// step is one warp's chain of instructions.
template <int N, int PHYS>
struct RunCfg1D : CfgW<1, N, PHYS> {
    static constexpr int NT = run1d_threads(N);
    static constexpr int NCB = run1d_cells(N);  // cells per chunk including the two halo cells
};

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Grid-wide barrier on a counter that only grows: every block adds one per
// barrier and waits until the count reaches `target` (the number of arrivals due
// by the end of this barrier), so no block resets anything and the last arrival
// wakes the others by its own add.  The fence before the add publishes the
// block's writes (ordered before it by the block barrier); the acquire load
// orders the reads after it.  The waiting thread then reads the attempt's
// admissibility flag, rate and limited-cell count together (one round trip)
// and hands them to the block.  Bounded wait (2 s of %globaltimer): returns false
// when it expired, and the caller then leaves its step loop.
struct SlotRead {
    int flag;
    unsigned long long rate, nlim;
};
__device__ bool grid_barrier(RunCtl *R, unsigned target, const RunSlot *SL, SlotRead &out) {
    __shared__ int s_ok;
    __shared__ SlotRead s_rd;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(&R->bar_count) : "memory");
        const unsigned long long t0 = global_ns();
        for (;;) {
            unsigned c;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(&R->bar_count) : "memory");
            if ((int)(c - target) >= 0) break;  // wrap-safe: the count never runs 2^31 ahead
            if (global_ns() - t0 > 2000000000ull) {
                ok = 0;
                break;
            }
            __nanosleep(40);
        }
        s_rd.flag = *(const volatile int *)&SL->flag;
        s_rd.rate = *(const volatile unsigned long long *)&SL->rate;
        s_rd.nlim = *(const volatile unsigned long long *)&SL->nlim;
        s_ok = ok;
    }
    __syncthreads();
    out = s_rd;
    return s_ok != 0;
}

// The stages run on the integer units as in the per-step kernels (eval_G_fx, lift_faces), and the
// final stage combines jumps of the weighted flux sums: of the FP64 instructions of a step, each 64 to
// 76 cycles behind the one before it, about a quarter is left.  Latency bounds the loop: 4096 cells of the blast
// tube 17.4 us a step (FP64 forms 20.2), where the blocks at the front wait for the limiter's FP64 form; Burgers,
// 200 cells, 7.4 (7.7).
// FX as in inner_body.
template <int N, int PHYS, bool FX>
__global__ void __launch_bounds__(RunCfg1D<N, PHYS>::NT) k_run1d(const __grid_constant__ Params P, double *U0, double *U1,
                                                                 RunCtl *R, int cown) {
    using C = RunCfg1D<N, PHYS>;
    constexpr int M = C::M;
    constexpr int kUnroll = PHYS == PH_EULER ? 1 : MAXS;  // four Euler stages would not fit the instruction cache
    const int COWN = cown;  // own cells per chunk (1 .. NCB - 2); slots beyond COWN + 1 stay idle
    __shared__ Smem<C> S;
    __shared__ BlockTab<C> Tb;
    __shared__ double sTr[MAXS][C::NCB][2][M];
    __shared__ double sAv[MAXS][C::NCB][M];  // cell averages of the traced stage values
    __shared__ double sFs[C::NCB][2][M];     // sum_i b_i f(trace^(i)) of a cell's two faces
    __shared__ double sSp[MAXS][C::NCB][2];  // spectral radii of the traces
    int lc, node;
    place<C>(lc, node);
    const int nchunks = (P.ncell + COWN - 1) / COWN;
    const bool periodic = P.bc[0] == BC_PERIODIC;
    fill_tab<C>(P, Tb);  // its dt products are replaced for every attempt
    __syncthreads();

    double t = R->t;
    const double t_end = R->t_end, cfl = R->cfl;
    const int nsteps = R->nsteps, maxh = R->max_halvings;
    int cur = R->cur, steps = 0, restarts = 0, halv = 0, it = 0, status = RUN_OK;
    unsigned long long nlim_total = 0;
    double rate_last = -1.0;
    double dt_try = fmin(R->dt0, t_end - t);

    while (steps < nsteps && t < t_end) {
        RunSlot *SL = &R->slot[it % 3];
        Bufs B;
        B.flag = &SL->flag;
        B.nlim = &SL->nlim;
        B.thmin = &SL->thmin;
        B.a0 = &SL->rate;
        const double *un = cur ? U1 : U0;
        double *unew = cur ? U0 : U1;
        const double dt = dt_try;

        for (int chunk = blockIdx.x; chunk < nchunks; chunk += gridDim.x) {
            const int c0 = chunk * COWN;        // first own cell of the chunk
            const int graw = c0 - 1 + lc;       // unwrapped global index of this slot
            const bool exists = lc <= COWN + 1 && (periodic || (graw >= 0 && graw < P.ncell));
            const int gc = periodic ? (graw % P.ncell + P.ncell) % P.ncell : graw;
            const bool own = lc >= 1 && lc <= COWN && graw < P.ncell;
            if (threadIdx.x >= 32 && threadIdx.x < 32 + MAXS * MAXS + MAXS) {  // this attempt's dt a_ij, dt b_i
                const int k = (int)threadIdx.x - 32;
                if (k < MAXS * MAXS)
                    Tb.dtA[k / MAXS][k % MAXS] = dt * P.A[k / MAXS][k % MAXS];
                else
                    Tb.dtb[k - MAXS * MAXS] = dt * P.b[k - MAXS * MAXS];
            }
            double u0[M], cur_u[M], u[M], fs[M], gh[MAXS][M];
            load_node<1, N, PHYS>(P, un, gc, node, exists, u0);
#pragma unroll
            for (int c = 0; c < M; ++c) {
                cur_u[c] = u[c] = u0[c];
                fs[c] = 0.0;
            }
            __syncthreads();
            // inner stages of every cell of the chunk, halo included
#pragma unroll kUnroll
            for (int i = 0; i < MAXS; ++i) {
                if (i >= P.s) break;
                if (i > 0) {
#pragma unroll
                    for (int c = 0; c < M; ++c) cur_u[c] = u0[c];
#pragma unroll kUnroll
                    for (int j = 0; j < i; ++j)
                        if (nonzero_bits(P.A[i][j]))
#pragma unroll
                            for (int c = 0; c < M; ++c) cur_u[c] = fma(Tb.dtA[i][j], gh[j][c], cur_u[c]);
                    double pts[C::PPT][M];
                    float rhi;
                    limit_block(P, B, S, lc, node, own, cur_u, pts, true, true, false, rhi);
                }
                const int q = P.slot[i];
                double g[M];
                auto put = [&](int, const double *tr, const double *f, double sp) {  // one face point per thread
                    if (q < 0) return;
#pragma unroll
                    for (int c = 0; c < M; ++c) {
                        sTr[q][lc][node][c] = tr[c];
                        fs[c] = fma(P.b[i], f[c], fs[c]);
                    }
                    sSp[q][lc][node] = sp;
                };
                auto avg = [&](int c, double v) { sAv[q][lc][c] = v; };
                if constexpr (FX)
                    eval_G_fx<C>(P, S, Tb, lc, node, cur_u, g, q >= 0, q >= 0, put, avg);
                else
                    eval_G_64<C>(P, S, lc, node, cur_u, g, true, q >= 0, q >= 0, put, avg);
#pragma unroll
                for (int c = 0; c < M; ++c) {
                    gh[i][c] = g[c];
                    if (nonzero_bits(P.b[i])) u[c] = fma(Tb.dtb[i], g[c], u[c]);
                }
            }
            if (node < 2)
#pragma unroll
                for (int c = 0; c < M; ++c) sFs[lc][node][c] = fs[c];
            __syncthreads();
            // final stage, as final_body: this thread's face of its cell, from the trace sums and radii
            // of the two sides; the exterior side of a boundary face from the boundary condition
            double dc[C::FPT][M];
#pragma unroll
            for (int c = 0; c < M; ++c) dc[0][c] = 0.0;
            if (own && node < 2) {
                const int ln = node ? lc + 1 : lc - 1, gn = node ? graw + 1 : graw - 1;
                const bool inside = periodic || (gn >= 0 && gn < P.ncell);
                double fe[M];
#pragma unroll
                for (int c = 0; c < M; ++c) fe[c] = 0.0;
                for (int i = 0; i < P.s; ++i) {
                    const int q = P.slot[i];
                    if (q < 0) continue;
                    double ui[M], ue[M], alpha = sSp[q][lc][node];
#pragma unroll
                    for (int c = 0; c < M; ++c) ui[c] = sTr[q][lc][node][c];
                    if (inside) {
#pragma unroll
                        for (int c = 0; c < M; ++c) ue[c] = sTr[q][ln][node ^ 1][c];
                        alpha = fmax_nonneg(alpha, sSp[q][ln][node ^ 1]);
                    } else {
                        double f[M];
                        exterior_state<PHYS, 1>(P, node, ui, sAv[q][lc], ue);
                        alpha = fmax_nonneg(alpha, face_flux<PHYS, 1>(P, ue, 0, true, f));
#pragma unroll
                        for (int c = 0; c < M; ++c) fe[c] = fma(P.b[i], f[c], fe[c]);
                    }
                    const double h = half_of(P.b[i]), ba = (node ? -h : h) * alpha;
#pragma unroll
                    for (int c = 0; c < M; ++c) dc[0][c] = fma(ba, ue[c] - ui[c], dc[0][c]);
                }
#pragma unroll
                for (int c = 0; c < M; ++c)
                    dc[0][c] = fma(0.5, (inside ? sFs[ln][node ^ 1][c] : fe[c]) - fs[c], dc[0][c]);
            }
            cell_sync<C>();
            lift_faces<C>(P, dt, S.c[lc], node, node, 0, dc, u);
            double pts[C::PPT][M];
            float rhi;
            const bool cleared = limit_block(P, B, S, lc, node, own, u, pts, true, true, true, rhi);
            post_rate<C>(P, B, S, lc, node, own, cleared, rhi, pts);
            if (own) store_node<1, N, PHYS>(P, unew, gc, node, true, u);
            __syncthreads();
        }
        SlotRead rd;
        if (!grid_barrier(R, (unsigned)(it + 1) * (gridDim.x + (unsigned)R->extra_arrivals), SL, rd)) {
            status = RUN_TIMEOUT;
            break;
        }
        const int fl = rd.flag;
        if (blockIdx.x == 0 && threadIdx.x == 0) {  // the slot used two attempts ahead
            RunSlot *Z = &R->slot[(it + 2) % 3];
            Z->flag = 0;
            Z->nlim = 0ull;
            Z->thmin = dbits(1.0);
            Z->rate = 0ull;
        }
        ++it;
        if (fl == 0) {
            const double rate = bitsd(rd.rate);
            nlim_total += rd.nlim;
            t += dt;
            if (t_end - t <= 1e-14 * fabs(t_end)) t = t_end;
            ++steps;
            restarts += halv;
            halv = 0;
            cur ^= 1;
            rate_last = rate;
            // adaptive: the trial step of the new state; fixed (cfl <= 0): dt0 every step
            dt_try = fmin(cfl > 0.0 ? (rate > 0.0 ? cfl / rate : INFINITY) : R->dt0, t_end - t);
        } else {
            if (++halv > maxh) {
                status = RUN_BOUNDS;
                break;
            }
            dt_try = 0.5 * dt;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        R->t_out = t;
        R->rate_out = rate_last;
        R->steps = steps;
        R->restarts = restarts;
        R->cur_out = cur;
        R->status = status;
        R->nlim_total = nlim_total;
    }
}

template <int N, int PHYS>
cudaError_t run1d_launch(cudaStream_t st, const Params &P, double *u0, double *u1, RunCtl *R, int chunk,
                         int *nblocks) {
    using C = RunCfg1D<N, PHYS>;
    constexpr int NCB = C::NCB;
    auto *kernel = PHYS != PH_EULER || P.fx.on ? k_run1d<N, PHYS, true> : k_run1d<N, PHYS, PHYS != PH_EULER>;
    int dev = 0, nsm = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, C::NT, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    // chunks of NCB - 2 own cells by default: smaller chunks put more blocks on the GPU but
    // recompute more halo cells and add arrivals at the grid barrier
    const int slots = nsm * per_sm;
    int cown = chunk > 0 ? chunk : NCB - 2;
    if (cown > NCB - 2) cown = NCB - 2;
    if (cown < 1) cown = 1;
    int nchunks = (P.ncell + cown - 1) / cown;
    int grid = nchunks < slots ? nchunks : slots;
    *nblocks = grid;
    Params Pc = P;
    void *args[] = {&Pc, &u0, &u1, &R, &cown};
    return cudaLaunchCooperativeKernel((void *)kernel, dim3(grid), dim3(C::NT), args, 0, st);
}

}  // namespace crkdg

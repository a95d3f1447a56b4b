// dg_types.h -- plain data shared by the host API and the kernels of the cRKDG
// library (no device code here).  Nodal Q^k tables, step parameters and the
// device buffer set one launch works on.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "dg_fixed.h"

namespace crkdg {

constexpr int MAXN = 4;  // nodes per direction (k <= 3)
constexpr int MAXM = 4;  // conservative components (2D Euler)
constexpr int MAXS = 4;  // Runge--Kutta stages

enum Phys { PH_ADV = 0, PH_BURG = 1, PH_EULER = 2 };
enum Bc { BC_PERIODIC = 0, BC_OUTFLOW = 1, BC_REFLECT = 2, BC_DIRICHLET = 3 };

// Operator modes of the inner / final kernels.
enum Mode {
    MODE_STEP = 0,   // one limited cRKDG step (Scheme 1L)
    MODE_OP_G = 1,   // inner kernel writes G(u) instead of the stage accumulation
    MODE_OP_F = 2,   // final kernel adds the face correction only (no limiter, no checks)
    MODE_RATE = 3,   // scan kernels: the trial-step rate only (no bound margins)
    MODE_LIMIT_CHECK = 4,  // limiter kernel: also test the averages and count limited cells
    MODE_LIMIT_FINAL = 5,  // as MODE_LIMIT_CHECK, and post the trial-step rate of the result
};

__host__ __device__ constexpr int ncomp(int phys, int dim) { return phys == PH_EULER ? dim + 2 : 1; }
// Gauss--Lobatto points of S_K: L = ceil((k+3)/2), the smallest rule exact for degree k.
__host__ __device__ constexpr int nlob(int n) { return (n + 3) / 2; }
__host__ __device__ constexpr int gcd_c(int a, int b) { return b == 0 ? a : gcd_c(b, a % b); }
// Cells per block of the thread-per-node kernels: whole warps of whole cells,
// at least 128 threads.
__host__ __device__ constexpr int warp_cells(int nn) { return nn * 32 / gcd_c(nn, 32); }  // lcm(nn, 32)
__host__ __device__ constexpr int cells_per_block(int dim, int n) {
    return (warp_cells(dim == 2 ? n * n : n) / (dim == 2 ? n * n : n)) *
           (warp_cells(dim == 2 ? n * n : n) >= 128 ? 1 : 128 / warp_cells(dim == 2 ? n * n : n));
}

// 2D meshes from this many cells on take the faces' corrections in a pass of their own (k_faces): below, the pass
// is one launch too many.  Final stage with it and without, Riemann problem: Q^1 192^2 44 against 43 us, 256^2 58
// against 59, 362^2 83 against 90; Q^2 64^2 32 against 30, 80^2 35.2 against 35.1, 96^2 45 against 48, 128^2 52
// against 60, 512^2 294 against 489; Q^3 64^2 42 against 37, 80^2 51 against 53, 128^2 75 against 80, 512^2
// 465 against 668.  The bits are the same.
__host__ __device__ constexpr int faces_cells(int n) { return n == 2 ? 65536 : 6400; }

// The FP64 kernels instead keep whole cells per warp (32 / nn of them, see CfgW).
constexpr int kWarpThreads = 128;
__host__ __device__ constexpr int warp_cells_per_block(int nn) { return (32 / nn) * (kWarpThreads / 32); }

// The 1D step loop: threads of a block, and cells of its chunk including the two halo cells.
__host__ __device__ constexpr int run1d_threads(int n) { return n == 2 ? 64 : 128; }
__host__ __device__ constexpr int run1d_cells(int n) { return (32 / n) * (run1d_threads(n) / 32); }

// Device memory that an optional array leaves for what is allocated after it (work items, graphs, features).
constexpr size_t kSpareBytes = (size_t)256 << 20;

// One-dimensional nodal tables for n = k+1 Gauss points on [-1, 1].
struct NodalTables {
    double xg[MAXN], wg[MAXN];  // Gauss--Legendre nodes / weights (sum 2)
    double xl[MAXN], wl[MAXN];  // Gauss--Lobatto nodes / weights
    double Dhat[MAXN][MAXN];    // Dhat[a][q] = w_q l_a'(x_q) / w_a  (volume term)
    double lm[MAXN], lp[MAXN];  // l_a(-1), l_a(+1)                 (traces)
    double liftm[MAXN], liftp[MAXN];  // l_a(-1)/w_a, l_a(+1)/w_a    (lift)
    double Igl[MAXN][MAXN];     // Igl[alpha][a] = l_a(xl_alpha)   (S_K interpolation)
    double w1[MAXN];            // w_a / 2                          (1D average weights)
    double w2[MAXN * MAXN];     // (w_a/2)(w_b/2) at node b*n+a      (2D average weights)
    // products of the tables the troubled-cell and feature kernels weigh node values by,
    // host-computed with the kernels' association of the factors (the sums are unchanged)
    double mom2[MAXN * MAXN];        // (3 w1_a) w1_b at node b*n+a: 2D first moments
    double trw2[2][2][MAXN * MAXN];  // [dir][R, L] w1_across l_along(+1 / -1): 2D face averages
    double pm2[2][MAXN * MAXN];      // [dir] ((3 w1_a) w1_b) x_along: 2D first moments along dir
    double pm1[MAXN];                // (3 w1_a) x_a: 1D first moment
    float momxf[MAXN * MAXN], momyf[MAXN * MAXN];  // FP32 ((3 w1_a) w1_b) x_a, ... x_b: 2D first moments
    // FP32 copies for the split-precision path
    float Dhatf[MAXN][MAXN], lmf[MAXN], lpf[MAXN], liftmf[MAXN], liftpf[MAXN], Iglf[MAXN][MAXN];
    float w1f[MAXN], w2f[MAXN * MAXN];
    // the L2 projection of Q^k nodal values onto the total-degree space P^k (2D): node b*n+a
    // from node q, sum over the Legendre modes i + j <= k of L_i(x_a) L_j(x_b) times the
    // Gauss-rule coefficient of that mode at node q
    double pk[MAXN * MAXN][MAXN * MAXN];
    // fixed-point copies (dg_fixed.h): l_a(-1), l_a(+1) scaled by 2^kFxTrace, the average weights
    // by 2^kFxAvg
    Fx tlx[2][MAXN], w1x[MAXN], w2x[MAXN * MAXN];
    Fx pm2x[2][MAXN * MAXN];              // pm2 scaled by 2^kFxAvg (its magnitudes sum to less than 2)
    Fx trw2x[2][2][MAXN * MAXN];          // trw2 scaled by 2^kFxTrace (their magnitudes sum to less than 4)
    float xgf[2][MAXN];       // xg as a sum of two floats
};
constexpr int kFxTrace = 56;  // sum_a |l_a(+-1)| < 4
constexpr int kFxAvg = 57;    // the weights sum to 1

// Fixed-point coefficients of G scaled by 2^k: row a of the x term, 2/h_x Dhat[a][q] against the
// x-fluxes of the node's row and -+ 2/h_x l_a(+-1)/w_a against its two x-face fluxes, and the y
// term likewise; k makes the largest row sum of magnitudes at most 2^58.  on = 0: the scales
// are outside the range of the fixed-point path (the FP64 form runs).
struct FxOp {
    Fx cx[MAXN][MAXN], cy[MAXN][MAXN];
    Fx lx[MAXN][2], ly[MAXN][2];  // [0] the lower face, [1] the upper one
    FxGas gas;                    // Euler, 1 < gamma < 2 (on = 0 otherwise)
    int k, on;
    // face sums of the split path's averages: w1_pos / (2 h_x), w1_pos / (2 h_y) scaled by 2^kk (2D; kon:
    // the scales are in range)
    Fx kx[MAXN], ky[MAXN];
    int kk, kon;
};

// FP32 copies of the parameters for the split-precision kernels, rounded once by
// the host at launch (the kernels then never convert a double parameter).
struct ParamsF {
    float rhx, rhy, gamma, gm1, velx, vely, lo, hi, eps;
    float thr[2];  // (float) of Params::thr
    float bcs[4][MAXM];
    float dtA[MAXS][MAXS];  // (float)(dt a_ij)
    float dtb[MAXS];        // (float)(dt b_i)
    float b[MAXS];
    float dt;
};

struct Params {
    int nx, ny, ncell;
    double rhx, rhy;  // 2/hx, 2/hy
    double gamma, velx, vely;
    double lo, hi, eps;
    int bc[4];
    double bcs[4][MAXM];
    int s;
    double A[MAXS][MAXS];
    double b[MAXS];
    int slot[MAXS];  // trace slot of stage i, -1 when b_i = 0
    int nslot;
    double dt;
    int mode;
    int defer_limit;  // final kernel leaves the limiter to the troubled-cell kernel
    double tvb_M;     // TVB constant of the plain indicator
    double thr[2];    // its thresholds M h_x^2, M h_y^2 (h_d = 2 / rh_d), set by tvb_thresholds
    double thr_feat;  // M h_x h_y: the learned indicator's feature scale floor
    // FP32 bounds of the FP64 limiter's screen, set by screen_bounds: eps and lo rounded up,
    // hi rounded down (scr_on = 0: the screen clears nothing)
    int scr_on;
    float scr_eps, scr_lo, scr_hi;
    float scr_rh[2], scr_gg;  // rate_bound: 2/h_x, 2/h_y and gamma (gamma - 1), rounded up
    int ind_stage;    // troubled-cell kernel: 0 decide and limit, 2 limit the given flags (the feature
                      // kernel decided), 3 combine the given plain flags with the learned
                      // probabilities, then limit; 4 (split path) decide, combine with the
                      // learned probabilities, then limit
    ParamsF f;        // split-precision kernels only
    // Owned box of a subdomain (domain decomposition): cells [own[0], own[1]) x [own[2], own[3])
    // of this mesh.  With own_on, only those cells count in the admissibility flag, the limiter
    // statistics, the trial-step rate and the bound margins; the other cells (the halo ring)
    // are still computed, so that the owned cells' final stage reads their traces.
    int own_on;
    int own[4];
    // theta_2 of the Euler limiter: 0 the concavity ratio of eq. (Euler-limiter2), 1 the exact
    // per-point solve (theta2_point)
    int theta2_exact;
    // the manufactured source of Example 4.2's scenario I (2D Euler) added to G at the nodes:
    // 0 off, 1 on; t0 the time of u^n (stage i at t0 + c_i dt), x0, y0 the mesh's lower corner
    int source;
    double t0, x0, y0;
    // 1: the total-degree space P^k (2D): stage values, u* and u^{n+1} projected (NodalTables::pk)
    int pk;
    // Non-rectangular domain (Examples 4.8 and 4.9) or null: one word per cell (device memory),
    // bits 4s..4s+3 the boundary kind of side s (GEO_*), GEO_SOLID a cell outside the domain.
    // Solid cells keep u^n (their operators are zero) and count in no test, statistic or rate.
    const unsigned *geo;
    FxOp fx;  // set by fx_operator
    double gstate[2][MAXM];          // the fixed states A and B of the GEO_STATE_* / GEO_SHOCK kinds
    double shock_x0, shock_speed;    // GEO_SHOCK: state A where x < shock_x0 + shock_speed t
};

// Boundary kinds of a side in a geometry word: the mesh rule (the neighbouring cell, or the
// rectangle side's condition), reflective wall, outflow, fixed state A, fixed state B, and a
// planar shock's exact trace (state A behind x_s(t) = shock_x0 + shock_speed t, B ahead).
enum GeoKind { GEO_MESH = 0, GEO_WALL = 1, GEO_OUTFLOW = 2, GEO_STATE_A = 3, GEO_STATE_B = 4, GEO_SHOCK = 5 };
constexpr unsigned GEO_SOLID = 0x10000u;

// A cell outside a non-rectangular domain (device side; never without a geometry).
__device__ __forceinline__ bool solid_cell(const Params &P, int cell) {
    return P.geo != nullptr && (P.geo[cell] & GEO_SOLID) != 0u;
}

// Cells outside the owned box are halo cells (never when own_on is 0).
__host__ __device__ __forceinline__ bool owned(const Params &P, int cell) {
    if (!P.own_on) return true;
    const int cy = cell / P.nx, cx = cell - cy * P.nx;
    return cx >= P.own[0] && cx < P.own[1] && cy >= P.own[2] && cy < P.own[3];
}

// The TVB thresholds from rhx, rhy and tvb_M (host side, once per parameter set).
inline void tvb_thresholds(Params &P) {
    const double hx = 2.0 / P.rhx, hy = 2.0 / P.rhy;
    P.thr[0] = P.tvb_M * hx * hx;
    P.thr[1] = P.tvb_M * hy * hy;
    P.thr_feat = P.tvb_M * (2.0 / P.rhx) * (2.0 / P.rhy);
}

// The fixed-point coefficients of G from rhx, rhy and the tables of the degree (host side).
inline void fx_operator(Params &P, const NodalTables &T, int dim, int n, int phys) {
    FxOp &F = P.fx;
    memset(&F, 0, sizeof(F));
    double sx = 0.0, sy = 0.0;  // largest row sums
    for (int a = 0; a < n; ++a) {
        double s = fabs(T.liftm[a]) + fabs(T.liftp[a]);
        for (int q = 0; q < n; ++q) s += fabs(T.Dhat[a][q]);
        sx = fmax(sx, fabs(P.rhx) * s);
        if (dim == 2) sy = fmax(sy, fabs(P.rhy) * s);
    }
    auto moderate = [](double x) { return x == 0.0 || (fabs(x) > 0x1p-100 && fabs(x) < 0x1p100); };
    if (dim == 2) {
        const double r = fabs(P.rhx) + fabs(P.rhy);
        F.kon = isfinite(r) && r > 0x1p-100 && r < 0x1p100;
        if (F.kon) {
            int e;
            frexp(r, &e);  // the four faces' weights sum to r
            F.kk = 58 - e;
            for (int a = 0; a < n; ++a) {
                F.kx[a] = fx_coef(0.5 * T.w1[a] * P.rhx, F.kk);
                F.ky[a] = fx_coef(0.5 * T.w1[a] * P.rhy, F.kk);
            }
        }
    }
    const double s = sx + sy;
    F.on = isfinite(s) && s > 0x1p-100 && s < 0x1p100 && moderate(P.gamma) && moderate(P.velx) && moderate(P.vely);
    if (phys == PH_EULER) F.on = F.on && P.gamma > 1.0 && P.gamma < 2.0;
    if (!F.on) return;
    if (phys == PH_EULER) {
        F.gas.g1 = fx_limb(llrint(ldexp(P.gamma - 1.0, 62)));
        F.gas.g = fx_limb(llrint(ldexp(P.gamma, 61)));
    }
    int e;
    frexp(s, &e);  // s < 2^e
    F.k = 58 - e;
    for (int a = 0; a < n; ++a) {
        for (int q = 0; q < n; ++q) {
            F.cx[a][q] = fx_coef(P.rhx * T.Dhat[a][q], F.k);
            F.cy[a][q] = dim == 2 ? fx_coef(P.rhy * T.Dhat[a][q], F.k) : Fx{0, 0};
        }
        F.lx[a][0] = fx_coef(P.rhx * T.liftm[a], F.k);
        F.lx[a][1] = fx_coef(-P.rhx * T.liftp[a], F.k);
        F.ly[a][0] = dim == 2 ? fx_coef(P.rhy * T.liftm[a], F.k) : Fx{0, 0};
        F.ly[a][1] = dim == 2 ? fx_coef(-P.rhy * T.liftp[a], F.k) : Fx{0, 0};
    }
}

// The FP32 bounds of the FP64 limiter's screen (host side): floats on the safe side of
// eps, lo and hi, moved a further 2^-20 inwards.
inline float float_at_least(double x) {
    float f = (float)x;
    if ((double)f < x) f = nextafterf(f, INFINITY);
    return f;
}
inline float float_at_most(double x) {
    float f = (float)x;
    if ((double)f > x) f = nextafterf(f, -INFINITY);
    return f;
}
inline void screen_bounds(Params &P) {
    const float in = 9.5367431640625e-07f;  // 2^-20
    P.scr_eps = float_at_least(P.eps) * (1.0f + in);
    P.scr_lo = float_at_least(P.lo);
    P.scr_lo = P.scr_lo + in * fabsf(P.scr_lo);
    P.scr_hi = float_at_most(P.hi);
    P.scr_hi = P.scr_hi - in * fabsf(P.scr_hi);
    P.scr_rh[0] = float_at_least(P.rhx);
    P.scr_rh[1] = float_at_least(P.rhy);
    P.scr_gg = float_at_least(P.gamma * (P.gamma - 1.0));
    P.scr_on = 1;
}

// The FP32 copies of the split path (host side).
inline void fill_f32(Params &P) {
    ParamsF &F = P.f;
    F.rhx = (float)P.rhx;
    F.rhy = (float)P.rhy;
    F.gamma = (float)P.gamma;
    F.gm1 = (float)(P.gamma - 1.0);
    F.velx = (float)P.velx;
    F.vely = (float)P.vely;
    F.lo = (float)P.lo;
    F.hi = (float)P.hi;
    F.eps = (float)P.eps;
    F.thr[0] = (float)P.thr[0];
    F.thr[1] = (float)P.thr[1];
    for (int s = 0; s < 4; ++s)
        for (int c = 0; c < MAXM; ++c) F.bcs[s][c] = (float)P.bcs[s][c];
    for (int i = 0; i < MAXS; ++i) {
        for (int j = 0; j < MAXS; ++j) F.dtA[i][j] = (float)(P.dt * P.A[i][j]);
        F.dtb[i] = (float)(P.dt * P.b[i]);
        F.b[i] = (float)P.b[i];
    }
    F.dt = (float)P.dt;
}

struct Bufs {
    const double *un;   // u^n (nodal, state layout)
    double *ustar;      // u^n + dt sum_i b_i G(u~^(i))   (or G(u) in MODE_OP_G)
    double *unew;       // u^{n+1}
    double *tr;         // face traces of u~^(i): [slot][m][cell][face point]
    double *tavg;       // cell averages of the same u~^(i): [slot][m][cell] (outflow exterior state)
    // optional (both or none; without them the final kernel recomputes): sum_i b_i f(u_int^(i)) . nu of
    // the traces [m][cell][face point], and each traced stage's largest radius over a face's
    // points [slot][cell][face]
    double *tsum = nullptr, *tsp = nullptr;
    // 2D, with tsum, from faces_cells on: the faces' corrections for the cells above and below them
    // [direction][above, below][m][cell of the lower face][face point]
    double *fc = nullptr;
    int *flag;          // set when a stage average leaves B
    unsigned long long *nlim;   // limited cells
    unsigned long long *thmin;  // bits of the smallest theta (non-negative double)
    unsigned long long *a0;     // bits of the largest spectral radius (non-negative double)
    double *aux;        // per-cell output of the utility kernels
    unsigned long long *ord;    // two order-preserving mins (margins)
    int *tflags;        // troubled-cell flags (one per cell) or nullptr
    unsigned long long *ntrb;   // number of troubled cells
    float *feat;        // MLP features [cell][44]
    const float *prob;  // MLP probabilities [cell]
};

enum KernelId { K_INNER = 0, K_FINAL = 1, K_LIMIT = 2, K_A0 = 3, K_MARGINS = 4, K_AVG = 5, K_TROUBLE = 6,
                K_FEATURES = 7 };

// Buffers of the split-precision path: FP64 cell averages plus FP32 nodal
// deviations (the polynomial is ubar + (dev - mean_w dev)).
struct MixBufs {
    const double *ub;   // averages of u^n            [m][cell]
    const float *dv;    // deviations of u^n          [m][cell][n^d]
    float *dv_s;        // deviations of u* = u^n + dt sum_i b_i G(u~^(i))
    double *ub_n;       // averages of u^{n+1}
    float *dv_n;        // deviations of u^{n+1}
    float *tr;          // FP32 face traces           [slot][m][cell][face point]
    float *tavg;        // FP32 cell averages of the traced stages [slot][m][cell]
    const double *nod_in;  // FP64 nodal input (split, operators)
    double *nod_out;       // FP64 nodal output (merge, operators)
    int *flag;
    unsigned long long *nlim, *thmin, *a0, *ord;
    double *aux;
    int *tflags;              // troubled-cell flags (indicator on)
    const float *prob;        // learned probabilities (ind_stage 3, 4)
    float *feat;              // learned indicator's features [cell][44] (k_features_x)
    unsigned long long *ntrb; // troubled cells
};

enum MixKernelId { KX_SPLIT = 0, KX_MERGE = 1, KX_LIMIT = 2, KX_INNER = 3, KX_FINAL = 4, KX_SCAN = 5, KX_AVG = 6,
                   KX_TROUBLE = 7, KX_FEATURES = 8 };

// ---------------------------------------------------------------- ensembles (2D Euler)

// Scalars of one problem's current attempt.
struct EnsScal {
    int flag;                 // a stage average left B^eps
    int pad;
    unsigned long long nlim;  // limited cells
    unsigned long long thmin; // bits of the smallest theta
    unsigned long long a0;    // bits of the rate of the new state
    unsigned long long ord[2];
    unsigned long long ntrb;  // troubled cells
};

// Descriptor of one problem of an ensemble (device table, one per problem).
struct EnsProblem {
    Params P;                // its parameters; P.dt is the step of the current attempt
    double *u[2];            // u[cur] holds u^n, u[cur ^ 1] receives u^{n+1}
    double *ustar, *tr, *tavg, *aux;
    int *tflags;
    float *feat;
    const float *prob;
    EnsScal *sc;
    int n;                   // k + 1
    int cur;
    int pending;             // takes part in the current attempt
    int done;                // reached t_end
    int status;              // 0, or CRKDG_E_BOUNDS after max_halvings
    int restarts;            // halvings of the current step
    int klass;               // (n - 3) * 3 + size class, for tuning
    int stored;              // tr also holds the flux sums and the faces' radii
    double t, t_end, cfl, a0;
    long long steps, restarts_total;
    // the last accepted step
    double last_dt, last_thmin;
    long long last_nlim, last_ntrb;
    int last_restarts, pad2;
};

// Work item: blocks [blk, blk + nblk) of problem prob.
struct EnsItem {
    int prob, blk, nblk, pad;
};

enum { ENS_COUNTERS = 16 };
// ENS_FINAL_BARE: the final stage of ensembles whose flux sums and radii do not fit (EnsProblem::stored);
// ENS_INNER_64: the inner stages of ensembles out of the fixed-point range (gamma >= 2)
enum EnsKernelKind { ENS_INNER = 0, ENS_FINAL = 1, ENS_TROUBLE = 2, ENS_FEATURES = 3, ENS_FINAL_BARE = 4, ENS_INNER_64 = 5, ENS_KINDS = 6 };
struct EnsCtl {
    unsigned int counter[ENS_COUNTERS];  // one work counter per persistent launch of an attempt
    int any_pending;
    int pad[3];
};

// Scalars of one attempt of the device-resident step loop (three rotate).
struct RunSlot {
    int flag;
    int pad;
    unsigned long long nlim;
    unsigned long long thmin;
    unsigned long long rate;  // bits of max over S_K of sum_d lambda_d / h_d
};

// Control block of the persistent 1D run kernel (device memory).
struct RunCtl {
    // inputs
    double t, t_end, dt0, cfl;
    int nsteps, max_halvings, cur;
    int extra_arrivals;  // testing aid: > 0 makes the barrier wait for blocks that never come
    // outputs
    double t_out, rate_out;
    int steps, restarts, cur_out, status;
    unsigned long long nlim_total;
    // grid barrier: arrivals so far (zero at launch)
    unsigned bar_count, pad_;
    RunSlot slot[3];
};

// Status values written by the run kernel (match crkdg_status).
enum RunStatus { RUN_OK = 0, RUN_BOUNDS = 4, RUN_TIMEOUT = 5 };

}  // namespace crkdg

// Per-dimension launchers (defined in dg_1d.cu / dg_2d.cu).
extern "C++" {
cudaError_t crkdg_upload_tables_1d(const crkdg::NodalTables *t);
cudaError_t crkdg_upload_tables_2d(const crkdg::NodalTables *t);
cudaError_t crkdg_launch_1d(int kernel, int n, int phys, cudaStream_t st, const crkdg::Params &P,
                            const crkdg::Bufs &B);
cudaError_t crkdg_launch_2d(int kernel, int n, int phys, cudaStream_t st, const crkdg::Params &P,
                            const crkdg::Bufs &B);
cudaError_t crkdg_launch_mx_1d(int kernel, int n, int phys, int nblocks, cudaStream_t st,
                               const crkdg::Params &P, const crkdg::MixBufs &B);
cudaError_t crkdg_launch_mx_2d(int kernel, int n, int phys, int nblocks, cudaStream_t st,
                               const crkdg::Params &P, const crkdg::MixBufs &B);
// Ensembles of 2D Euler problems (defined in dg_ens.cu).
cudaError_t crkdg_upload_tables_ens(const crkdg::NodalTables *t);
cudaError_t crkdg_ens_launch(int kind, int n, int grid, cudaStream_t st, crkdg::EnsProblem *E,
                             const crkdg::EnsItem *items, int nitems, crkdg::EnsCtl *ctl, int counter, int stage);
int crkdg_ens_occupancy(int kind, int n);
int crkdg_ens_cells_per_block(int kind, int n);
// which: 0 open a step (arg: size class or -1), 1 clear the counters, 2 close an attempt (arg: max_halvings)
cudaError_t crkdg_ens_control(int which, cudaStream_t st, crkdg::EnsProblem *E, int np, crkdg::EnsCtl *ctl, int arg);
// Inner stages of the split-precision path on the tensor cores (2D Euler, n = 4, MODE_STEP,
// tableaux whose A has only a sub-diagonal; defined in dg_2d.cu).
cudaError_t crkdg_launch_inner_tc(cudaStream_t st, const crkdg::Params &P, const crkdg::MixBufs &X);
// The split path's passes of 2D Euler, n = 2, 3, 4: the stages by lines (KX_INNER for the same tableaux,
// KX_FINAL, MODE_STEP), the others with one thread per cell (KX_TROUBLE, KX_MERGE, KX_SPLIT, with
// MODE_RATE also as KX_LIMIT); defined in dg_2d.cu.
cudaError_t crkdg_launch_cell(int kernel, int n, cudaStream_t st, const crkdg::Params &P, const crkdg::MixBufs &X);
// Closed-form nodal tables for n = 2, 3, 4 (defined in crkdg_api.cu).
void crkdg_build_tables(crkdg::NodalTables *tab);
// The same tables, built once per process (host memory).
const crkdg::NodalTables *crkdg_host_tables();
// Persistent 1D step loop (cooperative launch); chunk: own cells per block chunk (0: fill
// every block slot of the GPU); *nblocks receives the grid used.
cudaError_t crkdg_run_1d(int n, int phys, cudaStream_t st, const crkdg::Params &P, double *u0, double *u1,
                         crkdg::RunCtl *ctl, int chunk, int *nblocks);
}

// ac_kernels.cuh -- the fused pseudo-time stage sweep and its control kernels.
//
// One launch of stage_kernel performs Runge-Kutta stage s of one
// pseudo-iteration (Alg. 1, Eq. RK2) over the whole grid:
//   ghost synthesis (Sec. 2.5) -> limited gradients of rho, u, v (Sec. 2.3.1)
//   -> pressure gradient (Eq. new_gradp, or a limiter on p) -> MUSCL face
//   states (Eqs. muscl1-2) -> Osher flux on every x- and y-face (Sec. 2.4.3,
//   y-faces through the rotation of Alg. 2) -> flux divergence + real-time
//   term + body force (Sec. 2.2.1) -> point-implicit stage update
//   (Eqs. RK2, point_implicit) -> stage-1 residual partial sums.
// Each CTA owns a TX x TY tile; the tile plus a two-cell halo is staged in
// shared memory, so every field of every cell is read from HBM once per
// stage (halo re-reads hit L2).
//
// Which of the three state buffers holds Q^{m}, the stage inputs and the
// stage outputs is decided on the device from ctl->cur, so one captured
// graph serves every pseudo-iteration.
#pragma once

#include "ac_device.cuh"

namespace acgb {

// Device-resident control block of one physical step.
struct alignas(16) Ctl {
    int iter;        // pseudo-iterations completed
    int done;        // 1: stop iterating
    int cur;         // buffer index (0..2) holding Q^{m}
    int status;      // 0 converged / 1 not converged / -3 non-finite
    int max_iters;
    int fixed;       // 1: tol < 0, run exactly max_iters
    double tol;
    double dt, inv_dt;
    double R[4], R0[4];
    double abs_tol[4];
    unsigned long long dtau_bits;  // global pseudo-time step (bit pattern of a positive double)
    int rebase;      // mixed form: fold the pressure increment into its FP64 level before the next iteration
    double tau, tau_end;  // pure pseudo-time run: pseudo-time reached and its end (+inf in a physical step)
};

// What every stage kernel needs of the control block, in two loads issued
// together (the pass through L2 that each costs in sequence was 10 % of a small
// grid's stage).
template <typename T>
struct CtlHead {
    int done, cur;
    T inv_dt;
};
template <typename T>
__device__ __forceinline__ CtlHead<T> ctl_head(const Ctl *ctl) {
    CtlHead<T> h;
    int it, st;
    double inv_dt;
    asm volatile("ld.global.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(it), "=r"(h.done), "=r"(h.cur), "=r"(st) : "l"(ctl));
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(inv_dt) : "l"(&ctl->inv_dt));
    h.inv_dt = T(inv_dt);
    return h;
}

// The global pseudo-time step of the current iteration, shortened so that a
// pure pseudo-time run lands on its end (tau_end is +inf otherwise).
__device__ __forceinline__ double global_dtau(const Ctl *ctl) {
    return fmin(__longlong_as_double((long long)ctl->dtau_bits), ctl->tau_end - ctl->tau);
}

// What the end of a pseudo-iteration needs (see end_iteration).
// The mixed form rebases its pressure level after these pseudo-iterations of
// a step (1, 2, 4, ..., kRebaseLast): the first ones are where a step that
// starts from an unbalanced state moves the pressure the most.
constexpr int kRebaseLast = 8;
__host__ __device__ __forceinline__ bool rebase_after(int it) { return it <= kRebaseLast && (it & (it - 1)) == 0; }

struct IterEnd {
    int rebase_pow2;           // mixed form with a pressure level: rebase after iterations 1, 2, 4, 8
    int nparts;                // residual partial slots written by stage 1
    int s_max;
    int use_cond;              // set the graph's while-condition
    double inv_cells;
    unsigned long long cond;   // its handle
};
constexpr int kEndLanes = 128;  // threads that take part in end_iteration

template <typename T>
struct SweepArgs {
    int nx, ny;
    int bc[4];
    int gradp, limiter_k, realtime, local_dtau, alpha_pi_p_row;
    int riemann;                   // kOsher / kBassi / kRoe
    int stage, s_max;
    T dx, dy, half_dx, half_dy, dx_over_dy, dy_over_dx;
    T beta, inv_beta, gx, gy;
    int fixed;                     // the Osher flux may run in fixed point (beta and the cell sizes allow it)
    FixedBeta fbeta;               // beta for the fixed-point Osher flux
    T hidx, hidy, phidx, phidy;    // 1/(2 dx), 1/(2 dy), and beta times them
    FixedScale fhx, fhy, fphx, fphy;   // the same for the fixed-point flux
    T inv_alpha, inv_cfl_area;
    T cfl_area;                    // CFL_tau * |Omega|
    T *buf[3][4];                  // three state buffers: rho, rho u, rho v, p
    T *lev[4];                     // real-time level Q^n (rho, rho u, rho v, p)
    T *lev1[3], *lev2[3];          // Q^{n-1}, Q^{n-2} (rho, rho u, rho v) for BDF2/BDF3
    int order;                     // backward-difference order used in this step (1..3)
    T B[4];                        // its coefficients B0..B3 (Table BDF)
    double *partials;              // per-CTA residual partial sums [nblocks][4]
    Ctl *ctl;
    // Per-cell values that stay fixed through a pseudo-iteration (they come
    // from Q^{m} and the real-time levels): 1/dtau (local) and the real-time
    // terms of rho, rho u, rho v.  With reuse set, stage 1 writes them and
    // later stages read them back instead of recomputing; null otherwise.
    T *aux[4];
    int reuse;
};

// The constants of the fixed-point flux and of the scaled fluxes; stage, s_max and cfl_area are set.
inline void set_flux_scales(SweepArgs<double> &a, double beta, double dx, double dy) {
    a.fixed = fixed_beta_ok(beta) && fixed_beta_ok(dx) && fixed_beta_ok(dy);
    a.fbeta = make_fixed_beta(beta);
    a.hidx = 0.5 / dx;
    a.hidy = 0.5 / dy;
    a.phidx = beta * a.hidx;
    a.phidy = beta * a.hidy;
    a.fhx = make_fixed_scale(a.hidx);
    a.fhy = make_fixed_scale(a.hidy);
    a.fphx = make_fixed_scale(a.phidx);
    a.fphy = make_fixed_scale(a.phidy);
    a.inv_alpha = double(a.s_max - a.stage + 1);
    a.inv_cfl_area = 1.0 / a.cfl_area;
}

// Frozen real-time term (Eq. bdf) of field f at index s, Q^{m} value qm, Q^n
// value ql: (B0 Q^{m} + B1 Q^n + B2 Q^{n-1} + B3 Q^{n-2}) / dt, always in this order.
template <typename T>
__device__ __forceinline__ T realtime_term(const SweepArgs<T> &a, T qm, T ql, int f, size_t s, T inv_dt) {
    if (a.order == 1) return (qm - ql) * inv_dt;   // Backward-Euler: B0 = 1, B1 = -1
    T r = fma(a.B[1], ql, a.B[0] * qm);
    if (a.order >= 2) r = fma(a.B[2], a.lev1[f][s], r);
    if (a.order >= 3) r = fma(a.B[3], a.lev2[f][s], r);
    return r * inv_dt;
}
template <typename T>
__device__ __forceinline__ T realtime_term(const SweepArgs<T> &a, T qm, int f, size_t s, T inv_dt) {
    return realtime_term(a, qm, a.lev[f][s], f, s, inv_dt);
}

// Buffer roles within a pseudo-iteration: stage s reads `in` and writes
// `out`; Q^{m} (stage 0) stays in `cur` until the iteration ends.
__device__ __forceinline__ void stage_buffers(int cur, int s, int &in, int &out) {
    const int o1 = (cur + 1) % 3, o2 = (cur + 2) % 3;
    out = (s & 1) ? o1 : o2;
    in = (s == 1) ? cur : (((s - 1) & 1) ? o1 : o2);
}
__host__ __device__ __forceinline__ int final_buffer(int cur, int s_max) {
    return (s_max & 1) ? (cur + 1) % 3 : (cur + 2) % 3;
}

// Sum over a warp of four values per lane: lanes 0, 8, 16, 24 receive the sums
// of v[0], v[1], v[2], v[3].  The first two exchanges leave each lane one of the
// four, so that a warp spends 6 FP64 additions instead of 20.
__device__ __forceinline__ double warp_sum4(const double v[4]) {
    const int lane = threadIdx.x & 31;
    const bool up16 = lane & 16, up8 = lane & 8;
    double a = (up16 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, up16 ? v[0] : v[2], 16);
    const double b = (up16 ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, up16 ? v[1] : v[3], 16);
    a = (up8 ? b : a) + __shfl_xor_sync(0xffffffffu, up8 ? a : b, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}

// Sum of the stage-1 residual partials (4 per slot, nparts slots) in a fixed
// order: 128 strided sums, a shuffle tree in each of four warps, the four
// warp sums left to right.  Called by every thread of a CTA of at least
// kEndLanes threads; thread f < 4 receives field f's sum.  The single-tank end
// of iteration and the batch's per-tank end both use it, so a tank's norms do
// not depend on which of them ran.
__device__ __forceinline__ double sum_partials_fixed(const double *partials, int nparts) {
    __shared__ double wsum[kEndLanes / 32][4];
    const int tid = threadIdx.x;
    if (tid < kEndLanes) {
        double s[4] = {0.0, 0.0, 0.0, 0.0};
        for (int b = tid; b < nparts; b += kEndLanes) {
#pragma unroll
            for (int f = 0; f < 4; ++f) s[f] += partials[(size_t)b * 4 + f];
        }
        const double v = warp_sum4(s);
        if ((tid & 7) == 0) wsum[tid >> 5][(tid & 31) >> 3] = v;
    }
    __syncthreads();
    double sum = 0.0;
    if (tid < 4) {
        sum = wsum[0][tid];
        for (int w = 1; w < kEndLanes / 32; ++w) sum += wsum[w][tid];
    }
    return sum;
}

// The control block's part in the stopping test, read by threads f < 4 before
// the partial sums (whose loads it overlaps) and judged by them after.
struct EndTest {
    int it, cur, max_iters, fixed;
    double tol, R0, abs_tol;
    bool finite, conv;
    __device__ __forceinline__ void load(const Ctl *ctl) {
        const int f = threadIdx.x;
        if (f >= 4) return;
        it = ctl->iter + 1;
        cur = ctl->cur;
        max_iters = ctl->max_iters;
        fixed = ctl->fixed;
        tol = ctl->tol;
        R0 = ctl->R0[f];
        abs_tol = ctl->abs_tol[f];
    }
    // threads f < 4 only: field f's norm, stored, and the test over all fields
    __device__ __forceinline__ void judge(Ctl *ctl, double sum, double inv_cells) {
        const int f = threadIdx.x;
        const double R = sqrt(sum * inv_cells);
        ctl->R[f] = R;
        if (it == 1) ctl->R0[f] = R0 = R;
        finite = __all_sync(0xfu, isfinite(R));
        conv = __all_sync(0xfu, R <= fmax(tol * R0, abs_tol));
    }
};

// End of a pseudo-iteration: the residual norms from the stage-1 partials,
// the stopping test (Alg. 1), the buffer rotation and, inside a captured
// loop, the while-condition.  Called by every thread of one CTA of at least
// kEndLanes threads.
__device__ __forceinline__ void end_iteration(Ctl *ctl, const double *partials, const IterEnd &e) {
    EndTest t;
    t.load(ctl);
    double tau = 0.0, tau_end = 0.0, dtau = 0.0;
    const int tid = threadIdx.x;
    if (tid == 0) {
        tau = ctl->tau;
        tau_end = ctl->tau_end;
        dtau = global_dtau(ctl);
    }
    const double sum = sum_partials_fixed(partials, e.nparts);
    if (tid >= 4) return;
    t.judge(ctl, sum, e.inv_cells);
    if (tid == 0) {
        ctl->iter = t.it;
        ctl->cur = final_buffer(t.cur, e.s_max);
        bool reached = false;   // a pure pseudo-time run reached its end
        if (tau_end < INFINITY) {
            tau += dtau;
            ctl->tau = tau;
            reached = tau >= tau_end;
        }
        int done = 0;
        if (!t.finite) { ctl->status = -3; done = 1; }
        else if (reached) { ctl->status = 0; done = 1; }
        else if (!t.fixed && t.conv) { ctl->status = 0; done = 1; }
        else if (t.it >= t.max_iters) {
            // a fixed iteration count is complete; a pseudo-time run short of its end is not
            ctl->status = (t.fixed && !(tau_end < INFINITY)) ? 0 : 1;
            done = 1;
        }
        ctl->done = done;
        ctl->rebase = (e.rebase_pow2 && !done && rebase_after(t.it)) ? 1 : 0;
        ctl->dtau_bits = 0x7ff0000000000000ull;
        if (e.use_cond) cudaGraphSetConditional(e.cond, done ? 0u : 1u);
    }
}

template <typename T>
__device__ __forceinline__ T wall_ghost_sign(int gi, int gj, int nx, int ny, const int bc[4]) {
    const bool w = (gi < 0 && is_wall(bc[0])) || (gi >= nx && is_wall(bc[1])) ||
                   (gj < 0 && is_wall(bc[2])) || (gj >= ny && is_wall(bc[3]));
    return w ? T(-1) : T(1);
}

// Programmatic dependent launch: let the next kernel in the stream be
// scheduled (its CTAs then wait in pdl_wait), and wait until the previous
// kernel has finished and its writes are visible.  No-ops for a kernel
// launched without the programmatic-serialization attribute.  Every kernel
// waits first and triggers then: CTAs that triggered before their wait let the
// kernel after them in as well, and the waiting CTAs of two kernels filled the
// SMs' free slots unevenly (per iteration, trigger first -> wait first:
// 256x256 mixed tiles 26.9 -> 26.0 us, 1024x512 in 16-row strips 57.8 -> 54.8,
// 1024x1024 in 32-row strips 93.1 -> 84.5; FP64 and larger grids as before).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Threads of the FP64 sweep's CTA on a TX x TY tile: one per cell, but 16 warps
// on the 32x14 tile, whose two groups then have two warps on each of the four
// SM sub-partitions (14 warps leave one warp alone on some), and two per cell
// on the 8x8 tile, whose faces then take two passes.
__host__ __device__ constexpr int f64_threads(int tx, int ty) {
    return tx == 32 && ty == 14 ? 512 : tx * ty == 64 ? 128 : tx * ty;
}

template <typename T, int TX, int TY>
struct StageSmem {
    static constexpr int RW = TX + 4, RH = TY + 4;   // tile + 2-cell halo
    static constexpr int GW = TX + 2, GH = TY + 2;   // tile + 1-cell ring
    static constexpr int NXF = (TX + 1) * TY;        // x-faces
    static constexpr int NYF = TX * (TY + 1);        // y-faces
    T w[4][RW * RH];      // rho, u, v, p
    T wir[RW * RH];       // 1/rho of w (stage 1's local pseudo-time step takes it, with u and v)
    T rt[2][GW * GH];     // frozen real-time term of rho u, rho v on the ring
    T gx[4][GW * GH];     // whole slopes along x: rho, u, v, p (the face states take half of each)
    T gy[4][GW * GH];     // whole slopes along y
    T fx[4][NXF];         // x-face fluxes: mass, x-mom, y-mom, p/beta
    T fy[4][NYF];         // y-face fluxes
    double red[4][f64_threads(TX, TY) / 32];
};

// CTAs per SM the register allocation is asked to allow.  Tiles of 448 cells
// run one per SM and take the whole register file; 256-thread tiles run three
// (80 registers and a few spills: 568 us per pseudo-iteration of a 1024x512
// tank, 660-706 us at two or four), so that the FP64-bound phases of one CTA
// run beside the integer-bound faces of another; 128-thread tiles four.
constexpr int f64_min_blocks(int nt) { return nt >= 448 ? 1 : nt == 256 ? 3 : nt == 128 ? 4 : 0; }

// Named barriers of a CTA: wait for, or only signal, barrier id of n threads.
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

template <typename T, int TX, int TY, int RS = kOsher>
__global__ void __launch_bounds__(f64_threads(TX, TY), f64_min_blocks(TX * TY))
stage_kernel(const SweepArgs<T> a) {
    using S = StageSmem<T, TX, TY>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S &sm = *reinterpret_cast<S *>(smem_raw);
    constexpr int NT = f64_threads(TX, TY);
    constexpr int RW = S::RW, RH = S::RH, GW = S::GW, GH = S::GH;
    // A 32x14 tile runs alone on its SM, so nothing else fills the FP64 unit
    // while its faces keep the integer pipes busy.  Its warps therefore work in
    // two groups, one per half of the rows, the second a phase behind: the
    // first group's faces run beside the second's slopes, and its update
    // beside the second's faces (256x256 tank: 105 -> 91 us per pseudo-iteration;
    // 87 with what is now done less between the stages).
    constexpr int GR = (TX == 32 && TY == 14) ? 2 : 1, NTG = NT / GR;

    pdl_wait();
    pdl_trigger();
    const Ctl *ctl = a.ctl;
    const CtlHead<T> head = ctl_head<T>(ctl);
    if (head.done) return;
    int in, out;
    const int cur = head.cur;
    stage_buffers(cur, a.stage, in, out);
    const T *const *qin = a.buf[in];
    const T *const *q0 = a.buf[cur];
    T *const *qout = a.buf[out];
    const T inv_dt = a.realtime ? head.inv_dt : T(0);

    const int nx = a.nx, ny = a.ny;
    const int tid = threadIdx.x;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    // Rows of the tile inside the domain: tiles of under 256 cells load, slope
    // and solve nothing for the rows past them (100x1: 55 -> 32 us per
    // pseudo-iteration).  Larger tiles, picked only on grids of many rows,
    // keep constant bounds: there the rows saved are few and the bounds' extra
    // registers cost more (600x401 on 32x8: 297 -> 303 us, 256x256 on 32x14:
    // 86.0 -> 86.7).
    constexpr bool TRIM = TX * TY < 256;
    const int th = TRIM ? min(TY, ny - y0) : TY;

    // A tile whose halo lies inside the domain needs no ghost folding.  The
    // ring's real-time inputs are loaded first and used last, and interior
    // tiles load all their halo cells before the first is used, so that one
    // round trip to memory covers them.
    const bool interior = x0 >= 2 && x0 + TX + 2 <= nx && y0 >= 2 && y0 + TY + 2 <= ny;
    const bool need_rt = (a.gradp == kGradNew) && a.realtime;
    const bool reuse_now = a.reuse && a.stage > 1;   // fixed per-cell values from stage 1
    constexpr int NR = (GW * GH + NT - 1) / NT, NW = (RW * RH + NT - 1) / NT;
    T rt_q[NR][2], rt_l[NR][2];   // real-time terms (later stages) or Q^{m} and Q^n (stage 1) of rho u, rho v
    int rt_s[NR], rt_f[NR];       // source cell and signs of the ring cell
    if (need_rt) {
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int k = tid + r * NT;
            rt_f[r] = 0;
            if (k >= GW * (th + 2)) continue;
            const int gi = x0 + (k % GW) - 1, gj = y0 + (k / GW) - 1;
            if (interior) {
                rt_s[r] = gj * nx + gi;
            } else {
                int nfx, tfx, nfy, tfy;
                const int si = fold_axis(gi, nx, a.bc[0], a.bc[1], nfx, tfx);
                const int sj = fold_axis(gj, ny, a.bc[2], a.bc[3], nfy, tfy);
                rt_s[r] = sj * nx + si;
                rt_f[r] = ((nfx + tfy) & 1) | (((nfy + tfx) & 1) << 1);
            }
            if (reuse_now) {
                rt_q[r][0] = a.aux[2][rt_s[r]];
                rt_q[r][1] = a.aux[3][rt_s[r]];
            } else {
                rt_q[r][0] = q0[1][rt_s[r]];
                rt_q[r][1] = q0[2][rt_s[r]];
                rt_l[r][0] = a.lev[1][rt_s[r]];
                rt_l[r][1] = a.lev[2][rt_s[r]];
            }
        }
    }
    // ---- 1. stage Q^{s-1} (+ two-cell halo, ghosts synthesised) as W ----
    auto put_w = [&](int k, T r, T m, T n, T p) {
        const T ir = Ar<T>::rcp(r);
        sm.w[0][k] = r;
        sm.w[1][k] = m * ir;
        sm.w[2][k] = n * ir;
        sm.w[3][k] = p;
        sm.wir[k] = ir;
    };
    if (interior) {
        T in4[NW][4];
        const int base = (y0 - 2) * nx + (x0 - 2);
#pragma unroll
        for (int r = 0; r < NW; ++r) {
            const int k = tid + r * NT;
            if (k >= RW * RH) continue;
            const int s = base + (k / RW) * nx + k % RW;
#pragma unroll
            for (int f = 0; f < 4; ++f) in4[r][f] = qin[f][s];
        }
#pragma unroll
        for (int r = 0; r < NW; ++r)
            if (tid + r * NT < RW * RH) put_w(tid + r * NT, in4[r][0], in4[r][1], in4[r][2], in4[r][3]);
    } else {
        for (int k = tid; k < RW * (th + 4); k += NT) {
            const int gi = x0 + (k % RW) - 2, gj = y0 + (k / RW) - 2;
            int nfx, tfx, nfy, tfy;
            const int si = fold_axis(gi, nx, a.bc[0], a.bc[1], nfx, tfx);
            const int sj = fold_axis(gj, ny, a.bc[2], a.bc[3], nfy, tfy);
            const size_t s = (size_t)sj * nx + si;
            T m = qin[1][s], n = qin[2][s];
            if ((nfx + tfy) & 1) m = -m;
            if ((nfy + tfx) & 1) n = -n;
            put_w(k, qin[0][s], m, n, qin[3][s]);
        }
    }
    // ---- frozen real-time term of the momenta on the ring (Eq. bdf) ----
    if (need_rt) {
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int k = tid + r * NT;
            if (k >= GW * (th + 2)) continue;
            T rx = rt_q[r][0], ry = rt_q[r][1];
            if (!reuse_now) {
                rx = realtime_term(a, rx, rt_l[r][0], 1, rt_s[r], inv_dt);
                ry = realtime_term(a, ry, rt_l[r][1], 2, rt_s[r], inv_dt);
            }
            sm.rt[0][k] = rt_f[r] & 1 ? -rx : rx;
            sm.rt[1][k] = rt_f[r] & 2 ? -ry : ry;
        }
    }
    __syncthreads();

    // ---- 2. limited slopes and pressure gradient on the ring ----
    // Whole slopes (the limited difference across one cell, dx d_x rho and
    // so on); the face states take half of each with one FMA.  Halving is
    // exact, so these are the half slopes of the limiter's definition to
    // the last bit, formed with fewer FP64 instructions.
    const T klim = T(a.limiter_k);
    const T kp = (a.gradp == kGradSuperbee || a.gradp == kGradSplitSuperbee) ? T(2) : T(1);
    const int grp = GR == 2 ? tid / NTG : 0, tg = tid - grp * NTG;
    constexpr int R0 = GR == 2 ? TY / 2 + 2 : GH;      // ring rows the first group's faces need
    if (GR == 2 && grp == 1) bar_sync(3, NT);          // the first group's slopes first
    static_assert(!TRIM || GR == 1, "a trimmed tile works in one group");
    const int kend = GR == 2 && grp == 0 ? R0 * GW : GW * (th + 2);
    for (int k = grp * (R0 * GW) + tg; k < kend; k += NTG) {
        const int li = k % GW, lj = k / GW;            // ring coords (cell li-1, lj-1)
        const int c = (lj + 1) * RW + (li + 1);
        const int e = c + 1, wv = c - 1, nn = c + RW, ss = c - RW;
        const T *R = sm.w[0], *U = sm.w[1], *V = sm.w[2], *P = sm.w[3];
        T srx, sry, sux, suy, svx, svy;
        if (a.limiter_k == 1) {
            srx = minmod_bits(R[e] - R[c], R[c] - R[wv]);
            sry = minmod_bits(R[nn] - R[c], R[c] - R[ss]);
            sux = minmod_bits(U[e] - U[c], U[c] - U[wv]);
            suy = minmod_bits(U[nn] - U[c], U[c] - U[ss]);
            svx = minmod_bits(V[e] - V[c], V[c] - V[wv]);
            svy = minmod_bits(V[nn] - V[c], V[c] - V[ss]);
        } else {
            srx = limiter(R[e] - R[c], R[c] - R[wv], klim);
            sry = limiter(R[nn] - R[c], R[c] - R[ss], klim);
            sux = limiter(U[e] - U[c], U[c] - U[wv], klim);
            suy = limiter(U[nn] - U[c], U[c] - U[ss], klim);
            svx = limiter(V[e] - V[c], V[c] - V[wv], klim);
            svy = limiter(V[nn] - V[c], V[c] - V[ss], klim);
        }
        T spx, spy;
        if (a.gradp == kGradNew) {
            // Eq. new_gradp times dx, with dx d_x rho = srx etc.
            const int gi = x0 + li - 1, gj = y0 + lj - 1;
            const T rho = R[c], u = U[c], v = V[c];
            // the body force with gravity reversed in wall ghosts: a sign, not a product
            const T rho_g = wall_ghost_sign<T>(gi, gj, nx, ny, a.bc) < T(0) ? -rho : rho;
            const T rtx = need_rt ? sm.rt[0][k] : T(0);
            const T rty = need_rt ? sm.rt[1][k] : T(0);
            // d(rho u u) = u A + rho u du with A = d(rho u) along x, d(rho u v) = v A + rho u dv, and so on: 20 FP64
            // instructions in place of 27 term by term
            const T ru = rho * u, rv = rho * v;
            const T A = fma(rho, sux, u * srx), B = fma(rho, svy, v * sry);
            const T xx = fma(u, A, ru * sux), xy = fma(u, B, rv * suy);
            const T yy = fma(v, B, rv * svy), yx = fma(v, A, ru * svx);
            spx = fma(-a.dx_over_dy, xy, fma(a.dx, fma(rho_g, a.gx, -rtx), -xx));
            spy = fma(-a.dy_over_dx, yx, fma(a.dy, fma(rho_g, a.gy, -rty), -yy));
        } else if (a.gradp == kGradSplitMinmod || a.gradp == kGradSplitSuperbee) {
            // Qian et al. split (Sec. 2.3.2): limit the kinematic part of the
            // one-sided pressure differences, add the cell's hydrostatic
            // slope back; gravity reversed in wall ghosts as for Eq. new_gradp
            const int gi = x0 + li - 1, gj = y0 + lj - 1;
            const T sg = wall_ghost_sign<T>(gi, gj, nx, ny, a.bc);
            const T gxs = a.gx * sg, gys = a.gy * sg;
            spx = limiter(P[e] - P[c] - a.half_dx * (R[c] + R[e]) * gxs,
                          P[c] - P[wv] - a.half_dx * (R[wv] + R[c]) * gxs, kp) + a.dx * R[c] * gxs;
            spy = limiter(P[nn] - P[c] - a.half_dy * (R[c] + R[nn]) * gys,
                          P[c] - P[ss] - a.half_dy * (R[ss] + R[c]) * gys, kp) + a.dy * R[c] * gys;
        } else {
            spx = limiter(P[e] - P[c], P[c] - P[wv], kp);
            spy = limiter(P[nn] - P[c], P[c] - P[ss], kp);
        }
        sm.gx[0][k] = srx; sm.gx[1][k] = sux; sm.gx[2][k] = svx; sm.gx[3][k] = spx;
        sm.gy[0][k] = sry; sm.gy[1][k] = suy; sm.gy[2][k] = svy; sm.gy[3][k] = spy;
    }
    if (GR == 2) {
        if (grp == 0) bar_arrive(3, NT);
        bar_sync(1 + grp, NTG);
    } else {
        __syncthreads();
    }

    // ---- 3. face states and Osher fluxes ----
    // A group's faces are dealt out so that the four SM sub-partitions get
    // equal numbers of warp-passes (a pass costs the same with idle lanes).
    // The warps of a CTA sit on contiguous slots, so warps w and w + 4 share a
    // sub-partition; its share, faces [32 P s, 32 P (s + 1)) of the group's F,
    // P = ceil(F / 128), goes to its warps of the group in passes of 32, round-robin.
    // The faces of th rows are a prefix of each kind; on a grid of few rows
    // they are one or two passes, not three.
    constexpr int NWG = NTG / 32, HG = TY / GR;       // warps and rows of a group
    static_assert(NWG >= 4, "face schedule needs four warps");
    const int rows = TRIM ? th : HG;                               // the group's rows
    const int XG = rows * (TX + 1), xf0 = grp * (HG * (TX + 1));   // its x-faces and the first of them
    const int yf0 = grp * ((HG + 1) * TX);                         // its first y-face and their number: the first
    const int yfn = (grp == 0 ? rows + 1 : rows) * TX;             // group takes the faces between the groups
    const int nf = XG + yfn, fp = (nf + 127) / 128;
    const int fw = tid >> 5, sub = fw & 3;
    const int w0 = grp * NWG + ((sub - grp * NWG) & 3);            // the sub-partition's first warp of the group
    const int fwarps = (grp * NWG + NWG - w0 + 3) >> 2;
    const int fbeg = sub * 32 * fp, fend = min(nf, fbeg + 32 * fp);
    for (int fq = (fw - w0) >> 2; fbeg + 32 * fq < fend; fq += fwarps) {
        const int kf = fbeg + 32 * fq + (tid & 31);
        if (kf >= fend) continue;
        const int k = kf < XG ? xf0 + kf : S::NXF + yf0 + (kf - XG);
        const bool isx = k < S::NXF;
        // face states: density, normal and tangential velocity (rotation,
        // Alg. 2: (u, v) on x-faces, (v, u) on y-faces), pressure
        T rL, nL, tL, pL, rR, nR, tR, pR;
        int fo;   // face index within its kind
        if (isx) {
            const int fi = k % (TX + 1), fj = k / (TX + 1);  // face between cells fi-1 and fi
            const int ga = (fj + 1) * GW + fi, gb = ga + 1;
            const int ca = (fj + 2) * RW + fi + 1, cb = ca + 1;
            rL = fma(T(0.5), sm.gx[0][ga], sm.w[0][ca]); rR = fma(T(-0.5), sm.gx[0][gb], sm.w[0][cb]);
            nL = fma(T(0.5), sm.gx[1][ga], sm.w[1][ca]); nR = fma(T(-0.5), sm.gx[1][gb], sm.w[1][cb]);
            tL = fma(T(0.5), sm.gx[2][ga], sm.w[2][ca]); tR = fma(T(-0.5), sm.gx[2][gb], sm.w[2][cb]);
            pL = fma(T(0.5), sm.gx[3][ga], sm.w[3][ca]); pR = fma(T(-0.5), sm.gx[3][gb], sm.w[3][cb]);
            fo = k;
        } else {
            const int kk = k - S::NXF;
            const int fi = kk % TX, fj = kk / TX;            // face between cells fj-1 and fj
            const int ga = fj * GW + fi + 1, gb = ga + GW;
            const int ca = (fj + 1) * RW + fi + 2, cb = ca + RW;
            rL = fma(T(0.5), sm.gy[0][ga], sm.w[0][ca]); rR = fma(T(-0.5), sm.gy[0][gb], sm.w[0][cb]);
            tL = fma(T(0.5), sm.gy[1][ga], sm.w[1][ca]); tR = fma(T(-0.5), sm.gy[1][gb], sm.w[1][cb]);
            nL = fma(T(0.5), sm.gy[2][ga], sm.w[2][ca]); nR = fma(T(-0.5), sm.gy[2][gb], sm.w[2][cb]);
            pL = fma(T(0.5), sm.gy[3][ga], sm.w[3][ca]); pR = fma(T(-0.5), sm.gy[3][gb], sm.w[3][cb]);
            fo = kk;
        }
        // one flux call for both kinds: no divergence where a warp holds both.
        // Fluxes are stored as F/dx or F/dy (formed as 2F times 1/(2 dx)), the
        // pressure row times beta, so that the divergence is sums only.
        T F[4];
        if (RS == kOsher && a.fixed && fixed_flux_ok(rL, nL, tL, pL, rR, nR, tR, pR, a.fbeta)) {
            osher_flux_fixed(rL, nL, tL, pL, rR, nR, tR, pR, a.fbeta, isx ? a.fhx : a.fhy, isx ? a.fphx : a.fphy, F);
        } else {
            riemann_flux<RS, T, true>(rL, nL, tL, pL, rR, nR, tR, pR, a.beta, a.inv_beta, F);
            const T h = isx ? a.hidx : a.hidy;
            F[0] *= h;
            F[1] *= h;
            F[2] *= h;
            F[3] *= isx ? a.phidx : a.phidy;
        }
        T *fd = isx ? &sm.fx[0][fo] : &sm.fy[0][fo];
        const int fs = isx ? S::NXF : S::NYF;
        fd[0] = F[0];
        fd[fs] = isx ? F[1] : F[2];
        fd[2 * fs] = isx ? F[2] : F[1];
        fd[3 * fs] = F[3];
    }
    if (GR == 2) {
        // the second group's lowest cells take the y-faces between the groups
        if (grp == 0) {
            bar_arrive(4, NT);
            bar_sync(1, NTG);
        } else {
            bar_sync(4, NT);
        }
    } else {
        __syncthreads();
    }

    // ---- 4. divergence + sources + point-implicit stage update ----
    constexpr int CG = TX * TY / GR;   // cells of a group
    const int cell = grp * CG + tg;
    const int li = cell % TX, lj = cell / TX;
    const int gi = x0 + li, gj = y0 + lj;
    const bool inside = (tg < CG) && (gi < nx) && (gj < ny);
    double sq[4] = {0.0, 0.0, 0.0, 0.0};
    if (inside) {
        const size_t g = (size_t)gj * nx + gi;
        const int fw = lj * (TX + 1) + li, fe = fw + 1;
        const int fs = lj * TX + li, fn = fs + TX;
        T div[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) div[f] = (sm.fx[f][fe] - sm.fx[f][fw]) + (sm.fy[f][fn] - sm.fy[f][fs]);
        const T r0 = q0[0][g], m0 = q0[1][g], n0 = q0[2][g], p0 = q0[3][g];
        // At stage 1 the input Q^{s-1} is Q^{m} itself, so the cell's W (never
        // a folded ghost here) holds the 1/rho, u and v of Q^{m}, and the ring
        // already holds its momenta's real-time terms: taken as they are, the
        // same values to the last bit.
        const bool from_tile = a.stage == 1;
        const int ct = (lj + 2) * RW + (li + 2), cr = (lj + 1) * GW + (li + 1);
        T rt0 = T(0), rt1 = T(0), rt2 = T(0);
        if (a.realtime) {
            if (reuse_now) {
                rt0 = a.aux[1][g];
                rt1 = a.aux[2][g];
                rt2 = a.aux[3][g];
            } else {
                rt0 = realtime_term(a, r0, 0, g, inv_dt);
                if (from_tile && need_rt) {
                    rt1 = sm.rt[0][cr];
                    rt2 = sm.rt[1][cr];
                } else {
                    rt1 = realtime_term(a, m0, 1, g, inv_dt);
                    rt2 = realtime_term(a, n0, 2, g, inv_dt);
                }
                if (a.reuse) {
                    a.aux[1][g] = rt0;
                    a.aux[2][g] = rt1;
                    a.aux[3][g] = rt2;
                }
            }
        }
        const T b0 = -div[0] - rt0;
        T b1 = -div[1] - rt1;
        T b2 = -div[2] - rt2;
        if (a.gx != T(0)) b1 = fma(r0, a.gx, b1);
        if (a.gy != T(0)) b2 = fma(r0, a.gy, b2);
        const T b3 = -div[3];   // in pressure units
        // pseudo-time step from Q^{m} (Sec. 2.2.3), kept as 1/dtau: Eq. point_implicit's
        // alpha dtau / (1 + B0 alpha dtau/dt) is 1 / (1/(alpha dtau) + B0/dt), one reciprocal
        T idt;
        if (a.local_dtau && reuse_now) {
            idt = a.aux[0][g];
        } else if (a.local_dtau) {
            T ir, u, v;
            if (from_tile) {
                ir = sm.wir[ct];
                u = sm.w[1][ct];
                v = sm.w[2][ct];
            } else {
                ir = Ar<T>::rcp(r0);
                u = m0 * ir;
                v = n0 * ir;
            }
            const T fb = (T(4) * a.beta) * ir;
            T cx, cy, unused;
            Ar<T>::sqrt_rsqrt(fma(u, u, fb), cx, unused);
            Ar<T>::sqrt_rsqrt(fma(v, v, fb), cy, unused);
            idt = fma(fabs(u) + cx, a.half_dy, (fabs(v) + cy) * a.half_dx) * a.inv_cfl_area;
            if (a.reuse) a.aux[0][g] = idt;
        } else {
            idt = Ar<T>::rcp(T(global_dtau(ctl)));
        }
        const T coef = Ar<T>::rcp(fma(idt, a.inv_alpha, a.B[0] * inv_dt));
        const T coef_p = a.alpha_pi_p_row ? coef : Ar<T>::rcp(idt * a.inv_alpha);
        qout[0][g] = fma(coef, b0, r0);
        qout[1][g] = fma(coef, b1, m0);
        qout[2][g] = fma(coef, b2, n0);
        qout[3][g] = fma(coef_p, b3, p0);
        if (a.stage == 1) {
            sq[0] = double(b0) * double(b0);
            sq[1] = double(b1) * double(b1);
            sq[2] = double(b2) * double(b2);
            sq[3] = double(b3) * double(b3);
        }
    }
    if (a.stage == 1) {
        // deterministic block reduction of the squared bracket (FP64)
        const double v = warp_sum4(sq);
        if ((tid & 7) == 0) sm.red[(tid & 31) >> 3][tid >> 5] = v;
        __syncthreads();
        if (tid < 4) {
            double s = 0.0;
            for (int w = 0; w < NT / 32; ++w) s += sm.red[tid][w];
            a.partials[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 4 + tid] = s;
        }
    }
}

// Global pseudo-time step option: min over cells of the local step
// (Sec. 2.2.3), from Q^{m}.  Positive doubles order like their bit patterns.
template <typename T>
__global__ void dtau_min_kernel(const SweepArgs<T> a) {
    pdl_wait();
    pdl_trigger();
    const Ctl *ctl = a.ctl;
    if (ctl->done) return;
    const T *const *q = a.buf[ctl->cur];
    const size_t N = (size_t)a.nx * a.ny;
    double mn = INFINITY;
    for (size_t g = blockIdx.x * (size_t)blockDim.x + threadIdx.x; g < N; g += (size_t)gridDim.x * blockDim.x) {
        const T r0 = q[0][g];
        const T ir = Ar<T>::rcp(r0);
        const T u = q[1][g] * ir, v = q[2][g] * ir, fb = T(4) * a.beta * ir;
        const T cx = Ar<T>::sqrt_(u * u + fb), cy = Ar<T>::sqrt_(v * v + fb);
        const T den = T(0.5) * (fabs(u) + cx) * a.dy + T(0.5) * (fabs(v) + cy) * a.dx;
        mn = fmin(mn, double(Ar<T>::div(a.cfl_area, den)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mn = fmin(mn, __shfl_down_sync(0xffffffffu, mn, o));
    if ((threadIdx.x & 31) == 0)
        atomicMin(&a.ctl->dtau_bits, (unsigned long long)__double_as_longlong(mn));
}

// Global real-time step (Sec. 2.2.4): min over cells of
// CFL_t |Omega| / (|u| dS_x + |v| dS_y), from buffer `cur`; +inf at rest.
template <typename T>
__global__ void realtime_dt_kernel(const SweepArgs<T> a, int cur, double cfl_area, unsigned long long *out) {
    const T *const *q = a.buf[cur];
    const size_t N = (size_t)a.nx * a.ny;
    double mn = INFINITY;
    for (size_t g = blockIdx.x * (size_t)blockDim.x + threadIdx.x; g < N; g += (size_t)gridDim.x * blockDim.x) {
        const double ir = 1.0 / double(q[0][g]);
        const double u = double(q[1][g]) * ir, v = double(q[2][g]) * ir;
        const double den = fabs(u) * double(a.dy) + fabs(v) * double(a.dx);
        mn = fmin(mn, cfl_area / den);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mn = fmin(mn, __shfl_down_sync(0xffffffffu, mn, o));
    if ((threadIdx.x & 31) == 0) atomicMin(out, (unsigned long long)__double_as_longlong(mn));
}

// Start of a physical step: Q^n <- Q (Alg. 1) and reset of the control block.
template <typename T>
__global__ void begin_step_kernel(const SweepArgs<T> a, double dt, double tol, int max_iters, double tau_end) {
    Ctl *ctl = a.ctl;
    const int cur = ctl->cur;
    const size_t N = (size_t)a.nx * a.ny;
    for (size_t g = blockIdx.x * (size_t)blockDim.x + threadIdx.x; g < N; g += (size_t)gridDim.x * blockDim.x) {
        // older levels move back one step: Q^{n-2} <- Q^{n-1} <- Q^n
        if (a.lev2[0])
#pragma unroll
            for (int f = 0; f < 3; ++f) a.lev2[f][g] = a.lev1[f][g];
        if (a.lev1[0])
#pragma unroll
            for (int f = 0; f < 3; ++f) a.lev1[f][g] = a.lev[f][g];
#pragma unroll
        for (int f = 0; f < 4; ++f) a.lev[f][g] = a.buf[cur][f][g];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->iter = 0;
        ctl->done = 0;
        ctl->status = 1;
        ctl->max_iters = max_iters;
        ctl->fixed = tol < 0.0;
        ctl->tol = tol;
        ctl->dt = dt;
        ctl->inv_dt = 1.0 / dt;
        ctl->dtau_bits = 0x7ff0000000000000ull;  // +inf
        ctl->tau = 0.0;
        ctl->tau_end = tau_end;
    }
}

// End of a pseudo-iteration (kEndLanes threads, one CTA).  Sets the graph's
// while-condition when launched inside a captured loop.
static __global__ void __launch_bounds__(kEndLanes)
end_iteration_kernel(Ctl *ctl, const double *partials, const IterEnd e) {
    pdl_wait();
    pdl_trigger();
    if (ctl->done) {
        if (e.use_cond && threadIdx.x == 0) cudaGraphSetConditional(e.cond, 0);
        return;
    }
    end_iteration(ctl, partials, e);
}

}  // namespace acgb

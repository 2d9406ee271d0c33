// Device side of one step of the AB-/BA-GMRES loop (paper Sec. 2,
// algorithm box): the FP64 Givens update of the Hessenberg least-squares
// problem, y_k, and the end of a step (advance k, or stop the solve and end
// the CUDA graph's while loops).  Shared by the loop's own Givens kernel
// (gmres_loop.cu) and the one-launch CGS2 step, whose block 0 runs it once
// the new Hessenberg column is known (arnoldi.cu).
#pragma once
#include "vecops.cuh"

namespace {

__device__ __forceinline__ void end_loops(const LoopBufs &B, int which) {
    const int w = which & B.loops;
    if (w & kLoopSmall) cudaGraphSetConditional(B.c_small, 0u);
    if (w & kLoopFused) cudaGraphSetConditional(B.c_fused, 0u);
    if (w & kLoopPass) cudaGraphSetConditional(B.c_pass, 0u);
}

// End of step k (one thread): stop the solve with `stop` (a CTG_STOP_*
// value + 1, 0 to go on) returning x_iters, or move to step k + 1.  A
// timed-out grid barrier (counter[2] set) stops the solve too; the host
// reports it.
// k, steps and timed_out: S.k, S.steps and counter[2].
__device__ void end_step(const LoopBufs &B, int stop, int iters, int k, int steps, unsigned timed_out) {
    GmresState &S = *B.S;
    S.steps = steps + 1;
    if (timed_out != 0u) {
        stop = CTG_STOP_MAXIT + 1;
        S.timed_out = 1;
    }
    if (stop) {
        S.active = 0;
        S.stop_reason = stop - 1;
        S.iters = iters;
        end_loops(B, kLoopSmall | kLoopFused | kLoopPass);
    } else {
        const int k1 = k + 1;
        S.k = k1;
        if (k1 > B.small_max) end_loops(B, kLoopSmall);
        if (k1 > B.fused_max) end_loops(B, kLoopFused);
    }
}

__device__ __forceinline__ void end_step(const LoopBufs &B, int stop, int iters) {
    end_step(B, stop, iters, B.S->k, B.S->steps, B.counter[2]);
}

// Modes of the Givens update (kGivY, kGivZ, kGivEnd in ctg_internal.cuh):
//   kGivY  y_k into y and yring[k % 3] (BA with a residual rule, AB NCP),
//   kGivZ  z = beta e1 - H_k y_k, the residual's coefficients in W_{k+1}
//          (AB NCP), by the rotations applied backwards,
//   kGivEnd  end the step here (AB with DP / maxit): stop at breakdown, at
//          rho_k <= target (DP) or at k = maxit, else k + 1.
// Otherwise a breakdown or k = maxit is left in S.pending for the step's
// last kernel.  hist[k] = rho_k unless BA with the discrepancy rule (its
// history is the true residual).
constexpr int kGivStage = 512;     // steps staged in shared memory; beyond, lane 0 reads global memory

// Step k after its CGS2 step: Hessenberg column h[0..k] (global or shared
// memory) and ||q before CGS2||^2 = qpre2.  Run by one whole warp (lane =
// threadIdx.x & 31).  The column, the rotations and the rotated column are
// staged in s_stage (3 k + 1 doubles; NULL: global memory) so that lane 0's
// recurrence does no global round trips; the packed triangle of R for y_k
// in s_pack when k <= pack_cap.  A NaN column (a CGS2 step that gave up at
// a grid barrier) counts as a breakdown; end_step then reports the timeout.
__device__ void loop_givens_warp(const LoopBufs &B, int k, const double *h, double qpre2, int mode,
                                 double *s_pack, int pack_cap, double *s_stage) {
    GmresState &S = *B.S;
    const int lane = threadIdx.x & 31;
    double *Rk = B.R + (size_t)(k - 1) * B.ldr;
    double *s_h = s_stage, *s_gc = s_stage ? s_stage + (k + 1) : nullptr, *s_gs = s_gc ? s_gc + k : nullptr;
    if (s_stage) {
        for (int i = lane; i <= k; i += 32) s_h[i] = h[i];
        for (int i = lane; i < k - 1; i += 32) {
            s_gc[i] = B.gc[i];
            s_gs[i] = B.gs[i];
        }
    }
    __syncwarp();
    const double *hh = s_stage ? s_h : h;
    const double *gcc = s_stage ? s_gc : B.gc;
    const double *gss = s_stage ? s_gs : B.gs;
    double rho = 0.0;
    int brk = 0;
    if (lane == 0) {
        double r_prev = hh[0];
        for (int i = 0; i < k - 1; ++i) {
            const double a = r_prev, b = hh[i + 1];
            const double t = gcc[i] * a + gss[i] * b;
            if (s_stage) s_h[i] = t;           // rotated column, stored below
            else Rk[i] = t;
            r_prev = -gss[i] * a + gcc[i] * b;
        }
        const double a = r_prev, b = hh[k];
        double c, sn, rinv;
        givens_rotation(a, b, c, sn, rinv);
        B.gc[k - 1] = c;
        B.gs[k - 1] = sn;
        if (s_stage) s_h[k - 1] = rinv;        // R's diagonal as its reciprocal
        else Rk[k - 1] = rinv;
        B.gg[k] = -sn * B.gg[k - 1];
        B.gg[k - 1] = c * B.gg[k - 1];
        rho = fabs(B.gg[k]);
        S.rho = rho;
        B.rhoh[k] = rho;
        // b <= 1e-6 ||q before CGS2||, squared (b >= 0): no square root
        brk = (!(b == b) || b * b <= 1e-12 * qpre2) ? 1 : 0;
    }
    rho = __shfl_sync(0xffffffffu, rho, 0);
    brk = __shfl_sync(0xffffffffu, brk, 0);
    if (s_stage)
        for (int i = lane; i < k; i += 32) Rk[i] = s_h[i];
    __syncwarp();
    if (mode & kGivY) {
        solve_y_warp(B.R, B.ldr, B.gg, k, B.y, s_pack, pack_cap);
        double *yr = B.yring + (size_t)(k % 3) * B.ldr;
        for (int i = lane; i < k; i += 32) yr[i] = B.y[i];
    }
    if ((mode & kGivZ) && lane == 0) {
        // z = G_1^T ... G_k^T (g_{k+1} e_{k+1}), G_i acting on entries i-1, i
        for (int i = 0; i <= k; ++i) B.z[i] = 0.0;
        B.z[k] = B.gg[k];
        for (int i = k - 1; i >= 0; --i) {
            const double a = B.z[i], b = B.z[i + 1];
            B.z[i] = B.gc[i] * a - B.gs[i] * b;
            B.z[i + 1] = B.gs[i] * a + B.gc[i] * b;
        }
    }
    if (lane != 0) return;
    if (!(S.variant == CTG_BA && S.rule == kRuleDP)) B.hist[k] = rho;
    const int pending = brk ? CTG_STOP_BREAKDOWN + 1 : (k == S.maxit ? CTG_STOP_MAXIT + 1 : 0);
    if (mode & kGivEnd) {
        int stop = pending;
        if (!brk && S.rule == kRuleDP && rho <= S.io.target) stop = CTG_STOP_DP + 1;
        end_step(B, stop, k);
    } else {
        S.pending = pending;
    }
}

// The same update inside the one-launch CGS2 step, without a round trip to
// global memory: what earlier steps left (the rotations, the rotated right-hand
// side, the state and, for y_k, R's columns) is fetched into shared memory
// while the step's passes run (all threads of a block; cp.async), and the
// column comes from there too.  k <= 128 (64 with kGivY).  With lane 0's
// loads and stores in the chain and y_k by solve_y_warp it took 9,400 cycles at
// k = 8 and 22,000 with y_k at k = 9, of 29,500 and 48,600 of the whole step;
// a solve at 512^2, 720 angles went from 1,779 to 1,757 us (AB, 11 steps) and
// from 1,830 to 1,793 us (BA with y_k, 9 steps).
constexpr int kGivLanes = 4;          // entries of the column per lane
struct GivensStage {
    double *h;            // k + 1: the step's column
    double *gc, *gs;      // k - 1 rotations
    double *gg;           // k entries and the new one
    double *pack;         // R packed (kGivY)
    GmresState *S;
};
__host__ __device__ constexpr int givens_stage_doubles(int k) {
    return 4 * k + 2 + (int)((sizeof(GmresState) + sizeof(double) - 1) / sizeof(double));
}
__device__ __forceinline__ GivensStage givens_stage(double *s, int kcap, double *pack) {
    return GivensStage{s, s + kcap + 1, s + 2 * kcap + 1, s + 3 * kcap + 1, pack,
                       reinterpret_cast<GmresState *>(s + 4 * kcap + 2)};
}

__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}

// One block; complete after the threads' cp.async.wait_all and a barrier.
__device__ __forceinline__ void givens_fetch(const LoopBufs &B, int k, int mode, const GivensStage &g) {
    static_assert(sizeof(GmresState) % sizeof(double) == 0, "fetched as doubles");
    const int tid = threadIdx.x;
    for (int i = tid; i < (int)(sizeof(GmresState) / sizeof(double)); i += kThreads)
        cp_async8(reinterpret_cast<double *>(g.S) + i, reinterpret_cast<const double *>(B.S) + i);
    for (int i = tid; i < k; i += kThreads) {
        if (i < k - 1) {
            cp_async8(g.gc + i, B.gc + i);
            cp_async8(g.gs + i, B.gs + i);
        }
        cp_async8(g.gg + i, B.gg + i);
    }
    if (mode & kGivY)
        for (int j = tid >> 5; j < k - 1; j += kWarps)
            for (int i = tid & 31; i <= j; i += 32)
                cp_async8(g.pack + j * (j + 1) / 2 + i, B.R + (size_t)j * B.ldr + i);
}

// y = R^{-1} g by one warp for k <= 64, R packed in shared memory, its diagonal
// as reciprocals: lane l holds g_j / R_jj for j = l and l + 32, and each column
// of R, over its rows' diagonals, takes y_i off them, so that the chain of a
// step is one shuffle and one FMA.  y goes to y and y2.
__device__ void solve_y_packed(const double *s_pack, const double *g, int k, double *__restrict__ y,
                               double *__restrict__ y2) {
    const int lane = threadIdx.x & 31, j1 = lane + 32;
    const double d0 = lane < k ? s_pack[lane * (lane + 3) / 2] : 0.0, d1 = j1 < k ? s_pack[j1 * (j1 + 3) / 2] : 0.0;
    double t0 = lane < k ? g[lane] * d0 : 0.0, t1 = j1 < k ? g[j1] * d1 : 0.0;
    int i = k - 1;
    for (; i >= 32; --i) {
        const double *col = s_pack + i * (i + 1) / 2;
        const double r0 = col[lane] * d0, r1 = j1 < i ? col[j1] * d1 : 0.0;
        const double yi = __shfl_sync(0xffffffffu, t1, i - 32);
        t0 = fma(-r0, yi, t0);
        t1 = fma(-r1, yi, t1);
    }
    for (; i >= 1; --i) {
        const double r0 = lane < i ? s_pack[i * (i + 1) / 2 + lane] * d0 : 0.0;
        t0 = fma(-r0, __shfl_sync(0xffffffffu, t0, i), t0);
    }
    if (lane < k) y[lane] = y2[lane] = t0;
    if (j1 < k) y[j1] = y2[j1] = t1;
}

// One warp, the column in g.h.  The arithmetic of loop_givens_warp, with what
// the recurrence along the column need not wait for done by all lanes at
// once (FP64 issues slowly): before it the products with the column's entries,
// after it the rotated column.
__device__ void loop_givens_staged(const LoopBufs &B, int k, double qpre2, int mode, const GivensStage &g) {
    GmresState &S = *B.S;
    const int lane = threadIdx.x & 31;
    const unsigned timed_out = lane == 0 ? B.counter[2] : 0u;   // needed at the end
    double *Rk = B.R + (size_t)(k - 1) * B.ldr;
    double rho = 0.0;
    int brk = 0;
    const double hk = g.h[k];
    double b[kGivLanes];
#pragma unroll
    for (int u = 0; u < kGivLanes; ++u) {
        const int i = lane + 32 * u;
        b[u] = i < k - 1 ? g.h[i + 1] : 0.0;
    }
    __syncwarp();
    // h[i + 1] = c_i b_i; then h[i + 1] = r_{i + 1} = c_i b_i - s_i r_i
#pragma unroll
    for (int u = 0; u < kGivLanes; ++u) {
        const int i = lane + 32 * u;
        if (i < k - 1) g.h[i + 1] = g.gc[i] * b[u];
    }
    __syncwarp();
    if (lane == 0) {
        double r = g.h[0];
        int i = 0;
        for (; i + 4 <= k - 1; i += 4) {
            double s4[4], p4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                s4[u] = g.gs[i + u];
                p4[u] = g.h[i + 1 + u];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                r = fma(-s4[u], r, p4[u]);
                g.h[i + 1 + u] = r;
            }
        }
        for (; i < k - 1; ++i) {
            r = fma(-g.gs[i], r, g.h[i + 1]);
            g.h[i + 1] = r;
        }
        double c, sn, rinv;
        givens_rotation(r, hk, c, sn, rinv);
        g.h[k] = rinv;
        const double g0 = g.gg[k - 1], g1 = -sn * g0, gk = c * g0;
        g.gg[k - 1] = gk;
        B.gc[k - 1] = c;
        B.gs[k - 1] = sn;
        B.gg[k] = g1;
        B.gg[k - 1] = gk;
        rho = fabs(g1);
        S.rho = rho;
        B.rhoh[k] = rho;
        brk = (!(hk == hk) || hk * hk <= 1e-12 * qpre2) ? 1 : 0;
    }
    rho = __shfl_sync(0xffffffffu, rho, 0);
    brk = __shfl_sync(0xffffffffu, brk, 0);
    __syncwarp();
#pragma unroll
    for (int u = 0; u < kGivLanes; ++u) {
        const int i = lane + 32 * u;
        if (i >= k) break;
        const double t = i < k - 1 ? fma(g.gc[i], g.h[i], g.gs[i] * b[u]) : g.h[k];   // rotated; 1 / R_kk
        Rk[i] = t;
        if (mode & kGivY) g.pack[k * (k - 1) / 2 + i] = t;
    }
    __syncwarp();
    if (mode & kGivY) solve_y_packed(g.pack, g.gg, k, B.y, B.yring + (size_t)(k % 3) * B.ldr);
    if ((mode & kGivZ) && lane == 0) {
        for (int i = 0; i <= k; ++i) B.z[i] = 0.0;
        B.z[k] = B.gg[k];
        for (int i = k - 1; i >= 0; --i) {
            const double a = B.z[i], b = B.z[i + 1];
            B.z[i] = B.gc[i] * a - B.gs[i] * b;
            B.z[i + 1] = B.gs[i] * a + B.gc[i] * b;
        }
    }
    if (lane != 0) return;
    if (!(g.S->variant == CTG_BA && g.S->rule == kRuleDP)) B.hist[k] = rho;
    const int pending = brk ? CTG_STOP_BREAKDOWN + 1 : (k == g.S->maxit ? CTG_STOP_MAXIT + 1 : 0);
    if (mode & kGivEnd) {
        int stop = pending;
        if (!brk && g.S->rule == kRuleDP && rho <= g.S->io.target) stop = CTG_STOP_DP + 1;
        end_step(B, stop, k, k, g.S->steps, timed_out);
    } else {
        S.pending = pending;
    }
}

// Shared memory loop_givens_warp needs beside the caller's own: the packed
// triangle for y_k (pack_cap (pack_cap + 1) / 2 doubles) and the staging
// (3 k + 1 doubles).
__host__ __device__ inline int loop_pack_cap(int maxit) { return maxit < 160 ? maxit : 160; }

}  // namespace

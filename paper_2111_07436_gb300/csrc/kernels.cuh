// Kernels of the batched solve and of its per-step test entry points,
// templated on the LU precision LT (float: mixed form, double: plain form),
// the lanes per cell G and the register slots per lane NPL; W selects the
// build with the water parameter's per-state work (mechanisms whose section
// constants carry powers of 1/L(y)), so that no other mechanism pays for it.
#pragma once
#include "cellsolve.cuh"
#include "launch.h"

namespace campdev {

template <int G>
__device__ __forceinline__ unsigned group_mask() {
    if constexpr (G >= 32) {
        return 0xffffffffu;
    } else {
        const int sub = (threadIdx.x & 31) / G;
        return ((1u << G) - 1u) << (sub * G);
    }
}

// The whole solve: each group of G lanes integrates one cell at a time.  With
// `queue` null the mapping is static (cell = block * cpb + group); otherwise
// the groups take cells from the counter until it passes n_cells.
// Register caps: the FP32-LU form with one-warp cells takes 168 a lane, the
// most that leaves three warps to each of an SM's four sub-partitions (12
// cells; 184 to 232 leave two, 8 cells: 62 -> 69 ms for 16384 gas-72 cells,
// though a lone cell is 15% faster without the spills); 64-thread cells with
// 4 slots take 168 in both forms (6 cells per SM; 200, five cells, 40.8 ->
// 42.7 ms for 4096 multiphase-232 cells); 128-thread cells take 168 in the
// FP64 form (3 cells per SM instead of 2: 7% faster despite spills; the
// FP32-LU form gains nothing); the FP64 form and the other block cells may
// take the architectural maximum.
//
// What bounds it: a cell is one dependent chain (about 4700 instructions a
// Newton iteration of a gas-72 cell, 115 of them FP64 at 64 cycles each), so
// a lone warp takes 25k cycles an iteration and 12 of them an SM 40k: of the
// issue slots 34% are used, and a warp waits on fixed latencies and the FP64
// port (24%), shared memory and shuffles (23%), instruction fetch (16%; the
// loop, the setup and the step code exceed the 32 KB of first-level
// instruction cache) and table loads (11%; 28 KB of L1 beside 12 cells).
template <int G, int NPL, typename LT, bool W>
__global__ void __maxnreg__(camp_solve_regs(G, NPL, (int)sizeof(LT)))
    k_solve(const __grid_constant__ DevMech m, const __grid_constant__ SolveArgs a) {
    const int group = threadIdx.x / G, lane = threadIdx.x % G;
    const unsigned gm = group_mask<G>();
    const CellPtr<LT> c(group * CellPtr<LT>::layout(m).bytes, m);
    long long cell = a.queue ? 0 : (long long)blockIdx.x * a.cpb + group;
    for (;;) {
        if (a.queue) {
            if constexpr (G <= 32) {
                unsigned long long v = 0;
                if (lane == 0) v = atomicAdd(a.queue, 1ull);
                cell = (long long)__shfl_sync(gm, v, 0, G);
            } else {  // one cell per block: broadcast through shared memory
                __shared__ unsigned long long next;
                if (threadIdx.x == 0) next = atomicAdd(a.queue, 1ull);
                __syncthreads();
                cell = (long long)next;
                __syncthreads();
            }
        }
        if (cell >= a.n_cells) break;
        CellStats st, tot{0, 0, 0, 0, 0};
        int s = ST_OK;
        // one or more consecutive outer steps of dt, each an independent call
        // of the integrator (a cold start unless step sizes are carried);
        // with a trajectory, the state after each one is also written there
        for (int o = 0; o < a.n_outer && s == ST_OK; o++) {
            s = integrate_cell<G, NPL, LT, W>(m, c, a.state + cell * m.n, a.env + cell * m.n_env, a.dt, a.rtol,
                                              a.atol, a.atol_len, a.max_steps, a.hmin_frac,
                                              a.step ? a.step + cell : nullptr, lane, gm, st,
                                              a.traj ? a.traj + ((long long)o * a.n_cells + cell) * m.n : nullptr);
            tot.steps += st.steps;
            tot.newton += st.newton;
            tot.jac += st.jac;
            tot.errfail += st.errfail;
            tot.ordsum += st.ordsum;
            if (o + 1 < a.n_outer) gsync<G>(gm);  // the state written back is the next step's input
        }
        if (lane == 0) {
            a.status[cell] = s;
            if (a.stats) {
                int32_t *o = a.stats + 5 * cell;
                o[0] = tot.steps;
                o[1] = tot.newton;
                o[2] = tot.jac;
                o[3] = tot.errfail;
                o[4] = tot.ordsum;
            }
        }
        if (!a.queue) break;
        gsync<G>(gm);
    }
}

// Rate constants of every process of every cell, [cell][R] in process order.
template <int G>
__global__ void k_rates(const __grid_constant__ DevMech m, long long n_cells, const double *env, double *kf, double *kr) {
    const long long cell = (long long)blockIdx.x * (blockDim.x / G) + threadIdx.x / G;
    const int lane = threadIdx.x % G;
    if (cell >= n_cells) return;
    for (int k = lane; k < m.R; k += G) {
        double a, b;
        rate_constant(m, k, env + cell * m.n_env, a, b);
        kf[cell * m.R + k] = a;
        kr[cell * m.R + k] = b;
    }
}

template <int G, int NPL, typename LT, bool W>
__device__ __forceinline__ void load_cell(const DevMech &m, const CellPtr<LT> &c, const double *y,
                                          const double *env, double (&yr)[NPL], int lane, unsigned gm) {
    for (int k = lane; k < m.R; k += G) {
        double a, b;
        rate_constant(m, k, env, a, b);
        c.kf[k] = a;
        const int rv = __ldg(m.rrev + k);
        if (rv >= 0) c.kr[rv] = b;
    }
#pragma unroll
    for (int s = 0; s < NPL; s++) {
        int p = lane + G * s;
        yr[s] = p < m.n ? y[__ldg(m.perm + p)] : 0.0;
        if (p < m.n) c.ys[p] = yr[s];
    }
    gsync<G>(gm);
    if constexpr (W) water_setup<G>(m, c.pw, env, lane, gm);
}

// f(y) of every cell, [cell][n] in declaration order.
template <int G, int NPL, typename LT, bool W>
__global__ void k_forcing(const __grid_constant__ DevMech m, long long n_cells, const double *state, const double *env,
                          double *f_out) {
    const int group = threadIdx.x / G, lane = threadIdx.x % G;
    const unsigned gm = group_mask<G>();
    const long long cell = (long long)blockIdx.x * (blockDim.x / G) + group;
    if (cell >= n_cells) return;
    const CellPtr<LT> c(group * CellPtr<LT>::layout(m).bytes, m);
    double y[NPL], f[NPL];
    load_cell<G, NPL, LT, W>(m, c, state + cell * m.n, env + cell * m.n_env, y, lane, gm);
    eval_f<G, NPL, LT, W>(m, c, y, f, lane, gm);
#pragma unroll
    for (int s = 0; s < NPL; s++) {
        int p = lane + G * s;
        if (p < m.n) f_out[cell * m.n + __ldg(m.perm + p)] = f[s];
    }
}

// The same with one cell per lane, 32 cells a warp: every lane evaluates the
// same process, so that an FP64 instruction -- 64 cycles a warp whatever its
// active lanes -- serves 32 cells, and the rate constants' exp, pow and log,
// which bound this kernel, run without divergence.  The rates of the warp's
// cells lie in shared memory ([process][cell]); the state and env rows are
// read in place (each lane its own row: the loads are few beside the FP64
// work).  The sums take their entries in the order, and in the two
// accumulators, of the cell kernels: the same f bit for bit.  (L is always 32;
// as a template the kernel may stand in a header of several units.)
template <int L>
__global__ void __launch_bounds__(L) k_forcing_lanes(const __grid_constant__ DevMech m, long long n_cells,
                                                      const double *state, const double *env, double *f_out) {
    double *rs = (double *)block_smem;
    const int lane = threadIdx.x;
    const long long cell = (long long)blockIdx.x * L + lane, at = cell < n_cells ? cell : n_cells - 1;
    const double *y = state + at * m.n, *e = env + at * m.n_env;
#pragma unroll 1
    for (int k = 0; k < m.R; k++) {
        double kf, kr;
        rate_constant(m, k, e, kf, kr);
        const int4 rp = __ldg(m.rpack + k);
        const int a0 = lo16(rp.x), a1 = hi16(rp.x), a2 = lo16(rp.y), rv = hi16(rp.y);
        auto at_pos = [&](int p) { return y[__ldg(m.perm + p)]; };
        double a = kf;
        if (a0 != NONE16) a *= at_pos(a0);
        if (a1 != NONE16) a *= at_pos(a1);
        if (a2 != NONE16) a *= at_pos(a2);
        if (rv != NONE16) {
            const int b0 = lo16(rp.z), b1 = hi16(rp.z), b2 = lo16(rp.w);
            double b = kr;
            if (b0 != NONE16) b *= at_pos(b0);
            if (b1 != NONE16) b *= at_pos(b1);
            if (b2 != NONE16) b *= at_pos(b2);
            a -= b;
        }
        rs[k * L + lane] = a;
    }
    __syncwarp();
    for (int p = 0; p < m.n; p++) {
        const int q1 = __ldg(m.fsum_ptr + p + 1);
        double acc = 0.0, acc2 = 0.0;
        int q = __ldg(m.fsum_ptr + p);
#pragma unroll 1
        for (; q + 1 < q1; q += 2) {
            acc = fma(__ldg(m.fsum_c + q), rs[__ldg(m.fsum_k + q) * L + lane], acc);
            acc2 = fma(__ldg(m.fsum_c + q + 1), rs[__ldg(m.fsum_k + q + 1) * L + lane], acc2);
        }
        if (q < q1) acc = fma(__ldg(m.fsum_c + q), rs[__ldg(m.fsum_k + q) * L + lane], acc);
        if (cell < n_cells) f_out[cell * m.n + __ldg(m.perm + p)] = acc + acc2;
    }
}

// Jacobian values of every cell, [cell][nnzJ] in species-CSR order, computed
// in precision LT (the assembly precision of the corresponding solve form).
template <int G, int NPL, typename LT, bool W>
__global__ void k_jacobian(const __grid_constant__ DevMech m, long long n_cells, const double *state, const double *env,
                           double *jac) {
    const int group = threadIdx.x / G, lane = threadIdx.x % G;
    const unsigned gm = group_mask<G>();
    const long long cell = (long long)blockIdx.x * (blockDim.x / G) + group;
    if (cell >= n_cells) return;
    const CellPtr<LT> c(group * CellPtr<LT>::layout(m).bytes, m);
    double y[NPL];
    load_cell<G, NPL, LT, W>(m, c, state + cell * m.n, env + cell * m.n_env, y, lane, gm);
    assemble<G, LT, W>(m, c, 0.0, lane, gm, 1, jac + cell * (long long)m.nnzJ);
}

// Solve (I - gamma J(y)) x = b for every cell with the device LU in
// precision LT; b and x [cell][n] in declaration order; status 4 on a
// tiny pivot (x then left unwritten).
template <int G, int NPL, typename LT, bool W>
__global__ void k_lu_solve(const __grid_constant__ DevMech m, long long n_cells, const double *state, const double *env,
                           double gamma, const double *b, double *x, int *status) {
    const int group = threadIdx.x / G, lane = threadIdx.x % G;
    const unsigned gm = group_mask<G>();
    const long long cell = (long long)blockIdx.x * (blockDim.x / G) + group;
    if (cell >= n_cells) return;
    const CellPtr<LT> c(group * CellPtr<LT>::layout(m).bytes, m);
    double y[NPL];
    load_cell<G, NPL, LT, W>(m, c, state + cell * m.n, env + cell * m.n_env, y, lane, gm);
    const bool ok = setup_matrix<G, NPL, LT, W>(m, c.base, gamma, lane, gm);
    if (lane == 0) status[cell] = ok ? 0 : ST_SINGULAR;
    if (!ok) return;
    for (int p = lane; p < m.n; p += G) c.x[p] = (LT)b[cell * m.n + __ldg(m.perm + p)];
    substitute<G, NPL, LT>(m, c, lane, gm);
    for (int p = lane; p < m.n; p += G) x[cell * m.n + __ldg(m.perm + p)] = (double)c.x[p];
}

}  // namespace campdev

// Per-cell device routines of the batched chemistry solve (sm_103a).
//
// One group of G lanes (G = 32: one warp) owns one grid cell.  Lane l holds
// the FP64 Nordsieck rows, error weights and corrections of positions
// p = l + G*s (s < NPL) in registers.  Shared memory per cell holds the
// current iterate y, the process rates, the rate constants, the LU values and
// the substitution vector.  Every decision of the step controller is taken on
// group-reduced (hence identical) values, so the lanes of a cell never
// diverge from each other; different cells never synchronise.
//
// Paper references (CAMP, arXiv 2111.07436): rate constants, Table 2;
// forcing f_i = sum_k (dy_i/dt)_k and Jacobian df_i/dy_j = sum_k (...)_k,
// Sect. 2.4.2; the implicit BDF + Newton + sparse LU solve, Sect. 2.4.1.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "devmech.h"

namespace campdev {

// ---- controller constants (identical meaning to the oracle's) ------------
constexpr int QMAX = CAMP_QMAX;
constexpr int NEWTON_MAXIT = 3;
constexpr double NEWTON_TOL = 0.1;
constexpr double RHO_DIV = 2.0;
constexpr double DGMAX = 0.3;
constexpr int MSBJ = 20;
constexpr double ETA_MAX = 10.0;
constexpr double ETA_THRESH = 1.5;
constexpr double ETA_CF = 0.25;
constexpr int MAX_NEF = 7;
constexpr int MAX_NCF = 10;

enum { ST_OK = 0, ST_MAXSTEPS = 1, ST_ERRTEST = 2, ST_NEWTON = 3, ST_SINGULAR = 4, ST_NONFINITE = 5 };

// ---- physical constants (SI 2019, exact) ----------------------------------
constexpr double KB = 1.380649e-23;
constexpr double NAV = 6.02214076e23;
constexpr double RG = KB * NAV;
constexpr double PI_D = 3.14159265358979323846;

// ---- one cell's shared memory (cell_smem) -----------------------------------
// The arrays of one cell in the block's dynamic shared memory, from the cell's
// byte offset in it.  The layout comes precomputed with the mechanism (in the
// constant bank), and every pointer is visibly one into shared memory, also
// in the functions kept out of line.
extern __shared__ __align__(16) char block_smem[];
template <typename LT>
struct CellPtr {
    double *ys, *rs, *kf, *kr, *pw, *fb;
    LT *x, *lu;
    int base;
    __device__ __forceinline__ CellPtr(int b, const DevMech &m) : base(b) {
        const CellSmem &c = layout(m);
        ys = (double *)(block_smem + b + c.ys);
        rs = (double *)(block_smem + b + c.rs);
        kf = (double *)(block_smem + b + c.kf);
        kr = (double *)(block_smem + b + c.kr);
        pw = (double *)(block_smem + b + c.pw);
        x = (LT *)(block_smem + b + c.x);
        lu = (LT *)(block_smem + b + c.lu);
        fb = (double *)(block_smem + b + c.fb);
    }
    static __device__ __forceinline__ const CellSmem &layout(const DevMech &m) {
        return sizeof(LT) == 4 ? m.smem4 : m.smem8;
    }
    // whether the odd halves of the forcing sums have their own array (fb)
    static __device__ __forceinline__ bool halves(const DevMech &m) { return layout(m).fb >= 0; }
};

// ---- group primitives --------------------------------------------------------
// A cell is integrated by a group of G lanes: G = 32 lanes of one warp, or a
// whole block of G > 32 threads (one cell per block, for mechanisms too large
// for one warp's registers).  Control flow is uniform across a group, so
// these are safe wherever the group takes them together.
template <int G>
__device__ __forceinline__ void gsync(unsigned gm) {
    if constexpr (G <= 32) __syncwarp(gm);
    else __syncthreads();
}
template <int G>
__device__ __forceinline__ bool gany(bool v, unsigned gm) {
    if constexpr (G <= 32) return __any_sync(gm, v) != 0;
    else return __syncthreads_or(v) != 0;
}
// Sum over the group, the same value in every lane (for a block: a fixed
// order over its warps' partial sums, so every thread gets identical bits)
template <int G, typename T>
__device__ __forceinline__ T gsum_t(T v, unsigned gm) {
    if constexpr (G <= 32) {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(gm, v, o, G);
        return __shfl_sync(gm, v, 0, G);
    } else {
        __shared__ double part[G / 32];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        __syncthreads();  // the previous sum's reads are done
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = (double)v;
        __syncthreads();
        double t = 0.0;
#pragma unroll
        for (int i = 0; i < G / 32; i++) t += part[i];
        return (T)t;
    }
}
template <int G>
__device__ __forceinline__ double gsum(double v, unsigned gm) {
    return gsum_t<G, double>(v, gm);
}

// ---- rate constants (Table 2), per process, from the cell's env ------------
__device__ __forceinline__ double ipowd(double x, int k) {
    double r = 1.0;
    for (int i = 0; i < k; i++) r *= x;
    return r;
}

// exp(c / T) and (T / d)^b.  With c = 0 or b = 0 (most mechanisms' case) they
// are exactly 1 for a positive T, without the ~20 and ~80 FP64 instructions,
// each a warp's for 64 cycles, of the functions.
__device__ __forceinline__ double exp_over(double c, double T) {
    return c == 0.0 && T > 0.0 ? 1.0 : exp(c / T);
}
__device__ __forceinline__ double pow_over(double T, double d, double b) {
    return b == 0.0 ? 1.0 : pow(T / d, b);
}
// A exp(C/T) (T/300)^B: the Arrhenius terms of the Troe and custom rate
// constants (D = 300 K, E = 0)
__device__ __forceinline__ double arr300(const double *par, double T) {
    return __ldg(par) * exp_over(__ldg(par + 2), T) * pow_over(T, 300.0, __ldg(par + 1));
}

// Condensation constant of one section, s^-1: N particles of radius rad,
// each 4 pi rad Dg f_fs(Kn, alpha) with the Fuchs-Sutugin factor and
// Kn = 3 Dg / (cbar rad), cbar = sqrt(8 R T / (pi MW))
__device__ __forceinline__ double condensation(double rad, double Np, double alpha, double Dg,
                                               double MW, double T) {
    double cbar = sqrt(8.0 * RG * T / (PI_D * MW));
    double Kn = 3.0 * Dg / cbar / rad;
    double ffs = 0.75 * alpha * (1.0 + Kn) / (Kn * Kn + Kn + 0.283 * Kn * alpha + 0.75 * alpha);
    return Np * 4.0 * PI_D * rad * Dg * ffs;
}

// Liquid volume of a section in the rate constants: the env value (the
// section's (r, N, L) triple in sec), or 1 when the water parameter makes it a
// function of the state (the constants are then per unit volume and the
// powers of 1/L are applied at each state)
__device__ __forceinline__ double section_volume(const DevMech &m, const double *__restrict__ sec) {
    return m.n_wsec > 0 ? 1.0 : sec[2];
}

// Rate constants of process k: env holds T, P and the runtime rates; sec the
// (radius, number concentration, liquid volume) of the section (or particle)
// a section process acts in (unused by the others)
static __device__ __noinline__ void rate_constant_at(const DevMech &m, int k, const double *__restrict__ env,
                                        const double *__restrict__ sec, double &kf, double &kr) {
    const double T = env[0], P = env[1];
    const double Mair = P / (KB * T) * 1e-6;  // molec cm^-3
    const double mppb = Mair * 1e-9;          // molec cm^-3 per ppb
    const double *par = m.rpar + CAMP_NPAR * k;
    const int nr = __ldg(m.rnr + k);
    kf = 0.0;
    kr = 0.0;
    switch (__ldg(m.rtype + k)) {
    case CAMP_P_ARRHENIUS: {
        // k = A exp(C/T) (T/D)^B (1 + E P)
        double kk = __ldg(par) * exp_over(__ldg(par + 2), T) * pow_over(T, __ldg(par + 3), __ldg(par + 1)) *
                    (1.0 + __ldg(par + 4) * P);
        kf = kk * ipowd(mppb, nr - 1);
        break;
    }
    case CAMP_P_TROE: {
        // k0[M] / (1 + k0[M]/kinf) * Fc^(1 / (1 + (log10(k0[M]/kinf)/N)^2))
        double k0 = arr300(par, T);
        double ki = arr300(par + 3, T);
        double x = k0 * Mair / ki;
        double lg = log10(x) / __ldg(par + 7);
        double kk = k0 * Mair / (1.0 + x) * pow(__ldg(par + 6), 1.0 / (1.0 + lg * lg));
        kf = kk * ipowd(mppb, nr - 1);
        break;
    }
    case CAMP_P_CUSTOM_H2O2:
        // k1 + k2 [M]
        kf = (arr300(par, T) + arr300(par + 3, T) * Mair) * ipowd(mppb, nr - 1);
        break;
    case CAMP_P_CUSTOM_OH_HNO3: {
        // k0 + k3[M] / (1 + k3[M] / k2)
        double k3M = arr300(par + 6, T) * Mair;
        kf = (arr300(par, T) + k3M / (1.0 + k3M / arr300(par + 3, T))) * ipowd(mppb, nr - 1);
        break;
    }
    case CAMP_P_PHOTOLYSIS:
    case CAMP_P_EMISSION:
    case CAMP_P_LOSS:
        kf = env[__ldg(m.rslot + k)];
        break;
    case CAMP_P_HENRY:
    case CAMP_P_SIMPOL: {
        // condensation k_c per section; evaporation k_c / (H_cc L) with
        // H_cc = 1000 H R T.  Henry: H(T) [M/Pa] from H298 and C.  SIMPOL:
        // H = c_tot / p0 with the SIMPOL.1 vapour pressure
        // log10 p0 [atm] = B1/T + B2 + B3 T + B4 ln T (Raoult's law in a
        // condensed phase of fixed total molarity c_tot)
        const double rad = sec[0];
        const double Np = sec[1];
        const double L = section_volume(m, sec);
        if (!(L > 0.0 && Np > 0.0 && rad > 0.0)) break;
        double H, kb;
        if (__ldg(m.rtype + k) == CAMP_P_HENRY) {
            H = __ldg(par) * exp(__ldg(par + 1) * (1.0 / T - 1.0 / 298.0));
            kb = condensation(rad, Np, __ldg(par + 2), __ldg(par + 3), __ldg(par + 4), T);
        } else {
            double lg = __ldg(par) / T + __ldg(par + 1) + __ldg(par + 2) * T + __ldg(par + 3) * log(T);
            H = __ldg(par + 7) / (101325.0 * exp10(lg));
            kb = condensation(rad, Np, __ldg(par + 4), __ldg(par + 5), __ldg(par + 6), T);
        }
        kf = kb;
        kr = kb / (1000.0 * H * RG * T * L);
        break;
    }
    case CAMP_P_AQREV: {
        // K_eq = A exp(C (1/T - 1/298)); rates in M/s, molarity = y * phi,
        // phi = 1e-9 P / (R T 1000 L) M per ppb
        const double L = section_volume(m, sec);
        if (!(L > 0.0)) break;
        double Keq = __ldg(par) * exp(__ldg(par + 1) * (1.0 / T - 1.0 / 298.0));
        double krev = __ldg(par + 2);
        double phi = 1e-9 * P / (RG * T * 1000.0 * L);
        kf = Keq * krev * ipowd(phi, nr - 1);
        kr = krev * ipowd(phi, __ldg(m.rnp + k) - 1);
        break;
    }
    case CAMP_P_COND_ARRHENIUS: {
        // Arrhenius in the section's condensed phase, M^(1-nr) s^-1:
        // kf = k phi^(nr - 1) in ppb units
        const double L = section_volume(m, sec);
        if (!(L > 0.0)) break;
        double kk = __ldg(par) * exp_over(__ldg(par + 2), T) * pow_over(T, __ldg(par + 3), __ldg(par + 1)) *
                    (1.0 + __ldg(par + 4) * P);
        double phi = 1e-9 * P / (RG * T * 1000.0 * L);
        kf = kk * ipowd(phi, nr - 1);
        break;
    }
    }
}

__device__ __forceinline__ bool section_type(int t) {
    return t == CAMP_P_HENRY || t == CAMP_P_SIMPOL || t == CAMP_P_AQREV || t == CAMP_P_COND_ARRHENIUS;
}

// Rate constants of process k of a compiled mechanism (section processes
// read their section's triple from env)
__device__ __forceinline__ void rate_constant(const DevMech &m, int k, const double *__restrict__ env,
                                              double &kf, double &kr) {
    const int t = __ldg(m.rtype + k);
    const double *sec = section_type(t) ? env + m.env_sec_base + 3 * __ldg(m.rslot + k) : env;
    rate_constant_at(m, k, env, sec, kf, kr);
}

// ---- FP64 without the FP64 pipe -----------------------------------------------
// Every FP64 instruction of a warp -- conversions between FP32 and FP64 and
// FP64 comparisons included -- holds its SM sub-partition's FP64 port for 64
// cycles, however many lanes are active and however independent it is of the
// others (measured: 64 cycles an instruction for one warp at any ILP, one per
// 16-19 cycles over a whole SM).  The integer pipe issues tens of instructions
// in that time, so the conversions and comparisons of the solve's inner loops
// run there, with the same results bit for bit.

// (float)x, rounded to nearest even.  In range (an FP32 normal result): the
// exponent is re-biased and the 29 dropped bits rounded in by an integer
// carry.  Zeros and values below half the smallest FP32 denormal are signed
// zeros; FP32 denormals, overflows, infinities and NaN take the conversion
// instruction.
__device__ __forceinline__ float narrow(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned ex = (hi >> 20) & 0x7ffu, sign = hi & 0x80000000u;
    unsigned u = __funnelshift_l(lo, hi, 3) + 0x40000000u;  // (ex - 896) << 23 | top 23 fraction bits
    u += ((lo & 0x1fffffffu) + 0x0fffffffu + (u & 1u)) >> 29;
    if (ex - 897u >= 254u) {
        if (ex < 873u) u = 0u;
        else return (float)x;
    }
    return __uint_as_float(u | sign);
}
// (double)x, exact: normal values and zeros by shifts, the rest by the
// conversion instruction
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), a = b & 0x7fffffffu, sign = b & 0x80000000u;
    if (a - 0x00800000u >= 0x7f000000u) {
        if (a == 0u) return __hiloint2double((int)sign, 0);
        return (double)x;
    }
    return __hiloint2double((int)(((a >> 3) + 0x38000000u) | sign), (int)(b << 29));
}
// a > b and a >= b for b >= +0 and any a (false for a NaN or negative a, as
// the FP64 comparisons are; a = -0 compares below +0 here, which no caller
// can pass)
constexpr long long INF_BITS = 0x7ff0000000000000ll;
__device__ __forceinline__ bool pos_gt(double a, double b) {
    const long long x = __double_as_longlong(a);
    return x > __double_as_longlong(b) && x <= INF_BITS;
}
__device__ __forceinline__ bool pos_ge(double a, double b) {
    const long long x = __double_as_longlong(a);
    return x >= __double_as_longlong(b) && x <= INF_BITS;
}

// FP64 values into and out of the LU precision
template <typename LT> __device__ __forceinline__ LT to_lu(double x);
template <> __device__ __forceinline__ float to_lu<float>(double x) { return narrow(x); }
template <> __device__ __forceinline__ double to_lu<double>(double x) { return x; }
__device__ __forceinline__ double from_lu(float x) { return widen(x); }
__device__ __forceinline__ double from_lu(double x) { return x; }

// One lane's term (x w)^2 of the Newton update's squared norm, in the LU
// precision.  In FP32 a weight beyond the format's range (atol below ~3e-39
// on a species near zero) is held at its largest value and the product at
// 1e18, so the sum stays finite; either only arises far from convergence.
// A non-finite x is caught separately.  norm_weight: the weight as the norm
// takes it, in the LU precision (once per step).
template <typename LT> __device__ __forceinline__ LT norm_weight(double w);
template <> __device__ __forceinline__ float norm_weight<float>(double w) { return fminf(narrow(w), 3.4e38f); }
template <> __device__ __forceinline__ double norm_weight<double>(double w) { return w; }
__device__ __forceinline__ float upd_term(float x, float w) {
    const float t = fminf(fabsf(x * w), 1e18f);
    return t * t;
}
__device__ __forceinline__ double upd_term(double x, double w) {
    const double t = x * w;
    return t * t;
}

// finite test on the exponent bits (integer pipe, not the FP64 pipe)
__device__ __forceinline__ bool finite_bits(double x) {
    return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;
}

// ---- forcing f(y): rates of all processes, then a per-position gather --------
// r_k = kf prod(forward factors) - kr prod(reverse factors), from the
// process's packed record (16-bit fields, 0xffff = none).
__device__ __forceinline__ int lo16(int v) { return v & 0xffff; }
__device__ __forceinline__ int hi16(int v) { return (int)((unsigned)v >> 16); }
constexpr int NONE16 = 0xffff;

// r_k of every process into rs, G at a time.  The operands of the next
// processes are fetched under the present ones' FP64 products, without
// branches around the loads: a missing factor reads position 0 and is not
// multiplied in, and only the rare third factors and reverse terms branch.
template <int G>
__device__ __forceinline__ void rate_terms(const DevMech &m, const double *ys, const double *kfs, const double *kr,
                                           double *rs, int lane) {
    const int R = m.R;
    if (R == 0) return;
    auto at = [&](int p) { return ys[p != NONE16 ? p : 0]; };
    int k = min(lane, R - 1);
    int4 rp = __ldg(m.rpack + k);
    int4 rn = __ldg(m.rpack + min(lane + G, R - 1));
    double a = kfs[k], y0 = at(lo16(rp.x)), y1 = at(hi16(rp.x));
#pragma unroll 1
    for (int b = 0; b < R; b += G) {
        const int kn = min(lane + b + G, R - 1);
        const int4 r2 = __ldg(m.rpack + min(lane + b + 2 * G, R - 1));
        const double an = kfs[kn], n0 = at(lo16(rn.x)), n1 = at(hi16(rn.x));
        if (lo16(rp.x) != NONE16) a *= y0;
        if (hi16(rp.x) != NONE16) a *= y1;
        if (rp.y != -1) {
            const int a2 = lo16(rp.y), rv = hi16(rp.y);
            const int b0 = lo16(rp.z), b1 = hi16(rp.z), b2 = lo16(rp.w);
            if (a2 != NONE16) a *= ys[a2];
            if (rv != NONE16) {
                double r = kr[rv];
                const double u0 = at(b0), u1 = at(b1);
                if (b0 != NONE16) r *= u0;
                if (b1 != NONE16) r *= u1;
                if (b2 != NONE16) r *= ys[b2];
                a -= r;
            }
        }
        if (lane + b < R) rs[lane + b] = a;
        rp = rn;
        rn = r2;
        a = an;
        y0 = n0;
        y1 = n1;
    }
}

// The gather of f from the rate terms: each lane runs through its flat list
// of entry pairs (DevMech::gth), with the records two steps and the operands
// one step ahead, so that a step costs its two FP64 products-and-sums alone.
// A finished sum's two halves go to shared memory (ys or the partials, and
// fb), where the owners add them: one FP64 add per position slot instead of
// one in every step in which some lane finishes a sum.
template <int G, bool FB>
__device__ __forceinline__ void gather_terms(const DevMech &m, const double *rs, double *ys, double *fp, double *fb,
                                             int lane) {
    const int n = m.n, S = m.n_gstep;
    const int2 *rec = m.gth + lane;
    const double2 *cf = m.gcf + lane;
    int2 r0 = __ldg(rec), r1 = __ldg(rec + G);
    double2 c0 = __ldg(cf);
    rec += 2 * G;
    cf += G;
    double v0 = rs[r0.x & 0x7fff], v1 = rs[hi16(r0.x) & 0x7fff];
    double acc = 0.0, acc2 = 0.0;
#pragma unroll 2
    for (int s = 0; s < S; s++, rec += G, cf += G) {
        const int2 r2 = __ldg(rec);  // two steps of padding follow the last
        const double2 c1 = __ldg(cf);
        const double w0 = rs[r1.x & 0x7fff], w1 = rs[hi16(r1.x) & 0x7fff];
        if (!(r0.x & 0x8000)) acc = fma(c0.x, v0, acc);
        if (r0.x >= 0) acc2 = fma(c0.y, v1, acc2);
        const bool end = r0.y >= 0;
        double *to = (G == 32 || r0.y < n) ? ys + r0.y : fp + (r0.y - n);
        if constexpr (FB) {
            if (end) *to = acc;
            if (end) fb[r0.y] = acc2;
        } else {
            if (end) *to = acc + acc2;
        }
        acc = end ? 0.0 : acc;
        acc2 = end ? 0.0 : acc2;
        r0 = r1;
        r1 = r2;
        c0 = c1;
        v0 = w0;
        v1 = w1;
    }
}

// ---- the water parameter (Sect. 2.2.2; Table 4, ZSRAerosolWater) ----------
// With the parameter, the constants of the section processes stay per unit
// volume in kf / kr, and the powers of 1/L(y) are applied where they are
// used (the rate terms, the Jacobian's constants, the chain rule), from each
// process's record: bits 16-26 of rpack.w hold its section + 1 (0: not a
// section process), bits 27-28 la and bits 29-30 lb.  Per-cell scratch c.pw:
// the electrolyte weights, L_env and 1/L of each section (1/L stored as 0
// for a section whose water is not positive: its processes take no part),
// then, in the FP64 form only, the Jacobian's reverse constants.
__device__ __forceinline__ double *pw_wt(const DevMech &, double *pw) { return pw; }
__device__ __forceinline__ double *pw_lenv(const DevMech &m, double *pw) { return pw + m.n_el; }
__device__ __forceinline__ double *pw_invl(const DevMech &m, double *pw) { return pw + m.n_el + m.n_wsec; }
__device__ __forceinline__ double *pw_kr64(const DevMech &m, double *pw) { return pw + m.n_pw; }

struct WaterTag {
    int sec, la, lb;  // sec = -1: not a section process
};
__device__ __forceinline__ WaterTag water_tag(int w) {
    const int h = hi16(w);
    return {(h & 0x7ff) - 1, (h >> 11) & 3, (h >> 13) & 3};
}
// factor of kf (p = la) or kr (p = lb) at the current volumes
__device__ __forceinline__ double water_scale(int sec, int p, const double *invl) {
    if (sec < 0) return 1.0;
    const double il = invl[sec];
    return il > 0.0 ? ipowd(il, p) : 0.0;
}

// Water per ppb of electrolyte e [m^3 per m^3 air]: 1e-9 P / (R T) mol m^-3
// per ppb over the molality m_e(a_w) of its binary solution (ZSR:
// W = sum_i 1000 M_i / (MW_i m_i(a_w)) kg m^-3), over the density of water.
// The molality fit is sqrt(m) = sum_j Y_j a_w^j with a_w = RH, held at the
// fit's lowest activity below it; a fit that gives no positive molality
// holds no water.
__device__ inline double zsr_weight(const DevMech &m, int e, const double *__restrict__ env) {
    const double T = env[0], P = env[1];
    double aw = env[m.rh_slot];
    const double lo = __ldg(m.zsr_low + e);
    if (aw < lo) aw = lo;
    double s = 0.0, p = 1.0;
    for (int j = 0; j < CAMP_ZSR_NY; j++) {
        s += __ldg(m.zsr_Y + CAMP_ZSR_NY * e + j) * p;
        p *= aw;
    }
    const double mol = s * s;
    if (!(mol > 0.0) || !finite_bits(mol)) return 0.0;
    return 1e-9 * P / (RG * T) / mol / 1000.0;
}

// Per cell, once: the electrolyte weights and the sections' env volumes.
template <int G>
__device__ __forceinline__ void water_setup(const DevMech &m, double *pw, const double *__restrict__ env,
                                            int lane, unsigned gm) {
    double *wt = pw_wt(m, pw), *lenv = pw_lenv(m, pw);
    for (int e = lane; e < m.n_el; e += G) wt[e] = zsr_weight(m, e, env);
    for (int b = lane; b < m.n_wsec; b += G) lenv[b] = env[m.env_sec_base + 3 * b + 2];
    gsync<G>(gm);
}

// The parameter at the state in ys: L_b = L_env,b + sum_e w_e y_e, kept as
// 1/L_b (0 for a section whose water is not positive).
template <int G>
__device__ __forceinline__ void water_update(const DevMech &m, double *pw, const double *ys, int lane,
                                             unsigned gm) {
    const double *wt = pw_wt(m, pw), *lenv = pw_lenv(m, pw);
    double *invl = pw_invl(m, pw);
    for (int b = lane; b < m.n_wsec; b += G) {
        double v = lenv[b];
        const int q1 = __ldg(m.pw_ptr + b + 1);
        for (int q = __ldg(m.pw_ptr + b); q < q1; q++) {
            const int w = __ldg(m.pw + q);
            v += wt[hi16(w)] * ys[lo16(w)];
        }
        invl[b] = v > 0.0 ? 1.0 / v : 0.0;
    }
    gsync<G>(gm);
}

// a x^p without the products by one that ipowd's loop starts from
__device__ __forceinline__ double times_pow(double a, double x, int p) {
    if (p > 0) {
        double r = x;
        for (int i = 1; i < p; i++) r *= x;
        a *= r;
    }
    return a;
}

// r_k with the powers of 1/L of a section process applied (the water build's
// rate term)
__device__ __forceinline__ double rate_term_water(const DevMech &m, int k, const int4 rp, const double *ys,
                                                  const double *kf, const double *kr, const double *invl) {
    const WaterTag t = water_tag(rp.w);
    double il = 1.0;
    if (t.sec >= 0) {
        il = invl[t.sec];
        if (!pos_gt(il, 0.0)) return 0.0;
    }
    const int a0 = lo16(rp.x), a1 = hi16(rp.x), a2 = lo16(rp.y), rv = hi16(rp.y);
    double a = times_pow(kf[k], il, t.la);
    if (a0 != NONE16) a *= ys[a0];
    if (a1 != NONE16) a *= ys[a1];
    if (a2 != NONE16) a *= ys[a2];
    if (rv != NONE16) {
        const int b0 = lo16(rp.z), b1 = hi16(rp.z), b2 = lo16(rp.w);
        double b = times_pow(kr[rv], il, t.lb);
        if (b0 != NONE16) b *= ys[b0];
        if (b1 != NONE16) b *= ys[b1];
        if (b2 != NONE16) b *= ys[b2];
        a -= b;
    }
    return a;
}

// The chain-rule term J_p P_y of Sect. 2.2.2 after the direct assembly: for
// each (row i, section b) pair g, g = d f_i / d L_b = sum_j nu_ij dr_j/dL_b
// with dr/dL = -(la F - lb B) / L (F, B the forward and reverse terms at the
// assembly's state y), then J_ie += g w_e for each electrolyte e of b.  The
// entries of one g are its n_el consecutive chain records; every record is a
// distinct (row, electrolyte) pair, so lanes need no atomics.
template <int G, typename LT>
__device__ __forceinline__ void water_chain(const DevMech &m, double *pw, const double *kf, const double *kr,
                                            const LT *y, LT *lu, double gamma, int lane, int mode,
                                            double *out) {
    const double *wt = pw_wt(m, pw), *invl = pw_invl(m, pw);
    for (int g = lane; g < m.n_g; g += G) {
        double acc = 0.0;
        const int q1 = __ldg(m.g_ptr + g + 1);
        for (int q = __ldg(m.g_ptr + g); q < q1; q++) {
            const int4 r = __ldg(m.pp + __ldg(m.g_ent + q));
            const double il = invl[r.y];
            if (!(il > 0.0)) continue;
            const int la = r.z & 0xff, lb = r.z >> 8;
            const int4 rp = __ldg(m.rpack + r.x);
            const int a0 = lo16(rp.x), a1 = hi16(rp.x), a2 = lo16(rp.y);
            double F = kf[r.x] * ipowd(il, la);
            if (a0 != NONE16) F *= (double)y[a0];
            if (a1 != NONE16) F *= (double)y[a1];
            if (a2 != NONE16) F *= (double)y[a2];
            double B = 0.0;
            if (r.w >= 0) {
                const int b0 = lo16(rp.z), b1 = hi16(rp.z), b2 = lo16(rp.w);
                B = kr[r.w] * ipowd(il, lb);
                if (b0 != NONE16) B *= (double)y[b0];
                if (b1 != NONE16) B *= (double)y[b1];
                if (b2 != NONE16) B *= (double)y[b2];
            }
            acc += __ldg(m.g_coef + q) * (-((double)la * F - (double)lb * B) * il);
        }
        for (int e = 0; e < m.n_el; e++) {
            const int4 ch = __ldg(m.ch + g * m.n_el + e);
            const double v = acc * wt[e];
            if (mode == 0)
                lu[ch.x] -= to_lu<LT>(gamma * v);
            else
                out[ch.w] += v;
        }
    }
}

// y in c.ys (written by the caller, who also made it visible to the group)
// -> f in shared memory, as two halves in ys and fb (or whole in ys).  The per-position sums are spread over the cell's
// lanes by the compiler's balanced assignment (long sums in chunks) and
// handed back through shared memory (reusing ys).  On return a lane may
// write its own positions of ys and, after a group sync, anything.
template <int G, typename LT, bool W>
__device__ __forceinline__ void eval_f_ys(const DevMech &m, const CellPtr<LT> &c, int lane, unsigned gm) {
    if constexpr (W) {
        water_update<G>(m, c.pw, c.ys, lane, gm);
        const double *invl = pw_invl(m, c.pw);
        int4 rp = __ldg(m.rpack + max(min(lane, m.R - 1), 0));
#pragma unroll 1
        for (int k = lane; k < m.R; k += G) {
            const int4 rn = __ldg(m.rpack + min(k + G, m.R - 1));
            c.rs[k] = rate_term_water(m, k, rp, c.ys, c.kf, c.kr, invl);
            rp = rn;
        }
    } else {
        rate_terms<G>(m, c.ys, c.kf, c.kr, c.rs, lane);
    }
    gsync<G>(gm);
    double *fs = c.ys;  // y is no longer needed
    double *fp = c.rs + m.R;
    const bool two = c.halves(m);
    if (two) gather_terms<G, true>(m, c.rs, fs, fp, c.fb, lane);
    else gather_terms<G, false>(m, c.rs, fs, fp, nullptr, lane);
    gsync<G>(gm);
    if (G > 32 && m.n_fsplit > 0) {  // split sums: their partials in a fixed order
        for (int i = lane; i < m.n_fsplit; i += G) {
            const int2 sp = __ldg(m.fsplit + i);
            const int first = lo16(sp.y), cnt = hi16(sp.y);
            double t = 0.0;
#pragma unroll 1
            for (int j = 0; j < cnt; j++) t += two ? fp[first + j] + c.fb[m.n + first + j] : fp[first + j];
            fs[sp.x] = t;
            if (two) c.fb[sp.x] = 0.0;
        }
        gsync<G>(gm);
    }
}
template <int G, int NPL, typename LT>
__device__ __forceinline__ void take_f(const DevMech &m, const CellPtr<LT> &c, double (&f)[NPL], int lane) {
#pragma unroll
    for (int s = 0; s < NPL; s++) {
        const int p = lane + G * s;
        f[s] = p < m.n ? c.ys[p] : 0.0;
    }
    if (c.halves(m)) {
#pragma unroll
        for (int s = 0; s < NPL; s++) {
            const int p = lane + G * s;
            if (p < m.n) f[s] += c.fb[p];
        }
    }
}
// the same, out of line: the evaluations outside the Newton loop (a call's
// first two, a restart's) share one copy of the code, so that the loop's own
// stays in the instruction cache
template <int G, typename LT, bool W>
__device__ __noinline__ void eval_f_call(const DevMech &m, int base, int lane, unsigned gm) {
    const CellPtr<LT> c(base, m);
    eval_f_ys<G, LT, W>(m, c, lane, gm);
}

// f at y = a + b u (own positions), out of line
template <int G, int NPL, typename LT, bool W>
__device__ __forceinline__ void eval_f_at(const DevMech &m, const CellPtr<LT> &c, const double (&a)[NPL],
                                          double b, const double (&u)[NPL], double (&f)[NPL], int lane,
                                          unsigned gm) {
#pragma unroll
    for (int s = 0; s < NPL; s++) {
        int p = lane + G * s;
        if (p < m.n) c.ys[p] = a[s] + b * u[s];
    }
    gsync<G>(gm);
    eval_f_call<G, LT, W>(m, c.base, lane, gm);
    take_f<G, NPL, LT>(m, c, f, lane);
}

// f at y (own positions), out of line
template <int G, int NPL, typename LT, bool W>
__device__ __forceinline__ void eval_f(const DevMech &m, const CellPtr<LT> &c, const double (&y)[NPL],
                                       double (&f)[NPL], int lane, unsigned gm) {
#pragma unroll
    for (int s = 0; s < NPL; s++) {
        int p = lane + G * s;
        if (p < m.n) c.ys[p] = y[s];
    }
    gsync<G>(gm);
    eval_f_call<G, LT, W>(m, c.base, lane, gm);
    take_f<G, NPL, LT>(m, c, f, lane);
}

// f at y = z + e (own positions), e zero in a step's first iteration
template <int G, int NPL, typename LT, bool W>
__device__ __forceinline__ void eval_f_newton(const DevMech &m, const CellPtr<LT> &c, const double (&z)[NPL],
                                              const double (&e)[NPL], bool first, double (&f)[NPL], int lane,
                                              unsigned gm) {
#pragma unroll
    for (int s = 0; s < NPL; s++) {
        int p = lane + G * s;
        double y = z[s];
        if (!first) y += e[s];
        if (p < m.n) c.ys[p] = y;
    }
    gsync<G>(gm);
    eval_f_ys<G, LT, W>(m, c, lane, gm);
    take_f<G, NPL, LT>(m, c, f, lane);
}

// ---- Jacobian gather: J (or M = I - gamma J) at ys into LU storage -----------
// mode 0: write M = I - gamma J into c.lu (zeroing fill and block entries)
// mode 1: write J values to out[nnzJ] (species-CSR order)
// In FP32 the rate constants and y are converted once into scratch that is
// free at this point (the rate array and the substitution vector), so the
// per-entry gather does no FP64/FP32 conversion.
template <int G, typename LT, bool W>
__device__ __forceinline__ void assemble(const DevMech &m, const CellPtr<LT> &c, double gamma,
                                         int lane, unsigned gm, int mode, double *out) {
    const LT *kfv, *krv, *yv;
    // the water build: 1/L at this state, and the constants with their
    // powers of 1/L applied (FP64 form: into the rate scratch and the
    // parameter block)
    auto water_constants = [&](LT *kfw, LT *krw) {
        const double *invl = pw_invl(m, c.pw);
        for (int k = lane; k < m.R; k += G) {
            const int4 rp = __ldg(m.rpack + k);
            const WaterTag t = water_tag(rp.w);
            kfw[k] = to_lu<LT>(c.kf[k] * water_scale(t.sec, t.la, invl));
            const int rv = hi16(rp.y);
            if (rv != NONE16) krw[rv] = to_lu<LT>(c.kr[rv] * water_scale(t.sec, t.lb, invl));
        }
    };
    if constexpr (W) water_update<G>(m, c.pw, c.ys, lane, gm);
    if constexpr (sizeof(LT) == 4) {
        LT *kf32 = (LT *)c.rs, *kr32 = kf32 + m.R, *y32 = (LT *)c.ys;
        if constexpr (W) {
            water_constants(kf32, kr32);
        } else {
#pragma unroll 1
            for (int k = lane; k < m.R; k += G) kf32[k] = to_lu<LT>(c.kf[k]);
#pragma unroll 1
            for (int k = lane; k < m.n_rev; k += G) kr32[k] = to_lu<LT>(c.kr[k]);
        }
        // y to FP32 in place, G positions at a time: a chunk's FP32 values
        // overwrite only FP64 values of this or earlier chunks, and the
        // group reads its chunk before any lane writes it
#pragma unroll 1
        for (int b0 = 0; b0 < m.n; b0 += G) {
            const int p = b0 + lane;
            const double v = p < m.n ? c.ys[p] : 0.0;
            gsync<G>(gm);
            if (p < m.n) y32[p] = to_lu<LT>(v);
        }
        kfv = kf32;
        krv = kr32;
        yv = y32;
    } else {
        if constexpr (W) {
            LT *kf64 = (LT *)c.rs, *kr64 = (LT *)pw_kr64(m, c.pw);
            water_constants(kf64, kr64);
            kfv = kf64;
            krv = kr64;
        } else {
            kfv = (const LT *)c.kf;
            krv = (const LT *)c.kr;
        }
        yv = (const LT *)c.ys;
    }
    if (mode == 0) {  // 16-byte stores: the LU array starts 16-byte aligned
        constexpr int V = 16 / sizeof(LT);
        float4 *z4 = (float4 *)c.lu;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        const int nv = m.nlu / V;
#pragma unroll 1
        for (int i = lane; i < nv; i += G) z4[i] = zero;
        for (int i = nv * V + lane; i < m.nlu; i += G) c.lu[i] = (LT)0;
    }
    gsync<G>(gm);
    // flat per-lane entry lists: coalesced records read one step ahead, one
    // store per non-zero
    const LT g = (LT)gamma;
    const int4 *rec = m.jls + lane;
    const double *cf = m.jlc + lane;
    LT acc = (LT)0;
    int4 r = __ldg(rec);
    const int steps = m.n_jstep[G > 32 ? lane >> 5 : 0];
#pragma unroll 1
    for (int i = 0; i < steps; i++) {
        rec += G;
        int4 rn = make_int4(0, (int)0xffff0000u, 1 << 18, 0xffff);  // a lane past its list reads no more
        if (!(r.z & (1 << 18))) rn = __ldg(rec);
        const int k = (int)(short)(r.y & 0xffff);
        const int o1 = hi16(r.y), o2 = lo16(r.w);
        LT v;
        if constexpr (sizeof(LT) == 4) v = __int_as_float(r.x);
        else v = r.z & (1 << 18) && !(r.z & (1 << 17)) ? (LT)0 : (LT)__ldg(cf);
        cf += G;
        const LT *kp = k >= 0 ? kfv + k : krv + (-k - 1);
        const LT kv = *kp, y1 = yv[o1 != NONE16 ? o1 : 0], y2 = yv[o2 != NONE16 ? o2 : 0];
        v *= kv;
        if (o1 != NONE16) v *= y1;
        if (o2 != NONE16) v *= y2;
        acc += v;
        const bool end = r.z & (1 << 17);
        if (mode == 0) {
            const LT M = ((r.z >> 16) & 1 ? (LT)1 : (LT)0) - g * acc;
            if (end) c.lu[r.z & 0xffff] = M;
        } else {
            if (end) out[hi16(r.w)] = (double)acc;
        }
        acc = end ? (LT)0 : acc;
        r = rn;
    }
    gsync<G>(gm);
    if constexpr (W) {
        water_chain<G, LT>(m, c.pw, c.kf, c.kr, yv, c.lu, gamma, lane, mode, out);
        gsync<G>(gm);
    }
}

template <typename LT> __device__ __forceinline__ LT tiny_pivot();
template <> __device__ __forceinline__ float tiny_pivot<float>() { return 1e-30f; }
template <> __device__ __forceinline__ double tiny_pivot<double>() { return 1e-300; }

// ---- LU factorisation in place; returns true if every pivot is usable -------
// Pivots are checked, then replaced by their reciprocals: the substitutions
// and later rows multiply instead of dividing.
// 1 / u, correctly rounded, without the general division's range handling
__device__ __forceinline__ float recip(float u) { return __frcp_rn(u); }
__device__ __forceinline__ double recip(double u) { return 1.0 / u; }

template <typename LT>
__device__ __forceinline__ bool bad_pivot(LT u) {
    return !(fabs(u) > tiny_pivot<LT>()) || !isfinite(u);
}

// f(integral_constant NS) for a dense block of D rows, NS = rows per lane of
// its warp (at most 4; a cell of at most MAXN positions has no more)
template <int V> struct IntC { static constexpr int value = V; };
template <int MAXN, class F>
__device__ __forceinline__ void dense_rows(int D, F f) {
    constexpr int TOP = MAXN >= 128 ? 4 : (MAXN + 31) / 32;
    const int ns = (D + 31) >> 5;
    if (ns == 0) return;
    if (TOP == 1 || ns == 1) f(IntC<1>());
    else if (TOP == 2 || ns == 2) f(IntC<(TOP >= 2 ? 2 : 1)>());
    else if (TOP == 3 || ns == 3) f(IntC<(TOP >= 3 ? 3 : 1)>());
    else f(IntC<(TOP >= 4 ? 4 : 1)>());
}

// 16-byte pieces of the dense block's rows (4 FP32 or 2 FP64 values)
template <typename LT> struct Vec16;
template <> struct Vec16<float> {
    static constexpr int N = 4;
    static __device__ __forceinline__ void ld(const float *p, float (&v)[4]) {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    }
    static __device__ __forceinline__ void st(float *p, const float (&v)[4]) {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
};
template <> struct Vec16<double> {
    static constexpr int N = 2;
    static __device__ __forceinline__ void ld(const double *p, double (&v)[2]) {
        const double2 t = *reinterpret_cast<const double2 *>(p);
        v[0] = t.x; v[1] = t.y;
    }
    static __device__ __forceinline__ void st(double *p, const double (&v)[2]) {
        *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
    }
};

// Dense trailing block, right-looking in panels of DENSE_W pivots, lane l
// owning rows l + 32 t.  For each panel: (1) its columns are factored in the
// owners' registers, the pivot row's entries broadcast by shuffles, so that a
// pivot's chain is a shuffle, a reciprocal and two operations; (2) the pivot
// rows right of the panel are forward-substituted with the panel's unit lower
// triangle (lane l takes columns l + 32 s); (3) one rank-DENSE_W update of
// the trailing rows, 16 bytes of a row at a time, the multipliers already in
// registers and the pivot rows broadcast.  The row stride is 4 mod 8 FP32 or
// 2 mod 4 FP64 values where that costs no resident cells (choose_strides), so
// that 16-byte accesses of the rows spread over all banks.  Every entry
// takes its updates one by one in pivot order, as a plain elimination does.
// Pivots are checked and replaced by their reciprocals.
constexpr int DENSE_W = 8;
template <int NS, typename LT>
__device__ __noinline__ bool dense_factor(LT *A, int D, int LD, int lane, unsigned gm) {
    using V = Vec16<LT>;
    constexpr int N = V::N, W = DENSE_W;
    bool bad = false;
#pragma unroll
    for (int kb = 0; kb < NS; kb++) {
        const int k1 = min(D, 32 * kb + 32);
#pragma unroll 1
        for (int kp = 32 * kb; kp < k1; kp += W) {
            const int o = kp - 32 * kb;  // the panel's first row among the owners
            // (1) panel columns kp .. kp+W-1 of the rows from 32 kb on
            LT a[NS][W];
#pragma unroll
            for (int t = kb; t < NS; t++) {
                const LT *row = A + min(lane + 32 * t, D - 1) * LD + kp;
#pragma unroll
                for (int v = 0; v < W; v += N) {
                    LT x[N] = {};
                    if (kp + v < LD) V::ld(row + v, x);
#pragma unroll
                    for (int i = 0; i < N; i++) a[t][v + i] = x[i];
                }
            }
#pragma unroll
            for (int c = 0; c < W; c++) {
                if (kp + c < D) {
                    LT p[W];
#pragma unroll
                    for (int j = c; j < W; j++) p[j] = __shfl_sync(gm, a[kb][j], o + c);
                    bad |= bad_pivot(p[c]);
                    const LT rp = recip(p[c]);
#pragma unroll
                    for (int t = kb; t < NS; t++) {
                        if (t > kb || lane > o + c) {
                            const LT l = a[t][c] * rp;
                            a[t][c] = l;
#pragma unroll
                            for (int j = c + 1; j < W; j++) a[t][j] -= l * p[j];
                        }
                    }
                    if (lane == o + c) a[kb][c] = rp;
                }
            }
#pragma unroll
            for (int t = kb; t < NS; t++) {
                if ((t > kb || lane >= o) && lane + 32 * t < D) {
                    LT *row = A + (lane + 32 * t) * LD + kp;
#pragma unroll
                    for (int v = 0; v < W; v += N) {
                        LT x[N];
#pragma unroll
                        for (int i = 0; i < N; i++) x[i] = a[t][v + i];
                        if (kp + v < LD) V::st(row + v, x);
                    }
                }
            }
            __syncwarp(gm);
            const int j0 = kp + W;
            if (j0 >= D) break;
            // (2) pivot rows of the panel, columns right of it
            LT tr[W][W];
#pragma unroll
            for (int r = 1; r < W; r++) {
#pragma unroll
                for (int v = 0; v < r; v += N) {
                    LT x[N];
                    V::ld(A + (kp + r) * LD + kp + v, x);
#pragma unroll
                    for (int i = 0; i < N; i++) tr[r][v + i] = x[i];
                }
            }
#pragma unroll 1
            for (int j = j0 + lane; j < D; j += 32) {
                LT u[W];
#pragma unroll
                for (int r = 0; r < W; r++) u[r] = A[(kp + r) * LD + j];
#pragma unroll
                for (int r = 1; r < W; r++) {
#pragma unroll
                    for (int p = 0; p < r; p++) u[r] -= tr[r][p] * u[p];
                }
#pragma unroll
                for (int r = 1; r < W; r++) A[(kp + r) * LD + j] = u[r];
            }
            __syncwarp(gm);
            // (3) trailing rows
#pragma unroll 1
            for (int j = j0; j < D; j += N) {
                LT u[W][N];
#pragma unroll
                for (int r = 0; r < W; r++) V::ld(A + (kp + r) * LD + j, u[r]);
#pragma unroll
                for (int t = kb; t < NS; t++) {
                    if (t > kb || o + W < 32) {
                        LT *row = A + min(lane + 32 * t, D - 1) * LD + j;
                        LT x[N];
                        V::ld(row, x);
#pragma unroll
                        for (int r = 0; r < W; r++) {
#pragma unroll
                            for (int i = 0; i < N; i++) x[i] -= a[t][r] * u[r][i];
                        }
                        if ((t > kb || lane >= o + W) && lane + 32 * t < D) V::st(row, x);
                    }
                }
            }
        }
    }
    return bad;
}

// one op of the row-wise factorisation: a division makes the multiplier l
// (lu[src] holds 1 / U(k,k)), an update subtracts l U(k,j) from its target
template <typename LT>
__device__ __forceinline__ void factor_op(uint32_t op, LT *lu, LT &l) {
    const int t = CAMP_OP_TGT(op), s = CAMP_OP_SRC(op);
    if (op & CAMP_OP_DIV) {
        l = lu[t] * lu[s];
        lu[t] = l;
    } else {
        lu[t] = fma(-l, lu[s], lu[t]);
    }
}

template <typename LT>
__device__ __forceinline__ bool take_reciprocal(const DevMech &m, LT *lu, int i) {
    const int di = __ldg(m.udiag + i);
    const LT u = lu[di];
    lu[di] = recip(u);
    return bad_pivot(u);
}

template <int G, int NPL, typename LT>
__device__ bool factor(const DevMech &m, const CellPtr<LT> &c, int lane, unsigned gm) {
    LT *lu = c.lu;
    LT *part = (LT *)(c.rs + m.R);  // chunk partials: the rate scratch is free here
    bool bad = false;
    // sparse rows (and the sparse-pivot updates of the block rows), by level:
    // each lane runs through its op list, the next op's word read ahead
#pragma unroll 1
    for (int L = 0; L < m.n_flev; L++) {
        const int b = __ldg(m.fst_ptr + L), e = __ldg(m.fst_ptr + L + 1);
        if constexpr (G > 32) {
            const int np = __ldg(m.fst_part + L);
            if (np > 0) {
                for (int k = lane; k < np; k += G) part[k] = (LT)0;
                gsync<G>(gm);
            }
        }
        const uint32_t *ops = m.fst + (size_t)b * G + lane;
        LT l = (LT)0;
        uint32_t op = __ldg(ops);
#pragma unroll 1
        for (int q = b; q < e; q++) {
            ops += G;
            const uint32_t next = __ldg(ops);  // one step of padding follows the last
            const int t = CAMP_OP_TGT(op), s = CAMP_OP_SRC(op);
            const bool div = (op & CAMP_OP_DIV) != 0, act = s != CAMP_OP_NOSRC, pivot = !act && !div;
            LT *to = (G > 32 && (t & 0x8000) && !div) ? part + (t & 0x7fff) : lu + t;
            const LT tv = *to, sv = lu[act ? s : 0];
            const LT upd = fma(-l, sv, tv), quot = tv * sv;
            l = div ? quot : l;
            if (act) *to = div ? quot : upd;
            if (pivot) {  // the row's pivot
                *to = recip(tv);
                bad |= bad_pivot(tv);
            }
            op = next;
        }
        gsync<G>(gm);
        if constexpr (G > 32) {  // rows cut into chunks: partials in order, then the tail
            const int rb = __ldg(m.lred_ptr + L), re = __ldg(m.lred_ptr + L + 1);
            for (int k = rb + lane; k < re; k += G) {
                const int4 rd = __ldg(m.lred + k);
                const int ns = lo16(rd.z), nch = hi16(rd.z);
                for (int s = 0; s < ns; s++) {
                    const int off = __ldg(m.lred_off + rd.y + s);
                    LT t = lu[off];
                    for (int ch = 0; ch < nch; ch++) t += part[rd.w + ch * ns + s];
                    lu[off] = t;
                }
                const int2 tl = __ldg(m.ltail + k);
                LT l = (LT)0;
                for (int q = tl.x; q < tl.x + tl.y; q++) factor_op(__ldg(m.lops + q), lu, l);
                if (hi16(rd.x) & 1) bad |= take_reciprocal(m, lu, lo16(rd.x));
            }
            if (re > rb) gsync<G>(gm);
        }
    }
    // the dense block is one warp's work (a block group's first warp)
    LT *A = lu + m.dbase;
    if (G <= 32 || lane < 32) {
        const unsigned wm = G <= 32 ? gm : 0xffffffffu;
        dense_rows<G * NPL>(m.D, [&](auto ns) { bad |= dense_factor<decltype(ns)::value, LT>(A, m.D, m.LD, lane, wm); });
    }
    return !gany<G>(bad, gm);
}

// ---- substitution: solves (LU) x = x in place (c.x holds the right side) -----
// Sparse rows go level by level through shared memory.  The dense block's
// right side lives in registers (lane l holds rows l + 32 t), and the loops
// run one 32-row diagonal block at a time so that only that block's rows
// need a comparison.  Rows past the block end read the last row (a valid
// address) and are discarded.
//
// FP32: four pivots a round.  Their not yet final values come by independent
// shuffles, every lane finishes them with the broadcast 4 x 4 diagonal block,
// then the four columns, 16 bytes of a row at a time, update the rows: a
// round's chain is one shuffle and about a dozen FP32 operations.  The rows of
// the diagonal block take the same operations in the same order in their
// owner lanes as in the broadcast triangle; the backward pass scales them by
// their reciprocal pivots at the end.  (Eight pivots a round have a shorter
// chain per pivot but half again as many instructions: slower at full
// occupancy.)
template <int NS, int KB>
__device__ __forceinline__ void forward_block(const float *A, int D, int LD, const float *const (&row)[NS],
                                              float (&xr)[NS], int lane, unsigned gm) {
    using V = Vec16<float>;
    const int k0 = 32 * KB, k1 = min(D, k0 + 32);
    const float *dg = A + k0 * (LD + 1);
    int k = k0;
#pragma unroll 1
    for (; k + 4 <= k1; k += 4, dg += 4 * (LD + 1)) {
        const int o = k - k0, in = lane - o;
        float a[NS][4], d1[4], d2[4], d3[4], x[4];
        V::ld(dg + LD, d1);
        V::ld(dg + 2 * LD, d2);
        V::ld(dg + 3 * LD, d3);
#pragma unroll
        for (int t = KB; t < NS; t++) V::ld(row[t] + k, a[t]);
#pragma unroll
        for (int p = 0; p < 4; p++) x[p] = __shfl_sync(gm, xr[KB], o + p);
        x[1] -= d1[0] * x[0];
        x[2] -= d2[0] * x[0];
        x[2] -= d2[1] * x[1];
        x[3] -= d3[0] * x[0];
        x[3] -= d3[1] * x[1];
        x[3] -= d3[2] * x[2];
#pragma unroll
        for (int p = 0; p < 4; p++) {
            if (in > p) xr[KB] -= a[KB][p] * x[p];
#pragma unroll
            for (int t = KB + 1; t < NS; t++) xr[t] -= a[t][p] * x[p];
        }
    }
#pragma unroll 1
    for (; k < k1; k++) {  // the block's last pivots, one at a time
        const int o = k - k0;
        const float xk = __shfl_sync(gm, xr[KB], o);
#pragma unroll
        for (int t = KB; t < NS; t++) {
            const float a = row[t][k];
            if (t > KB || lane > o) xr[t] -= a * xk;
        }
    }
    if constexpr (KB + 1 < NS) forward_block<NS, KB + 1>(A, D, LD, row, xr, lane, gm);
}
template <int NS, int KB>
__device__ __forceinline__ void backward_block(const float *A, int D, int LD, const float *const (&row)[NS],
                                               float (&xr)[NS], int lane, unsigned gm) {
    using V = Vec16<float>;
    const int k0 = 32 * KB, k1 = min(D, k0 + 32);
    int k = k1;  // one past the next pivot
#pragma unroll 1
    for (; k > k0 && (k & 3); k--) {  // the ragged end, one pivot at a time
        const int o = k - 1 - k0;
        const float xk = __shfl_sync(gm, xr[KB], o) * A[(k - 1) * LD + k - 1];
#pragma unroll
        for (int t = 0; t <= KB; t++) {
            const float a = row[t][k - 1];
            if (t < KB || lane < o) xr[t] -= a * xk;
        }
    }
    k -= 4;
    const float *dg = A + k * (LD + 1);
#pragma unroll 1
    for (; k >= k0; k -= 4, dg -= 4 * (LD + 1)) {  // k0 is a multiple of 4
        const int o = k - k0, in = lane - o;
        float a[NS][4], d[4][4], x[4];
#pragma unroll
        for (int p = 0; p < 4; p++) V::ld(dg + p * LD, d[p]);
#pragma unroll
        for (int t = 0; t <= KB; t++) V::ld(row[t] + k, a[t]);
#pragma unroll
        for (int p = 0; p < 4; p++) x[p] = __shfl_sync(gm, xr[KB], o + p);
#pragma unroll
        for (int p = 3; p >= 0; p--) {
#pragma unroll
            for (int q = 3; q > p; q--) x[p] -= d[p][q] * x[q];
            x[p] *= d[p][p];
        }
#pragma unroll
        for (int p = 3; p >= 0; p--) {
            if (in < p) xr[KB] -= a[KB][p] * x[p];
#pragma unroll
            for (int t = 0; t < KB; t++) xr[t] -= a[t][p] * x[p];
        }
    }
    xr[KB] *= row[KB][min(lane + k0, D - 1)];  // final up to the reciprocal pivots
    if constexpr (KB > 0) backward_block<NS, KB - 1>(A, D, LD, row, xr, lane, gm);
}
template <int NS>
__device__ __forceinline__ void dense_subst(const float *A, int D, int LD, float *xb, int lane, unsigned gm) {
    float xr[NS];
    const float *row[NS];
#pragma unroll
    for (int t = 0; t < NS; t++) {
        const int i = lane + 32 * t;
        row[t] = A + min(i, D - 1) * LD;
        xr[t] = i < D ? xb[i] : 0.0f;
    }
    forward_block<NS, 0>(A, D, LD, row, xr, lane, gm);
    backward_block<NS, NS - 1>(A, D, LD, row, xr, lane, gm);
#pragma unroll
    for (int t = 0; t < NS; t++) {
        const int i = lane + 32 * t;
        if (i < D) xb[i] = xr[t];
    }
}

// FP64: bound by the FP64 port, so one pivot at a time without redundant
// products; two columns of a row per load.
template <int NS>
__device__ __forceinline__ void dense_subst(const double *A, int D, int LD, double *xb, int lane, unsigned gm) {
    using V = Vec16<double>;
    double xr[NS];
    const double *row[NS];
#pragma unroll
    for (int t = 0; t < NS; t++) {
        const int i = lane + 32 * t;
        row[t] = A + min(i, D - 1) * LD;
        xr[t] = i < D ? xb[i] : 0.0;
    }
#pragma unroll
    for (int kb = 0; kb < NS; kb++) {
        const int k0 = 32 * kb, k1 = min(D, k0 + 32);
        int k = k0;
#pragma unroll 1
        for (; k < k1; k += 2) {
            const int o = k - k0;
            double a[NS][2];
#pragma unroll
            for (int t = kb; t < NS; t++) V::ld(row[t] + k, a[t]);
            const double x0 = __shfl_sync(gm, xr[kb], o);
#pragma unroll
            for (int t = kb; t < NS; t++)
                if (t > kb || lane > o) xr[t] -= a[t][0] * x0;
            if (k + 1 < k1) {
                const double x1 = __shfl_sync(gm, xr[kb], o + 1);
#pragma unroll
                for (int t = kb; t < NS; t++)
                    if (t > kb || lane > o + 1) xr[t] -= a[t][1] * x1;
            }
        }
    }
#pragma unroll
    for (int kb = NS - 1; kb >= 0; kb--) {
        const int k0 = 32 * kb, k1 = min(D, k0 + 32);
#pragma unroll 1
        for (int k = (k1 - 1) & ~1; k >= k0; k -= 2) {  // columns k + 1 and k
            const int o = k - k0;
            double a[NS][2];
#pragma unroll
            for (int t = 0; t <= kb; t++) V::ld(row[t] + k, a[t]);
            if (k + 1 < k1) {
                const double x1 = __shfl_sync(gm, xr[kb], o + 1) * A[(k + 1) * LD + k + 1];
#pragma unroll
                for (int t = 0; t <= kb; t++)
                    if (t < kb || lane < o + 1) xr[t] -= a[t][1] * x1;
            }
            const double x0 = __shfl_sync(gm, xr[kb], o) * A[k * LD + k];
#pragma unroll
            for (int t = 0; t <= kb; t++)
                if (t < kb || lane < o) xr[t] -= a[t][0] * x0;
        }
        const int i = lane + k0;
        xr[kb] *= row[kb][min(i, D - 1)];
    }
#pragma unroll
    for (int t = 0; t < NS; t++) {
        const int i = lane + 32 * t;
        if (i < D) xb[i] = xr[t];
    }
}

// The passes [p, pe) of a sparse substitution: in each, every lane takes one
// row (DevMech::sub_pass), its entries two a step; the first entry of a pair
// goes to the row's sum, the second to its odd accumulator.  The backward
// pass scales the row by its reciprocal pivot.  The next pass's record, with
// its first entries, and the next step's entries are read ahead, and operands
// are loaded without branches (a missing entry reads entry 0), so that a
// pass costs its chain of shared-memory loads alone.
template <int G, typename LT, bool BACK>
__device__ __forceinline__ void subst_passes(const DevMech &m, int p, int pe, const LT *lu, LT *x, LT *xp, int lane,
                                             unsigned gm) {
    if (p >= pe) return;
    const int4 *rec = m.sub_pass + (size_t)p * G + lane;
    int4 h = __ldg(rec);
    int L = 0;
#pragma unroll 1
    for (; p < pe; p++) {
        rec += G;
        const int4 hn = __ldg(rec);  // one pass of padding follows the last
        const int steps = h.w & 0xfff, i = lo16(h.x);
        const int2 *ent = m.sub + (size_t)((unsigned)h.w >> 14) * G + lane;
        int ea = h.y, eb = h.z;
        LT *to = x + (h.x >= 0 ? i : 0);
        LT s = *to, s2 = (LT)0;
        if constexpr (!BACK && G > 32) {
            if (h.x >= 0 && i >= m.n) {  // a chunk of a split row
                to = xp + (i - m.n);
                s = (LT)0;
            }
        }
        LT dg = (LT)1;
        if constexpr (BACK) dg = lu[h.x >= 0 ? hi16(h.x) : 0];
#pragma unroll 1
        for (int q = 0; q < steps; q++) {
            const int2 rn = __ldg(ent);  // one step of padding follows the last
            ent += G;
            const int e0 = max(ea, 0), e1 = max(eb, 0);
            const LT a0 = lu[lo16(e0)], b0 = x[hi16(e0)], a1 = lu[lo16(e1)], b1 = x[hi16(e1)];
            if (ea >= 0) s -= a0 * b0;
            if (eb >= 0) s2 += a1 * b1;
            ea = rn.x;
            eb = rn.y;
        }
        LT v = s - s2;
        if constexpr (BACK) v *= dg;
        if (h.x >= 0) *to = v;
        if (h.w & 0x1000) {  // the level's last pass
            gsync<G>(gm);
            if constexpr (!BACK && G > 32) {
                if (h.w & 0x2000) {  // split rows: their partials in order
                    const int sb = __ldg(m.ssplit_ptr + L), se = __ldg(m.ssplit_ptr + L + 1);
                    for (int k = sb + lane; k < se; k += G) {
                        const int2 sp = __ldg(m.ssplit + k);
                        const int first = lo16(sp.y), cnt = hi16(sp.y);
                        LT t = x[sp.x];
#pragma unroll 1
                        for (int j = 0; j < cnt; j++) t += xp[first + j];
                        x[sp.x] = t;
                    }
                    gsync<G>(gm);
                }
                L++;
            }
        }
        h = hn;
    }
}

template <int G, int NPL, typename LT>
__device__ void substitute(const DevMech &m, const CellPtr<LT> &c, int lane, unsigned gm) {
    LT *x = c.x;
    const LT *lu = c.lu;
    gsync<G>(gm);
    // forward, sparse rows and the L21 part of block rows (rows without L
    // entries keep their value); split rows through partials (LU precision,
    // after the rate terms: free while solving)
    LT *xp = (LT *)(c.rs + m.R);
    subst_passes<G, LT, false>(m, 0, m.n_fpass, lu, x, xp, lane, gm);
    const LT *A = lu + m.dbase;
    if (G <= 32 || lane < 32) {
        const unsigned wm = G <= 32 ? gm : 0xffffffffu;
        dense_rows<G * NPL>(m.D, [&](auto ns) { dense_subst<decltype(ns)::value>(A, m.D, m.LD, x + m.d, lane, wm); });
    }
    gsync<G>(gm);
    // backward, sparse rows by level
    subst_passes<G, LT, true>(m, m.n_fpass, m.n_fpass + m.n_bpass, lu, x, xp, lane, gm);
}

// J at the state in ys and the factorisation of I - gamma J, out of line;
// returns true if every pivot is usable
template <int G, int NPL, typename LT, bool W>
__device__ __noinline__ bool setup_matrix(const DevMech &m, int base, double gamma, int lane, unsigned gm) {
    const CellPtr<LT> c(base, m);
    assemble<G, LT, W>(m, c, gamma, lane, gm, 0, nullptr);
    return factor<G, NPL, LT>(m, c, lane, gm);
}

template <int G, int NPL>
__device__ __forceinline__ double wrms(const DevMech &m, const double (&v)[NPL], const double (&w)[NPL],
                                       unsigned gm) {
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < NPL; i++) {
        double a = v[i] * w[i];
        s += a * a;
    }
    return sqrt(gsum<G>(s, gm) / (double)m.n);
}

// ---- Nordsieck array operations (q uniform per cell; rows in registers) -----
template <int NPL>
__device__ __forceinline__ void nord_predict(double (&z)[QMAX + 1][NPL], int q) {
#pragma unroll
    for (int k = 0; k < QMAX; k++) {
        if (k < q) {
#pragma unroll
            for (int j = QMAX; j > k; j--) {
                if (j <= q) {
#pragma unroll
                    for (int s = 0; s < NPL; s++) z[j - 1][s] += z[j][s];
                }
            }
        }
    }
}
template <int NPL>
__device__ __forceinline__ void nord_retract(double (&z)[QMAX + 1][NPL], int q) {
#pragma unroll
    for (int k = QMAX - 1; k >= 0; k--) {
        if (k < q) {
#pragma unroll
            for (int j = 1; j <= QMAX; j++) {
                if (j > k && j <= q) {
#pragma unroll
                    for (int s = 0; s < NPL; s++) z[j - 1][s] -= z[j][s];
                }
            }
        }
    }
}
template <int NPL>
__device__ __forceinline__ void nord_rescale(double (&z)[QMAX + 1][NPL], int q, double eta) {
    double f = 1.0;
#pragma unroll
    for (int j = 1; j <= QMAX; j++) {
        if (j <= q) {
            f *= eta;
#pragma unroll
            for (int s = 0; s < NPL; s++) z[j][s] *= f;
        }
    }
}

// x^p for the step-size and order heuristics of the mixed form.  Only the
// accept/reject tests need FP64; a step-size factor needs a few digits, so
// this takes FP32 log2/exp2 (x = 0 gives 0 for p > 0 and +inf for p < 0).
__device__ __forceinline__ float ctl_powf(float x, float p) {
    return exp2f(p * __log2f(x));
}


// 1/d for d > 0 to ~1e-14 relative: an FP32 estimate refined by one
// Newton-Raphson step w <- w (2 - d w) in FP64; outside the FP32 normal
// range a division
__device__ __forceinline__ double recip_refined(double d) {
    if (pos_gt(d, 1e-37) && __double_as_longlong(d) < __double_as_longlong(1e37)) {
        const double w = widen(__frcp_rn(narrow(d)));
        return w * fma(-d, w, 2.0);
    }
    return 1.0 / d;
}

// The step controller's scalar arithmetic.  EXACT (the plain FP64 form)
// takes every scalar decision with the oracle's own FP64 operations --
// divisions, square roots and pow -- so that the two follow the same step
// sequence up to the roundoff of f, J and the LU; otherwise (the mixed form)
// the cheaper forms: reciprocals, squared norms and FP32 powers.  A norm v
// is carried as the norm itself (EXACT: v = c WRMS, from a root) or as its
// square (v = (c WRMS)^2, no root); either way the tests compare v with 1.
template <bool EXACT>
struct Ctl {
    // v from the sum s of n squared weighted terms and the coefficient c
    static __device__ __forceinline__ double norm(double c, double c2, double s, int n, double rn) {
        if constexpr (EXACT) return c * sqrt(s / (double)n);
        else return c2 * (s * rn);
    }
    // the step-size factor of order selection, 1 / ((k err)^(1/p) + 1e-6)
    // (the mixed form entirely in FP32: no FP64 division)
    static __device__ __forceinline__ double eta(double k, double v, int p) {
        if constexpr (EXACT) return 1.0 / (pow(k * v, 1.0 / (double)p) + 1e-6);
        else return (double)(1.0f / (ctl_powf((float)(k * k) * (float)v, 0.5f / (float)p) + 1e-6f));
    }
    // 0.9 err^(-1/p): the step factor after an error-test failure
    static __device__ __forceinline__ double fail_eta(double v, int p) {
        if constexpr (EXACT) return 0.9 * pow(v, -1.0 / (double)p);
        else return (double)(0.9f * ctl_powf((float)v, -0.5f / (float)p));
    }
    // a / b for the ratio of step-size coefficients (rb = 1 / b)
    static __device__ __forceinline__ double ratio(double a, double b, double rb) {
        if constexpr (EXACT) return a / b;
        else return a * rb;
    }
    // the error weight 1 / (rtol |y| + atol)
    static __device__ __forceinline__ double weight(double rtol, double y, double atol) {
        if constexpr (EXACT) return 1.0 / __dadd_rn(__dmul_rn(rtol, fabs(y)), atol);
        else return recip_refined(fma(rtol, fabs(y), atol));
    }
};

struct CellStats {
    int steps, newton, jac, errfail, ordsum;
};

// ---- one cell over [0, dt] ---------------------------------------------------
// y_cell/env_cell: this cell's rows (declaration order).  Returns the status;
// the state is written back only on success.  step_io (null: cold start):
// warm start, in: a value > 0 replaces the initial-step estimate; out: the
// step held before the final cut to dt, 0 on failure.  y_copy (or null)
// receives a second copy of the new state on success.
template <int G, int NPL, typename LT, bool W>
__device__ int integrate_cell(const DevMech &m, const CellPtr<LT> &c, double *__restrict__ y_cell,
                              const double *__restrict__ env_cell, double dt, double rtol,
                              const double *__restrict__ atol, int atol_len, int max_steps,
                              double hmin_frac, double *step_io, int lane, unsigned gm,
                              CellStats &st, double *__restrict__ y_copy = nullptr) {
    const int n = m.n;
    constexpr bool EXACT = sizeof(LT) == 8;  // the plain FP64 form
    // whether z1 / l1 is rounded before the Newton residual takes it or fused
    // into its sum.  Either form would do in every shape; the condition
    // reproduces what the compiler chose for each before it was written out, so
    // that results stay the same, now whatever a build contracts.  (A cell thus
    // takes one or the other with its shape, as it takes other orders of sums.)
    constexpr bool ROUND_Z1 = G == 32 && !W && (EXACT || NPL <= 3);
    using C = Ctl<EXACT>;
    const double h_in = step_io ? *step_io : 0.0;
    st.steps = st.newton = st.jac = st.errfail = st.ordsum = 0;

    // inputs must be finite
    bool bad = false;
    for (int i = lane; i < m.n_env; i += G) bad |= !finite_bits(env_cell[i]);
    double z[QMAX + 1][NPL], e[NPL], ep[NPL], w[NPL], f[NPL];
    LT wn[NPL];  // the weights as the Newton update's norm takes them
#pragma unroll
    for (int s = 0; s < NPL; s++) {
        int p = lane + G * s;
        double v = 0.0;
        if (p < n) v = y_cell[__ldg(m.perm + p)];
        bad |= !finite_bits(v);
#pragma unroll
        for (int j = 0; j <= QMAX; j++) z[j][s] = 0.0;
        z[0][s] = v;
        e[s] = ep[s] = 0.0;
    }
    // a cell that fails hands back no step (the next call starts cold)
    auto fail_early = [&](int code) {
        if (step_io && lane == 0) *step_io = 0.0;
        return code;
    };
    if (gany<G>(bad, gm)) return fail_early(ST_NONFINITE);

#pragma unroll 1
    for (int k = lane; k < m.R; k += G) {
        double a, b;
        rate_constant(m, k, env_cell, a, b);
        c.kf[k] = a;
        const int rv = __ldg(m.rrev + k);
        if (rv >= 0) c.kr[rv] = b;
    }
    gsync<G>(gm);
    if constexpr (W) water_setup<G>(m, c.pw, env_cell, lane, gm);

    // atol is re-read (an L1 hit) rather than held in registers
    auto set_weights = [&]() {
#pragma unroll
        for (int s = 0; s < NPL; s++) {
            int p = lane + G * s;
            double a = 1.0;
            if (p < n) a = atol_len == 1 ? __ldg(atol) : __ldg(atol + __ldg(m.perm + p));
            w[s] = (p < n) ? C::weight(rtol, z[0][s], a) : 0.0;
            wn[s] = norm_weight<LT>(w[s]);
        }
    };
    auto any_nonfinite = [&](const double(&v)[NPL]) {
        bool b2 = false;
#pragma unroll
        for (int s = 0; s < NPL; s++) b2 |= !finite_bits(v[s]);
        return gany<G>(b2, gm) != 0;
    };

    const double T = dt, hmin = hmin_frac * dt;
    set_weights();
    eval_f<G, NPL, LT, W>(m, c, z[0], f, lane, gm);
    if (any_nonfinite(f)) return fail_early(ST_NONFINITE);

    // initial step: the carried one, else Hairer, Norsett & Wanner's
    // starting-step estimate for order 1
    double h;
    if (h_in > 0.0) {
        h = fmin(h_in, T);
    } else {
        double d0 = wrms<G, NPL>(m, z[0], w, gm), d1 = wrms<G, NPL>(m, f, w, gm);
        double h0 = (d0 < 1e-5 || d1 < 1e-5) ? 1e-6 : 0.01 * d0 / d1;
        if (h0 > T) h0 = T;
        eval_f_at<G, NPL, LT, W>(m, c, z[0], h0, f, e, lane, gm);
#pragma unroll
        for (int s = 0; s < NPL; s++) ep[s] = e[s] - f[s];  // ep is free until the first step ends
        double d2 = wrms<G, NPL>(m, ep, w, gm) / h0;
        double dm = d1 > d2 ? d1 : d2;
        double h1 = (dm <= 1e-15) ? fmax(1e-6, h0 * 1e-3) : sqrt(0.01 / dm);
        h = fmin(100.0 * h0, h1);
        if (!(h <= T)) h = T;
    }
#pragma unroll
    for (int s = 0; s < NPL; s++) {
        z[1][s] = h * f[s];
        e[s] = 0.0;
    }

    int q = 1, qwait = 2, nst = 0, nst_lu = 0;
    double h_held = h;
    bool have_lu = false, need_setup = true, ep_valid = false;
    double t = 0.0, gamma_lu = 0.0;
    // gamma, its drift from the factored one beyond the limit and the
    // update's scaling are functions of (h, q, gamma_lu): kept, and formed
    // again only after one of them changed (`moved`)
    double gamma = 0.0, rl1 = 0.0;
    LT scale = (LT)1;
    bool moved = true, drifted = false;
    int status = ST_OK;
    // The mixed form takes the controller's tests on squared norms (the same
    // decisions as comparing the norms themselves, without roots): Newton
    // converged when dn^2 min(1, rho^2) <= tol^2, diverged when
    // rho^2 > RHO_DIV^2; the step is accepted when ecoef^2 mean((e w)^2) <= 1.
    // The FP64 form compares the norms themselves, as the oracle does
    // (err2 and dn2 then hold the norms, not their squares).
    constexpr double NEWTON_TOL2 = NEWTON_TOL * NEWTON_TOL;
    constexpr double RHO_DIV2 = RHO_DIV * RHO_DIV;

    while (pos_gt(T, t)) {
        if (nst >= max_steps) { status = ST_MAXSTEPS; break; }
        set_weights();
        int nef = 0, ncf = 0;
        bool last = false;
        double err2 = 0.0, t_new = 0.0;
        bool accepted = false;
        while (!accepted) {
            last = false;
            h_held = h;
            t_new = t + h;
            if (pos_ge(t_new, T)) {
                if (pos_gt(t_new, T)) {
                    double eta = (T - t) / h;
                    nord_rescale<NPL>(z, q, eta);
                    h = T - t;
                    moved = true;
                }
                last = true;
                t_new = T;
            }
            nord_predict<NPL>(z, q);
            if (moved) {
                rl1 = m.inv_l1[q];
                gamma = C::ratio(h, m.lcoef[q][1], rl1);
                drifted = false;
                scale = (LT)1;
                if (have_lu && __double_as_longlong(gamma) != __double_as_longlong(gamma_lu)) {
                    const double gr = C::ratio(gamma, gamma_lu, 1.0 / gamma_lu);
                    drifted = fabs(gr - 1.0) > DGMAX;
                    scale = (LT)2 / ((LT)1 + to_lu<LT>(gr));
                }
                moved = false;
            }
            bool jcur = false, lu_fail = false;
            if (!have_lu || need_setup || nst >= nst_lu + MSBJ || drifted) {
#pragma unroll
                for (int s = 0; s < NPL; s++) {
                    int p = lane + G * s;
                    if (p < n) c.ys[p] = z[0][s];
                }
                gsync<G>(gm);
                lu_fail = !setup_matrix<G, NPL, LT, W>(m, c.base, gamma, lane, gm);
                st.jac++;
                gamma_lu = gamma;
                drifted = false;
                scale = (LT)1;
                nst_lu = nst;
                have_lu = !lu_fail;
                need_setup = false;
                jcur = true;
            }
            // modified Newton on G(e) = e - gamma f(z0 + e) + z1 / l1
            bool conv = false;
            if (!lu_fail) {
                LT dprev2 = (LT)0;
#pragma unroll
                for (int s = 0; s < NPL; s++) e[s] = 0.0;
#pragma unroll 1
                for (int it = 0; it < NEWTON_MAXIT; it++) {  // one copy of the loop's code (instruction cache)
                    eval_f_newton<G, NPL, LT, W>(m, c, z[0], e, it == 0, f, lane, gm);
                    st.newton++;
                    if (any_nonfinite(f)) break;
#pragma unroll
                    for (int s = 0; s < NPL; s++) {
                        int p = lane + G * s;
                        const double r0 = fma(-gamma, f[s], e[s]);
                        const double r = ROUND_Z1 ? __dadd_rn(r0, __dmul_rn(z[1][s], rl1)) : fma(z[1][s], rl1, r0);
                        if (p < n) c.x[p] = to_lu<LT>(-r);
                    }
                    substitute<G, NPL, LT>(m, c, lane, gm);
                    // the update's norm in the LU precision (it only steers the iteration)
                    LT dsq = (LT)0;
                    bool nf = false;
#pragma unroll
                    for (int s = 0; s < NPL; s++) {
                        int p = lane + G * s;
                        LT xl = (p < n) ? c.x[p] : (LT)0;
                        xl *= scale;
                        if (it == 0) e[s] = from_lu(xl);  // e was zero
                        else e[s] += from_lu(xl);
                        dsq += upd_term(xl, wn[s]);
                        nf |= !isfinite(xl);
                    }
                    // EXACT: the norm itself, as the oracle tests it; mixed:
                    // its square in the LU precision
                    const LT dn2 = EXACT ? (LT)sqrt((double)gsum_t<G, LT>(dsq, gm) / (double)n)
                                         : gsum_t<G, LT>(dsq, gm) * (LT)m.rn;
                    if (gany<G>(nf, gm) || !isfinite(dn2)) break;
                    LT test2 = dn2;
                    if (it > 0) {
                        const LT rho2 = dn2 / dprev2;
                        if (rho2 > (LT)(EXACT ? RHO_DIV : RHO_DIV2)) break;
                        if (rho2 < (LT)1) test2 = dn2 * rho2;
                    }
                    if (test2 <= (LT)(EXACT ? NEWTON_TOL : NEWTON_TOL2)) { conv = true; break; }
                    dprev2 = dn2;
                }
            }
            if (!conv) {
                nord_retract<NPL>(z, q);
                if (!jcur) { need_setup = true; continue; }
                if (++ncf >= MAX_NCF) { status = lu_fail ? ST_SINGULAR : ST_NEWTON; break; }
                h *= ETA_CF;
                moved = true;
                if (h < hmin) { status = ST_ERRTEST; break; }
                nord_rescale<NPL>(z, q, ETA_CF);
                need_setup = true;
                qwait = q + 1;
                continue;
            }
            {
                double es = 0.0;
#pragma unroll
                for (int s = 0; s < NPL; s++) { double a = e[s] * w[s]; es += a * a; }
                err2 = C::norm(m.ecoef[q], m.ecoef2[q], gsum<G>(es, gm), n, m.rn);
            }
            if (pos_gt(err2, 1.0)) {
                nord_retract<NPL>(z, q);
                st.errfail++;
                moved = true;
                if (++nef >= MAX_NEF) { status = ST_ERRTEST; break; }
                if (nef >= 3) {
                    h *= 0.1;
                    if (h < hmin) { status = ST_ERRTEST; break; }
                    q = 1;
                    eval_f<G, NPL, LT, W>(m, c, z[0], f, lane, gm);
#pragma unroll
                    for (int s = 0; s < NPL; s++) z[1][s] = h * f[s];
                } else {
                    double eta = C::fail_eta(err2, q + 1);
                    if (eta < 0.2) eta = 0.2;
                    h *= eta;
                    if (h < hmin) { status = ST_ERRTEST; break; }
                    nord_rescale<NPL>(z, q, eta);
                }
                qwait = q + 1;
                continue;
            }
            accepted = true;
        }
        if (status != ST_OK) break;

        // accept: z += l (x) e
#pragma unroll
        for (int j = 0; j <= QMAX; j++) {
            if (j <= q) {
                const double lj = m.lcoef[q][j];
#pragma unroll
                for (int s = 0; s < NPL; s++) z[j][s] += lj * e[s];
            }
        }
        t = t_new;
        nst++;
        st.ordsum += q;
        if (any_nonfinite(z[0])) { status = ST_NONFINITE; break; }

        if (--qwait <= 0 && !last) {
            // eta = 1 / ((c err)^(1/(p+1)) + 1e-6), from the squared norms
            double eta_q = C::eta(1.2, err2, q + 1);
            double eta_m = 0.0, eta_p = 0.0;
            if (q > 1) {
                double zs = 0.0;
#pragma unroll
                for (int j = 1; j <= QMAX; j++) {
                    if (j == q) {
#pragma unroll
                        for (int s = 0; s < NPL; s++) { double a = z[j][s] * w[s]; zs += a * a; }
                    }
                }
                const double ce = m.ecoef[q - 1] * m.fact[q];
                const double em2 = C::norm(ce, ce * ce, gsum<G>(zs, gm), n, m.rn);
                eta_m = C::eta(1.3, em2, q);
            }
            if (q < QMAX && ep_valid) {
                double ds = 0.0;
#pragma unroll
                for (int s = 0; s < NPL; s++) { double a = (e[s] - ep[s]) * w[s]; ds += a * a; }
                const double ep2 = C::norm(m.ecoef[q + 1], m.ecoef2[q + 1], gsum<G>(ds, gm), n, m.rn);
                eta_p = C::eta(1.4, ep2, q + 2);
            }
            double eta = eta_q;
            int qn = q;
            if (eta_m > eta) { eta = eta_m; qn = q - 1; }
            if (eta_p > eta) { eta = eta_p; qn = q + 1; }
            if (eta < ETA_THRESH) {
                qwait = 2;
            } else {
                if (eta > ETA_MAX) eta = ETA_MAX;
                if (qn == q + 1) {
                    const double c_up = m.lcoef[q][q] / (double)(q + 1);
#pragma unroll
                    for (int j = 2; j <= QMAX; j++) {
                        if (j == q + 1) {
#pragma unroll
                            for (int s = 0; s < NPL; s++) z[j][s] = e[s] * c_up;
                        }
                    }
                }
                q = qn;
                h *= eta;
                moved = true;
                nord_rescale<NPL>(z, q, eta);
                qwait = q + 1;
            }
        }
#pragma unroll
        for (int s = 0; s < NPL; s++) ep[s] = e[s];
        ep_valid = true;
    }
    st.steps = nst;
    if (status == ST_OK) {
#pragma unroll
        for (int s = 0; s < NPL; s++) {
            int p = lane + G * s;
            if (p < n) {
                const int i = __ldg(m.perm + p);
                y_cell[i] = z[0][s];
                if (y_copy) y_copy[i] = z[0][s];
            }
        }
    }
    if (step_io && lane == 0) *step_io = status == ST_OK ? h_held : 0.0;
    return status;
}

}  // namespace campdev

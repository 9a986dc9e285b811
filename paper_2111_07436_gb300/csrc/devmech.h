// Device-side mechanism tables, shared by the host compiler (mech.cpp) and the
// CUDA kernels.  Every array lives in one device allocation; the struct is
// passed to kernels by value (it sits in the kernel-parameter constant bank).
//
// All species indices here are POSITIONS in the elimination order chosen by
// the compiler (position p holds species perm[p]); only the state/env/atol
// loads and stores translate back to declaration order.
#pragma once
#include <stddef.h>
#include <stdint.h>
#include <vector_types.h>

#define CAMP_QMAX 5
#define CAMP_MAXFAC 3  // at most 3 factors (with multiplicity) per rate term

enum {
    CAMP_P_ARRHENIUS = 0,
    CAMP_P_TROE = 1,
    CAMP_P_PHOTOLYSIS = 2,
    CAMP_P_EMISSION = 3,
    CAMP_P_LOSS = 4,
    CAMP_P_HENRY = 5,
    CAMP_P_AQREV = 6,
    CAMP_P_CUSTOM_H2O2 = 7,
    CAMP_P_CUSTOM_OH_HNO3 = 8,
    CAMP_P_COND_ARRHENIUS = 9,
    CAMP_P_SIMPOL = 10
};

#define CAMP_NPAR 10  // rate parameters per process
#define CAMP_ZSR_NY 8 // coefficients of one electrolyte's molality fit

// Lanes that integrate one cell of an n-species mechanism: one warp up to
// 192 species (up to 6 a lane), else one block of 64 threads (4 species a
// lane up to 256 species, 8 beyond), 128 or 256 threads (8 a lane).  For
// 193-256 species two warps with 4 slots each measured 1.3x one warp with 8
// (fewer registers a lane, more warps a SM).  The per-lane tables below are
// built for this many lanes.
inline int camp_cell_lanes(int n) {
    if (n <= 192) return 32;
    if (n <= 512) return 64;
    if (n <= 1024) return 128;
    return 256;
}

// The other lane count the launch autotuner tries for an n-species
// mechanism (0: none): 129-256 species run on one warp (6 or 8 slots a
// lane) or on 64 threads (4 slots a lane), whichever measures faster.
inline int camp_alt_lanes(int n) {
    if (n > 128 && n <= 192) return 64;
    if (n > 192 && n <= 256) return 32;
    return 0;
}

// LU op encoding for the sparse (row-wise) part of the factorisation
#define CAMP_OP_DIV 0x80000000u
#define CAMP_OP_TGT(op) ((int)((op)&0xFFFFu))
#define CAMP_OP_SRC(op) ((int)(((op) >> 16) & 0x7FFFu))
#define CAMP_OP_NOSRC 0x7FFF  // no source: with DIV no op, without it a pivot's reciprocal

// Dynamic shared memory one block may use (227 KB less room for a block
// group's static reduction scratch).
constexpr int CAMP_MAX_SMEM = 227 * 1024 - 256;

// Register slots a lane of an n-species cell (the water builds hold one
// one-warp shape)
inline int camp_cell_slots(int n, int lanes, bool water) {
    if (lanes == 32 && !water) {
        const int need = (n + 31) / 32;
        return need <= 4 ? need : need <= 6 ? 6 : 8;
    }
    return lanes == 64 && n <= 256 ? 4 : 8;
}

// Registers a lane of the solve kernel (kernels.cuh has the reasons)
constexpr int camp_solve_regs(int lanes, int slots, int lu_elem) {
    return (lanes == 64 && slots == 4) || (lanes == 128 && lu_elem == 8) ? 168
           : lu_elem == 8 || lanes > 32                                  ? 255
                                                                         : (slots >= 6 ? 224 : 168);
}

// Cells of `bytes` of shared memory that an SM holds, at the best cells per
// block: 228 KB less 1 KB a block (and a block group's reduction scratch), and
// whole warps to each of four register files of 16384, 256 at a time.
inline int camp_resident_cells(int bytes, int n, int lanes, bool water, int lu_elem) {
    const int regs = (camp_solve_regs(lanes, camp_cell_slots(n, lanes, water), lu_elem) * 32 + 255) & ~255;
    const int warps = 4 * (16384 / regs), fixed = 1024 + (lanes > 32 ? 256 : 0);
    int best = 0;
    for (int c = 1; c <= (lanes == 32 ? 4 : 1) && c * bytes <= CAMP_MAX_SMEM; c++) {
        const int by_smem = 228 * 1024 / (c * bytes + fixed), by_regs = warps / (c * lanes / 32);
        const int cells = c * (by_smem < by_regs ? by_smem : by_regs);
        if (cells > best) best = cells;
    }
    return best;
}

// Shared-memory layout of one cell (byte offsets).  rs holds the R rate
// terms, then n_part partial sums (of split forcing sums inside an f
// evaluation, of split substitution and factorisation rows inside a solve);
// pw the water parameter's per-cell values (n_pw doubles, and n_pw64 more in
// the FP64 form; none without one); fb the odd halves of the
// forcing sums (n + n_fpart doubles), which saves FP64 adds where a lane owns
// few positions: one-warp cells and block cells of up to 4 positions a lane.
// Other cells, and a mechanism of which an SM holds more cells without it, have
// none (fb = -1) and add the two halves of a sum where the sum ends (117
// species, FP64: 2 cells an SM with it, 189 ms for 2048 cells; 3 without,
// 143 ms).
struct CellSmem {
    int ys, rs, kf, kr, pw, x, lu, fb, bytes;
};
inline int camp_align16(int b) { return (b + 15) & ~15; }
inline CellSmem cell_smem(int n, int R, int n_rev, int nlu, int lu_elem, int n_part, int n_fpart, int n_pw, int n_pw64,
                          int lanes) {
    CellSmem c;
    int o = 0;
    c.ys = o; o = camp_align16(o + 8 * n);
    c.rs = o; o = camp_align16(o + 8 * (R + n_part));
    c.kf = o; o = camp_align16(o + 8 * R);
    c.kr = o; o = camp_align16(o + 8 * n_rev);
    c.pw = o; o = camp_align16(o + 8 * (n_pw + (lu_elem == 8 ? n_pw64 : 0)));
    // the substitution vector shares the rate-term scratch when it fits:
    // the rate terms live only inside one f evaluation, the vector only
    // inside one Newton solve, and the Jacobian assembly keeps its FP32
    // copy of y in ys instead
    if (8 * R >= lu_elem * n) {
        c.x = c.rs;
    } else {
        c.x = o;
        o = camp_align16(o + lu_elem * n);
    }
    c.lu = o; o = camp_align16(o + lu_elem * nlu);
    const int with = camp_align16(o + 8 * (n + n_fpart));
    const bool few = n <= (lanes == 32 ? 8 : 4) * lanes;
    auto cells = [&](int bytes) { return camp_resident_cells(bytes, n, lanes, n_pw > 0, lu_elem); };
    c.fb = few && with <= CAMP_MAX_SMEM && cells(with) >= cells(o) ? o : -1;
    c.bytes = c.fb >= 0 ? with : o;
    return c;
}

struct DevMech {
    CellSmem smem4, smem8;  // shared memory of one cell, FP32 and FP64 LU
    int n;            // species
    int R;            // process instances
    int n_env;
    int env_sec_base; // env index of section 0's radius
    int lanes;        // lanes per cell the per-lane tables were built for

    // --- rate constants (process order) ---
    const int *rtype;     // [R]
    const double *rpar;   // [R][CAMP_NPAR]
    const int *rslot;     // [R] env slot (runtime types) or section (section types)
    const int *rnr;       // [R] total reactant multiplicity
    const int *rnp;       // [R] total product multiplicity (reversible types)
    int n_rev;            // reversible processes (the only ones with a kr)
    const int *rrev;      // [R] index into the cell's kr array, -1 if irreversible

    // --- rate terms r_k = kf prod(fwd) - kr prod(rev), one 16-byte record each:
    // x = fwd0 | fwd1 << 16, y = fwd2 | rv << 16, z = rev0 | rev1 << 16,
    // w = rev2 (positions; 16-bit fields, 0xffff = none; rv = kr index)
    const int4 *rpack;    // [R]

    // --- forcing gather f_p = sum_q c_q r_k(q), as one flat list per lane ---
    // step * lanes + lane, n_gstep steps (two more of padding follow for the
    // read-ahead).  gth: x = a pair of entries of the lane's current sum, their
    // processes in 15 bits each (low half: to the sum's even accumulator, high
    // half: to its odd one; 0x8000 in a half: no entry), y = the sum's
    // destination at its last pair, else -1; gcf: the pair's coefficients.  A
    // destination d < n is the position's f, d >= n the partial sum d - n of a
    // position whose sum was split into chunks (block cells only).
    const int2 *gth;
    const double2 *gcf;
    int n_gstep;
    int n_fpart;          // partial sums of split forcing sums
    // the sums by position, for a lane that holds a whole cell: entries
    // fsum_ptr[p] .. fsum_ptr[p+1]: process, coefficient
    const int *fsum_ptr;  // [n+1]
    const int *fsum_k;
    const double *fsum_c;
    int n_part;           // partial sums of split forcing sums, substitution
                          // rows and factorisation rows (scratch after the
                          // rate terms; counted in FP64 values)
    int n_fsplit;         // positions whose sums are split
    // split position i: x = position, y = first partial | chunk count << 16
    const int2 *fsplit;   // [n_fsplit]

    // --- Jacobian, assembled straight into I - gamma J ---
    int nnzJ;
    // Per-lane flat entry lists (nonzeros spread over the lanes by entry
    // count), jls[step * lanes + lane].  Record: x = bits of the FP32
    // coefficient, y = k (signed 16 bits; -(r+1) for a reverse constant) |
    // o1 << 16 (0xffff: none), z = LU offset | diag << 16 | last entry of the
    // nonzero << 17, w = o2 | CSR index << 16; jlc: the coefficients in FP64.
    // The last record of a lane's list has bit 18 of z set; warp w of the cell
    // has lists of at most n_jstep[w].
    const int4 *jls;
    const double *jlc;
    int n_jstep[8];

    // --- LU storage: sparse rows [0, nsp) then a dense trailing block ---
    int nlu;              // storage entries (this form's: an FP32 or an FP64 LU)
    int d;                // first position of the dense block (= n when there is none)
    int D;                // dense block size n - d
    int LD;               // dense block row stride of this form (jls, fst, lops,
                          // lred_off and ch hold offsets that follow it)
    int dbase;            // storage offset of the dense block

    // factorisation of the sparse part: row-wise (up-looking) ops, level by
    // level as one list per lane, fst[step * lanes + lane] for the steps
    // fst_ptr[L] .. fst_ptr[L+1] of level L (one padding step follows the
    // last).  Op: DIV flag | source << 16 | target (LU offsets; a division
    // makes the multiplier, an update subtracts it times the source); with
    // the source CAMP_OP_NOSRC it takes the reciprocal of its target (a
    // row's pivot) or, with the DIV flag, does nothing.  An update whose
    // target has bit 15 set adds to a partial sum instead of an LU value (the
    // level's fst_part[L] partials start at zero).  Per level, the rows cut
    // into chunks then get a reduction (x = row | reciprocal flag << 16, y =
    // first entry of lred_off, z = shared columns ns | chunks << 16, w =
    // partial base; chunk c's slot s is w + c ns + s) and their tail ops (x =
    // first op in lops, y = count).
    int n_flev;
    const int *fst_ptr;   // [n_flev+1]
    const int *fst_part;  // [n_flev]
    const uint32_t *fst;
    const uint32_t *lops;
    const int *lred_ptr;  // [n_flev+1] into lred / ltail
    const int4 *lred;
    const int *lred_off;  // LU offsets of the shared columns
    const int2 *ltail;

    // Substitution of the sparse part, as passes over the lanes: in pass p
    // lane l takes the record sub_pass[p * lanes + l]: x = its row (-1: none),
    // y, z = the first two entries (LU offset | column << 16, -1: none), w =
    // entry pairs of the pass | 0x1000 on its level's last pass | 0x2000 if
    // that level has split rows | first step in `sub` << 14; sub[step * lanes
    // + l] holds the pairs from the second on.  One padding pass and step
    // follow the last.  The first n_fpass passes are the forward substitution
    // of the rows that have L entries, level by level; a row number >= n is
    // the partial dot product (row - n) of a row cut into chunks, and level
    // L's split rows (ssplit_ptr[L] ..: x = row, y = first partial | chunk
    // count << 16) then subtract their partials in order.  The n_bpass passes
    // after them are the backward substitution of the sparse rows (i < d), row
    // | LU offset of its reciprocal pivot << 16 in x.
    const int4 *sub_pass;
    const int2 *sub;
    int n_fpass, n_bpass;
    const int *ssplit_ptr;
    const int2 *ssplit;
    const int *udiag;     // [n] storage offset of U(i,i) for sparse rows

    const int *perm;      // [n] position -> species (declaration order)

    // --- ZSR aerosol water as a parameter (Sect. 2.2.2): with n_wsec > 0 the
    // liquid volume of section b is L_b(y) = L_env,b + sum_e w_e y_e over its
    // electrolytes, w_e = 1e-9 P / (R T) / (1000 m_e(a_w)) with the molality
    // fit sqrt(m_e) = sum_j Y_j a_w^j at a_w = RH (held at the fit's lowest
    // activity below it).  Section processes then keep per-unit-volume
    // constants in kf / kr; the kernels apply L^-la, L^-lb where the
    // constants are used (each section process's rpack record carries
    // section + 1 in bits 16-26 of w, la in bits 27-28 and lb in bits 29-30),
    // and the Jacobian adds the chain-rule term J_p P_y.
    int n_wsec;           // sections with a water parameter (0: none)
    int n_el;             // electrolytes
    int rh_slot;          // env index of the relative humidity
    const double *zsr_Y;  // [n_el][CAMP_ZSR_NY]
    const double *zsr_low;// [n_el]
    const int *pw_ptr;    // [n_wsec+1] into pw
    const int *pw;        // electrolyte entries: position | electrolyte << 16
    int n_pp;             // section processes with a power of 1/L (chain rule)
    // x = process, y = section, z = la | lb << 8, w = kr index (-1: none)
    const int4 *pp;       // [n_pp]
    // d f_i / d L_b for each (row, section) pair g: sum over entries of
    // coefficient * d r_j / d L_b of parameterised process j
    int n_g;
    const int *g_ptr;     // [n_g+1] into g_ent, g_coef
    const int *g_ent;     // parameterised process index
    const double *g_coef; // net stoichiometric coefficient
    // chain-rule entries J_ij += g_(i,b) w_e, n_el consecutive records per
    // g: x = LU offset of (i, e), y = g index, z = electrolyte e, w =
    // species-CSR non-zero
    int n_ch;
    const int4 *ch;
    int n_pw;             // per-cell FP64 values of the parameter (0: none)
    int n_pw64;           // more of them in the FP64 form (reverse constants)

    // BDF coefficients: l-vector of prod_{i=1..q}(1 + x/i), local-error
    // constants 1/((q+1) l_1(q)), factorials
    double lcoef[CAMP_QMAX + 2][CAMP_QMAX + 2];
    double ecoef[CAMP_QMAX + 2];
    double fact[CAMP_QMAX + 2];
    // the same, arranged so the step controller multiplies instead of
    // dividing and compares squares instead of taking roots
    double inv_l1[CAMP_QMAX + 2];   // 1 / l_1(q)
    double ecoef2[CAMP_QMAX + 2];   // ecoef(q)^2
    double rn;                      // 1 / n
};

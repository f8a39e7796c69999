// rgf_cell.cuh -- four columns of the recursion (one unit cell's worth) in one
// inverse.
//
// Columns a, b, c, d that follow one another in the recursion, a and b joined
// by t I (one bond per row), b and c by the bidiagonal stencil, c and d by t I
// (c0 c1 c2 c3 of a cell, c2 c3 c0' c1', and their mirrors).  No column has a
// bond inside itself.  Row by row c and d are dimers with 2 x 2 inverses,
//     g_cc = d_d / D,  g_cd = h = t / D,  g_dd = n = d_c / D,   D = d_c d_d - t^2
// (d_x = z - eps_x; an atom whose partner is absent is alone: 1 / d_x), whose
// levels lie near +-t, so D stays of order t^2 for every energy in use.
// Eliminating them leaves b with the tridiagonal matrix
//     T = d_b - t^2 S g_cc S^T                    (S the bond stencil b - c),
// and with A = z - eps_a - W_a^T g_q W_a (a after the columns before it) the
// pair a, b is [[A, -t], [-t, T]].  Then
//     B = T A - t^2,  V = B^-1:   G_ab = t V,  G_bb = A V,  G_aa = V T,
//     Q   = (P_q W_a) V,          P_d = t Q X,   g_d = n + X^T (A V) X,
//     X   = t S h                                 (bidiagonal),
// one inverse and two products for four columns, where two pairs
// (rgf_steps.cuh) take two inverses and two products.  Neither A nor T is
// inverted, so nothing grows when a level of the partial system or an isolated
// atom of b meets the energy (T and A are then small against t^2 and B is
// close to -t^2): near E = 0 the steps are better conditioned than the pair
// steps' shifted inverse, and no energy has to be excluded but those near the
// dimers' own levels (cell_ok).  Strongly detuned atoms are excluded: B holds
// products of two columns' diagonals, so an atom of a and its partner in b shut
// off by an on-site energy V put V^2 beside the other rows' t^2, which the
// inverse's pivot test (relative to max |B|) takes for a singular matrix (from V =
// 1e7 eV in double-float and 1e8 in binary64), and D leaves binary32 in c and d.
//
// Removed atoms: kappa_i = both atoms of row i of a and b kept.  B = T A -
// t^2 diag(kappa), where a row of A whose atom is removed (an identity row) is
// scaled by t if its partner in b is kept: the unknown of that row is then
// b's.  A removed atom of b has an identity row in T, which makes B's row A's;
// its row and column of A V are not used by X.
//
// What it saves is an inverse (about 0.75 ms of the 2.3 ms that a unit cell of
// N = 245 takes in pair steps on one SM, RGF_MIXED_TC).  Measured against pair
// steps: N = 245, 320 cells, 69 energies (RGF_MIXED_TC) 394.7 -> 263.8 ms;
// N = 101, 200 cells, 64 energies (RGF_FP64) 132.7 -> 93.4 ms; 192 uneven
// chains of N = 51 .. 401 952 -> 658 ms.  It is taken for every size.
#pragma once

#include "rgf_steps.cuh"

namespace rgf {

// Per-row quantities of columns c and d of a cell step and the tridiagonal T,
// in the Gauss-Jordan scratch (free between inverses; filled again after one).
template <class R>
struct CellCoef {
    cx<R>* Td;       // [Ka]  diagonal of T
    cx<R>* To;       // [Ka]  T_i,i+1
    cx<R>* x;        // [Kd]  t h
    cx<R>* n;        // [Kd]  n
};
template <class R>
__device__ __forceinline__ CellCoef<R> cell_coef(const SweepSmem<R>& s) {
    return CellCoef<R>{s.gj.panel, s.gj.panel2, s.gj.mult, s.gj.xrow};
}

// Entries of b bonded to entry i of c: i0 and i0 + 1 (within 0 .. Ka - 1),
// i0 = i for an even-row a (KL entries; c has odd rows), i - 1 for an odd-row a.
__device__ __forceinline__ int cell_nb(int ka_type, int i) { return i - ka_type; }

__device__ __forceinline__ bool site_keep(const ChainCtx& c, int k, int i) {
    return !c.rem || c.rem[(size_t)(k >> 2) * c.M + 4 * i + (k & 3)] == 0;
}

// Fills the coefficients of the cell a = k and returns whether the step may be
// taken: |D| >= t^2 / 4 on every dimer and |d| >= 0.05 |t| / 2.7 on every atom
// of c and d left alone (their 1 / D and 1 / d stay small against what they
// are added to), and |d| <= kCellMaxD |t| on every atom of the four columns (B
// then stays below about 4e3 t^2; left out with check = false, where a step
// taken already needs its coefficients again).  Needs s.kc and s.kn (keep masks
// of a and b) and s.eps of a.  Every thread; ends with a barrier.
//
// kCellMaxD: errors of T with one detuned dimer or 3 % of detuned atoms (N = 21, 24;
// 2 and 3 domains) are those of the pair steps up to 1e3 eV; with c and the next
// cell's a detuned, three domains, double-float, 8e-13 at 1e5 eV, 2e-11 at 1e6, 2e-7
// at 1e10 where pairs have 1e-13.
constexpr double kCellMaxD = 64.0;
template <class R>
__device__ bool cell_ok(const ChainCtx& c, int k, SweepSmem<R>& s, bool check = true) {
    const CellCoef<R> w = cell_coef(s);
    const int st = c.dir ? -1 : 1, kb = k + st, kc = k + 2 * st, kd = k + 3 * st;
    const int Ka = col_size(c, k), Kd = col_size(c, kd), ty = (k & 3) < 2 ? 0 : 1;
    const float lim = 0.25f * c.t2f.hi, alone = fabsf(c.tf.hi) * (0.05f / 2.7f);
    const float far2 = (float)(kCellMaxD * kCellMaxD) * c.t2f.hi;
    bool bad = false;
    auto near = [&](cx<R> d) {
        if (check && !(cabs2f(d) <= far2)) bad = true;
        return d;
    };
    // g_cc of row i of c (0 where c is removed)
    auto dimer = [&](int i, cx<R>& gcc, cx<R>& h, cx<R>& n) {
        const bool kpc = site_keep(c, kc, i), kpd = site_keep(c, kd, i);
        gcc = h = czero<R>();
        n = from_z<R>(1.0, 0.0);
        if (kpc && kpd) {
            const cx<R> dc = near(pair_d<R>(c, kc, i)), dd = near(pair_d<R>(c, kd, i));
            const cx<R> D = csub(cmul(dc, dd), from_z<R>(c.t2, 0.0));
            if (!(cabs2f(D) >= lim * lim)) bad = true;
            const cx<R> r = crecip(D);
            gcc = cmul(dd, r);
            h = cscale(r, Hop<R>::t(c));
            n = cmul(dc, r);
        } else if (kpc) {
            const cx<R> dc = near(pair_d<R>(c, kc, i));
            if (!(cabs2f(dc) >= alone * alone)) bad = true;
            gcc = crecip(dc);
        } else if (kpd) {
            const cx<R> dd = near(pair_d<R>(c, kd, i));
            if (!(cabs2f(dd) >= alone * alone)) bad = true;
            n = crecip(dd);
        }
    };
    for (int i = threadIdx.x; i < Kd; i += NT) {
        cx<R> gcc, h, n;
        dimer(i, gcc, h, n);
        w.x[i] = cscale(h, Hop<R>::t(c));
        w.n[i] = n;
    }
    for (int i = threadIdx.x; i < Ka; i += NT) {
        cx<R> Td = from_z<R>(1.0, 0.0), To = czero<R>();
        if (s.kc[i]) near(from_z<R>(c.z.re - s.eps[i], c.z.im));
        if (s.kn[i]) {
            Td = near(pair_d<R>(c, kb, i));
            // the entries of c bonded to i: cl below, cu above (towards i + 1)
            const int cl = i - 1 + ty, cu = i + ty;
            cx<R> gcc, h, n;
            if (cl >= 0) {
                dimer(cl, gcc, h, n);
                Td = csub(Td, cscale(gcc, Hop<R>::t2(c)));
            }
            if (cu < Kd) {
                dimer(cu, gcc, h, n);
                gcc = cscale(gcc, Hop<R>::t2(c));
                Td = csub(Td, gcc);
                if (i + 1 < Ka && s.kn[i + 1]) To = csub(czero<R>(), gcc);
            }
        }
        w.Td[i] = Td;
        w.To[i] = To;
    }
    return __syncthreads_or(bad) == 0;
}

// B = T A - t^2 diag(kappa) into X (ld KL) from A in F (ld ldf).  Needs s.kc,
// s.kn and the coefficients.  Returns max |X_il|^2.
template <class R>
__device__ double cell_B(const ChainCtx& c, int k, const cx<R>* F, int ldf, cx<R>* X, SweepSmem<R>& s) {
    const CellCoef<R> w = cell_coef(s);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int KL = c.KL, K = col_size(c, k);
    double amax2 = 0.0;
    for (int i = warp; i < K; i += NWARP) {
        const cx<R> td = w.Td[i], tu = w.To[i], tl = i > 0 ? w.To[i - 1] : czero<R>();
        const bool kappa = s.kc[i] && s.kn[i];
        for (int l = lane; l < K; l += 32) {
            cx<R> v = cmul(td, F[(size_t)i * ldf + l]);
            if (i > 0) v = cmac(v, tl, F[(size_t)(i - 1) * ldf + l], false);
            if (i + 1 < K) v = cmac(v, tu, F[(size_t)(i + 1) * ldf + l], false);
            if (i == l && kappa) v = csub(v, cscale(from_z<R>(1.0, 0.0), Hop<R>::t2(c)));
            X[(size_t)i * KL + l] = v;
            const double a2 = (double)cabs2f(v);
            amax2 = (a2 > amax2 || isnan(a2)) ? a2 : amax2;
        }
    }
    return block_max(amax2, s.red);
}

// Y <- Y T in place (rows x Ka, ld): the right operand of an interior domain's
// G_aa update, G_aa += (Y V) (Y T)^T.  A warp per row, the previous chunk's
// last old value carried along.  Every thread; ends with a barrier.
template <class R>
__device__ void cell_apply_T(int rows, int K, cx<R>* Y, int ld, SweepSmem<R>& s) {
    const CellCoef<R> w = cell_coef(s);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int r = warp; r < rows; r += NWARP) {
        cx<R>* y = Y + (size_t)r * ld;
        cx<R> carry = czero<R>();
        for (int l0 = 0; l0 < K; l0 += 32) {
            const int l = l0 + lane;
            const bool in = l < K;
            cx<R> lo = czero<R>(), me = czero<R>(), up = czero<R>();
            if (in) {
                me = y[l];
                if (lane > 0) lo = y[l - 1];
                if (l + 1 < K) up = y[l + 1];
            }
            __syncwarp();
            if (lane == 0) lo = carry;
            if (lane == 31 && in) carry = me;
            carry = shfl_from(carry, 31);
            if (in) {
                cx<R> v = cmul(me, w.Td[l]);
                if (l > 0) v = cmac(v, lo, w.To[l - 1], false);
                if (l + 1 < K) v = cmac(v, up, w.To[l], false);
                y[l] = v;
            }
            __syncwarp();
        }
    }
    __syncthreads();
}

// g_d = diag(n) + X^T Gbb X into G (Kd x Kd), and P_d = t Q X in place in P
// (rows x Ka -> rows x Kd).  Needs s.kn and the coefficients.  P's rows are
// overwritten behind the entries still to be read: upwards where c's entry i
// reads b's i, i + 1, downwards where it reads i - 1, i.  Every thread; ends
// with a barrier.
template <class R>
__device__ void cell_finish(const ChainCtx& c, int k, int rows, const cx<R>* Gbb, cx<R>* G, cx<R>* P,
                            SweepSmem<R>& s) {
    const CellCoef<R> w = cell_coef(s);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int KL = c.KL, Ka = col_size(c, k), Kd = c.KL + c.KR - Ka, ty = (k & 3) < 2 ? 0 : 1;
    for (int i = warp; i < Kd; i += NWARP) {
        const int p0 = cell_nb(ty, i), p1 = p0 + 1;
        const bool k0 = p0 >= 0 && s.kn[p0], k1 = p1 < Ka && s.kn[p1];
        const cx<R> xi = w.x[i];
        for (int l = lane; l < Kd; l += 32) {
            const int q0 = cell_nb(ty, l), q1 = q0 + 1;
            const bool m0 = q0 >= 0 && s.kn[q0], m1 = q1 < Ka && s.kn[q1];
            cx<R> v = czero<R>();
            if (k0 && m0) v = cadd(v, Gbb[(size_t)p0 * KL + q0]);
            if (k0 && m1) v = cadd(v, Gbb[(size_t)p0 * KL + q1]);
            if (k1 && m0) v = cadd(v, Gbb[(size_t)p1 * KL + q0]);
            if (k1 && m1) v = cadd(v, Gbb[(size_t)p1 * KL + q1]);
            v = cmul(cmul(v, xi), w.x[l]);
            if (i == l) v = cadd(v, w.n[i]);
            G[(size_t)i * KL + l] = v;
        }
    }
    const int nch = (Kd + 31) >> 5;
    for (int r = warp; r < rows; r += NWARP) {
        cx<R>* p = P + (size_t)r * KL;
        for (int h = 0; h < nch; ++h) {
            const int l = 32 * (ty ? nch - 1 - h : h) + lane;
            const int q0 = cell_nb(ty, l), q1 = q0 + 1;
            cx<R> v = czero<R>();
            if (l < Kd) {
                if (q0 >= 0 && s.kn[q0]) v = cadd(v, p[q0]);
                if (q1 < Ka && s.kn[q1]) v = cadd(v, p[q1]);
                v = cmul(cscale(v, Hop<R>::t(c)), w.x[l]);
            }
            __syncwarp();
            if (l < Kd) p[l] = v;
            __syncwarp();
        }
    }
    __syncthreads();
}

}  // namespace rgf

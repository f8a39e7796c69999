// rgf_grad.cu -- dT/d eps for every on-site energy, and the local density of
// states of ribbons without removed atoms; one thread block per chain.
//
// The paper does not differentiate; the derivative follows from Eq. 1 and
// Eq. 2.  With A = z - H - Sigma and dA/d eps_i = -e_i e_i^T, dG = G e_i e_i^T G,
// so for T = Tr[Gamma_L G_1L Gamma_R G_1L^dagger]:
//
//   dT/d eps_i = 2 Re (G_kL M G_1k)_ii,   M = Gamma_R G_1L^dagger Gamma_L,
//
// for site i of column k.  The blocks of the whole system's G come from the
// Dyson equation (Eq. 3) across a bond that cuts the ribbon in two, with the
// recursion of Eqs. 4-5 run from both leads (this two-sided form keeps its
// accuracy next to the poles of the half systems, E near 0, where a reverse sweep
// through the left recursion amplifies rounding at isolated sites).
//
// (G_c2c2 from the sum of what both sides put on column c2, not as gr (1 - Sigma
// gr)^-1: next to a pole of a half system gr or gl is large, and the product form
// then loses its square: on the chains of kLargeGrad, binary64, a mean error of
// 1.8e-8 of the scale and a largest of 5e-6.)
//
// Four columns at a time.  Both recursions take cell steps (rgf_cell.cuh): from
// the left they stop at the columns c1 of every cell (gl, Pl = G_1,c1 of the
// columns left of the cut), from the right at the columns c2 (gr, and S = M^T
// G_L,c2 of the columns right of it).  The two meet at the bond c1 - c2 (W its
// coupling) of every cell:
//
//   G_c2c2 = (gr^-1 - Sigma)^-1,  Sigma = W^T gl W,
//   G_1,c2 = (Pl W) G_c2c2,                 (G_c2,L M)^T = (S gr^-1) G_c2c2,
//   G_1,c1 = Pl + (G_1,c2 W^T) gl,          (G_c1,L M)^T = ((G_c2,L M)^T W^T) gl,
//
// where gl is large (kLargeGrad) the cut taken at c1 instead,
//
//   G_c1c1 = (gl^-1 - W gr W^T)^-1,
//   G_1,c1 = (Pl gl^-1) G_c1c1,             (G_c1,L M)^T = (S W^T) G_c1c1.
//
// The columns between two cells' cuts follow from the rows of z - H at c1 and c2
// themselves, where G_1x and G_xL have no source,
//
//   t psi_c0 = (z - eps_c1) psi_c1 - W psi_c2,   t psi_c3 = (z - eps_c2) psi_c2 - W^T psi_c1
//
// (psi_k = G_1k or G_kL M, row by row).  An atom of c3 or the next c0 whose partner in the
// row is removed (an orphan) has no such row; the chain of rows formed by c3 and
// the next c0 gives it from its neighbours' rows.  Where that would amplify rounding
// (orphans_tame), or an atom of c1 or c2 is far from the energy (far_row), both columns
// get blocks of their own from the parts on either side; in the lead-attached columns
// a Dyson step from their own block does.  Per cell: an inverse and two
// products for each of the two recursions, the same again for the recomputed
// left recursion, and two inverses and five products (three right operands) at
// the cut, where forming every column's block took 16 inverses and 24 products.
//
// Passes: the left-to-right recursion stores (gl, Pl) at every segment of
// seg_cells cells and yields G_1L, T and M; the right-to-left pass recomputes each
// segment's (gl, Pl) from its checkpoint, then walks it backwards.
//
// Local density of states rho_i(E) = -Im (G_ii) / pi (the paper notes that the
// Green's function of Eq. 1 gives the charge density; rho is its integrand over
// energy): with the same cuts, G_c1c2 = gl W G_c2c2, G_c1c1 from its inverse above,
// and for c0 and c3 the rows above taken on both sides,
//   t^2 G_c3c3 = d^2 G_c2c2 - d - 2 d W^T G_c1c2 + W^T G_c1c1 W   (diagonal, d = z - eps_c2).
// Ribbons with removed atoms: rgf_ldos.cu.
//
// What bounds it: the inverses and products, as the half sweep, one block per
// chain.  Against the column-wise sweeps: N = 101, L = 60, 64 energies
// (mixed, tensor cores) 364 -> 105 ms; N = 61, L = 40, 48 energies (binary64)
// 235 -> 65 ms; LDOS of N = 151, L = 32, 40 energies 465 -> 192 ms.
#include "rgf_cell.cuh"

namespace rgf {

namespace {

// |t| max|gl| from which on the gradient's cut is also taken at c1 (G_1,c1 = Pl + ... gl
// cancels to about 1 / |t| and loses that factor).  Errors next to poles (36 chains
// of N = 20, |E| <= 0.12 eV, of the scale, mean / largest; column by column before):
// binary64 3.6e-11 / 5.2e-10 before, 1.2e-11 / 2.9e-10 at 16, 1.3e-11 / 2.9e-10 at 64, 3.0e-10 /
// 9.0e-7 without;  mixed 1.3e-9 / 2.5e-8, 1.9e-10 / 3.6e-9, 2.5e-10 / 4.5e-9, 7.7e-9 / 1.1e-5
// (without: end columns by Dyson steps as well).  At 64 the N = 101 gradient takes 105
// ms, at 16 114.  The LDOS takes it in every cell: gl + G_c1c2 W^T gl cancels at any
// energy (60 chains of N = 34 .. 89, 0.3 to 1.2 eV, mean error of the LDOS, column by column /
// from |t| max|gl| = 8 on / everywhere: binary64 1.3e-14 / 3.1e-14 / 1.3e-14, mixed 9.1e-14 /
// 4.2e-13 / 1.0e-13; below 0.3 eV 1.8e-13 / 4.4e-13 / 1.4e-13 and 5.9e-12 / 1.1e-11 / 2.3e-12), in
// the same time, N = 151 192 ms.
constexpr double kLargeGrad = 64.0;

// The inverse out of line (one copy per kernel): flags << 16 | mbarrier parities.
template <class R, bool TC>
static __device__ __noinline__ uint32_t invert_nl(cx<R>* A, int K, int lda, cx<R>* G, int Kmax, double amax2,
                                                  tc::Area ar, uint32_t phase) {
    SweepSmem<R> s = carve<R>(rgf_dyn_smem, Kmax, TC);
    tc::State st{ar, phase};
    if constexpr (TC) s.gj.tcs = &st;
    const int flag = cta_gj_invert<R, TC && std::is_same<R, double>::value>(A, K, lda, G, lda, s.gj, amax2);
    return st.phase | ((uint32_t)flag << 16);
}

// One step of a recursion at column k: a cell step where want and cell_ok, else
// a single column.  G: g of the column before, replaced; P (rows rows, may be
// none): the corner block.  Out of line, the context in shared memory.  Returns
// the columns taken << 24 | flags << 16 | mbarrier parities.
template <class R, bool TC>
static __device__ __noinline__ uint32_t advance_nl(int k, bool want, cx<R>* G, cx<R>* P, int rows, cx<R>* X,
                                                   cx<R>* F, int Kmax, tc::Area ar, uint32_t phase) {
    constexpr bool TC64 = TC && std::is_same<R, double>::value;
    SweepSmem<R> s = carve<R>(rgf_dyn_smem, Kmax, TC);
    tc::State st{ar, phase};
    if constexpr (TC) {
        s.tcs = &st;
        s.gj.tcs = &st;
    }
    const ChainCtx& c = *s.ctx;
    const int KL = c.KL, K = col_size(c, k), kb = c.dir ? k - 1 : k + 1;
    load_col(c, k, s.kc, s.eps);
    load_col(c, prev_col(c, k), s.kp, nullptr);
    if (want) load_col(c, kb, s.kn, nullptr);
    __syncthreads();
    const bool cell = want && cell_ok<R>(c, k, s);
    double amax2 = build_column<R>(c, k, G, cell ? F : X, cell ? K : KL, s, -1, cell);
    if (cell) amax2 = cell_B<R>(c, k, F, K, X, s);
    const int flag = cta_gj_invert<R, TC64>(X, K, KL, G, KL, s.gj, amax2);
    if (rows > 0) strip_rows<R>(c, k, P, X, rows, s);
    if (cell) {
        if (rows > 0) two_products<R, TC64>(rows, K, K, X, KL, F, K, G, KL, P, X, KL, s);
        else dense_product<R, false, TC64>(K, K, K, F, K, G, KL, X, KL, s);
        cell_ok<R>(c, k, s, false);                  // the coefficients again
        cell_finish<R>(c, k, rows, X, G, P, s);
    } else if (rows > 0) {
        dense_product<R, false, TC64>(rows, K, K, X, KL, G, KL, P, KL, s);
    }
    return st.phase | ((uint32_t)flag << 16) | ((cell ? 4u : 1u) << 24);
}

// X (ld KL) = [z - eps_k on kept atoms, identity rows and columns at removed
// ones] - Sigma (ld K) + (add: what X holds).  Needs s.kc, s.eps.  Returns max
// |X_il|^2; ends with a barrier.
template <class R>
__device__ double lead_matrix(const ChainCtx& c, int K, const zd* Sig, bool onto, cx<R>* X, SweepSmem<R>& s) {
    double amax2 = 0.0;
    for (int e = threadIdx.x; e < K * K; e += NT) {
        const int i = e / K, l = e - i * K;
        cx<R>* x = X + (size_t)i * c.KL + l;
        cx<R> v;
        if (!s.kc[i] || !s.kc[l]) {
            v = (i == l) ? from_z<R>(1.0, 0.0) : czero<R>();
        } else {
            v = onto ? *x : (i == l) ? from_z<R>(c.z.re - s.eps[i], c.z.im) : czero<R>();
            v = csub(v, ld_z<R>(Sig + (size_t)i * K + l));
        }
        *x = v;
        const double a2 = (double)cabs2f(v);
        amax2 = (a2 > amax2 || isnan(a2)) ? a2 : amax2;
    }
    return block_max(amax2, s.red);
}

// D_ii = z - eps of entry i of column k in the working precision.
template <class R>
__device__ __forceinline__ cx<R> site_d(const ChainCtx& c, int k, int i) { return pair_d<R>(c, k, i); }

template <class R>
__device__ __forceinline__ double re_mul(cx<R> a, cx<R> b) {
    const zd u = to_z(a), g = to_z(b);
    return u.re * g.re - u.im * g.im;
}

// out[i] = 2 Re sum_b A[b][i] B[b][i] (b < rows) for the kept entries i of column
// k.  The 16 warps take 16 interleaved sets of rows, summed in order; the
// partial sums lie in the Gauss-Jordan scratch.  Every thread; barriers.
template <class R>
__device__ void contract(const ChainCtx& c, int k, const cx<R>* A, const cx<R>* B, int rows, double* out,
                         SweepSmem<R>& s) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, K = col_size(c, k), KL = c.KL;
    double* part = reinterpret_cast<double*>(s.gj.panel);        // [16][K]
    for (int i = lane; i < K; i += 32) {
        double acc = 0.0;
        for (int b = warp; b < rows; b += NWARP) acc += re_mul(A[(size_t)b * KL + i], B[(size_t)b * KL + i]);
        part[warp * K + i] = acc;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < K; i += NT) {
        double acc = 0.0;
        for (int w = 0; w < NWARP; ++w) acc += part[w * K + i];
        if (site_keep(c, k, i)) out[(size_t)(k >> 2) * c.M + 4 * i + (k & 3)] = 2.0 * acc;
    }
    __syncthreads();
}

// The rows formed by c3 of cell j (odd rows, psi3) and c0 of cell j + 1 (even rows,
// psi0), r = 0 .. N-1, in order across the ribbon.  fl: 0 no atom, 1 known (its
// partner kept), 2 orphan; d: z - eps.  Rows without an atom cut them into
// segments.  Two neighbouring rows that are both known (beyond a segment's ends psi
// is 0, which counts) give every other row of their segment, one after the other
// in both directions: the equation of row r, whose r and r - 1 are known, gives
// r + 1.
// Finds the segment lo .. hi from row lo on and rows p, p + 1 of it that are both
// known.  Returns 0 for nothing to fill (no atom at lo, or no known row: isolated
// from both leads, zero), 1 for such rows, 2 where known rows never meet each
// other or a known end.
__device__ __forceinline__ int orphan_segment(const uint8_t* fl, int N, int lo, int& hi, int& p) {
    hi = lo;
    if (fl[lo] == 0) return 0;
    bool known = fl[lo] == 1;
    while (hi + 1 < N && fl[hi + 1] != 0) known |= fl[++hi] == 1;
    if (!known) return 0;
    p = lo - 1;
    if (fl[lo] == 1) return 1;
    for (p = lo; p < hi; ++p)
        if (fl[p] == 1 && fl[p + 1] == 1) return 1;
    return fl[hi] == 1 ? 1 : 2;                 // p = hi: the last row and the one beyond it
}

// Whether the orphans of those rows may be filled from their neighbours: what an
// error of the known rows grows to on the way, row q from its neighbours by
//     e_q = |d / t|_{q-1} e_{q-1} + e_{q-2} (+ 1 for the partner of a known q - 1),
// stays below kMaxGrowth.  By one thread.  Without the bound the growing solution of
// the recurrence takes over where |d| > 2 |t| (24 orphans at 9 eV, N = 50: gradient
// errors of 1e-5 in binary64, 7e-4 in double-float; at 20 eV 5e8).  Runs of three or
// less and |d| up to |t| stay below it, ordinary vacancies therefore.
constexpr float kMaxGrowth = 16.0f;
template <class R>
__device__ bool orphans_tame(const uint8_t* fl, const cx<R>* d, int N, float at) {
    float worst = 0.0f;
    auto run = [&](int p, int q, int o, int end) {      // rows p, p + o are known
        float e2 = p >= 0 && p < N && fl[p] ? 1.0f : 0.0f, e1 = p + o >= 0 && p + o < N && fl[p + o] ? 1.0f : 0.0f;
        for (; q != end; q += o) {
            const float e = fl[q] == 1 ? 1.0f : sqrtf(cabs2f(d[q - o])) / at * e1 + e2 + (fl[q - o] == 1 ? 1.0f : 0.0f);
            worst = e <= worst ? worst : e;             // NaN is kept
            e2 = e1;
            e1 = e;
        }
    };
    for (int lo = 0, hi; lo < N; lo = hi + 1) {
        int p;
        const int g = orphan_segment(fl, N, lo, hi, p);
        if (g == 2) return false;
        if (g == 0) continue;
        if (p + 2 <= hi) run(p, p + 2, 1, hi + 1);
        if (p - 1 >= lo) run(p + 1, p - 1, -1, lo - 1);
    }
    return worst <= kMaxGrowth;
}

// The orphans' psi of those rows (orphans_tame).  psi1: c1 of cell j + 1, psi2: c2 of
// cell j (the partners of known rows).  One thread per row of psi.
template <class R>
__device__ void fill_orphans(const ChainCtx& c, int rows, const uint8_t* fl, const cx<R>* d, cx<R>* psi0,
                             cx<R>* psi3, const cx<R>* psi1, const cx<R>* psi2) {
    const int N = c.N, KL = c.KL;
    for (int b = threadIdx.x; b < rows; b += NT) {
        auto val = [&](int r) -> cx<R>& { return ((r & 1) ? psi3 : psi0)[(size_t)b * KL + (r >> 1)]; };
        auto has = [&](int r) { return r >= 0 && r < N && fl[r] != 0; };
        // the row's equation solved for the neighbour on side o
        auto from = [&](int r, int o) {
            cx<R> v = cmul(d[r], val(r));
            if (fl[r] == 1) v = csub(v, cscale(((r & 1) ? psi2 : psi1)[(size_t)b * KL + (r >> 1)], Hop<R>::t(c)));
            if (has(r - o)) v = csub(v, cscale(val(r - o), Hop<R>::t(c)));
            return cscale(v, 1.0 / c.t);
        };
        for (int lo = 0, hi; lo < N; lo = hi + 1) {
            int p;
            if (orphan_segment(fl, N, lo, hi, p) != 1) continue;
            for (int q = p + 2; q <= hi; ++q)
                if (fl[q] == 2) val(q) = from(q - 1, 1);
            for (int q = p - 1; q >= lo; --q)
                if (fl[q] == 2) val(q) = from(q + 1, -1);
        }
    }
    __syncthreads();
}

// Whether z - eps of entry i of column k is beyond kMaxRow |t|: psi of its partner in
// c0 or c3 from its row, (d psi_k - ..) / t, then cancels to about |t / d|.  Mean errors
// of 40 chains (N = 18 .. 39) with 2 % of the atoms at +-V, column by column / the rows
// everywhere / rows up to 2 |t|:
//   V = 8 |t|     gradient, mixed 7.7e-14 / 1.0e-13 / 8.2e-14, LDOS 9.5e-14 / 3.2e-13 / 1.2e-13
//   V = 1e3 |t|   gradient, mixed 3.6e-14 / 1.2e-13 / 3.5e-14, LDOS 8.0e-14 / 2.4e-12 / 8.3e-14
//   V = 4e5 |t|   gradient, binary64 3.3e-15 / 9.6e-14 / 2.9e-15 (the largest 5e-14 / 5e-11 /
//                 8e-14), LDOS 8.3e-15 / 1.5e-11 / 8.0e-15
// Ordinary disorder and the bands (|E| up to 3 |t|, next to no atom detuned) stay with the
// rows, 2.3 times faster on such chains.
constexpr float kMaxRow = 2.0f;
__device__ __forceinline__ bool far_row(const ChainCtx& c, int k, int i) {
    const float dr = (float)(c.z.re - site_eps(c, k, i)), dm = (float)c.z.im;
    return !(dr * dr + dm * dm <= kMaxRow * kMaxRow * (float)c.t2);
}

// Row flags and d of the rows between cells j and j + 1 (fill_orphans), in the
// Gauss-Jordan scratch.
template <class R>
struct BondRows {
    uint8_t* fl;     // [N]
    cx<R>* d;        // [N]
};
enum : int { BOND_ROWS = 0, BOND_ORPHANS = 1, BOND_COLUMNS = 2 };

// How c3 of cell j and c0 of cell j + 1 are had: from the rows of z - H at c2 and c1
// (BOND_ROWS), with orphans filled in (BOND_ORPHANS, w then holds the rows), or from
// blocks of their own (BOND_COLUMNS).  Every thread; barriers.
template <class R>
__device__ int bond_route(const ChainCtx& c, int j, const BondRows<R>& w, SweepSmem<R>& s) {
    const int c2 = 4 * j + 2, c3 = c2 + 1;
    bool any = false, far = false;
    for (int r = threadIdx.x; r < c.N; r += NT) {
        const int k = (r & 1) ? c3 : c3 + 1, kp = (r & 1) ? c2 : c3 + 2, i = r >> 1;
        const bool kk = site_keep(c, k, i), known = site_keep(c, kp, i);
        far = far || (kk && known && far_row(c, kp, i));
        if (!c.rem) continue;
        w.fl[r] = !kk ? 0 : known ? 1 : 2;
        w.d[r] = site_d<R>(c, k, i);
        any = any || w.fl[r] == 2;
    }
    if (__syncthreads_or(far) != 0) return BOND_COLUMNS;
    if (__syncthreads_or(any) == 0) return BOND_ROWS;
    if (threadIdx.x == 0) s.gj.ctl[2] = orphans_tame<R>(w.fl, w.d, c.N, (float)fabs(c.t));
    __syncthreads();
    const bool tame = s.gj.ctl[2] != 0;
    __syncthreads();
    return tame ? BOND_ORPHANS : BOND_COLUMNS;
}

// A (ld KL) -= W^T g W at column k, g the Green's function of the part that ends with
// the column before k in the recursion of direction c.dir.  Needs s.kc and s.kp of
// the two.  Returns max |A_il|^2; ends with a barrier.
template <class R>
__device__ double take_side(const ChainCtx& c, int k, const cx<R>* g, cx<R>* A, SweepSmem<R>& s) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int KL = c.KL, K = col_size(c, k), Kq = col_size(c, prev_col(c, k));
    double amax2 = 0.0;
    for (int i = warp; i < K; i += NWARP) {
        int a0, a1;
        prev_src(c, k, i, Kq, a0, a1);
        const bool ka0 = a0 >= 0 && s.kp[a0], ka1 = a1 >= 0 && s.kp[a1];
        for (int l = lane; l < K; l += 32) {
            cx<R> f = A[(size_t)i * KL + l];
            if (s.kc[i] && s.kc[l]) {
                int b0, b1;
                prev_src(c, k, l, Kq, b0, b1);
                const bool kb0 = b0 >= 0 && s.kp[b0], kb1 = b1 >= 0 && s.kp[b1];
                cx<R> v = czero<R>();
                if (ka0 && kb0) v = cadd(v, g[(size_t)a0 * KL + b0]);
                if (ka0 && kb1) v = cadd(v, g[(size_t)a0 * KL + b1]);
                if (ka1 && kb0) v = cadd(v, g[(size_t)a1 * KL + b0]);
                if (ka1 && kb1) v = cadd(v, g[(size_t)a1 * KL + b1]);
                f = csub(f, cscale(v, Hop<R>::t2(c)));
                A[(size_t)i * KL + l] = f;
            }
            const double a2 = (double)cabs2f(f);
            amax2 = (a2 > amax2 || isnan(a2)) ? a2 : amax2;
        }
    }
    return block_max(amax2, s.red);
}

// Whether entry i of column k (c0 or c3) follows from the row of its partner in kp,
// and whether column k holds an atom for which it does not.
__device__ __forceinline__ bool by_row(const ChainCtx& c, int k, int kp, int i) {
    return site_keep(c, k, i) && site_keep(c, kp, i) && !far_row(c, kp, i);
}
__device__ __forceinline__ bool any_not_by_row(const ChainCtx& c, int k, int kp) {
    bool any = false;
    for (int i = threadIdx.x; i < col_size(c, k); i += NT) any = any || (site_keep(c, k, i) && !by_row(c, k, kp, i));
    return __syncthreads_or(any) != 0;
}

struct GradArgs {
    const ChainDev* chains;
    const int* order;
    int Kmax;
    double eta_d;
    const zd* leadout;
    const int* lead_status;
    const LeadDev* leads;
    void* ws;
    const int* seg_cells;
    double* T;
    double* out;
    int32_t* status;
};

}  // namespace

template <class R, bool TC, bool LDOS>
__global__ void __launch_bounds__(NT, 1) grad_kernel(GradArgs a) {
    constexpr bool TC64 = TC && std::is_same<R, double>::value;
    SweepSmem<R> s = carve<R>(rgf_dyn_smem, a.Kmax, TC);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ci = a.order[blockIdx.x];
    const ChainDev& ch = a.chains[ci];
    const int lst = lead_state(a.lead_status, ch.lead);
    if (lst != ST_OK) {                                      // for every chain, rgf_ldos.cu's too
        if (threadIdx.x == 0) { a.T[ci] = NAN; if (a.status) a.status[ci] = lst; }
        return;
    }
    if (LDOS && ch.rem) return;                              // rgf_ldos.cu
    if (threadIdx.x == 0) *s.ctx = make_ctx(ch, a.leads[ch.lead], a.leadout, a.eta_d, 0);
    __syncthreads();
    const ChainCtx& c = *s.ctx;
    auto set_dir = [&](int d) {
        __syncthreads();
        if (threadIdx.x == 0) s.ctx->dir = d;
        __syncthreads();
    };
    const int KL = c.KL, KR = c.KR, L = c.L, n = c.ncol;
    const int sc = a.seg_cells[ci], nseg = (L + sc - 1) / sc;
    const size_t B = (size_t)KL * KL;
    cx<R>* base = reinterpret_cast<cx<R>*>(a.ws) + ch.ws_off;
    auto blk = [&](int i) { return base + (size_t)i * B; };
    cx<R> *X = blk(0), *X2 = blk(1), *F = blk(2), *gl = blk(3), *Pl = blk(4), *gr = blk(5), *S = blk(6);
    cx<R> *T1 = blk(7), *G12 = blk(8), *R2 = blk(9), *Y2G = blk(10), *Y2R = blk(11);
    cx<R> *psi0G = blk(16), *psi0R = blk(17), *g0 = blk(18), *G1L = blk(19);
    // (G_1,c1, (G_c1,L M)^T) of cell j: two sets, the other one cell j + 1's
    auto G11 = [&](int j) { return blk(12 + 2 * (j & 1)); };
    auto R1 = [&](int j) { return blk(13 + 2 * (j & 1)); };
    cx<R>* ckpt = blk(20);                                   // (gl, Pl) at cell seg * sc
    cx<R>* seg = ckpt + (size_t)nseg * 2 * B;                // (gl, Pl) of the segment's cells
    double* out = a.out + ch.grad_off;
    tc::State tst{};
    if constexpr (TC) tc_attach<R>(a.Kmax, s, tst);
    int flag = 0;
    auto invert = [&](cx<R>* A, int K, cx<R>* G, double amax2) {
        const uint32_t r = invert_nl<R, TC>(A, K, KL, G, a.Kmax, amax2, TC ? tst.ar : tc::Area{0}, TC ? tst.phase : 0u);
        if (TC) tst.phase = r & 0xFFFFu;
        flag |= (int)(r >> 16);
    };
    auto advance = [&](int k, bool want, cx<R>* G, cx<R>* P, int rows) {
        const uint32_t r = advance_nl<R, TC>(k, want, G, P, rows, X, F, a.Kmax, TC ? tst.ar : tc::Area{0}, TC ? tst.phase : 0u);
        if (TC) tst.phase = r & 0xFFFFu;
        flag |= (int)((r >> 16) & 0xFFu);
        return (int)(r >> 24);
    };
    // the LDOS of column k from its block (ld KL)
    auto column_ldos = [&](int k, const cx<R>* G) {
        for (int i = threadIdx.x; i < col_size(c, k); i += NT)
            out[(size_t)(k >> 2) * c.M + 4 * i + (k & 3)] = -to_z(G[(size_t)i * KL + i]).im * kInvPi;
        __syncthreads();
    };
    auto finish = [&](int st, double T) {
        if (threadIdx.x == 0) {
            a.T[ci] = st == ST_OK ? T : NAN;
            if (a.status) a.status[ci] = st;
        }
        if constexpr (TC) tc::teardown(tst.ar);
    };

    // ---- left to right --------------------------------------------------
    // column 0, then column 1 (c1 of cell 0), then cell steps from c1 to c1
    load_col(c, 0, s.kc, s.eps);
    __syncthreads();
    invert(X, KL, gl, lead_matrix<R>(c, KL, c.SigL(), false, X, s));
    copy_blk(g0, gl, B);
    copy_blk(Pl, gl, B);
    advance(1, false, gl, Pl, KL);
    for (int j = 0; j < L; ++j) {
        if (j % sc == 0) {
            cx<R>* cp = ckpt + (size_t)(j / sc) * 2 * B;
            copy_blk(cp, gl, B);
            copy_blk(cp + B, Pl, B);
        }
        if (j + 1 < L)
            for (int q = 0; q < 4;) q += advance(4 * j + 2 + q, q == 0, gl, Pl, KL);
    }
    advance(n - 2, false, gl, Pl, KL);
    {
        // the last column: both the left part and the right lead
        load_col(c, n - 1, s.kc, s.eps);
        load_col(c, n - 2, s.kp, nullptr);
        __syncthreads();
        build_column<R>(c, n - 1, gl, X, KL, s, -1, false);
        invert(X, KR, gl, lead_matrix<R>(c, KR, c.SigR(), true, X, s));
        strip_rows<R>(c, n - 1, Pl, X, KL, s);
        dense_product<R, false, TC64>(KL, KR, KR, X, KL, gl, KL, G1L, KL, s);
    }
    if constexpr (TC) {
        if (*(volatile int*)tst.ar.err()) flag |= 4;
    }
    const double T = trace_T<R>(c, G1L, X, X2, F, s);
    {
        const int st = chain_status(c, flag, T);
        if (st != ST_OK) {
            finish(st, T);
            return;
        }
    }
    if constexpr (LDOS) column_ldos(n - 1, gl);

    // ---- right to left ----------------------------------------------------
    // column n - 1, then n - 2 (c2 of the last cell), then cell steps from c2 to c2
    cx<R>*gR = blk(12), *Sn = blk(13);                       // of column n - 1, for the last cell only
    if (L & 1) { gR = blk(14); Sn = blk(15); }               // (the set that its own c1 does not use)
    load_col(c, n - 1, s.kc, s.eps);
    __syncthreads();
    invert(X, KR, gr, lead_matrix<R>(c, KR, c.SigR(), false, X, s));
    if constexpr (!LDOS) {
        // M^T = Gamma_L^T conj(G_1L) Gamma_R^T (KL x KR), S = M^T gr
        for (int e = threadIdx.x; e < KL * KL; e += NT) {
            const int i = e / KL, l = e - i * KL;
            X[(size_t)i * KL + l] = ld_z<R>(c.GamL() + (size_t)l * KL + i);
            if (l < KR) X2[(size_t)i * KL + l] = cconj(G1L[(size_t)i * KL + l]);
        }
        for (int e = threadIdx.x; e < KR * KR; e += NT) {
            const int i = e / KR, l = e - i * KR;
            F[(size_t)i * KL + l] = ld_z<R>(c.GamR() + (size_t)l * KR + i);
        }
        __syncthreads();
        dense_product<R, false, TC64>(KL, KR, KL, X, KL, X2, KL, T1, KL, s);
        dense_product<R, false, TC64>(KL, KR, KR, T1, KL, F, KL, X, KL, s);
        dense_product<R, false, TC64>(KL, KR, KR, X, KL, gr, KL, S, KL, s);
        copy_blk(gR, gr, B);
        copy_blk(Sn, S, B);
    }
    const int rrows = LDOS ? 0 : KL;
    int route = BOND_ROWS;                                   // of the bond behind the cell at hand
    set_dir(1);
    advance(n - 2, false, gr, S, rrows);
    for (int sg = nseg - 1; sg >= 0; --sg) {
        const int ja = sg * sc, jb = min(L, ja + sc);
        // (gl, Pl) of cells ja .. jb - 1 from the checkpoint
        set_dir(0);
        {
            const cx<R>* cp = ckpt + (size_t)sg * 2 * B;
            copy_blk(gl, cp, B);
            if (!LDOS) copy_blk(Pl, cp + B, B);
            for (int j = ja; j < jb; ++j) {
                cx<R>* sl = seg + (size_t)(j - ja) * 2 * B;
                copy_blk(sl, gl, B);
                if (!LDOS) copy_blk(sl + B, Pl, B);
                if (j + 1 < jb)
                    for (int q = 0; q < 4;)
                        q += advance(4 * j + 2 + q, q == 0, gl, Pl, LDOS ? 0 : KL);
            }
        }
        for (int j = jb - 1; j >= ja; --j) {
            const cx<R>*glj = seg + (size_t)(j - ja) * 2 * B, *Plj = glj + B;
            const int c0 = 4 * j, c1 = c0 + 1, c2 = c0 + 2, c3 = c0 + 3;
            // the cut c1 - c2: gr^-1 into F, S gr^-1 into T1, gr^-1 - W^T gl W into F
            // (no pivot threshold: gr is as small as 1 / eps where an atom is shut off)
            copy_blk(X, gr, B);
            invert(X, KR, F, 0.0);
            if (!LDOS) dense_product<R, false, TC64>(KL, KR, KR, S, KL, F, KL, T1, KL, s);
            set_dir(0);
            load_col(c, c2, s.kc, s.eps);
            load_col(c, c1, s.kp, nullptr);
            __syncthreads();
            invert(F, KR, X, take_side<R>(c, c2, glj, F, s));    // G_c2c2 into X
            strip_rows<R>(c, c2, LDOS ? glj : Plj, X2, KL, s);
            bool large = false;
            if constexpr (!LDOS) {
                double g2 = 0.0;
                for (int e = threadIdx.x; e < KL * KL; e += NT) g2 = fmax(g2, (double)cabs2f(glj[e]));
                large = block_max(g2, s.red) * c.t2 > kLargeGrad * kLargeGrad;
            }
            // c3 and the next cell's c0 column by column: G_kk from the parts that end
            // beside k on both sides, G_1k = (Pl W) G_kk, (G_kL M)^T = (S W^T) G_kk
            auto bond_columns = [&]() {
                copy_blk(gl, glj, B);
                if (!LDOS) copy_blk(Pl, Plj, B);
                for (int k = c3; k <= c3 + 1; ++k) {
                    set_dir(0);
                    advance(k - 1, false, gl, Pl, rrows);
                    load_col(c, k, s.kc, s.eps);
                    load_col(c, k - 1, s.kp, nullptr);
                    __syncthreads();
                    build_column<R>(c, k, gl, X, KL, s, -1, false);
                    if (!LDOS) strip_rows<R>(c, k, Pl, X2, KL, s);
                    set_dir(1);
                    load_col(c, k + 1, s.kp, nullptr);
                    __syncthreads();
                    const int K = col_size(c, k);
                    invert(X, K, F, take_side<R>(c, k, k == c3 ? psi0G : G11(j + 1), X, s));
                    if constexpr (LDOS) {
                        column_ldos(k, F);
                    } else {
                        dense_product<R, false, TC64>(KL, K, K, X2, KL, F, KL, T1, KL, s);
                        strip_rows<R>(c, k, k == c3 ? psi0R : R1(j + 1), X2, KL, s);
                        dense_product<R, false, TC64>(KL, K, K, X2, KL, F, KL, G12, KL, s);
                        contract<R>(c, k, T1, G12, KL, out, s);
                    }
                }
                set_dir(0);
            };
            if constexpr (LDOS) {
                // G_c1c2 = (gl W) G_c2c2 into G12, G_c1c1 = (gl^-1 - W gr W^T)^-1 into T1
                dense_product<R, false, TC64>(KL, KR, KR, X2, KL, X, KL, G12, KL, s);
                set_dir(1);
                copy_blk(T1, glj, B);
                invert(T1, KL, F, 0.0);
                load_col(c, c1, s.kc, s.eps);
                load_col(c, c2, s.kp, nullptr);
                __syncthreads();
                invert(F, KL, T1, take_side<R>(c, c1, gr, F, s));
                const double t = c.t, t2 = c.t2;
                auto G11z = [&](int p, int p2) { return to_z(T1[(size_t)min(p, p2) * KL + max(p, p2)]); };
                auto G22z = [&](int i, int l) { return to_z(X[(size_t)i * KL + l]); };
                auto G12z = [&](int p, int i) { return to_z(G12[(size_t)p * KL + i]); };
                double* o = out + (size_t)j * c.M;
                for (int p = threadIdx.x; p < KL; p += NT) {
                    const zd d = {c.z.re - site_eps(c, c1, p), c.z.im}, g = G11z(p, p);
                    o[4 * p + 1] = -g.im * kInvPi;
                    // c0: c1's row on both sides; its neighbours in c2 are p - 1, p
                    zd v = csub(cmul(cmul(d, d), g), d);
                    zd h = {0.0, 0.0}, w = {0.0, 0.0};
                    for (int q = max(p - 1, 0); q <= min(p, KR - 1); ++q) {
                        h = cadd(h, G12z(p, q));
                        for (int q2 = max(p - 1, 0); q2 <= min(p, KR - 1); ++q2) w = cadd(w, G22z(q, q2));
                    }
                    v = cadd(csub(v, cscale(cmul(d, h), 2.0 * t)), cscale(w, t2));
                    o[4 * p] = -v.im / t2 * kInvPi;
                }
                for (int i = threadIdx.x; i < KR; i += NT) {
                    const zd d = {c.z.re - site_eps(c, c2, i), c.z.im}, g = G22z(i, i);
                    o[4 * i + 2] = -g.im * kInvPi;
                    zd v = csub(cmul(cmul(d, d), g), d);
                    zd h = {0.0, 0.0}, w = {0.0, 0.0};
                    for (int p = i; p <= min(i + 1, KL - 1); ++p) {
                        h = cadd(h, G12z(p, i));
                        for (int p2 = i; p2 <= min(i + 1, KL - 1); ++p2) w = cadd(w, G11z(p, p2));
                    }
                    v = cadd(csub(v, cscale(cmul(d, h), 2.0 * t)), cscale(w, t2));
                    if (j < L - 1) o[4 * i + 3] = -v.im / t2 * kInvPi;
                }
                __syncthreads();
                if (j < L - 1 && route == BOND_COLUMNS) bond_columns();
                if (j == 0 && any_not_by_row(c, c0, c1)) {
                    // column 0 from its own block: the right recursion up to c1
                    set_dir(1);
                    advance(c1, false, gr, S, 0);
                    load_col(c, c0, s.kc, s.eps);
                    load_col(c, c1, s.kp, nullptr);
                    __syncthreads();
                    build_column<R>(c, c0, gr, X, KL, s, -1, false);
                    invert(X, KL, F, lead_matrix<R>(c, KL, c.SigL(), true, X, s));
                    column_ldos(c0, F);
                }
            } else {
                cx<R>*g11 = G11(j), *r1 = R1(j);
                two_products<R, TC64>(KL, KL, KR, X2, KL, T1, KL, X, KL, G12, R2, KL, s);
                set_dir(1);
                load_col(c, c1, s.kc, s.eps);
                load_col(c, c2, s.kp, nullptr);
                __syncthreads();
                strip_rows<R>(c, c1, G12, Y2G, KL, s);
                strip_rows<R>(c, c1, R2, Y2R, KL, s);
                if (large) {
                    copy_blk(X, glj, B);
                    invert(X, KL, F, 0.0);
                    dense_product<R, false, TC64>(KL, KL, KL, Plj, KL, F, KL, T1, KL, s);
                    invert(F, KL, X, take_side<R>(c, c1, gr, F, s));     // G_c1c1 = (gl^-1 - W gr W^T)^-1 into X
                    strip_rows<R>(c, c1, S, X2, KL, s);
                    two_products<R, TC64>(KL, KL, KL, T1, KL, X2, KL, X, KL, g11, r1, KL, s);
                } else {
                    two_products<R, TC64>(KL, KL, KL, Y2G, KL, Y2R, KL, glj, KL, g11, r1, KL, s);
                    for (size_t e = threadIdx.x; e < B; e += NT) g11[e] = cadd(g11[e], Plj[e]);
                    __syncthreads();
                }
                const double ti = 1.0 / c.t;
                // c3 into X2 (G_1,c3) and T1 ((G_c3,L M)^T)
                set_dir(0);
                load_col(c, c2, s.kc, s.eps);
                load_col(c, c1, s.kp, nullptr);
                __syncthreads();
                strip_rows<R>(c, c2, g11, X2, KL, s);
                strip_rows<R>(c, c2, r1, T1, KL, s);
                for (int e = threadIdx.x; e < KL * KR; e += NT) {
                    const int b = e / KR, i = e - b * KR;
                    const size_t o = (size_t)b * KL + i;
                    const bool kap = by_row(c, c3, c2, i);
                    const cx<R> d = site_d<R>(c, c2, i);
                    X2[o] = kap ? cscale(csub(cmul(d, G12[o]), X2[o]), ti) : czero<R>();
                    T1[o] = kap ? cscale(csub(cmul(d, R2[o]), T1[o]), ti) : czero<R>();
                }
                __syncthreads();
                if (j == L - 1 && any_not_by_row(c, c3, c2)) {
                    // the last column's others: G_1L, and S_n + ((G_c2,L M)^T t kappa) gR
                    for (int e = threadIdx.x; e < KL * KR; e += NT) {
                        const int b = e / KR, i = e - b * KR;
                        const size_t o = (size_t)b * KL + i;
                        X[o] = site_keep(c, c2, i) && site_keep(c, c3, i) ? cscale(R2[o], Hop<R>::t(c)) : czero<R>();
                    }
                    __syncthreads();
                    dense_product<R, false, TC64>(KL, KR, KR, X, KL, gR, KL, F, KL, s);
                    for (int e = threadIdx.x; e < KL * KR; e += NT) {
                        const int b = e / KR, i = e - b * KR;
                        const size_t o = (size_t)b * KL + i;
                        if (!site_keep(c, c3, i) || by_row(c, c3, c2, i)) continue;
                        X2[o] = G1L[o];
                        T1[o] = cadd(F[o], Sn[o]);
                    }
                    __syncthreads();
                }
                contract<R>(c, c2, G12, R2, KL, out, s);
                if (j == L - 1 || route != BOND_COLUMNS) contract<R>(c, c3, X2, T1, KL, out, s);
                if (j < L - 1 && route == BOND_ORPHANS) {
                    const BondRows<R> w{reinterpret_cast<uint8_t*>(s.gj.mult), s.gj.xrow};
                    bond_route<R>(c, j, w, s);               // the rows again
                    fill_orphans<R>(c, KL, w.fl, w.d, psi0G, X2, G11(j + 1), G12);
                    fill_orphans<R>(c, KL, w.fl, w.d, psi0R, T1, R1(j + 1), R2);
                    for (int r = warp; r < c.N; r += NWARP) {
                        if (w.fl[r] != 2) continue;
                        const cx<R>*pg = (r & 1) ? X2 : psi0G, *pr = (r & 1) ? T1 : psi0R;
                        double acc = 0.0;
                        for (int b = lane; b < KL; b += 32)
                            acc += re_mul(pg[(size_t)b * KL + (r >> 1)], pr[(size_t)b * KL + (r >> 1)]);
                        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                        const int k = (r & 1) ? c3 : c3 + 1;
                        if (lane == 0) out[(size_t)(k >> 2) * c.M + 4 * (r >> 1) + (k & 3)] = 2.0 * acc;
                    }
                    __syncthreads();
                }
                if (j < L - 1 && route == BOND_COLUMNS) bond_columns();
                // c0 into psi0
                for (int e = threadIdx.x; e < KL * KL; e += NT) {
                    const int i = e % KL;
                    const bool kap = by_row(c, c0, c1, i);
                    const cx<R> d = site_d<R>(c, c1, i);
                    psi0G[e] = kap ? cscale(csub(cmul(d, g11[e]), Y2G[e]), ti) : czero<R>();
                    psi0R[e] = kap ? cscale(csub(cmul(d, r1[e]), Y2R[e]), ti) : czero<R>();
                }
                __syncthreads();
                if (j == 0 && any_not_by_row(c, c0, c1)) {
                    // column 0's others: g0 + (G_1,c1 t kappa) g0, ((G_c1,L M)^T t kappa) g0
                    for (int e = threadIdx.x; e < KL * KL; e += NT) {
                        const int i = e % KL;
                        const bool kap = site_keep(c, c0, i) && site_keep(c, c1, i);
                        X[e] = kap ? cscale(g11[e], Hop<R>::t(c)) : czero<R>();
                        F[e] = kap ? cscale(r1[e], Hop<R>::t(c)) : czero<R>();
                    }
                    __syncthreads();
                    dense_product<R, false, TC64>(KL, KL, KL, X, KL, g0, KL, X2, KL, s);
                    dense_product<R, false, TC64>(KL, KL, KL, F, KL, g0, KL, X, KL, s);
                    for (int e = threadIdx.x; e < KL * KL; e += NT) {
                        const int i = e % KL;
                        if (!site_keep(c, c0, i) || by_row(c, c0, c1, i)) continue;
                        psi0G[e] = cadd(X2[e], g0[e]);
                        psi0R[e] = X[e];
                    }
                    __syncthreads();
                }
                contract<R>(c, c1, g11, r1, KL, out, s);
                contract<R>(c, c0, psi0G, psi0R, KL, out, s);
            }
            // the right recursion on to c2 of cell j - 1; on the way, where that cell's
            // c3 and this one's c0 are had column by column, (gr, S) of c1 into
            // the c1 blocks of this cell, which is done, and of c0 into psi0
            if (j > 0) {
                route = bond_route<R>(c, j - 1, BondRows<R>{reinterpret_cast<uint8_t*>(s.gj.mult), s.gj.xrow}, s);
                set_dir(1);
                for (int q = 0; q < 4;) {
                    q += advance(c1 - q, q == 0 && route != BOND_COLUMNS, gr, S, rrows);
                    if (route == BOND_COLUMNS && q <= 2) {
                        copy_blk(q == 1 ? G11(j) : psi0G, gr, B);
                        if (!LDOS) copy_blk(q == 1 ? R1(j) : psi0R, S, B);
                    }
                }
            }
        }
    }
    if constexpr (TC) {
        if (*(volatile int*)tst.ar.err()) flag |= 4;
    }
    const int st = chain_status(c, flag, T);
    if (st != ST_OK)
        for (size_t e = threadIdx.x; e < (size_t)L * c.M; e += NT) out[e] = 0.0;
    finish(st, T);
}

size_t grad_ws_elems(int N, int L, int seg_cells) {
    const size_t KL = (size_t)col_KL(N), nseg = ((size_t)L + seg_cells - 1) / seg_cells;
    const size_t cut = (20 + 2 * nseg + 2 * (size_t)seg_cells) * KL * KL;
    const size_t col = ldos_ws_elems(N, L, seg_cells);
    return cut > col ? cut : col;
}

cudaError_t launch_grad(int precision, const ChainDev* chains, const int* order, int nchains,
                        int Kmax, double eta_device, const void* leadout, const int* lead_status,
                        const LeadDev* leads, void* ws, const int* seg_cells, double* T, double* out,
                        int out_mode, bool any_removed, int32_t* status, cudaStream_t st) {
    if (nchains <= 0) return cudaSuccess;
    // the _TC precisions on the pipes where the tensor-core layout does not fit
    if ((precision == 2 || precision == 3) && !tc_layout_fits(Kmax)) precision = precision == 2 ? 1 : 0;
    const bool tc = precision == 2 || precision == 3;
    const size_t smem = sweep_smem_bytes(Kmax, tc);
    const GradArgs a{chains, order, Kmax, eta_device, (const zd*)leadout, lead_status, leads, ws, seg_cells, T, out, status};
    const bool ldos = out_mode == OUT_LDOS;
    auto kern = precision == 3   ? (ldos ? grad_kernel<double, true, true> : grad_kernel<double, true, false>)
                : precision == 2 ? (ldos ? grad_kernel<df32, true, true> : grad_kernel<df32, true, false>)
                : precision == 1 ? (ldos ? grad_kernel<df32, false, true> : grad_kernel<df32, false, false>)
                                 : (ldos ? grad_kernel<double, false, true> : grad_kernel<double, false, false>);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<nchains, NT, smem, st>>>(a);
    e = cudaGetLastError();
    if (e == cudaSuccess && ldos && any_removed)
        e = launch_ldos_removed(precision, chains, order, nchains, Kmax, eta_device, leadout, lead_status, leads,
                                ws, seg_cells, T, out, status, st);
    return e;
}

}  // namespace rgf

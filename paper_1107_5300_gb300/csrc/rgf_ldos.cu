// rgf_ldos.cu -- the local density of states of ribbons with removed atoms,
// column by column, one thread block per chain (without removed atoms:
// rgf_grad.cu, four columns at a time).
//
// rho_i(E) = -Im (G_kk)_ii / pi for site i of column k, with
//   G_kk = (A_k - W_k^T gl_{k-1} W_k - W_{k+1} gr_{k+1} W_{k+1}^T)^-1
// from the recursion of Eqs. 4-5 run from both leads (Eq. 3 with the bonds on both
// sides of column k cut).  The right-to-left recursion stores gr at the end of
// every segment; the left-to-right pass recomputes each segment's gr from its
// checkpoint, then walks it forwards carrying gl and Pl = G_1k, which gives T.
#include "rgf_cell.cuh"

namespace rgf {

namespace {

// X = (z - eps_k) I - [left] SigmaL_k - [right] SigmaR_k for column k, identity
// rows and columns at removed atoms.  SigmaL_k: Sigma_L at k = 0, else
// W_k^T glp W_k; SigmaR_k: Sigma_R at the last column, else
// W_{k+1} grn W_{k+1}^T (W = t times the bond pattern between two columns,
// applied as a stencil).  Needs s.kc, s.eps of column k, s.kp of k-1 and s.kn
// of k+1.  Returns max |X_il|^2 over the block (ends with a barrier).
template <class R>
__device__ double build_A(const ChainCtx& c, int k, bool left, const cx<R>* glp, bool right,
                          const cx<R>* grn, cx<R>* X, SweepSmem<R>& s) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int KL = c.KL, ct = k & 3, K = col_size(c, k);
    const bool first = k == 0, last = k == c.ncol - 1;
    const int Kp = first ? 0 : col_size(c, k - 1), Kn = last ? 0 : col_size(c, k + 1);
    const int ctn = (k + 1) & 3;
    const auto t2 = Hop<R>::t2(c);
    double amax2 = 0.0;
    for (int i = warp; i < K; i += NWARP) {
        int a0 = -1, a1 = -1, n0 = -1, n1 = -1;
        if (left && !first) col_src(ct, i, Kp, a0, a1);
        if (right && !last) col_src_T(ctn, i, Kn, n0, n1);
        const bool ki = s.kc[i];
        const bool ka0 = a0 >= 0 && s.kp[a0], ka1 = a1 >= 0 && s.kp[a1];
        const bool kn0 = n0 >= 0 && s.kn[n0], kn1 = n1 >= 0 && s.kn[n1];
        for (int l = lane; l < K; l += 32) {
            cx<R> v;
            if (!ki || !s.kc[l]) {
                v = (i == l) ? from_z<R>(1.0, 0.0) : czero<R>();
            } else {
                // the left term as the forward sweep forms it (build_column), so
                // that the left recursion reproduces the forward sweep bit for bit
                cx<R> sig = czero<R>();
                if (left && first) sig = ld_z<R>(c.SigL() + (size_t)i * KL + l);
                if (left && !first) {
                    int b0, b1;
                    col_src(ct, l, Kp, b0, b1);
                    const bool kb0 = b0 >= 0 && s.kp[b0], kb1 = b1 >= 0 && s.kp[b1];
                    if (ka0 && kb0) sig = cadd(sig, glp[(size_t)a0 * KL + b0]);
                    if (ka0 && kb1) sig = cadd(sig, glp[(size_t)a0 * KL + b1]);
                    if (ka1 && kb0) sig = cadd(sig, glp[(size_t)a1 * KL + b0]);
                    if (ka1 && kb1) sig = cadd(sig, glp[(size_t)a1 * KL + b1]);
                    sig = cscale(sig, t2);
                }
                if (right && last) sig = cadd(sig, ld_z<R>(c.SigR() + (size_t)i * c.KR + l));
                if (right && !last) {
                    int m0, m1;
                    col_src_T(ctn, l, Kn, m0, m1);
                    const bool km0 = m0 >= 0 && s.kn[m0], km1 = m1 >= 0 && s.kn[m1];
                    cx<R> w = czero<R>();
                    if (kn0 && km0) w = cadd(w, grn[(size_t)n0 * KL + m0]);
                    if (kn0 && km1) w = cadd(w, grn[(size_t)n0 * KL + m1]);
                    if (kn1 && km0) w = cadd(w, grn[(size_t)n1 * KL + m0]);
                    if (kn1 && km1) w = cadd(w, grn[(size_t)n1 * KL + m1]);
                    sig = cadd(sig, cscale(w, t2));
                }
                v = (i == l) ? from_z<R>(c.z.re - s.eps[i], c.z.im) : czero<R>();
                v = csub(v, sig);
            }
            X[(size_t)i * KL + l] = v;
            const double a2 = (double)cabs2f(v);
            amax2 = (a2 > amax2 || isnan(a2)) ? a2 : amax2;
        }
    }
    return block_max(amax2, s.red);
}

// Column k's matrix (build_A) inverted into Gout; one out-of-line copy for
// the four call sites.  Returns the Gauss-Jordan flags.
template <class R, bool TC64>
static __device__ __noinline__ int build_invert(const ChainCtx& c, int k, bool left, const cx<R>* glp,
                                                bool right, const cx<R>* grn, cx<R>* X, cx<R>* Gout,
                                                SweepSmem<R>& s) {
    const double amax2 = build_A<R>(c, k, left, glp, right, grn, X, s);
    return cta_gj_invert<R, TC64 && std::is_same<R, double>::value>(X, col_size(c, k), c.KL, Gout, c.KL, s.gj, amax2);
}

// Y = Pl W_k (KL x K): Y[r][l] = t sum over the kept sources a of l in column
// k-1 of Pl[r][a]; zero for a removed l.  Ends with a barrier.
template <class R>
__device__ void stencil_left(const ChainCtx& c, int k, const cx<R>* Pl, cx<R>* Y, SweepSmem<R>& s) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int KL = c.KL, ct = k & 3, K = col_size(c, k), Kp = col_size(c, k - 1);
    const auto t = Hop<R>::t(c);
    for (int r = warp; r < KL; r += NWARP)
        for (int l = lane; l < K; l += 32) {
            cx<R> v = czero<R>();
            if (s.kc[l]) {
                int a0, a1;
                col_src(ct, l, Kp, a0, a1);
                if (a0 >= 0 && s.kp[a0]) v = cadd(v, Pl[(size_t)r * KL + a0]);
                if (a1 >= 0 && s.kp[a1]) v = cadd(v, Pl[(size_t)r * KL + a1]);
                v = cscale(v, t);
            }
            Y[(size_t)r * KL + l] = v;
        }
    __syncthreads();
}

// Masks and on-site energies of column k and its neighbours into shared memory.
template <class R>
__device__ void load_cols(const ChainCtx& c, int k, SweepSmem<R>& s) {
    load_col(c, k, s.kc, s.eps);
    load_col(c, k - 1, s.kp, nullptr);
    load_col(c, k + 1, s.kn, nullptr);
    __syncthreads();
}

}  // namespace

template <class R, bool TC>
__global__ void __launch_bounds__(NT, 1)
ldos_kernel(const ChainDev* __restrict__ chains, const int* __restrict__ order, int Kmax, double eta_d,
            const zd* __restrict__ leadout, const int* __restrict__ lead_status,
            const LeadDev* __restrict__ leads, cx<R>* __restrict__ ws, const int* __restrict__ seg_cells,
            double* __restrict__ Tout, double* __restrict__ rho, int32_t* __restrict__ status) {
    SweepSmem<R> s = carve<R>(rgf_dyn_smem, Kmax, TC);
    const int ci = order[blockIdx.x];
    const ChainDev ch = chains[ci];
    const int lst = lead_state(lead_status, ch.lead);
    if (!ch.rem || lst != ST_OK) return;                     // rgf_grad.cu; a failed lead is reported there
    const ChainCtx c = make_ctx(ch, leads[ch.lead], leadout, eta_d);
    const int KL = c.KL, ncol = c.ncol;
    const int Sc = 4 * seg_cells[ci];
    const int nseg = (ncol + Sc - 1) / Sc;
    const size_t B = (size_t)KL * KL;
    cx<R>* base = ws + ch.ws_off;
    cx<R> *X = base, *Y = base + B, *Z = base + 2 * B, *U = base + 3 * B, *Gkk = base + 4 * B;
    cx<R> *gl = base + 5 * B, *Pl = base + 6 * B, *gr = base + 7 * B;
    cx<R>* ckpt = base + 8 * B;                        // gr at column (j + 1) Sc
    cx<R>* seg = ckpt + (size_t)nseg * B;              // Sc + 1 blocks
    double* ldos = rho + ch.grad_off;
    tc::State tst;
    if constexpr (TC) tc_attach<R>(Kmax, s, tst);
    int flag = 0;
    for (int k = ncol - 1; k >= Sc; --k) {
        load_cols(c, k, s);
        flag |= build_invert<R, TC>(c, k, k == 0, nullptr, true, gr, X, gr, s);
        if (k % Sc == 0) copy_blk(ckpt + (size_t)(k / Sc - 1) * B, gr, B);
    }
    for (int j = 0; j < nseg; ++j) {
        const int k0 = j * Sc, k1 = min(ncol, k0 + Sc);
        if (k1 < ncol) copy_blk(seg + (size_t)(k1 - k0) * B, ckpt + (size_t)j * B, B);
        for (int k = k1 - 1; k >= k0; --k) {
            cx<R>* sk = seg + (size_t)(k - k0) * B;
            load_cols(c, k, s);
            flag |= build_invert<R, TC>(c, k, k == 0, nullptr, true, sk + B, X, sk, s);
        }
        for (int k = k0; k < k1; ++k) {
            const cx<R>* sn = seg + (size_t)(k - k0 + 1) * B;
            const int K = col_size(c, k), n = k >> 2, ct = k & 3;
            load_cols(c, k, s);
            flag |= build_invert<R, TC>(c, k, true, gl, true, sn, X, Gkk, s);
            for (int i = threadIdx.x; i < K; i += NT)
                ldos[(size_t)n * c.M + 4 * i + ct] = s.kc[i] ? -to_z(Gkk[(size_t)i * KL + i]).im * kInvPi : 0.0;
            if (k > 0) stencil_left<R>(c, k, Pl, Y, s);     // Y = Pl_{k-1} W_k
            // gl_k and Pl_k (the forward recursion)
            flag |= build_invert<R, TC>(c, k, true, gl, k == ncol - 1, nullptr, X, gl, s);
            if (k == 0) copy_blk(Pl, gl, B);
            else dense_product<R, false, TC && std::is_same<R, double>::value>(KL, K, K, Y, KL, gl, KL, Pl, KL, s);
        }
    }
    if constexpr (TC) {
        if (*(volatile int*)tst.ar.err()) flag |= 4;
    }
    // T from Pl = G_1L of the left recursion
    const double T = trace_T<R>(c, Pl, X, Z, U, s);
    const int st = chain_status(c, flag, T);
    if (st != ST_OK)
        for (size_t e = threadIdx.x; e < (size_t)c.L * c.M; e += NT) ldos[e] = 0.0;
    if (threadIdx.x == 0) {
        Tout[ci] = (st == ST_OK) ? T : NAN;
        if (status) status[ci] = st;
    }
    if constexpr (TC) tc::teardown(tst.ar);
}

size_t ldos_ws_elems(int N, int L, int seg_cells) {
    const size_t KL = (size_t)col_KL(N), nseg = ((size_t)L + seg_cells - 1) / seg_cells;
    return (8 + nseg + 4 * (size_t)seg_cells + 1) * KL * KL;
}

cudaError_t launch_ldos_removed(int precision, const ChainDev* chains, const int* order, int nchains,
                                int Kmax, double eta_device, const void* leadout, const int* lead_status,
                                const LeadDev* leads, void* ws, const int* seg_cells, double* T, double* rho,
                                int32_t* status, cudaStream_t st) {
    const bool tc = precision == 2 || precision == 3;
    const size_t smem = sweep_smem_bytes(Kmax, tc);
    auto run = [&](auto kern, auto* w) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<nchains, NT, smem, st>>>(chains, order, Kmax, eta_device, (const zd*)leadout, lead_status, leads, w,
                                        seg_cells, T, rho, status);
        return cudaGetLastError();
    };
    if (precision == 3) return run(ldos_kernel<double, true>, (zd*)ws);
    if (precision == 2) return run(ldos_kernel<df32, true>, (zf*)ws);
    if (precision == 1) return run(ldos_kernel<df32, false>, (zf*)ws);
    return run(ldos_kernel<double, false>, (zd*)ws);
}

}  // namespace rgf

// rgf_device.cuh -- thread-block (CTA) level dense complex kernels used by the
// RGF sweeps: a tiled GEMM and an in-place Gauss-Jordan inverse with partial
// pivoting.  All matrices are row-major in global memory (L2-resident per
// chain); every routine is called by all threads of the block and ends with a
// __syncthreads().  The block size is RGF_NT threads.
#pragma once

#include <type_traits>

#include "rgf_common.cuh"
#include "rgf_tc.cuh"

namespace rgf {

// ---------------------------------------------------------------------------
// Block reductions
// ---------------------------------------------------------------------------
// Max of a non-negative binary64 value over the block; NaN wins (so that a
// non-finite matrix is noticed).  red: >= NWARP doubles of shared memory.
__device__ __forceinline__ double block_max(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) {
        double w = __shfl_xor_sync(0xffffffffu, v, o);
        v = (isnan(w) || w > v) ? w : v;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double r = red[0];
    for (int w = 1; w < NWARP; ++w) {
        double x = red[w];
        r = (isnan(x) || x > r) ? x : r;
    }
    __syncthreads();
    return r;
}

__device__ __forceinline__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double r = 0.0;
    for (int w = 0; w < NWARP; ++w) r += red[w];
    __syncthreads();
    return r;
}

// ---------------------------------------------------------------------------
// C (m x n) {=, +=} op(A) (m x kd) * op(B) (kd x n)
// op(X) = X or X^T (no conjugation).  64 x 64 output tiles, k-chunks of 8,
// each thread owns a 2 x 4 register tile (columns a quarter of the tile's apart, so
// that neighbouring threads read and write neighbouring entries).  The threads
// are laid over the outputs that a tile has, in order, so that the warps past
// them and the inner entries past kd cost nothing: the FP64 pipe (about two FMAs a
// cycle and SM) bounds it, and a fixed 16 x 32 grid of threads spends four times
// the arithmetic at K = 31, 1.6 times at 51.
// binary64, N = 101, L = 200, 64 energies 92.9 -> 75.6 ms; gradient of N = 61 115 -> 65.
// C must not alias A or B.
// smem: 2 * 8 * 64 elements of cx<R>.
// ---------------------------------------------------------------------------
enum GemmMode { GEMM_SET = 0, GEMM_ADD = 1 };

template <class R, bool TA, bool TB>
__device__ void cta_gemm(int m, int n, int kd, const cx<R>* __restrict__ A, int lda,
                         const cx<R>* __restrict__ B, int ldb, cx<R>* __restrict__ C, int ldc,
                         int mode, cx<R>* sm) {
    cx<R>* As = sm;            // [8][64], k-major
    cx<R>* Bs = sm + 8 * 64;   // [8][64]
    const int tid = threadIdx.x;
    static_assert(NT == 512, "cta_gemm assumes 512 threads");
    for (int i0 = 0; i0 < m; i0 += 64) {
        for (int j0 = 0; j0 < n; j0 += 64) {
            const int mg = (min(64, m - i0) + 1) >> 1, ng = (min(64, n - j0) + 3) >> 2;
            const int ty = tid / ng, tx = tid - ty * ng;
            cx<R> acc[2][4];
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[r][c] = czero<R>();
            for (int k0 = 0; k0 < kd; k0 += 8) {
                {
                    int r, kk;
                    if (TA) { kk = tid >> 6; r = tid & 63; }   // A^T: rows of A are k
                    else    { r = tid >> 3;  kk = tid & 7;  }
                    int gi = i0 + r, gk = k0 + kk;
                    cx<R> v = czero<R>();
                    if (gi < m && gk < kd) v = TA ? A[(size_t)gk * lda + gi] : A[(size_t)gi * lda + gk];
                    As[kk * 64 + r] = v;
                }
                {
                    int kk, c;
                    if (TB) { c = tid >> 3; kk = tid & 7; }
                    else    { kk = tid >> 6; c = tid & 63; }
                    int gk = k0 + kk, gj = j0 + c;
                    cx<R> v = czero<R>();
                    if (gk < kd && gj < n) v = TB ? B[(size_t)gj * ldb + gk] : B[(size_t)gk * ldb + gj];
                    Bs[kk * 64 + c] = v;
                }
                __syncthreads();
                const int kc = ty < mg ? min(8, kd - k0) : 0;
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {
                    if (kk >= kc) break;
                    cx<R> a0 = As[kk * 64 + ty * 2], a1 = As[kk * 64 + ty * 2 + 1];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        cx<R> b = Bs[kk * 64 + tx + c * ng];
                        acc[0][c] = cmac(acc[0][c], a0, b, false);
                        acc[1][c] = cmac(acc[1][c], a1, b, false);
                    }
                }
                __syncthreads();
            }
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                int gi = i0 + ty * 2 + r;
                if (ty >= mg || gi >= m) continue;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    int gj = j0 + tx + c * ng;
                    if (gj >= n) continue;
                    cx<R>* p = C + (size_t)gi * ldc + gj;
                    const cx<R> v = acc[r][c];
                    if (mode == GEMM_SET) *p = v;
                    else *p = cadd(*p, v);
                }
            }
        }
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// Blocked Gauss-Jordan inverse with partial (row) pivoting.
//   A (K x K, leading dim lda, row-major on entry) is destroyed; A^-1 is written
//   to G (row-major, ldg).  The elimination runs on W = A^T, which the
//   row-major input already is when read column-major (W(i, l) = A[l*lda + i]):
//   the columns of W are contiguous, so every column-wise phase below reads
//   and writes contiguous memory.  The copy-out transposes back:
//   A^-1 = (W^-1)^T.
//   No row is ever moved: step j takes the largest entry of column j among the
//   rows that have not been pivots yet, row p_j, scales it by 1/W[p_j][j]
//   (keeping 1/W[p_j][j] in column j) and eliminates column j from every other
//   row (keeping -W[i][j]/W[p_j][j] in column j).  With S the array at the end,
//   W^-1[j][p_m] = S[p_j][m]: the copy-out applies p on both sides.
//   Pivots are taken in panels of b columns.  A panel lives in registers: thread
//   (l, g) of the block holds column l of rows g, g + 512/b, ... (four of them),
//   and a pivot costs two block barriers.  Before the first, the threads of
//   column j publish it (the multipliers c_j, [b][K] in shared memory) and the
//   sixteen of row p_j form the reciprocal and publish the scaled row; after it
//   every thread updates its four entries and those of column j + 1 rank the
//   candidates for the next pivot (a shared-memory atomic maximum on a (|a|^2 in
//   binary32, position) key), which the second barrier completes.  What bounds a
//   pivot is that serial chain, most of it the double-float reciprocal: about
//   3.9 thousand cycles at K = 123, where the arithmetic is 830 (with a team of
//   warps per panel and rows moved: 5 thousand).  The whole inverse with
//   tensor-core updates, one block alone: K = 123 609 -> 515 us, K = 201 2.76 ->
//   2.07 ms.
//   The columns outside the panel then take the panel's b steps at once.  Their
//   pivot rows first: the forward substitution
//       x_r = (W[p_r][l] - sum_{q < r} c_q[p_r] x_q) / W[p_r][j_r]
//   is applied through its b x b inverse T (unit lower triangular entries of at
//   most one times the reciprocals, by the choice of the pivots; formed by one
//   warp per two columns), x = T W[p][l], so that no barrier stands between its
//   steps.  Then one rank-b update of every row, W[i][l] -= sum_q c_q[i] x_q, the
//   pivot rows starting from x_r with their multipliers q <= r set to zero (their
//   later steps' eliminations): on the tensor cores (tc::zupdate) or on the FP32
//   / FP64 pipes.
//   Pivot reciprocals are formed in the working precision (a Newton step on the
//   binary32 reciprocal for double-float).  The pivot test runs in binary32 and
//   falls back to binary64 near its limits.
// Returns a flag: bit 0 = zero pivot, or a pivot below 64 u sqrt(amax2) with
// amax2 = max |A_ij|^2 supplied by the caller (0 disables the test); bit 1 =
// non-finite pivot.
// ---------------------------------------------------------------------------
// Ranking key of a pivot candidate: |a|^2 in binary32 (NaN ranked as +inf)
// in the high word, the complement of the row's position in the low word -- the
// largest key is the largest magnitude and, among equal magnitudes, the lowest
// position.
template <class R>
__device__ __forceinline__ unsigned long long pivot_key(cx<R> v, int i) {
    float m = cabs2f(v);
    if (isnan(m)) m = INFINITY;
    return ((unsigned long long)__float_as_uint(m) << 32) | (0xFFFFFFFFu - (unsigned)i);
}

// Broadcast of a lane's complex value across the warp.
__device__ __forceinline__ zd shfl_from(zd v, int src) {
    return {__shfl_sync(0xffffffffu, v.re, src), __shfl_sync(0xffffffffu, v.im, src)};
}
__device__ __forceinline__ zf shfl_from(zf v, int src) {
    return {{__shfl_sync(0xffffffffu, v.re.hi, src), __shfl_sync(0xffffffffu, v.re.lo, src)},
            {__shfl_sync(0xffffffffu, v.im.hi, src), __shfl_sync(0xffffffffu, v.im.lo, src)}};
}

template <class R>
struct GJSmem {
    cx<R>* panel;    // [bmax][Kmax]  pivot rows outside the panel before the substitution
    cx<R>* panel2;   // [gj_panel2_elems]  T [bmax][bmax], then the published pivot rows [2][bmax]
    cx<R>* mult;     // [bmax][Kmax]  multipliers c_jj[i] at mult[jj*K + i]
    cx<R>* xrow;     // [bmax][Kmax]  substituted pivot rows outside the panel
    cx<R>* pinv;     // [bmax]   pivot reciprocals
    int* perm;       // [Kmax]   p_j
    int* ctl;        // [4]: [1] = the pivot flags
    unsigned long long* key;   // [3]  pivot keys, one per step, rotating
    int bmax;        // panel width, a power of two
    tc::State* tcs;  // tensor-core state for the rank-b update, or nullptr
};

// Panels up to this width update on the FP64 pipe also where the block holds the
// tensor cores: a narrow panel's update costs the pipe little (8 K^2 b operations) and
// zupdate its passes, barriers and slicing all the same.  FP64_TC, 16 energies, tensor
// cores / pipe, ms: single columns, panel 2, N = 41, L = 20 11.1 / 5.6, N = 64 20.5 / 8.6,
// N = 245, L = 4 60.9 / 40.9; panel 4 7.6 / 5.2, 12.5 / 7.7, 43.9 / 39.9; the widest
// panel that fits at N = 701 (4 energies, L = 2) 620 / 571, N = 1001 1585 / 1500.  Double-float
// panels (N = 245, panel 2 34.2 / 35.9, N = 1001 1325 / 1361) stay on the tensor cores.
constexpr int kPipePanel = 4;

constexpr int GJ_ROWS = 4;           // rows of a panel column per thread (pairs: see the update)

// TC64: with R = double, run the rank-b updates on the tensor cores (binary64
// slicing) when the block holds them.
template <class R, bool TC64 = false>
__device__ __forceinline__ int cta_gj_invert(cx<R>* __restrict__ A, int K, int lda, cx<R>* __restrict__ G,
                                             int ldg, GJSmem<R> s, double amax2 = 0.0) {
    constexpr bool kF64 = std::is_same<R, double>::value;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int bm = s.bmax;
    while (K * bm > GJ_ROWS * NT) bm >>= 1;         // four rows per thread
    cx<R>* Cm = s.mult;
    cx<R>* Xr = s.xrow;
    const double tiny2 = amax2 * (64.0 * Unit<R>::u) * (64.0 * Unit<R>::u);
    const float tiny2f = (float)tiny2;
    const int l = tid & (bm - 1), g = tid / bm, RG = NT / bm;
    // groups of rows that this warp holds below K: u = 0 .. nu - 1
    const int gw = (warp << 5) / bm, nu = gw >= K ? 0 : min(GJ_ROWS, (K - gw + RG - 1) / RG);
    // Position of row g + u RG, as if step j had swapped its pivot row with the
    // row in position j: rows in positions before j have been pivots, and of
    // equal candidates the lowest position wins.
    int pos[GJ_ROWS];
#pragma unroll
    for (int u = 0; u < GJ_ROWS; ++u) pos[u] = g + u * RG;
    for (int i = tid; i < K; i += NT) s.perm[i] = i;
    if (tid == 0) s.ctl[1] = 0;
    if (tid < 3) s.key[tid] = 0ull;
    __syncthreads();
    for (int j0 = 0; j0 < K; j0 += bm) {
        const int bb = min(bm, K - j0);
        cx<R>* Tm = s.panel2;                   // [bb][bm]
        cx<R>* prow = s.panel2 + bm * bm;       // [2][bm]
        cx<R> a[GJ_ROWS];
        {
            unsigned long long kmax = 0ull;
#pragma unroll
            for (int u = 0; u < GJ_ROWS; ++u) {
                const int i = g + u * RG;
                a[u] = czero<R>();
                if (i < K && l < bb) {
                    a[u] = A[(size_t)(j0 + l) * lda + i];
                    if (l == 0 && pos[u] >= j0) kmax = max(kmax, pivot_key(a[u], pos[u]));
                }
            }
            if (kmax) atomicMax(&s.key[j0 % 3], kmax);
        }
        __syncthreads();
        for (int jj = 0; jj < bb; ++jj) {
            const int j = j0 + jj;
            const int q = (int)(0xFFFFFFFFu - (unsigned)(s.key[j % 3] & 0xFFFFFFFFull));
            const int p = s.perm[q];
            const int gp = p & (RG - 1), up = p / RG;
            if (l == jj) {                      // the pivot column as it is: the multipliers
#pragma unroll
                for (int u = 0; u < GJ_ROWS; ++u) {
                    const int i = g + u * RG;
                    if (i < K) Cm[jj * K + i] = a[u];
                }
            }
            if ((gp * bm) >> 5 == warp) {       // the warp that holds row p
                cx<R> v = a[0];
#pragma unroll
                for (int u = 1; u < GJ_ROWS; ++u)
                    if (u == up) v = a[u];
                cx<R> pv = shfl_from(v, (gp * bm + jj) & 31);
                int bad = 0;
                const float df = cabs2f(pv);
                if (!cfinite(pv)) {
                    bad = 2;
                } else if (!(df >= 1e-30f && df <= 1e30f && df >= 2.0f * tiny2f)) {
                    const double d = cabs2(pv);       // borderline: decide in binary64
                    if (!isfinite(d)) bad = 2;
                    else if (!(d > 0.0)) bad = 1;
                    else if (d < tiny2) bad = 1;
                }
                if (bad) pv = from_z<R>(1.0, 0.0);
                const cx<R> inv = crecip(pv);
                if (g == gp && l < bb) {
                    prow[(jj & 1) * bm + l] = l == jj ? inv : cmul(v, inv);
                    if (l == jj) {
                        s.ctl[1] |= bad;
                        s.pinv[jj] = inv;
                        s.key[(j + 2) % 3] = 0ull;   // read one step ago, filled the next
                    }
                }
            }
            __syncthreads();
            unsigned long long kmax = 0ull;
            if (l < bb && nu > 0) {
                const cx<R> r = prow[(jj & 1) * bm + l];
                cx<R> m[GJ_ROWS];
#pragma unroll
                for (int u = 0; u < GJ_ROWS; ++u) {
                    m[u] = Cm[jj * K + min(g + u * RG, K - 1)];
                    if (l == jj) a[u] = czero<R>();
                }
                // No branch between the two rows of a pair: their chains of
                // dependent operations run side by side.  Groups past K are
                // left out: at K = 51 they are half the arithmetic, at K = 6 most.
                if (nu > 1) {
                    m[0] = cmac(a[0], m[0], r, true);
                    m[1] = cmac(a[1], m[1], r, true);
                } else {
                    m[0] = cmac(a[0], m[0], r, true);
                }
                if (nu > 2) {
                    m[2] = cmac(a[2], m[2], r, true);
                    m[3] = cmac(a[3], m[3], r, true);
                }
                const int pu = g == gp ? up : GJ_ROWS;
#pragma unroll
                for (int u = 0; u < GJ_ROWS; ++u) {
                    a[u] = u == pu ? r : m[u];
                    if (pos[u] == j) pos[u] = q;
                    if (u == pu) pos[u] = j;
                }
                if (g == gp && l == jj) {
                    s.perm[q] = s.perm[j];
                    s.perm[j] = p;
                }
                if (l == jj + 1) {
#pragma unroll
                    for (int u = 0; u < GJ_ROWS; ++u) {
                        const unsigned long long key = pivot_key(a[u], pos[u]);
                        if (g + u * RG < K && pos[u] > j) kmax = max(kmax, key);
                    }
                }
            }
            for (int o = bm; o < 32; o <<= 1) kmax = max(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
            if (lane == jj + 1 && kmax) atomicMax(&s.key[(j + 1) % 3], kmax);
            __syncthreads();
        }
        // the reduced panel back
#pragma unroll
        for (int u = 0; u < GJ_ROWS; ++u) {
            const int i = g + u * RG;
            if (i < K && l < bb) A[(size_t)(j0 + l) * lda + i] = a[u];
        }
        const int nown = K - bb;                // columns outside the panel
        if (nown > 0) {
            auto own_col = [&](int c) { return c < j0 ? c : c + bb; };
            cx<R>* Wp = s.panel;                // [bb][K]
            // their pivot rows, one column after the other
            for (int e = tid; e < bb * nown; e += NT) {
                const int c = e / bb, q = e - c * bb, lc = own_col(c);
                Wp[q * K + lc] = A[(size_t)lc * lda + s.perm[j0 + q]];
            }
            // T: half a warp per column q, lane r its row
            {
                const int r = lane & 15, q = 2 * warp + (lane >> 4);
                cx<R> t = r == q ? from_z<R>(1.0, 0.0) : czero<R>();
                const int pr = s.perm[j0 + min(r, bb - 1)];
                if (2 * warp < bb)
                    for (int st = 2 * warp; st < bb; ++st) {
                        const cx<R> ts = cmul(shfl_from(t, (lane & 16) + st), s.pinv[st]);
                        if (r == st) t = ts;
                        else if (r > st) t = cmac(t, Cm[st * K + pr], ts, true);
                    }
                if (q < bb && r < bb) Tm[r * bm + q] = t;
            }
            __syncthreads();
            // x = T W[p][l]: four rows of one column per thread, r, 7 - r, 8 + r,
            // 15 - r (for b = 16), which have the same number of terms together
            {
                const int h = (bm + 3) >> 2, half = max(bm >> 1, 1);
                for (int e = tid; e < h * nown; e += NT) {
                    const int rg = e / nown, lc = own_col(e - rg * nown);
                    int rr[4];
                    rr[0] = rg;
                    rr[1] = half - 1 - rg;
                    rr[2] = half + rg;
                    rr[3] = bm - 1 - rg;
                    if (bm <= 2) { rr[1] = bm; rr[2] = 1; rr[3] = bm; }        // rows 0 and 1 only
                    cx<R> x[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) x[u] = czero<R>();
                    for (int q = 0; q < bb; ++q) {
                        const cx<R> wv = Wp[q * K + lc];
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (q <= rr[u] && rr[u] < bb) x[u] = cmac(x[u], Tm[rr[u] * bm + q], wv, false);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (rr[u] < bb) {
                            Xr[rr[u] * K + lc] = x[u];
                            A[(size_t)lc * lda + s.perm[j0 + rr[u]]] = x[u];
                        }
                }
            }
            // the pivot rows' multipliers of their own and earlier steps: none
            for (int e = tid; e < bb * bb; e += NT) {
                const int r = e / bb, q = e - r * bb;
                if (q <= r) Cm[q * K + s.perm[j0 + r]] = czero<R>();
            }
            __syncthreads();
            bool tc_done = false;
            if constexpr (std::is_same<R, df32>::value || TC64) {
                if (s.tcs && !(kF64 && bm <= kPipePanel)) {
                    const int cm_off = tc::dyn_off(Cm), xr_off = tc::dyn_off(Xr);
                    for (int r0 = 0; r0 < K; r0 += 128)
                        s.tcs->phase = tc::zupdate<cx<R>>(cm_off, xr_off, K, bb, A, lda, r0, min(128, K - r0), j0,
                                                          nown, s.tcs->ar, s.tcs->phase);
                    tc_done = true;
                }
            }
            const int Kh = (K + 1) >> 1, Ch = tc_done ? 0 : (nown + 1) >> 1;
            for (int tt = tid; tt < Kh * Ch; tt += NT) {
                const int i0 = 2 * (tt % Kh), c0 = 2 * (tt / Kh);
                const bool ok_i1 = i0 + 1 < K, ok_c1 = c0 + 1 < nown;
                const int l0 = own_col(c0);
                const int l1 = ok_c1 ? own_col(c0 + 1) : l0;
                cx<R>* c0p = A + (size_t)l0 * lda;
                cx<R>* c1p = A + (size_t)l1 * lda;
                cx<R> a00 = c0p[i0], a01 = czero<R>(), a10 = czero<R>(), a11 = czero<R>();
                if (ok_c1) a01 = c1p[i0];
                if (ok_i1) {
                    a10 = c0p[i0 + 1];
                    if (ok_c1) a11 = c1p[i0 + 1];
                }
                for (int jj = 0; jj < bb; ++jj) {
                    const cx<R> p0 = Cm[jj * K + i0];
                    const cx<R> p1 = ok_i1 ? Cm[jj * K + i0 + 1] : czero<R>();
                    const cx<R> m0 = Xr[jj * K + l0];
                    const cx<R> m1 = ok_c1 ? Xr[jj * K + l1] : czero<R>();
                    a00 = cmac(a00, p0, m0, true);
                    a01 = cmac(a01, p0, m1, true);
                    a10 = cmac(a10, p1, m0, true);
                    a11 = cmac(a11, p1, m1, true);
                }
                c0p[i0] = a00;
                if (ok_c1) c1p[i0] = a01;
                if (ok_i1) {
                    c0p[i0 + 1] = a10;
                    if (ok_c1) c1p[i0 + 1] = a11;
                }
            }
        }
        __syncthreads();
    }
    // G[p_m][j] = S[p_j][m]
    for (int m = warp; m < K; m += NWARP) {
        const cx<R>* col = A + (size_t)m * lda;
        cx<R>* grow = G + (size_t)s.perm[m] * ldg;
        for (int j = lane; j < K; j += 32) grow[j] = col[s.perm[j]];
    }
    const int flag = s.ctl[1];
    __syncthreads();
    return flag;
}

}  // namespace rgf

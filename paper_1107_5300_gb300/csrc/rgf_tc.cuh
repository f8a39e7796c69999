// rgf_tc.cuh -- complex matrix products on the tcgen05 tensor cores at
// double-float accuracy (the dense contractions of the RGF step: the rank-b
// updates of the slice inverse and the corner-strip product of Eq. 5).
//
// Method: exact digit slicing (the Ozaki scheme; K. Ozaki, T. Ogita, S. Oishi,
// S. M. Rump, Numer. Algorithms 59 (2012) 95).  Each row of A (each column of
// B) gets a power-of-two scale 2^e with |entries| < 2^e.  A real double-float
// value x of that row is written as a sum of S signed base-256 digits,
//     x ~ 2^(e-7) sum_i d_i 2^(-8 i),   d_i integer, |d_i| <= 128,
// every digit exact in f16, the type of the tiles.  A product of digit tiles i
// (of A) and j (of B) carries the weight 2^(-8 (i + j)), applied when the
// accumulators are read; the tensor core accumulates it in binary32:
//     level l = i + j = 0 .. 3    one TMEM accumulator each.  Every term of a
//                                 level is an integer of at most 2^14, and a
//                                 level sums at most 4 x 256 of them (groups of
//                                 up to 128 complex
//                                 inner entries): at most 2^24, exact;
//     level 4                     two accumulators (its pairs with even and
//                                 with odd i, at most 3 x 256 terms): exact;
//     levels 5, 6                 one accumulator each.  The tensor core's
//                                 binary32 additions drop low-order bits at
//                                 every MMA (measured: levels 3 to 6 in one
//                                 accumulator cost 2^-44 of the scale, 4 to 6
//                                 about 2^-48 over the 288 MMAs of a 123-deep
//                                 product); at 2^-40 of the scale these
//                                 levels lose less than 2^-55;
//     levels >= S                 dropped (below 2^-(8S-1) of the scale).
// The eight accumulators are summed in double-float and scaled back by
// 2^(e_row - 7) 2^(e_col - 7).  With S = 7 digits (55 bits)
// the product is accurate to a few units of 2^-48 of (row max x column max x
// inner dimension), the accuracy of the double-float arithmetic it replaces.
//
// Complex products use the real 2 x 2 block form C' = A' B' with
//     A'[m][2k] = Re A[m][k],  A'[m][2k+1] = Im A[m][k],
//     B'[2k][2n] = Re B[k][n], B'[2k+1][2n] = -Im B[k][n]      (C'[m][2n] = Re C),
//     B'[2k][2n+1] = Im B[k][n], B'[2k+1][2n+1] = Re B[k][n]   (C'[m][2n+1] = Im C),
// so one MMA chain (M = 128, N = 2 x columns, K = 16 per instruction, f16 x
// f16 -> f32) gives both parts, side by side in TMEM.  Operands are staged in shared memory by the
// threads that slice them (K-major, no swizzle: 8-row x 16-byte core
// matrices, 128 B apart along K and 256 B apart along M/N); one elected
// lane issues the MMAs and commits them to an mbarrier; the accumulators
// live in TMEM (8 x 64 columns) and are read back with tcgen05.ld.
#pragma once

#include <cuda_fp16.h>

#include <type_traits>

#include "rgf_common.cuh"

namespace rgf {
namespace tc {

constexpr int S = 7;                 // digits per real value
constexpr int TILE = 128 * 16;       // elements of one digit tile of A' (128 rows x 16 k)
constexpr int MAXC = 32;             // complex output columns per pass
constexpr int TILEB = 2 * MAXC * 16; // elements of one digit tile of B' (64 rows x 16 k)
constexpr int NACC = 8;              // TMEM accumulators: levels 0..3, level 4 twice, 5, 6
constexpr int ACOLS = 2 * MAXC;      // TMEM columns per accumulator (8 x 64 = 512)
constexpr int KCH = 8;               // complex inner entries per chunk (16 real-block k)
constexpr int KGRP = 128;            // complex inner entries per exact accumulation group
constexpr int NBUF = 2;              // chunks whose digit tiles are staged at a time

// The MMAs of a chunk: digit i of A' times nd consecutive digits j0 .. of B'
// (their tiles lie one after another, so they are one operand of N = 64 nd
// rows) into nd consecutive accumulators.  Accumulators in TMEM order: levels 0,
// 1, 2, 3, 4 with even i, 5, 6, 4 with odd i.  An MMA of M = 128 takes 64 cycles
// at N = 64, 71 at N = 128, about 100 at 192 and 130 at 256 (A' is read anew
// for each), so these 13 take 1.1 thousand cycles where 28 of N = 64 take 1.8.
struct MmaOp {
    int i, j0, nd, acc;
};
constexpr int NMMA = 13;
__device__ constexpr MmaOp kMma[NMMA] = {{0, 0, 4, 0}, {0, 4, 3, 4}, {1, 0, 3, 1}, {1, 3, 1, 7}, {1, 4, 2, 5},
                                         {2, 0, 2, 2}, {2, 2, 3, 4}, {3, 0, 1, 3}, {3, 1, 1, 7}, {3, 2, 2, 5},
                                         {4, 0, 3, 4}, {5, 0, 2, 5}, {6, 0, 1, 6}};

// Byte offsets inside the tensor-core area of shared memory.
constexpr int OFF_A = 0;                            // [NBUF][S][TILE] f16 digit tiles of A'
constexpr int OFF_B = OFF_A + NBUF * S * TILE * 2;  // [NBUF][S][TILEB] f16 digit tiles of B'
constexpr int OFF_RSC = OFF_B + NBUF * S * TILEB * 2;   // [128] row slicing scales 2^(7-e)
constexpr int OFF_RFAC = OFF_RSC + 128 * 4;         // [128] row output factors 2^(e-7)
constexpr int OFF_CSC = OFF_RFAC + 128 * 4;         // [3][MAXC] column slicing scales of three passes
constexpr int OFF_CFAC = OFF_CSC + 3 * MAXC * 4;    // [3][MAXC] their output factors
constexpr int OFF_BAR = OFF_CFAC + 3 * MAXC * 4;    // mbarriers (8 bytes each):
constexpr int BAR_EMPTY = 0;                        //   [2] a chunk's MMAs (zupdate: a pass's) are complete
constexpr int BAR_FULL = 2;                         //   [2] a chunk's digit tiles are written
constexpr int BAR_UFULL = 4;                        //   [2] zupdate: a pass's digit tiles
constexpr int BAR_UDRAINED = 6;                     //   [2] zupdate: a pass's accumulators are read
constexpr int BAR_DRAINED = 8;                      //   a pass's accumulators are read
constexpr int BAR_DONE = 9;                         //   a pass's MMAs are complete
constexpr int BAR_LAST = 10;                        //   the MMAs in flight after a timeout
constexpr int NBAR = 11;
__host__ __device__ constexpr uint32_t bar_count(int i) {
    return i < BAR_FULL ? 1u : i < BAR_UFULL ? 12u : i < BAR_UDRAINED ? 4u : i < BAR_DONE ? (uint32_t)NWARP : 1u;
}
constexpr int OFF_LIMIT = OFF_BAR + 8 * NBAR;             // completion-wait limit, device clock cycles
constexpr int OFF_TSLOT = OFF_LIMIT + 8;            // TMEM base address (tcgen05.alloc)
constexpr int OFF_ERR = OFF_TSLOT + 4;              // sticky: an MMA wait gave up
constexpr int OFF_SKIP = OFF_ERR + 4;               // self-test: completion commits left out
constexpr int BYTES = (OFF_SKIP + 4 + 15) / 16 * 16;
static_assert(OFF_BAR % 8 == 0 && OFF_LIMIT % 8 == 0 && BYTES % 16 == 0, "tensor-core area layout");

// Default limit of a completion wait: about a second of device clock.
constexpr long long kWaitLimit = 2000000000ll;

__host__ __device__ constexpr size_t smem_bytes() { return (size_t)BYTES; }

}  // namespace tc
}  // namespace rgf

// The block's dynamic shared memory (every extern __shared__ array aliases it).
extern __shared__ __align__(1024) unsigned char rgf_dyn_smem[];

namespace rgf {
namespace tc {

__device__ __forceinline__ uint32_t su32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Byte offset of a shared-memory pointer from the start of dynamic shared memory.
__device__ __forceinline__ int dyn_off(const void* p) { return (int)(su32(p) - su32(rgf_dyn_smem)); }

// The tensor-core area, `off` bytes into dynamic shared memory.  Passed by
// value (one integer); every accessor is a shared-memory address.
struct Area {
    int off;
    __device__ unsigned char* base() const { return rgf_dyn_smem + off; }
    __device__ __half* a(int buf) const { return reinterpret_cast<__half*>(base() + OFF_A) + buf * (S * TILE); }
    __device__ __half* b(int buf) const { return reinterpret_cast<__half*>(base() + OFF_B) + buf * (S * TILEB); }
    __device__ float* rsc() const { return reinterpret_cast<float*>(base() + OFF_RSC); }
    __device__ float* rfac() const { return reinterpret_cast<float*>(base() + OFF_RFAC); }
    __device__ float* csc(int pass) const { return reinterpret_cast<float*>(base() + OFF_CSC) + (pass % 3) * MAXC; }
    __device__ float* cfac(int pass) const { return reinterpret_cast<float*>(base() + OFF_CFAC) + (pass % 3) * MAXC; }
    __device__ unsigned long long* bar(int i) const { return reinterpret_cast<unsigned long long*>(base() + OFF_BAR) + i; }
    __device__ long long* limit() const { return reinterpret_cast<long long*>(base() + OFF_LIMIT); }
    __device__ int* skip() const { return reinterpret_cast<int*>(base() + OFF_SKIP); }
    __device__ uint32_t* tslot() const { return reinterpret_cast<uint32_t*>(base() + OFF_TSLOT); }
    __device__ int* err() const { return reinterpret_cast<int*>(base() + OFF_ERR); }
};

// The area plus the parities of the mbarriers' next phases (bit i: mbarrier i).
struct State {
    Area ar;
    uint32_t phase;
};

// Element offset of (row r, k) inside one 128 x 16 K-major tile.
__device__ __forceinline__ int tile_off(int r, int k) {
    return (r >> 3) * 128 + (k >> 3) * 64 + (r & 7) * 8 + (k & 7);
}

// Shared-memory matrix descriptor: start address, leading-dimension byte
// offset 128 (next core matrix along K), stride-dimension byte offset 256
// (next 8-row group), descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t sdesc(const void* p) {
    return (uint64_t)((su32(p) >> 4) & 0x3FFFu) | ((uint64_t)(128 >> 4) << 16) |
           ((uint64_t)(256 >> 4) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: D f32, A and B f16, both K-major,
// M = 128, N = n (multiple of 16, <= 256).
__device__ __forceinline__ uint32_t idesc(int n) {
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 :: "r"(d), "l"(a), "l"(b), "r"(id), "r"(acc) : "memory");
}

// One lane of the (converged) warp; the same one every time.  The compiler
// issues a tcgen05.mma under this predicate directly; under an ordinary
// one-thread branch it takes 144 cycles each.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
constexpr int ISSUE_WARP = NWARP - 1;      // the warp whose elected lane issues the MMAs

__device__ __forceinline__ void commit(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 :: "r"(su32(bar)) : "memory");
}

__device__ __forceinline__ bool try_wait(unsigned long long* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(su32(bar)), "r"(parity) : "memory");
    return ok != 0;
}

// 32 lanes x 4 consecutive columns of TMEM (this warp's lane quarter).
__device__ __forceinline__ void ld4(uint32_t addr, float* v) {
    uint32_t r[4];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = __uint_as_float(r[j]);
}
__device__ __forceinline__ void ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Allocates all 512 TMEM columns (warp 0) and initialises the mbarriers, the
// completion-wait limit and the self-test switch (skip != 0: the completion of
// the MMAs is never committed, so the first wait runs into its limit).  Must
// be called by every thread of the block (it ends with a barrier); the block
// must be the only one on its SM that uses TMEM.  Returns the initial phase.
__device__ inline uint32_t setup(Area ar, long long limit = kWaitLimit, int skip = 0) {
    if ((threadIdx.x >> 5) == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;"
                     :: "r"(su32(ar.tslot())) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int i = 0; i < NBAR; ++i) {
            const uint32_t count = bar_count(i);
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(su32(ar.bar(i))), "r"(count) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        *ar.err() = 0;
        *ar.limit() = limit;
        *ar.skip() = skip;
    }
    fence_before();
    __syncthreads();
    fence_after();
    return 0u;
}

// Releases TMEM.  Every thread.  If a completion wait gave up, MMAs may still
// be in flight: the issuing thread commits them to the second mbarrier and the
// block waits for it (bounded by the default limit) before the release.
__device__ inline void teardown(Area ar) {
    fence_before();
    __syncthreads();
    if (*(volatile int*)ar.err()) {
        if (__shfl_sync(0xffffffffu, threadIdx.x >> 5, 0) == ISSUE_WARP) {
            if (elect_one()) commit(ar.bar(BAR_LAST));
            __syncwarp();
        }
        const long long t0 = clock64();
        while (!try_wait(ar.bar(BAR_LAST), 0u) && clock64() - t0 <= kWaitLimit) {
        }
        fence_after();
        fence_before();
        __syncthreads();
    }
    if ((threadIdx.x >> 5) == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" :: "r"(*ar.tslot()) : "memory");
}

// Waits for the phase of parity `par` of mbarrier i; gives up after the block's
// limit (about a second of device clock by default) and sets the sticky error
// flag, after which later waits return at once.
// Returns whether the phase is complete (a warp whose wait gave up arrives
// nowhere any more: its arrivals would run ahead of the phases).
__device__ __forceinline__ bool wait_bar(Area ar, int i, uint32_t par) {
    unsigned long long* bar = ar.bar(i);
    if (try_wait(bar, par)) return true;
    const long long t0 = clock64();
    while (!try_wait(bar, par)) {
        if (*(volatile int*)ar.err()) return false;
        if (clock64() - t0 > *(volatile long long*)ar.limit()) *(volatile int*)ar.err() = 1;
    }
    return true;
}
__device__ __forceinline__ void arrive(unsigned long long* bar, uint32_t count) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" :: "r"(su32(bar)), "r"(count) : "memory");
}

// The S signed base-256 digits d_i of a value v below 2^e in magnitude, from
// X = round(v 2^(55 - e)) (|X| <= 2^55): balanced digits are the bytes of
// X + 0x0080808080808080, each less 128 (d_0: the top 16 bits, less 128), so
// v 2^(7 - e) ~ sum_i d_i 2^(-8 i) with d_i in [-128, 127], d_0 in [-128, 128].
// word_*: that sum's two halves.
//
// Double-float (h, l), slicing scale sc = 2^(7-e) (|h sc| < 128): the top sixteen
// bits of h, then its next 22 and those of l beside them, then what is left of
// both, each by adding 1.5 2^23: X to within 0.52 units.  The additions' offsets
// cancel in the integer sums (modulo 2^32, where the high half ends up).
__device__ __forceinline__ void words(float h, float l, float sc, uint32_t& hi, uint32_t& lo) {
    const float M = 12582912.0f, s8 = sc * 256.0f;
    const float t0 = __fmaf_rn(h, s8, M), f0 = __fsub_rn(t0, M);
    const float r0 = __fmaf_rn(h, s8, -f0);                       // exact, |r0| <= 1/2
    const float t1 = __fmaf_rn(r0, 4194304.0f, M), f1 = __fsub_rn(t1, M);
    const float r1 = __fmaf_rn(r0, 4194304.0f, -f1);              // exact, |r1| <= 1/2
    const float z = __fmul_rn(__fmul_rn(l, s8), 4194304.0f);      // |z| <= 2^13
    const float tz = __fadd_rn(z, M), rz = __fsub_rn(z, __fsub_rn(tz, M));
    const float t2 = __fadd_rn(__fmaf_rn(r1, 262144.0f, __fmul_rn(rz, 262144.0f)), M);
    const int i1 = (int)((uint32_t)__float_as_int(t1) + (uint32_t)__float_as_int(tz) - 0x96800000u);
    // X + bias = i0 2^40 + i1 2^18 + (i2 + 0x80808080) + 0x00808080 2^32
    const long long x = (long long)i1 * (1 << 18) +
                        (long long)(unsigned long long)((uint32_t)__float_as_int(t2) + (0x80808080u - 0x4B400000u));
    hi = (uint32_t)((unsigned long long)x >> 32) + ((uint32_t)__float_as_int(t0) << 8) + (0x00808080u - 0x40000000u);
    lo = (uint32_t)x;
}

// Binary64 v (|v| < 2^e), slicing scale sc = 2^(7-e): X from the significand by
// a shift, its rounding being the only error (half a unit of 2^(-48) of sc's
// unit, below the lowest digit).  Zero / subnormal v, or sc = 0, give zero.
__device__ __forceinline__ void words(double v, float sc, uint32_t& hi, uint32_t& lo) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int E = (int)((b >> 52) & 0x7FFull);
    const unsigned scb = __float_as_uint(sc);
    long long X = 0;
    if (E != 0 && E != 2047 && (scb & 0x7F800000u) != 0u) {
        const int e = 134 - (int)((scb >> 23) & 0xFFu);
        const unsigned long long M = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
        const int sh = E - 1020 - e;              // X = M 2^sh, sh <= 2
        unsigned long long mag = 0;
        if (sh >= 0) mag = M << sh;
        else if (sh > -60) mag = (M + (1ull << (-sh - 1))) >> (-sh);
        X = (b >> 63) ? -(long long)mag : (long long)mag;
    }
    X += 0x0080808080808080ll;
    hi = (uint32_t)((unsigned long long)X >> 32);
    lo = (uint32_t)X;
}

// The S pairs (Re low, Im high) of f16 digits of a complex value from its words:
// a byte b below f16's 1024 is 1024 + b, and one packed addition takes 1152 off.
__device__ __forceinline__ uint32_t digit_pair(uint32_t y) {
    uint32_t r;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(y), "r"(0xE480E480u));
    return r;
}
// Digits 2 h + 1 and 2 h + 2 (h = 0, 1, 2) of a complex value with words w (Re
// high, Re low, Im high, Im low), and digit 0.
__device__ __forceinline__ void two_digits(const uint32_t* w, int h, uint32_t& p, uint32_t& q) {
    const uint32_t c = 0x64646464u;
    const uint32_t x = h == 0 ? __byte_perm(w[0], w[2], 0x4051) : __byte_perm(w[1], w[3], h == 1 ? 0x6273 : 0x4051);
    p = digit_pair(__byte_perm(x, c, 0x4140));
    q = digit_pair(__byte_perm(x, c, 0x4342));
}
__device__ __forceinline__ uint32_t digit_0(const uint32_t* w) {
    return digit_pair(__byte_perm(w[0], w[2], 0x7632) + 0x64006400u);
}

// Max with NaN propagation (non-negative arguments).
__device__ __forceinline__ float nmax(float a, float b) { return (isnan(b) || b > a) ? b : a; }

// Slicing scale 2^(7-e) and output factor 2^(e-7) for a row / column maximum
// mx, with e the least integer such that mx < 2^e (from the exponent field:
// mx in [2^(E-127), 2^(E-126)) for a normal binary32 with biased exponent E).
__device__ __forceinline__ void scales(float mx, float& sc, float& fac) {
    const unsigned E = (__float_as_uint(mx) >> 23) & 0xFFu;
    if (!(mx <= 3.0e38f)) {          // NaN or Inf: poison the outputs of this row / column
        sc = 1.0f;
        fac = __int_as_float(0x7fc00000);
    } else if (E < 27u) {            // below 2^-100 (zeros, subnormals): treat as zero
        sc = 0.0f;
        fac = 0.0f;
    } else {
        const int e = (int)E - 126;
        sc = __int_as_float((134 - e) << 23);
        fac = __int_as_float((120 + e) << 23);
    }
}

// ---------------------------------------------------------------------------
// Binary64 operands (accessors with kF64 = true).  The scale of a row / column
// comes from the largest binary64 exponent field in it, and the digits of a
// value from its 53-bit integer significand: integer arithmetic only, no work
// on the FP64 pipe.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned exp64(double v) {
    return (unsigned)((unsigned long long)__double_as_longlong(v) >> 52) & 0x7FFu;
}

// Slicing scale 2^(7-e) and output factor 2^(e-7) for a largest biased
// binary64 exponent E (values below 2^(E-1022) in magnitude): e = E - 1022.
// E = 2047 (NaN, Inf) and e > 126 (beyond binary32) poison the outputs;
// below 2^-100 the row / column counts as zero -- as scales() does.
__device__ __forceinline__ void scales64(unsigned E, float& sc, float& fac) {
    const int e = (int)E - 1022;
    if (E == 2047u || e > 126) {
        sc = 1.0f;
        fac = __int_as_float(0x7fc00000);
    } else if (e < -99) {
        sc = 0.0f;
        fac = 0.0f;
    } else {
        sc = __int_as_float((134 - e) << 23);
        fac = __int_as_float((120 + e) << 23);
    }
}

// Whether an accessor works on binary64 (kF64 = true) or double-float values.
template <class T, class = void>
struct IsF64 : std::false_type {};
template <class T>
struct IsF64<T, std::void_t<decltype(T::kF64)>> : std::integral_constant<bool, T::kF64> {};

// One operand entry as it is loaded, its contribution to a maximum and its digits.
__device__ __forceinline__ unsigned maxbits(zf v) {      // NaN ranks above everything
    return __float_as_uint(nmax(fabsf(v.re.hi), fabsf(v.im.hi)));
}
__device__ __forceinline__ unsigned maxbits(zd v) { return max(exp64(v.re), exp64(v.im)); }
template <bool F64>
__device__ __forceinline__ void scale_of(unsigned mx, float& sc, float& fac) {
    if constexpr (F64) scales64(mx, sc, fac);
    else scales(__uint_as_float(mx), sc, fac);
}
__device__ __forceinline__ void words_of(zf v, float sc, uint32_t* w) {
    words(v.re.hi, v.re.lo, sc, w[0], w[1]);
    words(v.im.hi, v.im.lo, sc, w[2], w[3]);
}
__device__ __forceinline__ void words_of(zd v, float sc, uint32_t* w) {
    words(v.re, sc, w[0], w[1]);
    words(v.im, sc, w[2], w[3]);
}

// C op= A B, A: M x Kc (M <= 128), B: Kc x N, complex double-float, through the
// accessor object `op` (passed by value):
//   const zf* op.pa(m), op.pb(n)              a(m, 0), b(0, n) (shared or global memory)
//   int op.sa(), op.sb()                      elements from one inner entry to the next
//                                             (1: contiguous along k, as is taken to
//                                             mean; else contiguous in m / n)
//   void op.store(m, n, re, im, first)        sets (first: the first group) or
//                                             adds to the target of (m, n) the sum
//                                             re + i im of (A B)[m][n] over one group
//                                             of up to 128 inner entries.  32 lanes
//                                             hold 32 consecutive m.
// With Op::kF64 = true the entries are binary64 (zd), sliced from their 53-bit significands, and
// store receives re, im in binary64: the eight accumulators are summed
// error-free in binary32 to three terms s + t + w (|w| < 2^-40 |s|), which are
// added in binary64 -- a product accurate to a few units of 2^-53 of (row max
// x column max x inner dimension).
//
// What bounds it: the MMAs (about 1.1 thousand cycles per chunk of 8 complex
// inner entries, kMma) and the digit slicing (about 30 instructions per real
// value), which run at the same time.  Warps 0-7 slice 16 rows of A' each (four
// inner entries per lane and chunk, one 16-byte store per digit), warps 8-11 8
// columns of B' each (two per lane), into two buffers of digit tiles; an elected
// lane of the last warp issues a chunk's MMAs when its twelve warps have arrived
// on the buffer's "full" mbarrier, and their commit frees the buffer ("empty"),
// so no block barrier stands between chunks.  A chunk's raw entries are loaded
// while the chunk before is sliced, and turned into integers before the wait
// for its buffer.  After the last chunk of a pass (32 columns) the slicing warps
// go on into the next pass's first chunk, then every warp drains its share of
// the accumulators; the next pass's MMAs wait for the 16 warps' "drained".  With
// Kc <= 16 (the rank-b updates) A's two chunks stay in their buffers for all
// passes.
// Measured (246 x 123 x 123 double-float on one SM): 155 us where two products of
// 123 rows with M = 128, N = 64 MMAs and one thread issuing took 600 us.
// Called by every thread of the block (NT = 512); begins and ends with a
// barrier.  Returns the next mbarrier parities.
template <class Op>
__device__ __forceinline__ uint32_t zgemm(Op op, int M, int N, int Kc, Area ar, uint32_t phase) {
    static_assert(NT == 512, "zgemm assumes 512 threads");
    constexpr bool F64 = IsF64<Op>::value;
    using E = std::conditional_t<F64, zd, zf>;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wu = __shfl_sync(0xffffffffu, warp, 0);       // the same, known to be uniform
    const uint32_t tmem = *ar.tslot();
    const int q4 = warp & 3, mrow = 32 * q4 + lane, cgrp = warp >> 2;   // drain mapping
    const int ngrp = (Kc + KGRP - 1) / KGRP;
    const int gsz = ((Kc + ngrp - 1) / ngrp + KCH - 1) / KCH * KCH;     // <= KGRP
    const int npass = (N + MAXC - 1) / MAXC;
    const int pw = ((N + npass - 1) / npass + 3) & ~3;                  // columns per pass
    // slicing warps: the lane's row of A' (column of B') and its inner entries
    // kq .. of a chunk, 4 or 2
    const bool isA = wu < 8, isB = wu >= 8 && wu < 12;
    const int row = isA ? 16 * warp + (lane >> 1) : 8 * (warp & 3) + (lane >> 2);
    const int kq = isA ? 4 * (lane & 1) : 2 * (lane & 3);
    const bool anyA = 16 * warp < M;                    // an A' warp with rows
    const int sk = isA ? op.sa() : op.sb();
    __syncthreads();
    for (int g0 = 0; g0 < Kc; g0 += gsz) {
        const int kg = min(gsz, Kc - g0);
        const int nch = (kg + KCH - 1) / KCH;
        const bool keepA = nch <= NBUF;
        // scales of the columns of pass p
        auto col_max = [&](int p) {
            const int n0 = p * pw, nc = min(pw, N - n0);
            float *cs = ar.csc(p), *cf = ar.cfac(p);
            if (op.sb() == 1) {
                for (int c = warp; c < nc; c += NWARP) {
                    unsigned mx = 0u;
                    const E* q = op.pb(n0 + c) + g0;
                    for (int k = lane; k < kg; k += 32) mx = max(mx, maxbits(q[k]));
                    mx = __reduce_max_sync(0xffffffffu, mx);
                    if (lane == 0) scale_of<F64>(mx, cs[c], cf[c]);
                }
            } else if (warp == 0) {
                unsigned mx = 0u;
                if (lane < nc) {
                    const E* q = op.pb(n0 + lane) + (size_t)g0 * op.sb();
#pragma unroll 4
                    for (int k = 0; k < kg; ++k, q += op.sb()) mx = max(mx, maxbits(*q));
                }
                scale_of<F64>(mx, cs[lane], cf[lane]);
            }
        };
        // row scales over this group, column maxima of the first pass
        if (op.sa() != 1) {
            unsigned* part = reinterpret_cast<unsigned*>(ar.a(0));
            const int m = tid & 127;
            unsigned mx = 0u;
            if (m < M) {
                const E* q = op.pa(m) + (size_t)(g0 + (tid >> 7)) * op.sa();
#pragma unroll 4
                for (int k = tid >> 7; k < kg; k += 4, q += (ptrdiff_t)4 * op.sa()) mx = max(mx, maxbits(*q));
            }
            part[tid] = mx;
            col_max(0);
            if (npass > 1) col_max(1);
            __syncthreads();
            if (tid < 128)
                scale_of<F64>(max(max(part[tid], part[tid + 128]), max(part[tid + 256], part[tid + 384])),
                              ar.rsc()[tid], ar.rfac()[tid]);
        } else {
            for (int m = warp; m < 128; m += NWARP) {
                unsigned mx = 0u;
                if (m < M) {
                    const E* q = op.pa(m) + g0;
                    for (int k = lane; k < kg; k += 32) mx = max(mx, maxbits(q[k]));
                }
                mx = __reduce_max_sync(0xffffffffu, mx);
                if (lane == 0) scale_of<F64>(mx, ar.rsc()[m], ar.rfac()[m]);
            }
            col_max(0);
            if (npass > 1) col_max(1);
        }
        __syncthreads();
        // the raw entries of a chunk: loads without a condition (indices clamped
        // into the operands), so that nothing waits for them before they are
        // sliced; base: the row's (column's) entry g0 + kq
        E raw[4];
        const E* base = isA ? op.pa(min(row, M - 1)) : op.pb(min(row, N - 1));
        base += (ptrdiff_t)(g0 + kq) * sk;
        const int klast = kg - 1 - kq;                  // relative to base
        auto fetch = [&](int ch) {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (u < 2 || isA) raw[u] = base[(ptrdiff_t)min(ch * KCH + u, klast) * sk];   // 64 bits: sk is any int
        };
        // ... as words, which frees them for the next chunk's loads (scale 0
        // beyond the last inner entry and outside the rows), and the words'
        // digits into the tiles of buffer buf
        uint32_t w[4][4];
        float sc = isA && row < M ? ar.rsc()[row] : 0.0f;
        auto to_words = [&](int ch) {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (u < 2 || isA) words_of(raw[u], ch * KCH + u <= klast ? sc : 0.0f, w[u]);
        };
        auto slice = [&](int buf) {
            uint32_t d[4], e[4];
            if (isA) {
                __half* o = ar.a(buf) + tile_off(row, 2 * kq);
#pragma unroll
                for (int u = 0; u < 4; ++u) d[u] = digit_0(w[u]);
                *reinterpret_cast<uint4*>(o) = make_uint4(d[0], d[1], d[2], d[3]);
#pragma unroll
                for (int h = 0; h < 3; ++h) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) two_digits(w[u], h, d[u], e[u]);
                    *reinterpret_cast<uint4*>(o + (2 * h + 1) * TILE) = make_uint4(d[0], d[1], d[2], d[3]);
                    *reinterpret_cast<uint4*>(o + (2 * h + 2) * TILE) = make_uint4(e[0], e[1], e[2], e[3]);
                }
            } else {
                // rows (Re, -Im) and (Im, Re)
                __half *ore = ar.b(buf) + tile_off(2 * row, 2 * kq), *oim = ar.b(buf) + tile_off(2 * row + 1, 2 * kq);
                auto put = [&](int j, const uint32_t* v) {
                    *reinterpret_cast<uint2*>(ore + j * TILEB) = make_uint2(v[0] ^ 0x80000000u, v[1] ^ 0x80000000u);
                    *reinterpret_cast<uint2*>(oim + j * TILEB) =
                        make_uint2(__byte_perm(v[0], 0, 0x1032), __byte_perm(v[1], 0, 0x1032));
                };
                d[0] = digit_0(w[0]);
                d[1] = digit_0(w[1]);
                put(0, d);
#pragma unroll
                for (int h = 0; h < 3; ++h) {
                    two_digits(w[0], h, d[0], e[0]);
                    two_digits(w[1], h, d[1], e[1]);
                    put(2 * h + 1, d);
                    put(2 * h + 2, e);
                }
            }
        };
        // drain of pass p: warp w reads lanes 32 (w & 3) .. +31 (rows) and the
        // 8-column blocks (4 complex columns) w >> 2, + 4
        auto drain = [&](int p) {
            const int n0 = p * pw, nc = min(pw, N - n0);
            const float rf = ar.rfac()[mrow];
            const float* cf = ar.cfac(p);
#pragma unroll
            for (int b = 0; b < MAXC / 16; ++b) {
                const int cb = cgrp + 4 * b;
                if (4 * cb < nc) {
                    const uint32_t ad = tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)(8 * cb);
                    // two halves of 4 columns (2 complex columns)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint32_t ah = ad + 4u * h;
                        float a0[4], a1[4], a2[4], a3[4], a4[4], a5[4], a6[4], a7[4];
                        ld4(ah, a0);
                        ld4(ah + ACOLS, a1);
                        ld4(ah + 2 * ACOLS, a2);
                        ld4(ah + 3 * ACOLS, a3);
                        ld4(ah + 4 * ACOLS, a4);
                        ld4(ah + 5 * ACOLS, a5);
                        ld4(ah + 6 * ACOLS, a6);
                        ld4(ah + 7 * ACOLS, a7);
                        ld_wait();
                        if constexpr (F64) {
                            // s + t + w exactly up to the rounding of w
                            // (below 2^-70 of s), then binary64
                            double z[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                float s01, e01, s23, e23, r4, e4, r, er, s, e, p1, pe, q, qe, t, te;
                                two_sum(a0[j], a1[j] * 0x1p-8f, s01, e01);
                                two_sum(a2[j] * 0x1p-16f, a3[j] * 0x1p-24f, s23, e23);
                                two_sum(a4[j] * 0x1p-32f, a7[j] * 0x1p-32f, r4, e4);
                                two_sum(r4, __fmaf_rn(a6[j], 0x1p-48f, a5[j] * 0x1p-40f), r, er);
                                two_sum(s01, s23, s, e);
                                two_sum(e01, e, p1, pe);
                                two_sum(e23, r, q, qe);
                                two_sum(p1, q, t, te);
                                const float w1 = __fadd_rn(__fadd_rn(__fadd_rn(pe, qe), __fadd_rn(te, er)), e4);
                                z[j] = (double)s + ((double)t + (double)w1);
                            }
                            if (mrow < M) {
#pragma unroll
                                for (int jj = 0; jj < 2; ++jj) {
                                    const int j = 2 * h + jj, c = 4 * cb + j;
                                    if (c < nc) {
                                        const double f = (double)rf * (double)cf[c];
                                        op.store(mrow, n0 + c, z[2 * jj] * f, z[2 * jj + 1] * f, g0 == 0);
                                    }
                                }
                            }
                        } else {
                            // levels 0 + 1 and 2 + 3 pair up error-free, the
                            // others in binary32 (below 2^-32 of the scale),
                            // then one double-float sum
                            float hi[4], lo[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                float s01, e01, s23, e23, s, e;
                                two_sum(a0[j], a1[j] * 0x1p-8f, s01, e01);               // exact
                                two_sum(a2[j] * 0x1p-16f, a3[j] * 0x1p-24f, s23, e23);   // exact
                                const float r = __fmaf_rn(__fadd_rn(a4[j], a7[j]), 0x1p-32f,
                                                          __fmaf_rn(a6[j], 0x1p-48f, a5[j] * 0x1p-40f));
                                two_sum(s01, s23, s, e);
                                fast_two_sum(s, __fadd_rn(__fadd_rn(e01, e), __fadd_rn(e23, r)), hi[j], lo[j]);
                            }
                            if (mrow < M) {
#pragma unroll
                                for (int jj = 0; jj < 2; ++jj) {
                                    const int j = 2 * h + jj, c = 4 * cb + j;
                                    if (c < nc) {
                                        const float f = rf * cf[c];
                                        const df32 re{__fmul_rn(hi[2 * jj], f), __fmul_rn(lo[2 * jj], f)};
                                        const df32 im{__fmul_rn(hi[2 * jj + 1], f), __fmul_rn(lo[2 * jj + 1], f)};
                                        op.store(mrow, n0 + c, re, im, g0 == 0);
                                    }
                                }
                            }
                        }
                    }
                }
            }
        };
        // Step (p, ch): the slicing warps slice the chunk, the issuing warp issues
        // it; pass p - 1 is drained after its successor's first chunk is sliced.
        // Chunks go through the two buffers in turn (with A kept, chunk ch through
        // buffer ch).  ph: the parities of the phases this warp waits for next.
        // Every slicing warp takes every chunk in turn (with A kept, every pass's
        // one use of a buffer, two passes behind the drains), so none can take an
        // earlier phase of a barrier for the one it waits for.
        uint32_t ph = phase;
        uint32_t used = 0u;                             // buffers used before in this group
        bool ok = true;
        auto wait = [&](int bar) {
            ok = wait_bar(ar, bar, (ph >> bar) & 1u) && ok;
            ph ^= 1u << bar;
        };
        if (isA || isB) fetch(0);
        int buf = 0;
        for (int p = 0; p <= npass; ++p) {
            const int nc = min(pw, N - p * pw);
            const bool slicing = p < npass && (isB || (isA && !(keepA && p > 0)));
            for (int ch = 0; ch < nch; ++ch) {
                if (slicing) {
                    if (ch == 0 && isB) {
                        // the column scales, formed by all warps before "drained" of p - 2
                        if (p > 1) wait(BAR_DRAINED);
                        sc = row < nc ? ar.csc(p)[row] : 0.0f;
                    }
                    to_words(ch);
                    if (ch + 1 < nch) {
                        fetch(ch + 1);
                    } else if (p + 1 < npass) {
                        if (isB) base = op.pb(min((p + 1) * pw + row, N - 1)) + (ptrdiff_t)(g0 + kq) * sk;
                        fetch(0);
                    }
                    if ((used >> buf) & 1u) wait(BAR_EMPTY + buf);
                    used |= 1u << buf;
                    if (anyA || isB) {
                        slice(buf);
                        fence_async_smem();
                    }
                    __syncwarp();
                    // with A kept the first warp of B' arrives for those of A' too
                    if (lane == 0 && ok) arrive(ar.bar(BAR_FULL + buf), keepA && p > 0 && wu == 8 ? bar_count(BAR_FULL) - 3u : 1u);
                }
                if (ch == 0 && p > 0) {
                    // this warp's share of the drain of pass p - 1
                    wait(BAR_DONE);
                    fence_after();
                    drain(p - 1);
                    fence_before();
                    if (p + 1 < npass) col_max(p + 1);
                    __syncwarp();
                    if (lane == 0 && ok) arrive(ar.bar(BAR_DRAINED), 1u);
                }
                if (p == npass) break;
                if (wu == ISSUE_WARP) {
                    wait(BAR_FULL + buf);
                    if (ch == 0 && p > 0) wait(BAR_DRAINED);
                    fence_after();
                    __syncwarp();
                    if (elect_one()) {
                        // digit tile i starts TILE * 2 (TILEB * 2) bytes after tile
                        // i - 1: its descriptor's address field (16-byte units, every
                        // shared address below 2^18) is kTile(B)Desc further on
                        constexpr uint64_t kTileDesc = (uint64_t)(TILE * 2) >> 4, kTileBDesc = (uint64_t)(TILEB * 2) >> 4;
                        const uint64_t da = sdesc(ar.a(buf)), db = sdesc(ar.b(buf));
                        const uint32_t more = ch > 0;
#pragma unroll
                        for (int q = 0; q < NMMA; ++q) {
                            const MmaOp o = kMma[q];
                            mma(tmem + (uint32_t)(ACOLS * o.acc), da + (uint64_t)o.i * kTileDesc,
                                db + (uint64_t)o.j0 * kTileBDesc, idesc(ACOLS * o.nd),
                                (o.i == 0 || (o.i == 1 && o.acc == 7)) ? more : 1u);
                        }
                        if (!*ar.skip()) {
                            commit(ar.bar(BAR_EMPTY + buf));
                            if (ch == nch - 1) commit(ar.bar(BAR_DONE));
                        }
                    }
                    __syncwarp();
                }
                buf = keepA ? (ch + 1 < nch ? 1 : 0) : buf ^ 1;
            }
        }
        // every barrier's uses in this group, for the next parities
        const int nc = npass * nch;
        const uint32_t u0 = keepA ? npass : (nc + 1) >> 1, u1 = keepA ? (nch > 1 ? npass : 0) : nc >> 1;
        phase ^= ((u0 & 1u) << BAR_EMPTY) | ((u1 & 1u) << (BAR_EMPTY + 1)) | ((u0 & 1u) << BAR_FULL) |
                 ((u1 & 1u) << (BAR_FULL + 1)) | ((uint32_t)(npass & 1) << BAR_DRAINED) |
                 ((uint32_t)(npass & 1) << BAR_DONE);
        __syncthreads();
    }
    return phase;
}

// The binary32 sums of a level set (level l's integer sum in a[l], l = 0 .. 6) as
// a double-float value, or error-free as three terms in binary64.
__device__ __forceinline__ df32 level_sum(const float* a, df32) {
    float s01, e01, s23, e23, s, e;
    two_sum(a[0], a[1] * 0x1p-8f, s01, e01);                   // exact
    two_sum(a[2] * 0x1p-16f, a[3] * 0x1p-24f, s23, e23);       // exact
    const float r = __fmaf_rn(a[4], 0x1p-32f, __fmaf_rn(a[6], 0x1p-48f, a[5] * 0x1p-40f));
    two_sum(s01, s23, s, e);
    df32 v;
    fast_two_sum(s, __fadd_rn(__fadd_rn(e01, e), __fadd_rn(e23, r)), v.hi, v.lo);
    return v;
}
__device__ __forceinline__ double level_sum(const float* a, double) {
    float s01, e01, s23, e23, r, er, s, e, p1, pe, q, qe, t, te;
    two_sum(a[0], a[1] * 0x1p-8f, s01, e01);
    two_sum(a[2] * 0x1p-16f, a[3] * 0x1p-24f, s23, e23);
    two_sum(a[4] * 0x1p-32f, __fmaf_rn(a[6], 0x1p-48f, a[5] * 0x1p-40f), r, er);
    two_sum(s01, s23, s, e);
    two_sum(e01, e, p1, pe);
    two_sum(e23, r, q, qe);
    two_sum(p1, q, t, te);
    return (double)s + ((double)t + (double)__fadd_rn(__fadd_rn(pe, qe), __fadd_rn(te, er)));
}

// The rank-bb update of the inverse (bb <= 16): W[r0 + m][l] -= sum_q C[q][r0 + m]
// X[q][l] for m < M <= 128 and the N columns l outside the panel (column c: l = c
// below j0, c + bb from there on), W column-major with leading dimension lda, C
// and X [bb][K] at byte offsets cm_off and xr_off of dynamic shared memory.
//
// Few inner entries and many columns: what bounds it is reading the accumulators
// and W, so passes are narrow (16 columns) and the 7 accumulators (levels 0 .. 6,
// exact up to level 4 with 32 inner entries) are kept twice: while the tensor
// core works on pass p, all warps read pass p - 1.  C is sliced once (warps 0-7,
// 16 rows each), X pass by pass (warps 8-11, 4 columns each, all 16 inner entries
// in 8 lanes, so that a row's or column's scale is a shuffle away).  Per chunk of
// 8 inner entries the 28 digit products are 7 MMAs, digit i of C times digits
// 0 .. 6 - i of X into levels i .. 6, N = 32 (7 - i).
// Measured (K = 123, bb = 16, double-float, one SM): 18 us, with 64-column zgemm
// passes 37 us.
// Called by every thread of the block; begins and ends with a barrier.
template <class E>
__device__ __forceinline__ uint32_t zupdate(int cm_off, int xr_off, int K, int bb, E* W, int lda, int r0, int M,
                                            int j0, int N, Area ar, uint32_t phase) {
    static_assert(NT == 512, "zupdate assumes 512 threads");
    constexpr bool F64 = std::is_same<E, zd>::value;
    using Re = std::conditional_t<F64, double, df32>;
    constexpr int UC = 16, UTILE = 2 * UC * 16, UCOLS = 2 * UC;     // columns of a pass; B' tile; TMEM columns
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wu = __shfl_sync(0xffffffffu, warp, 0);
    const uint32_t tmem = *ar.tslot();
    const int q4 = warp & 3, mrow = 32 * q4 + lane, cgrp = warp >> 2;
    const int npass = (N + UC - 1) / UC, nch = (bb + KCH - 1) / KCH;
    const E* X = reinterpret_cast<const E*>(rgf_dyn_smem + xr_off);
    auto col = [&](int c) { return c < j0 ? c : c + bb; };
    __syncthreads();
    if (wu < 8 && 16 * wu < M) {
        // C's digits: row, entries kq .. kq + 3 of both chunks
        const E* C = reinterpret_cast<const E*>(rgf_dyn_smem + cm_off) + r0;
        const int row = 16 * warp + (lane >> 1), kq = 4 * (lane & 1), m = min(row, M - 1);
        E v[8];
        unsigned mx = 0u;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int k = (u & 4) * 2 + kq + (u & 3);
            v[u] = C[min(k, bb - 1) * K + m];
            if (k < bb) mx = max(mx, maxbits(v[u]));
        }
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        float sc, fac;
        scale_of<F64>(mx, sc, fac);
        if (kq == 0) ar.rfac()[row] = fac;
        if (row >= M) sc = 0.0f;
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
            if (ch >= nch) break;
            uint32_t w[4][4], d[4], e[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) words_of(v[4 * ch + u], 8 * ch + kq + u < bb ? sc : 0.0f, w[u]);
            __half* o = ar.a(ch) + tile_off(row, 2 * kq);
#pragma unroll
            for (int u = 0; u < 4; ++u) d[u] = digit_0(w[u]);
            *reinterpret_cast<uint4*>(o) = make_uint4(d[0], d[1], d[2], d[3]);
#pragma unroll
            for (int h = 0; h < 3; ++h) {
#pragma unroll
                for (int u = 0; u < 4; ++u) two_digits(w[u], h, d[u], e[u]);
                *reinterpret_cast<uint4*>(o + (2 * h + 1) * TILE) = make_uint4(d[0], d[1], d[2], d[3]);
                *reinterpret_cast<uint4*>(o + (2 * h + 2) * TILE) = make_uint4(e[0], e[1], e[2], e[3]);
            }
        }
        fence_async_smem();
    }
    __syncthreads();
    uint32_t ph = phase;
    bool ok = true;
    auto wait = [&](int bar) {
        ok = wait_bar(ar, bar, (ph >> bar) & 1u) && ok;
        ph ^= 1u << bar;
    };
    float* cfac = ar.csc(0);                             // [4][UC] column factors of four passes
    for (int p = 0; p <= npass; ++p) {
        const int set = p & 1;
        if (p < npass && wu >= 8 && wu < 12) {
            // X's digits of the pass's columns; buffer `set` was freed when pass
            // p - 2 was complete, which this warp has waited for to drain it
            const int c = 4 * (warp & 3) + (lane >> 3), k0 = 2 * (lane & 7);
            const bool in = p * UC + c < N;
            const E* q = X + col(min(p * UC + c, N - 1));
            const E v0 = q[min(k0, bb - 1) * K], v1 = q[min(k0 + 1, bb - 1) * K];
            unsigned mx = max(k0 < bb ? maxbits(v0) : 0u, k0 + 1 < bb ? maxbits(v1) : 0u);
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            float sc, fac;
            scale_of<F64>(in ? mx : 0u, sc, fac);
            if (k0 == 0) cfac[(p & 3) * UC + c] = fac;
            uint32_t w[2][4], d[2], e[2];
            words_of(v0, k0 < bb ? sc : 0.0f, w[0]);
            words_of(v1, k0 + 1 < bb ? sc : 0.0f, w[1]);
            // chunk (k0 >> 3)'s tiles of the set; rows (Re, -Im) and (Im, Re)
            __half* t = ar.b(0) + (set * 2 + (k0 >> 3)) * (S * UTILE);
            __half *ore = t + tile_off(2 * c, 2 * (k0 & 7)), *oim = t + tile_off(2 * c + 1, 2 * (k0 & 7));
            auto put = [&](int j, const uint32_t* x) {
                *reinterpret_cast<uint2*>(ore + j * UTILE) = make_uint2(x[0] ^ 0x80000000u, x[1] ^ 0x80000000u);
                *reinterpret_cast<uint2*>(oim + j * UTILE) =
                    make_uint2(__byte_perm(x[0], 0, 0x1032), __byte_perm(x[1], 0, 0x1032));
            };
            d[0] = digit_0(w[0]);
            d[1] = digit_0(w[1]);
            put(0, d);
#pragma unroll
            for (int h = 0; h < 3; ++h) {
                two_digits(w[0], h, d[0], e[0]);
                two_digits(w[1], h, d[1], e[1]);
                put(2 * h + 1, d);
                put(2 * h + 2, e);
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0 && ok) arrive(ar.bar(BAR_UFULL + set), 1u);
        }
        if (p < npass && wu == ISSUE_WARP) {
            wait(BAR_UFULL + set);
            if (p > 1) wait(BAR_UDRAINED + set);
            fence_after();
            __syncwarp();
            if (elect_one()) {
                for (int ch = 0; ch < nch; ++ch) {
                    const uint64_t da = sdesc(ar.a(ch)), db = sdesc(ar.b(0) + (set * 2 + ch) * (S * UTILE));
                    constexpr uint64_t kTileDesc = (uint64_t)(TILE * 2) >> 4;
                    const uint32_t acc = ch > 0;
#pragma unroll
                    for (int i = 0; i < S; ++i)
                        mma(tmem + (uint32_t)(256 * set + UCOLS * i), da + (uint64_t)i * kTileDesc, db,
                            idesc(UCOLS * (S - i)), i == 0 ? acc : 1u);
                }
                if (!*ar.skip()) commit(ar.bar(BAR_EMPTY + set));
            }
            __syncwarp();
        }
        if (p > 0) {
            // drain of pass p - 1: warp w reads rows 32 (w & 3) .. and columns 4 (w >> 2) ..
            const int pd = p - 1, sd = pd & 1, c0 = pd * UC + 4 * cgrp;
            E old[4];
            E* wc[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                wc[j] = W + (size_t)col(min(c0 + j, N - 1)) * lda + r0 + min(mrow, M - 1);
                old[j] = *wc[j];
            }
            wait(BAR_EMPTY + sd);
            fence_after();
            const float rf = ar.rfac()[mrow];
            const uint32_t ad = tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)(256 * sd + 8 * cgrp);
            if (c0 < N) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float a[S][4];
#pragma unroll
                    for (int i = 0; i < S; ++i) ld4(ad + (uint32_t)(UCOLS * i + 4 * h), a[i]);
                    ld_wait();
#pragma unroll
                    for (int jj = 0; jj < 2; ++jj) {
                        const int j = 2 * h + jj;
                        const float cf = cfac[(pd & 3) * UC + 4 * cgrp + j];
                        Re z[2];
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            float v[S];
#pragma unroll
                            for (int i = 0; i < S; ++i) v[i] = a[i][2 * jj + c];
                            z[c] = level_sum(v, Re{});
                            if constexpr (F64) z[c] *= (double)rf * (double)cf;
                            else z[c] = df32{__fmul_rn(z[c].hi, rf * cf), __fmul_rn(z[c].lo, rf * cf)};
                        }
                        if (mrow < M && c0 + j < N) *wc[j] = csub(old[j], E{z[0], z[1]});
                    }
                }
            }
            fence_before();
            __syncwarp();
            if (lane == 0 && ok) arrive(ar.bar(BAR_UDRAINED + sd), 1u);
        }
    }
    const uint32_t u0 = (uint32_t)((npass + 1) >> 1), u1 = (uint32_t)(npass >> 1);
    phase ^= ((u0 & 1u) * ((1u << BAR_EMPTY) | (1u << BAR_UFULL) | (1u << BAR_UDRAINED))) ^
             ((u1 & 1u) * ((2u << BAR_EMPTY) | (2u << BAR_UFULL) | (2u << BAR_UDRAINED)));
    __syncthreads();
    return phase;
}

}  // namespace tc
}  // namespace rgf

// Tensor-core form of the structure-factor pass (Alg. 1) and of the
// back-contraction (Alg. S1) for orthorhombic cells.
//
// In an orthorhombic cell the pair prefactor factorises over the three axes
// (Sec. 2.4, the orthorhombic fully separable case; App. D):
//   exp(-|G|^2/4p) exp(-i G.P) = X(n_a) Y(n_b) Z(n_c),
//   X(n) = exp(-c M_aa n^2) exp(-2 pi i f_a n),   c = 1/(4p),
// f_a the fractional coordinate of the pair centre.  With a pair record's
// Hermite densities D'_{ijk} (the walks' convention: the record adds
// X Y Z sum_ijk D'_ijk (-i n_a)^i (-i n_b)^j (-i n_c)^k to rho(n)),
//   rho(n_a, n_b, n_c) = sum_{(i,j)} (-i n_a)^i (-i n_b)^j sum_r X_r(n_a) Y_r(n_b) B_ij[r, n_c]
//   B_ij = Z_r(n_c) sum_k D'_{r,ijk} (-i n_c)^k         (per density).
//
// Real form.  X(-n) = conj X(n), so with X(s n) = X_0(n) + i s X_1(n) (real
// and imaginary part, s = +-1) the four sign combinations of (n_a, n_b) are
// sums of the four REAL products X_ta(|n_a|) Y_tb(|n_b|), ta, tb in {0, 1}:
//   X(s_a |n_a|) Y(s_b |n_b|) = sum_{ta,tb} i^{ta+tb} s_a^ta s_b^tb X_ta Y_tb.
// The matrix product over the records is therefore formed with real A
// (rows = "slots" (|n_a|, |n_b|, ta, tb), K = records) and complex B
// (columns = (Re, Im) of (i, j) x n_c >= 0 x densities); the signs are put
// back when the sums leave the kernel.  Against the complex form (rows
// (n_a, n_b), two K entries and two columns per complex product) this is half
// the multiply-adds, half the operand bytes, and one real product per A entry
// instead of a complex one.  For the records of one class L, all (i, j) with
// i + j <= L share A, so up to G column blocks B_ij go side by side.  A block
// contributes with (-i)^{i+j} n_a^i n_b^j, whose sign s_a^i s_b^j moves a
// product of type (ta, tb) to the sign character (ta + i, tb + j) mod 2: the
// four slots of a point sit in four adjacent lanes, and the drain exchanges
// their sums with one xor shuffle per block.  A carries only the Gaussian and
// the phase, so a row's entries over a window of records sorted by their width
// differ little in size, which is what keeps the slicing below at full
// relative precision.
//
// Precision.  bf16 products summed in FP32 carry 8 bits; the target is FP64-
// class.  The operands are therefore split after Ozaki, Ogita, Oishi and Rump
// ("Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication", Numer. Algorithms 59, 2012): every row
// of A and every column of B, over a window of at most 1024 records, gets a
// power-of-two bound 2^e of its entries, and each entry is cut into six slices
// m_s 2^{e-6-7s} with integers |m_s| <= 64.  The columns' exponents are taken
// relative to the largest of their window and density, which multiplies the
// sums when they are drained: a build scales with its density over FP64's range
// (the split form's terms over FP32's).  Slice s of A
// times slice t of B is a tcgen05.mma of kind::f16 (bf16 operands, FP32
// accumulator in tensor memory); products with s + t <= 5 are formed (21 per
// k-step), the others fall below 2^-40 of the window's scale.  Products of the
// same level s + t land in one accumulator: levels 0 to 3 are exact integer
// sums (|m| <= 64, at most 4 products per level and 1024 K terms keep every
// partial sum at or below 2^24), levels 4 and 5 share a fifth, rounded
// accumulator, 2^-28 of the first.  At each window's end the level sums are
// added in double-float (FP32 pairs, df.cuh) to sums kept in registers, which
// are written as FP64 partial rows and summed across window groups in fixed
// order by the row reduction.
//
// Kernel shape.  B does not depend on the row, and a sphere has several row
// tiles, so B is sliced once per build (k_tc_rho_b) into stage tiles in global
// memory, already in the core-matrix layout of the MMA descriptors, and comes
// in with one bulk copy per stage.  k_tc_rho runs one CTA per SM (512
// tensor-memory columns, ~200 KB of shared memory), 19 warps: warps 0-15, two
// groups in turn, form the A slices of a 16-record stage (one thread per row
// and eight records: one 16-byte core-matrix row per slice) into a ring of up
// to four buffers; one elected lane of warp 16 issues the MMAs; warp 17 brings
// the records' factor tables and warp 18 the B tiles in (cp.async.bulk,
// completion counted in bytes on mbarriers).  Warps 0-15 also drain tensor
// memory.  Stages are handed over with mbarriers (arrivals; tcgen05.commit for
// the MMA side).  Every wait is bounded: past ~2 s of clock a waiting thread
// raises the CTA's abort flag and the plan's device error word, every thread
// leaves its loops, the copies and MMAs in flight are waited for (again
// bounded), the CTA's outputs become NaN and tensor memory is freed before it
// exits.
//
// What bounds it (molecular crystal, 1056 AOs, 2 densities, GB300): the product
// takes 1.10 ms, of which the MMAs alone (operands left unformed) need 0.89 ms:
// their operand reads from shared memory (15 MMAs of N = 96 or 192 per k-step,
// 123 KB) beside the operand and table writes.  B tiles in global memory cost
// 0.28 ms more (0.49 GB written).  What took the pass from 4.76 ms there: the
// real form (half of everything), B formed once instead of once per row tile,
// one bulk copy per stage instead of one per record and block (each copy takes
// ~100 cycles of the copy engine whatever its size: 1.32 ms for the loads
// alone), and MMAs issued from warp-uniform code (1.57 -> 1.35 ms).
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <queue>
#include <type_traits>
#include <vector>

#include "df.cuh"
#include "ftcj_internal.h"

namespace ftcj {
namespace {

constexpr int kTcM = 128;                      // rows per tile (MMA M)
constexpr int kTcStageK = 16;                  // records per stage: one MMA k-step
constexpr int kTcWinMax = 1024;                // records per exact-accumulation window at most (FP64 form: half)
constexpr int kTcNmax = 96;                    // MMA N at most in the split form: five accumulators in 512 columns
constexpr int kTcNmax64 = 64;                  // in the FP64 form: eight
constexpr int kTcTmemCols = 512;
constexpr int kTcDensMax = 32;                 // densities per launch at most: one per lane of a drain warp
constexpr int kTcGmax = 15;                    // (i, j) blocks per window at most (class 4 has 15)
constexpr int kTcNbufMax = 4;                  // stage buffers at most
constexpr int kTcTabSlotsMax = 6;              // stage tables in flight at most
constexpr int kTcAsliceBytes = kTcM * kTcStageK * 2;      // 128 rows x 16 K x bf16
constexpr long long kTcBWorkMax = 8LL << 30;              // bytes of B tiles per pass at most
constexpr long long kTcSpinCycles = 1LL << 32;            // ~2 s of SM clock per wait
// Exponent bound of a column with a NaN or an infinity.  Slices hold neither
// (their digits come from integer operations or cancelling sums), so the sums
// of such a column become NaN where they leave the product.
constexpr int kNonFinite = 1 << 20;

// a slot: bits 0-7 |n_a|, 8-15 |n_b|, 16 ta, 17 tb, 18 / 19: the lane's bit 0
// (1) is the sign of n_a (n_b), 20: valid
__host__ __device__ constexpr int slot_pack(int na, int nb, int ta, int tb, int da, int db, int valid) {
    return na | (nb << 8) | (ta << 16) | (tb << 17) | (da << 18) | (db << 19) | (valid << 20);
}

struct TcArgs {
    const int* slots;    // row slots, a multiple of kTcM
    const int* map;      // [2 nam + 1][2 nbm + 1][ncols]: half-sphere index of (n_a, n_b, n_c), ~index where the
                         // stored point is -n, INT_MIN none
    const int4* winfo;   // [nwin]: class L, number of (i,j) blocks, first block index into wpairs,
                         // position of the window's first record in its class's K order
    const int* wcnt;     // [nwin]: records of the window
    const long long* boff;  // [nwin]: start of the window's B tiles in bs (16-byte units)
    const int* sched;    // [ngroups + 1] offsets, then window ids grouped by CTA group
    const int* wpairs;   // (i | j << 3) of each block
    const void* tabk;    // X(0..), Y(0..) as complex double-float or double (16 bytes either way), [tws] per record in
                         // the K order of all classes
    const void* tabz;    // Z(0..), [ncols] per record in the same order
    const float* clk;    // c log2(e) in the same order
    long long kbase[kNclass];  // first record of each class in that order
    const void* Dp;      // Hermite densities: split plans double-float in the K order, [dens][class][term][position];
                         // FP64 plans doubles in record order, [dens][class][term][record]
    const int* korder;   // FP64 form: class-local record of each position of the K order of all classes
    long long dp_total;
    long long dp_base[kNclass];
    long long dp_stride[kNclass];
    uint4* bs;           // sliced B stage tiles of this pass
    float* clw;          // [nwin]: smallest c log2(e) of each window's records
    int* ew;             // [nwin][nd]: exponent that the B slices of a window and density are relative to, kNonFinite
                         // where a term of its records is not finite
    double2* out;        // partial rows [dens][out_rows][ng_half], this pass's from out_row0
    long long ng_half;
    int out_rows, out_row0;
    int* err;            // device error word (bit 0: a bounded wait gave up)
    float Maa, Mbb, Mcc;
    int ax, bx, cx;      // lattice axes of the row indices (a, b) and of the column index (c)
    int nam, nbm;
    int tws, offY;       // table entries per record (X and Y, rounded up to odd), start of Y
    int ncols;           // complex columns per density and block: n_c = 0 .. ncols-1
    int nd, d0;          // densities of this launch, first density
    int colw;            // real columns per block: 2 nd ncols rounded up to 8
    int npad;            // MMA N of a full window: G colw rounded up to 16
    int w0;              // first window of this pass
    int nslots;
    long long spin;      // clock cycles a wait between roles may take before it gives up
};

// ---- PTX wrappers -----------------------------------------------------------

__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* b, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(saddr(b)) : "memory");
}

__device__ __forceinline__ bool mbar_test(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(saddr(b)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Waits for phase `parity` of b to complete; false when it gave up (after
// ~2 s of clock, or because another thread of the CTA already did).
__device__ bool mbar_wait(uint64_t* b, uint32_t parity, volatile int* abort_flag, long long spin) {
    const long long t0 = clock64();
    while (!mbar_test(b, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > spin) {
            *abort_flag = 1;
            return false;
        }
    }
    return true;
}

// One lane of a converged warp, always the same one.  The MMA warp runs its
// loops with all lanes on warp-uniform values and only the MMAs and commits
// under this predicate, so that descriptors stay in uniform registers: with
// the loops inside a one-lane branch every MMA cost ~90 cycles of register
// moves, whatever its width.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// shared-memory matrix descriptor: K-major, no swizzle, core matrices of 8
// rows x 16 B; K-adjacent core matrices 128 B apart (leading byte offset),
// 8-row groups 256 B apart (stride byte offset: 16 K per stage row)
__device__ __forceinline__ uint64_t sdesc(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(256u >> 4) << 32) |
           (1ull << 46);
}

__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void tc_commit(uint64_t* b) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(saddr(b))
                 : "memory");
}

// The slice products of one k-step, A_s B_t with s + t < S, into the level
// accumulators min(s + t, ACC - 1) (nw columns each, side by side).  The slices
// of B follow each other in shared memory in the same core-matrix layout, so up
// to W of them whose levels have accumulators of their own go into one MMA of
// N = W nw columns (<= 256): A_s is then read from shared memory once for all
// of them, and fewer MMAs are issued.  acc false: the window's first k-step,
// whose s = 0 products start each level's accumulator.
template <int S, int ACC, int W>
__device__ __forceinline__ void issue_kstep(uint32_t tmem, uint64_t ad, uint32_t astep, uint64_t bd, uint32_t bstep,
                                            uint32_t nw, uint32_t idesc, bool acc) {
#pragma unroll
    for (int s = 0; s < S; ++s) {
        const int nt = S - s;  // t = 0 .. nt - 1
#pragma unroll
        for (int t = 0; t < nt; ++t) {
            const int own = ACC - s;  // t below this has a level accumulator that no other t of this s shares
            const int lead = t < own ? t % W : 0;
            if (lead != 0) continue;  // part of the previous MMA
            const int lim = own < nt ? own : nt;
            const int n = t < own ? (lim - t < W ? lim - t : W) : 1;
            const int lv = s + t < ACC - 1 ? s + t : ACC - 1;
            const uint32_t on = s == 0 && t < ACC ? (acc ? 1u : 0u) : 1u;
            tc_mma(tmem + (uint32_t)lv * nw, ad + (uint64_t)(s * astep), bd + (uint64_t)(t * bstep),
                   idesc + ((((uint32_t)n * nw) >> 3) << 17), on);
        }
    }
}

// W slices side by side for nw columns each
template <int S, int ACC>
__device__ __forceinline__ void issue_kstep(uint32_t tmem, uint64_t ad, uint32_t astep, uint64_t bd, uint32_t bstep,
                                            uint32_t nw, uint32_t idesc, bool acc) {
    if (nw > 80) issue_kstep<S, ACC, 2>(tmem, ad, astep, bd, bstep, nw, idesc, acc);
    else if (nw > 64) issue_kstep<S, ACC, 3>(tmem, ad, astep, bd, bstep, nw, idesc, acc);
    else if (nw > 48) issue_kstep<S, ACC, 4>(tmem, ad, astep, bd, bstep, nw, idesc, acc);
    else issue_kstep<S, ACC, 5>(tmem, ad, astep, bd, bstep, nw, idesc, acc);
}

// Tensor-memory reads of 4 (8) columns of the five level accumulators, npad
// columns apart, with the wait for them in the same statement, so that no use
// of the values can be scheduled before it.
__device__ __forceinline__ void tc_ld_levels4(uint32_t taddr, uint32_t npad, float (&v)[5][4]) {
    uint32_t r[20];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%20];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%21];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8,%9,%10,%11}, [%22];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12,%13,%14,%15}, [%23];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%16,%17,%18,%19}, [%24];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19])
        : "r"(taddr), "r"(taddr + npad), "r"(taddr + 2 * npad), "r"(taddr + 3 * npad), "r"(taddr + 4 * npad)
        : "memory");
#pragma unroll
    for (int l = 0; l < 5; ++l)
#pragma unroll
        for (int i = 0; i < 4; ++i) v[l][i] = __uint_as_float(r[4 * l + i]);
}

__device__ __forceinline__ void tc_ld_levels4(uint32_t taddr, uint32_t npad, float (&v)[8][4]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%33];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8,%9,%10,%11}, [%34];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12,%13,%14,%15}, [%35];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%16,%17,%18,%19}, [%36];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%20,%21,%22,%23}, [%37];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%24,%25,%26,%27}, [%38];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%28,%29,%30,%31}, [%39];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr), "r"(taddr + npad), "r"(taddr + 2 * npad), "r"(taddr + 3 * npad), "r"(taddr + 4 * npad),
          "r"(taddr + 5 * npad), "r"(taddr + 6 * npad), "r"(taddr + 7 * npad)
        : "memory");
#pragma unroll
    for (int l = 0; l < 8; ++l)
#pragma unroll
        for (int i = 0; i < 4; ++i) v[l][i] = __uint_as_float(r[4 * l + i]);
}

// Triple-float: the unevaluated sum of three FP32 numbers, about 70 bits; the
// FP64 form adds its level sums in it on the FP32 pipe, 64 times the FP64 rate.
struct tf {
    float h, m, l;
};

__device__ __forceinline__ tf tf_add(tf a, tf b) {
    const df s = two_sum(a.h, b.h), t = two_sum(a.m, b.m), u = two_sum(t.hi, s.lo);
    const float l = __fadd_rn(__fadd_rn(a.l, b.l), __fadd_rn(t.lo, u.lo));
    const df h = fast_two_sum(s.hi, u.hi), m = two_sum(h.lo, l);
    return tf{h.hi, m.hi, m.lo};
}

__device__ __forceinline__ tf tf_mulf(tf a, float f) {
    const float p = __fmul_rn(a.h, f), q = __fmul_rn(a.m, f);
    const float e = __fmaf_rn(a.h, f, -p);
    const df s = two_sum(e, q);
    return tf{p, s.hi, __fadd_rn(s.lo, __fmaf_rn(a.l, f, __fmaf_rn(a.m, f, -q)))};
}

__device__ __forceinline__ tf tf_mul(tf a, tf b) {
    const float p = __fmul_rn(a.h, b.h), q = __fmul_rn(a.h, b.m), r = __fmul_rn(a.m, b.h);
    const float e = __fmaf_rn(a.h, b.h, -p);
    const df s = two_sum(q, r), t = two_sum(s.hi, e);
    float l = __fmaf_rn(a.m, b.m, __fadd_rn(__fmaf_rn(a.h, b.m, -q), __fmaf_rn(a.m, b.h, -r)));
    l = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, l));
    return tf{p, t.hi, __fadd_rn(l, __fadd_rn(s.lo, t.lo))};
}

__device__ __forceinline__ tf tf_neg(tf a) { return tf{-a.h, -a.m, -a.l}; }

__device__ __forceinline__ double tf_double(tf a) { return widen(a.h) + (widen(a.m) + widen(a.l)); }

// Operations that the kernels need on their sums, double-float or triple-float
__device__ __forceinline__ df sum_zero(df) { return df{0.f, 0.f}; }
__device__ __forceinline__ tf sum_zero(tf) { return tf{0.f, 0.f, 0.f}; }
__device__ __forceinline__ df sum_nan(df) { return df{NAN, 0.f}; }
__device__ __forceinline__ tf sum_nan(tf) { return tf{NAN, 0.f, 0.f}; }
__device__ __forceinline__ df sum_neg(df a) { return df_neg(a); }
__device__ __forceinline__ tf sum_neg(tf a) { return tf{-a.h, -a.m, -a.l}; }
__device__ __forceinline__ df sum_add(df a, df b) { return df_add(a, b); }
__device__ __forceinline__ tf sum_add(tf a, tf b) { return tf_add(a, b); }
__device__ __forceinline__ df sum_mulf(df a, float f) { return df_mulf_u(a, f); }
__device__ __forceinline__ tf sum_mulf(tf a, float f) { return tf_mulf(a, f); }
__device__ __forceinline__ double sum_double(df a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ double sum_double(tf a) { return tf_double(a); }
__device__ __forceinline__ df sum_xor(df a, int mask) {
    return df{__shfl_xor_sync(0xffffffffu, a.hi, mask), __shfl_xor_sync(0xffffffffu, a.lo, mask)};
}
__device__ __forceinline__ tf sum_xor(tf a, int mask) {
    return tf{__shfl_xor_sync(0xffffffffu, a.h, mask), __shfl_xor_sync(0xffffffffu, a.m, mask),
              __shfl_xor_sync(0xffffffffu, a.l, mask)};
}

// the level sums of one real output (column v of the levels read), in double-
// float (|lo| may exceed ulp(hi)/2 by a few units) and in triple-float
__device__ __forceinline__ df level_sum(const float (&t)[5][4], int v) {
    const df a = two_sum(t[0][v], t[1][v]), b = two_sum(t[2][v], t[3][v]);
    const df s = two_sum(a.hi, b.hi);
    return df{s.hi, __fadd_rn(__fadd_rn(s.lo, a.lo), __fadd_rn(b.lo, t[4][v]))};
}
__device__ __forceinline__ tf level_sum(const float (&t)[8][4], int v) {
    const df a = two_sum(t[0][v], t[1][v]), b = two_sum(t[2][v], t[3][v]), c = two_sum(t[4][v], t[5][v]);
    const df s = two_sum(a.hi, b.hi);
    const df m1 = two_sum(s.lo, a.lo), m2 = two_sum(m1.hi, b.lo), m3 = two_sum(m2.hi, c.hi);
    const float l = __fadd_rn(__fadd_rn(__fadd_rn(m1.lo, m2.lo), m3.lo),
                              __fadd_rn(c.lo, __fadd_rn(t[6][v], t[7][v])));
    const df m = two_sum(m3.hi, l);
    return tf{s.hi, m.hi, m.lo};
}

// ---- operand slices ---------------------------------------------------------

// 2^k for an exponent in the normal FP32 range (k clamped to it)
__device__ __forceinline__ float pow2f(int k) {
    k = max(-126, min(127, k));
    return __int_as_float((k + 127) << 23);
}

// Slices of x = h + l (|x| < 2^e): o[s] = m_s u 2^(-7s) with u = 2^(e-6) and
// integers |m_s| <= 64 (<= 72 for s = 3, which takes the low part's rounding),
// so that x = sum_s o[s] up to 2^(e-41).  Each slice rounds the remainder to a
// multiple of u 2^(-7s) by adding and subtracting 1.5 x 2^(23-7s) u (round to
// nearest even, no fast-math reassociation); slices 0-2 peel the high part
// exactly, the low part joins at slice 3 with one rounding below 2^(e-45).
struct Slicer6 {
    float c[6];
    __device__ __forceinline__ explicit Slicer6(float u) {
        c[0] = 0x1.8p23f * u;
        c[1] = 0x1.8p16f * u;
        c[2] = 0x1.8p9f * u;
        c[3] = 0x1.8p2f * u;
        c[4] = 0x1.8p-5f * u;
        c[5] = 0x1.8p-12f * u;
    }
    __device__ __forceinline__ void operator()(float h, float l, float (&o)[6]) const {
        o[0] = __fsub_rn(__fadd_rn(h, c[0]), c[0]);
        h = __fsub_rn(h, o[0]);
        o[1] = __fsub_rn(__fadd_rn(h, c[1]), c[1]);
        h = __fsub_rn(h, o[1]);
        o[2] = __fsub_rn(__fadd_rn(h, c[2]), c[2]);
        h = __fadd_rn(__fsub_rn(h, o[2]), l);
        o[3] = __fsub_rn(__fadd_rn(h, c[3]), c[3]);
        h = __fsub_rn(h, o[3]);
        o[4] = __fsub_rn(__fadd_rn(h, c[4]), c[4]);
        h = __fsub_rn(h, o[4]);
        o[5] = __fsub_rn(__fadd_rn(h, c[5]), c[5]);
    }
};

__device__ __forceinline__ uint32_t pack_bf2(float a, float b) {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);  // exact: every slice has <= 8 significant bits
    return *reinterpret_cast<uint32_t*>(&v);
}

// Seven slices of x = h + l (|x| < 2^e): o[s] = m_s u 2^(-7s), u = 2^(e-6),
// integers |m_s| <= 64, x = sum_s o[s] up to 2^(e-51).  As in the six-slice
// split, but the low part joins at slice 3 through an error-free sum, so that
// none of its bits above 2^-45 u is lost.
struct Slicer7 {
    float c[7];
    __device__ __forceinline__ explicit Slicer7(float u) {
        c[0] = 0x1.8p23f * u;
        c[1] = 0x1.8p16f * u;
        c[2] = 0x1.8p9f * u;
        c[3] = 0x1.8p2f * u;
        c[4] = 0x1.8p-5f * u;
        c[5] = 0x1.8p-12f * u;
        c[6] = 0x1.8p-19f * u;
    }
    __device__ __forceinline__ void operator()(float h, float l, float (&o)[7]) const {
        o[0] = __fsub_rn(__fadd_rn(h, c[0]), c[0]);
        h = __fsub_rn(h, o[0]);
        o[1] = __fsub_rn(__fadd_rn(h, c[1]), c[1]);
        h = __fsub_rn(h, o[1]);
        o[2] = __fsub_rn(__fadd_rn(h, c[2]), c[2]);
        h = __fsub_rn(h, o[2]);
        const df j = two_sum(h, l);  // h + l = j.hi + j.lo exactly
        o[3] = __fsub_rn(__fadd_rn(j.hi, c[3]), c[3]);
        h = __fadd_rn(__fsub_rn(j.hi, o[3]), j.lo);
        o[4] = __fsub_rn(__fadd_rn(h, c[4]), c[4]);
        h = __fsub_rn(h, o[4]);
        o[5] = __fsub_rn(__fadd_rn(h, c[5]), c[5]);
        h = __fsub_rn(h, o[5]);
        o[6] = __fsub_rn(__fadd_rn(h, c[6]), c[6]);
    }
};

// The FP64 form's slices: x (|x| < 2^e) in fixed point to 2^(e-55), truncated,
// cut into eight 7-bit digits m_s in [-64, 64], x = 2^(e-6) sum_s m_s 2^(-7s),
// with integer operations alone (GB300 has 64 FP32 and 32 integer lanes for
// each FP64 one).  The word holds the digits plus 64 each, digit s at bit
// 7 (7 - s); |x| <= 2^e (1 - 2^-11) keeps the word below 2^56 + 2^49.
__device__ __forceinline__ unsigned long long fixed8(double x, int e) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    // an exponent far below e, zero and subnormals among them, shifts everything out
    const int r = min(e + 1022 - (int)((u >> 52) & 0x7ff), 63);
    const unsigned long long f = (((u & 0xfffffffffffffULL) | 0x10000000000000ULL) << 2) >> r;
    constexpr unsigned long long bias = 64ULL * (((1ULL << 56) - 1) / 127);  // 64 in every digit
    const unsigned long long neg = (unsigned long long)((long long)u >> 63);
    return (f ^ neg) + (bias - neg);
}

// The digits of two words as bf16 pairs, digit s times 2^(-7s): 128 + u is the
// bf16 with u in its mantissa field (u = 128, digit 0 only, carries into the
// exponent: 256), and 192 = 128 + 64 comes off in one exact FMA.  A byte
// permutation puts 16 bits of each word side by side, so that one shift and one
// mask serve both.
__device__ __forceinline__ uint32_t digit_fma(uint32_t v, float w) {
    const __nv_bfloat162 r = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&v), __float2bfloat162_rn(w),
                                     __float2bfloat162_rn(-192.f * w));
    return *reinterpret_cast<const uint32_t*>(&r);
}
__device__ __forceinline__ void digit_pairs(unsigned long long a, unsigned long long b, uint32_t (&o)[8]) {
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    constexpr uint32_t kMask = 0x007f007fu, kOne = 0x43004300u;
    const uint32_t w0 = __byte_perm(al, bl, 0x5410);  // bits 0-15
    o[7] = digit_fma((w0 & kMask) | kOne, 0x1p-49f);
    o[6] = digit_fma(((w0 >> 7) & kMask) | kOne, 0x1p-42f);
    o[5] = digit_fma(((__byte_perm(al, bl, 0x6521) >> 6) & kMask) | kOne, 0x1p-35f);  // bits 8-23
    o[4] = digit_fma(((__byte_perm(al, bl, 0x7632) >> 5) & kMask) | kOne, 0x1p-28f);  // bits 16-31
    o[3] = digit_fma((__byte_perm(__funnelshift_r(al, ah, 28), __funnelshift_r(bl, bh, 28), 0x5410) & kMask) | kOne,
                     0x1p-21f);
    o[2] = digit_fma(((__byte_perm(ah, bh, 0x5410) >> 3) & kMask) | kOne, 0x1p-14f);
    o[1] = digit_fma(((__byte_perm(ah, bh, 0x6521) >> 2) & kMask) | kOne, 0x1p-7f);
    o[0] = digit_fma(((__byte_perm(ah, bh, 0x7632) >> 1) & 0x00ff00ffu) + kOne, 1.f);
}

// element offset of (row, k) in a stage tile [rows][16 K] of core matrices
__device__ __forceinline__ int tile_off(int row, int k) {
    return (((row >> 3) * 2 + (k >> 3)) << 6) + ((row & 7) << 3) + (k & 7);
}

// stage counter of a ring of n buffers: index and phase parity
struct Ring {
    int i = 0, n;
    uint32_t ph = 0;
    __device__ __forceinline__ explicit Ring(int n_) : n(n_) {}
    __device__ __forceinline__ void next() {
        if (++i == n) {
            i = 0;
            ph ^= 1u;
        }
    }
};

// (-i)^p z
__device__ __forceinline__ cdf rot_mi(cdf z, int p) {
    switch (p & 3) {
        case 0: return z;
        case 1: return cdf{z.im, df_neg(z.re)};
        case 2: return cdf{df_neg(z.re), df_neg(z.im)};
        default: return cdf{df_neg(z.im), z.re};
    }
}

// exponent of |x|, x < 2^(exponent + 1): one above FP32's (FP64's) largest for infinities and NaN, one below the
// smallest for zero and subnormals
__device__ __forceinline__ int exponent(float x) { return (int)((__float_as_uint(x) >> 23) & 0xffu) - 127; }
__device__ __forceinline__ int exponent(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) - 1023; }

// |x| 2^-es for es >= its exponent, rounded up; FP64 (off its pipe): 0 where it is below 2^-100
__device__ __forceinline__ float relative(float x, int es) { return fabsf(x) * (1.0001f * pow2f(-es)); }
__device__ __forceinline__ float relative(double x, int es) {
    const int k = exponent(x) - es;
    const unsigned hi = (unsigned)__double2hiint(x), mantissa = ((hi & 0xfffffu) << 3) | ((unsigned)__double2loint(x) >> 29);
    return k < -100 ? 0.f : __uint_as_float(((unsigned)(k + 127) << 23) + mantissa + 2u);
}

// log2 of a number that is zero (-infinity) or normal
__device__ __forceinline__ float log2_normal(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// x 2^k for a sum of FP32 numbers and |k| <= 860, so that the result is a normal number: by its exponent field, off the
// FP64 pipe
__device__ __forceinline__ double scale_pow2(double x, int k) {
    const int hi = __double2hiint(x);
    const bool normal = (unsigned)((hi & 0x7ff00000) - 0x100000) < 0x7fe00000u;  // neither zero nor infinite nor NaN
    return __hiloint2double(normal ? hi + (k << 20) : hi, __double2loint(x));
}

__device__ __forceinline__ int exp_bound(float log2_bound) {
    // smallest e with 2^e > the bound, from a log2 estimate good to ~1e-4
    if (!(log2_bound > -100.f)) return -100;
    return (int)floorf(log2_bound + 1e-3f) + 1;
}

__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(saddr(dst)), "l"(src), "r"(bytes), "r"(saddr(bar))
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive_tx(uint64_t* b, uint32_t tx) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(saddr(b)),
                 "r"(tx)
                 : "memory");
}

// index of D'_{p1 p2 p3} (powers of n_1, n_2, n_3) for powers (i, j, k) of (n_a, n_b, n_c)
__device__ __forceinline__ int term_of(int ax, int bx, int i, int j, int k) {
    const int p1 = ax == 0 ? i : (bx == 0 ? j : k);
    const int p2 = ax == 1 ? i : (bx == 1 ? j : k);
    const int lam = i + j + k;
    return lam_offset(lam) + mono_index(lam, p1, p2);
}

// |n|^k for k <= 4, exact
__device__ __forceinline__ float ipow(float n, int k) {
    float p = 1.f;
    for (int q = 0; q < k; ++q) p *= n;
    return p;
}

// columns of an MMA over nb blocks
__host__ __device__ __forceinline__ int mma_cols(int nb, int colw) { return (nb * colw + 15) / 16 * 16; }

// ---- the two precisions of the product -----------------------------------------
//
// S slices per operand, ACC level accumulators, Comp the table component (a
// real or imaginary part), Sum the type that adds level sums.  pair() multiplies
// the X and Y parts of two K entries and cuts both products; a row's bound 2^e
// is in the slices (split form) or comes back through row_scale (FP64 form,
// whose A digits carry only 2^(-7s)).

template <int NS, class Cutter>
struct SplitPrec {
    static constexpr int S = NS, ACC = 5;  // levels 0-3 exact, the rest in a rounded fifth accumulator
    using Comp = float2;
    using Sum = df;
    struct Cut {
        Cutter c;
        __device__ __forceinline__ explicit Cut(int e) : c(pow2f(e - 6)) {}
        __device__ __forceinline__ void pair(df a, df b, uint32_t (&o)[S]) const {
            float oa[S], ob[S];
            c(a.hi, a.lo, oa);
            c(b.hi, b.lo, ob);
#pragma unroll
            for (int s = 0; s < S; ++s) o[s] = pack_bf2(oa[s], ob[s]);
        }
    };
    using Entry = df;
    __device__ static __forceinline__ Entry product(float2 x, float2 y) { return df_mul_u(df{x.x, x.y}, df{y.x, y.y}); }
    __device__ static __forceinline__ Entry entry(float2 x) { return df{x.x, x.y}; }
    __device__ static __forceinline__ float row_scale(int) { return 1.f; }
    static constexpr int kWin = kTcWinMax, kNmax = kTcNmax;
    static constexpr int kRefMin = -120, kRefMax = 126, kColMin = -100;  // as for Prec64, in FP32
};
using PrecRho = SplitPrec<6, Slicer6>;
using PrecJ = SplitPrec<7, Slicer7>;

// Eight slices, 36 products s + t <= 7, every level in an accumulator of its
// own: 64^2 x 8 products x 512 K terms = 2^24 keeps all of them exact over a
// window of 512, and 56 bits below the bounds of the window leave the sums with
// a smaller error than FP64 accumulation.
struct Prec64 {
    static constexpr int S = 8, ACC = 8;
    using Comp = double;
    using Sum = tf;
    struct Cut {
        int e;
        __device__ __forceinline__ explicit Cut(int e_) : e(e_) {}
        __device__ __forceinline__ void pair(double a, double b, uint32_t (&o)[S]) const {
            digit_pairs(fixed8(a, e), fixed8(b, e), o);
        }
    };
    using Entry = double;
    __device__ static __forceinline__ Entry product(double x, double y) { return x * y; }
    __device__ static __forceinline__ Entry entry(double x) { return x; }
    __device__ static __forceinline__ float row_scale(int e) { return pow2f(e - 6); }
    static constexpr int kWin = kTcWinMax / 2, kNmax = kTcNmax64;
    // B's (V's) digits carry their column's exponent relative to the largest of their window (their (i, j)) and density:
    // at most 60 below it, where the last digit is 2^-115 of the largest bound and every product is still a normal FP32
    // number.  The reference itself covers FP64's range but for its ends (scale_pow2).
    static constexpr int kRefMin = -850, kRefMax = 850, kColMin = -60;
};

// the reference exponent of columns whose largest exponent is top, and a column's own relative to it
template <class P>
__device__ __forceinline__ int ref_exp(int top) {
    return max(P::kRefMin, min(P::kRefMax, top));
}
template <class P>
__device__ __forceinline__ int col_exp(int e, int ref) {
    return max(e - ref, P::kColMin);
}

// the exponent of a row bound of A (log2; at most 1), not below -60 in the FP64 form, where the last slice sits 2^-55
// under it
template <class P>
__device__ __forceinline__ int bound_exp(float log2_bound) {
    return P::S == 8 ? max(exp_bound(log2_bound), -60) : exp_bound(log2_bound);
}

constexpr int kTcProdWarps = 16;                    // two groups of eight, stages in turn
constexpr int kTcGroupWarps = kTcProdWarps / 2;
constexpr int kTcMmaWarp = 16;
constexpr int kTcTabWarp = 17;
constexpr int kTcLoadWarp = 18;
constexpr int kTcWarps = 19;
constexpr int kTcThreadsAll = kTcWarps * 32;

// ---- B: window scales and slices, once per build and density group ---------

constexpr int kTcBThreads = 512;

// One block per window.  First the scales: the window's smallest width c
// (every row of A gets the bound exp(-c_min Q)) and the column bounds of B,
// |B_ij| <= exp(-c Mcc n^2) sum_k |D'_ijk| n^k maximised over the window's
// records, per (block, n_c, density).  Then the slices: one thread per four
// records of one (block, n_c, density), both columns (Re, Im), as halves of
// 16-byte core-matrix rows; neighbouring lanes take the other half, neighbouring
// columns and record octets, so a warp's stores of one slice fill 512-byte runs.
// DF: D' as the split form's Hermite map writes it, double-float in the K
// order; otherwise (FP64 form) doubles in record order.
template <class P, bool DF>
__global__ void __launch_bounds__(kTcBThreads, P::S == 8 ? 1 : 2) k_tc_rho_b(TcArgs g) {
    constexpr bool kF64 = P::S == 8;
    static_assert(kF64 || DF, "the six-slice operands are cut from double-float terms");
    constexpr int kS = P::S;
    __shared__ int mx[kTcNmax / 2], top[kTcNmax / 2];  // exponents of the column bounds; the largest per density
    __shared__ int bad[kTcNmax / 2];
    __shared__ int pairs[kTcGmax], tidx[kTcGmax][5];
    __shared__ int clmin_bits;
    const int w = g.w0 + blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    const int4 wi = __ldg(g.winfo + w);
    const int L = wi.x, npair = wi.y, npo = g.nd * g.ncols, cnt = __ldg(g.wcnt + w);
    for (int i = tid; i < npair * npo; i += blockDim.x) mx[i] = INT_MIN / 2;
    if (tid < g.nd) {
        bad[tid] = 0;
        top[tid] = INT_MIN / 2;
    }
    if (tid < npair) {
        const int pr = __ldg(g.wpairs + wi.z + tid), i = pr & 7, j = pr >> 3;
        pairs[tid] = pr;
        for (int kk = 0; kk < 5; ++kk) tidx[tid][kk] = kk <= L - i - j ? term_of(g.ax, g.bx, i, j, kk) : -1;
    }
    if (tid == 0) clmin_bits = __float_as_int(INFINITY);
    __syncthreads();
    const long long stride = g.dp_stride[L];
    // double-float terms: this window's positions; doubles: the class's records
    const float2* dpw = reinterpret_cast<const float2*>(g.Dp) + g.dp_base[L] + (long long)g.d0 * g.dp_total + wi.w;
    const double* dp64 = reinterpret_cast<const double*>(g.Dp) + g.dp_base[L] + (long long)g.d0 * g.dp_total;
    const long long kb = g.kbase[L] + wi.w;  // the window's first record in the K order
    constexpr int kIt = P::kWin / kTcBThreads;
    float cr[kIt], cmin = INFINITY;
    int ko[kIt];
#pragma unroll
    for (int q = 0; q < kIt; ++q) {
        const int k = tid + q * kTcBThreads;
        cr[q] = k < cnt ? __ldg(g.clk + kb + k) : 0.f;
        if (k < cnt) cmin = fminf(cmin, cr[q]);
        ko[q] = !DF && k < cnt ? __ldg(g.korder + kb + k) : 0;
    }
    for (int gb = 0; gb < npair; ++gb)
        for (int d = 0; d < g.nd; ++d) {
            using Term = std::conditional_t<DF, float, double>;
            float cm[kIt][5], es[kIt];
#pragma unroll
            for (int q = 0; q < kIt; ++q) {
                const int k = tid + q * kTcBThreads;
                Term v[5];
#pragma unroll
                for (int kk = 0; kk < 5; ++kk) {
                    const int t = tidx[gb][kk];
                    v[kk] = 0;
                    if (t < 0 || k >= cnt) continue;
                    const long long off = (long long)d * g.dp_total + (long long)t * stride;
                    if constexpr (DF) v[kk] = __ldg(dpw + off + k).x;
                    else v[kk] = __ldg(dp64 + off + ko[q]);
                }
                // relative to the record's largest term, so that a bound neither overflows nor underflows
                int e = exponent(v[0]);
#pragma unroll
                for (int kk = 1; kk < 5; ++kk) e = max(e, exponent(v[kk]));
                if (e == (DF ? 128 : 1024)) bad[d] = 1;
#pragma unroll
                for (int kk = 0; kk < 5; ++kk) cm[q][kk] = k < cnt ? relative(v[kk], e) : 0.f;
                es[q] = (float)e;
            }
            int etop = INT_MIN / 2;
            for (int nc = 0; nc < g.ncols; ++nc) {
                const float x = (float)nc, mq = -g.Mcc * x * x;
                float m = -1e9f;
#pragma unroll
                for (int q = 0; q < kIt; ++q) {
                    const float sv = cm[q][0] + x * (cm[q][1] + x * (cm[q][2] + x * (cm[q][3] + x * cm[q][4])));
                    m = fmaxf(m, log2_normal(sv) + (es[q] + cr[q] * mq));
                }
                const int me = __reduce_max_sync(0xffffffffu, __float2int_rd(m + 1e-3f) + 1);
                etop = max(etop, me);
                if (lane == 0) atomicMax(&mx[gb * npo + nc * g.nd + d], me);
            }
            if (lane == 0) atomicMax(&top[d], etop);
        }
    for (int o = 16; o > 0; o >>= 1) cmin = fminf(cmin, __shfl_xor_sync(0xffffffffu, cmin, o));
    if (lane == 0 && cmin < INFINITY) atomicMin(&clmin_bits, __float_as_int(cmin));
    __syncthreads();
    if (tid == 0) g.clw[w] = __int_as_float(clmin_bits);
    if (tid < g.nd) g.ew[w * g.nd + tid] = bad[tid] ? kNonFinite : ref_exp<P>(top[tid]);
    const int nst = (cnt + kTcStageK - 1) / kTcStageK, npc = (npo + 3) / 4, nw = mma_cols(npair, g.colw);
    uint4* base = g.bs + __ldg(g.boff + w);
    const int ntask = nst * npair * npc * 16;
    for (int idx = tid; idx < ntask; idx += kTcBThreads) {
        int rest = idx >> 4;
        const int half = idx & 1, oc = (idx >> 3) & 1, p = 4 * (rest % npc) + ((idx >> 1) & 3);
        rest /= npc;
        const int gb = rest % npair, q = rest / npair;
        if (p >= npo) continue;  // columns past the block's outputs are never read back
        const int nc = p / g.nd, d = p - nc * g.nd;
        const int pr = pairs[gb], nk = L - (pr & 7) - (pr >> 3);  // k = 0 .. L - i - j
        const int k0 = q * kTcStageK + oc * 8 + half * 4;
        const int er = ref_exp<P>(top[d]), ec = col_exp<P>(mx[gb * npo + p], er);
        uint32_t s0[kS][2], s1[kS][2];
        if constexpr (kF64) {
            const float sc = pow2f(ec - 6);  // B's digits carry their column's relative bound
            const int eb = bad[d] ? kNonFinite : er + ec;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                unsigned long long fr[2], fi[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int k = k0 + 2 * u + e;
                    double br = 0.0, bi = 0.0;
                    if (k < cnt) {
                        const long long at = (long long)d * g.dp_total + (DF ? (long long)k : (long long)__ldg(g.korder + kb + k));
                        auto term = [&](int kk) {
                            const long long o = at + (long long)tidx[gb][kk] * stride;
                            if constexpr (DF) {
                                const float2 v = __ldg(dpw + o);
                                return join_df(df{v.x, v.y});
                            } else {
                                return __ldg(dp64 + o);
                            }
                        };
                        const double2 z = __ldg(reinterpret_cast<const double2*>(g.tabz) + (kb + k) * g.ncols + nc);
                        // sum_k D'_k (-i n_c)^k: terms of even k real, of odd k imaginary (few FP64 instructions:
                        // the pipe has 2 lanes per SM)
                        double re = term(0);
                        if (nk == 0) {
                            br = z.x * re;
                            bi = z.y * re;
                        } else {
                            const double x = widen((float)nc);
                            double im = -x * term(1);
                            if (nk > 1) re = fma(-widen((float)(nc * nc)), term(2), re);
                            if (nk > 2) im = fma(widen((float)(nc * nc * nc)), term(3), im);
                            if (nk > 3)
                                re = fma(widen((float)(nc * nc * nc * nc)), term(4), re);
                            br = z.x * re - z.y * im;
                            bi = z.x * im + z.y * re;
                        }
                    }
                    fr[e] = fixed8(br, eb);
                    fi[e] = fixed8(bi, eb);
                }
                float w = sc;
#pragma unroll
                for (int s = 0; s < kS; ++s, w *= 0x1p-7f) {
                    const int sh = 7 * (7 - s);
                    auto digit = [&](unsigned long long f) {
                        return (float)((int)((f >> sh) & (s == 0 ? 0xffULL : 0x7fULL)) - 64) * w;
                    };
                    s0[s][u] = pack_bf2(digit(fr[0]), digit(fr[1]));
                    s1[s][u] = pack_bf2(digit(fi[0]), digit(fi[1]));
                }
            }
        } else {
            const typename P::Cut cut(ec);
            const float unref = pow2f(-er);
            const float2* dpd = dpw + (long long)d * g.dp_total + k0;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                df re[2], im[2];
                re[0] = re[1] = im[0] = im[1] = df{0.f, 0.f};
                float pw = 1.f;
                for (int kk = 0; kk <= nk; ++kk) {
                    // two records' D'_k (16-byte aligned: classes, windows and halves start at even positions)
                    const float4 v = __ldg(reinterpret_cast<const float4*>(dpd + (long long)tidx[gb][kk] * stride + 2 * u));
                    const df a = df_mulf(df{v.x, v.y}, pw), b = df_mulf(df{v.z, v.w}, pw);  // D'_k n_c^k, exact power
                    switch (kk & 3) {                                                       // (-i)^k
                        case 0: re[0] = df_add(re[0], a); re[1] = df_add(re[1], b); break;
                        case 1: im[0] = df_sub(im[0], a); im[1] = df_sub(im[1], b); break;
                        case 2: re[0] = df_sub(re[0], a); re[1] = df_sub(re[1], b); break;
                        default: im[0] = df_add(im[0], a); im[1] = df_add(im[1], b); break;
                    }
                    pw *= (float)nc;
                }
                cdf bv[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int k = k0 + 2 * u + e;
                    bv[e] = cdf{{0.f, 0.f}, {0.f, 0.f}};
                    if (k < cnt) {
                        const float4 zv = __ldg(reinterpret_cast<const float4*>(g.tabz) + (kb + k) * g.ncols + nc);
                        const cdf t = cdf_mul(cdf{{zv.x, zv.y}, {zv.z, zv.w}}, cdf{re[e], im[e]});
                        bv[e] = cdf{{t.re.hi * unref, t.re.lo * unref}, {t.im.hi * unref, t.im.lo * unref}};
                    }
                }
                uint32_t o[kS];
                cut.pair(bv[0].re, bv[1].re, o);
#pragma unroll
                for (int s = 0; s < kS; ++s) s0[s][u] = o[s];
                cut.pair(bv[0].im, bv[1].im, o);
#pragma unroll
                for (int s = 0; s < kS; ++s) s1[s][u] = o[s];
            }
        }
        const int col = gb * g.colw + 2 * p;
        uint2* dst = reinterpret_cast<uint2*>(base + (size_t)q * kS * nw * 2 + ((col >> 3) * 2 + oc) * 8 + (col & 7)) + half;
#pragma unroll
        for (int s = 0; s < kS; ++s) {
            dst[(size_t)s * nw * 4] = make_uint2(s0[s][0], s0[s][1]);
            dst[(size_t)s * nw * 4 + 2] = make_uint2(s1[s][0], s1[s][1]);
        }
    }
}

// ---- the product ---------------------------------------------------------------

struct TcSmem {
    uint64_t afull[kTcNbufMax], bfull[kTcNbufMax], empty[kTcNbufMax], accf, acce, done;
    uint64_t tfull[kTcTabSlotsMax], tempty[kTcTabSlotsMax];
    uint32_t tmem;
    int abort_flag;
};

__host__ __device__ inline size_t tab_slot_bytes(int tws) { return (size_t)kTcStageK * tws * 16; }

// waits (bounded) until the copies counted on the barriers of a ring have
// landed, `issued` stages into it: nothing is in flight when the CTA exits
__device__ void ring_settle(uint64_t* bar, int n, long long issued) {
    for (int b = 0; b < n && b < issued; ++b) {
        const long long last = issued - 1 - ((issued - 1 - b) % n);  // last stage that used slot b
        const long long t0 = clock64();
        while (!mbar_test(bar + b, (uint32_t)((last / n) & 1)) && clock64() - t0 < kTcSpinCycles) {
        }
    }
}

template <class P, int NU>
__global__ void __launch_bounds__(kTcThreadsAll, 1) k_tc_rho(TcArgs g, int nbuf, int ntslots) {
    extern __shared__ __align__(1024) unsigned char tsm[];
    unsigned char* abuf = tsm;                                                // [nbuf][S][4096]
    unsigned char* bbuf = abuf + (size_t)nbuf * P::S * kTcAsliceBytes;         // [nbuf][S][npad*32]
    const int bbytes = P::S * g.npad * 32;
    unsigned char* tring = bbuf + (size_t)nbuf * bbytes;                       // [ntslots][slot]
    const size_t tslot = tab_slot_bytes(g.tws);
    TcSmem& sm = *reinterpret_cast<TcSmem*>(tring + (size_t)ntslots * tslot);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int kg = blockIdx.x, mt = blockIdx.y;
    const int j0 = __ldg(g.sched + kg), j1 = __ldg(g.sched + kg + 1);
    const int* wlist = g.sched + gridDim.x + 1;
    volatile int* abort_flag = &sm.abort_flag;

    if (tid == 0) {
        for (int b = 0; b < nbuf; ++b) {
            mbar_init(&sm.afull[b], kTcGroupWarps);
            mbar_init(&sm.bfull[b], 1);
            mbar_init(&sm.empty[b], 1);
        }
        for (int b = 0; b < ntslots; ++b) {
            mbar_init(&sm.tfull[b], 1);
            mbar_init(&sm.tempty[b], kTcGroupWarps);
        }
        mbar_init(&sm.accf, 1);
        mbar_init(&sm.acce, kTcProdWarps);
        mbar_init(&sm.done, 1);
        sm.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // the table slots start finite: records past a window's end are not copied, their A entries meet zeros of B
    for (int i = tid; i < (int)(ntslots * tslot / 16); i += kTcThreadsAll)
        reinterpret_cast<uint4*>(tring)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (warp == kTcMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&sm.tmem)),
                     "r"(kTcTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tmem;
    bool ok = true;

    if (warp == kTcTabWarp) {
        // the stages' X and Y tables: consecutive records of the K order, one bulk copy each
        if (lane == 0) {
            Ring t(ntslots);
            long long gt = 0;
            for (int jw = j0; jw < j1 && ok; ++jw) {
                const int w = __ldg(wlist + jw), cnt = __ldg(g.wcnt + w);
                const int4 wi = __ldg(g.winfo + w);
                const float4* src = reinterpret_cast<const float4*>(g.tabk) + (g.kbase[wi.x] + wi.w) * g.tws;
                for (int k0 = 0; k0 < cnt; k0 += kTcStageK, ++gt, t.next()) {
                    if (gt >= ntslots && !(ok = mbar_wait(&sm.tempty[t.i], t.ph ^ 1u, abort_flag, g.spin))) break;
                    const uint32_t bytes = (uint32_t)(min(kTcStageK, cnt - k0) * g.tws) * 16u;
                    mbar_arrive_tx(&sm.tfull[t.i], bytes);
                    bulk_copy(tring + (size_t)t.i * tslot, src + (size_t)k0 * g.tws, bytes, &sm.tfull[t.i]);
                }
            }
            ring_settle(sm.tfull, ntslots, gt);
        }
        __syncwarp();
    } else if (warp == kTcLoadWarp) {
        // the stages' B tiles, one bulk copy each
        if (lane == 0) {
            Ring b(nbuf);
            long long gs = 0;
            for (int jw = j0; jw < j1 && ok; ++jw) {
                const int w = __ldg(wlist + jw), nst = (__ldg(g.wcnt + w) + kTcStageK - 1) / kTcStageK;
                const uint32_t bb = (uint32_t)(P::S * mma_cols(__ldg(&g.winfo[w].y), g.colw) * 32);
                const unsigned char* src = reinterpret_cast<const unsigned char*>(g.bs + __ldg(g.boff + w));
                for (int q = 0; q < nst; ++q, ++gs, b.next()) {
                    if (gs >= nbuf && !(ok = mbar_wait(&sm.empty[b.i], b.ph ^ 1u, abort_flag, g.spin))) break;
                    mbar_arrive_tx(&sm.bfull[b.i], bb);
                    bulk_copy(bbuf + (size_t)b.i * bbytes, src + (size_t)q * bb, bb, &sm.bfull[b.i]);
                }
            }
            ring_settle(sm.bfull, nbuf, gs);
        }
        __syncwarp();
    } else if (warp == kTcMmaWarp) {
        const uint32_t a0 = saddr(abuf), b0 = saddr(bbuf);
        Ring b(nbuf);
        for (int jw = j0; jw < j1 && ok; ++jw) {
            const int w = __ldg(wlist + jw), nst = (__ldg(g.wcnt + w) + kTcStageK - 1) / kTcStageK;
            const uint32_t nw = (uint32_t)mma_cols(__ldg(&g.winfo[w].y), g.colw);
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTcM >> 4) << 24);
            // the window's first MMAs wait for the drain of the previous one
            if (jw > j0 && !(ok = __all_sync(0xffffffffu, mbar_wait(&sm.acce, (uint32_t)((jw - j0 - 1) & 1), abort_flag, g.spin))))
                break;
            tc_fence_after();
            for (int q = 0; q < nst; ++q, b.next()) {
                ok = __all_sync(0xffffffffu, mbar_wait(&sm.bfull[b.i], b.ph, abort_flag, g.spin) &&
                                                 mbar_wait(&sm.afull[b.i], b.ph, abort_flag, g.spin));
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) {
                    issue_kstep<P::S, P::ACC>(tmem, sdesc(a0 + b.i * P::S * kTcAsliceBytes), kTcAsliceBytes >> 4,
                                              sdesc(b0 + b.i * bbytes), nw * 2, nw, idesc, q > 0);
                    tc_commit(&sm.empty[b.i]);
                    if (q + 1 == nst) tc_commit(&sm.accf);
                }
                __syncwarp();
            }
        }
        // everything issued completes before tensor memory is freed
        if (elect_one()) {
            tc_commit(&sm.done);
            const long long t0 = clock64();
            while (!mbar_test(&sm.done, 0u) && clock64() - t0 < kTcSpinCycles) {
            }
        }
        __syncwarp();
    } else {
        // forms row `row` of A for the records 8 oct .. 8 oct + 7 of its group's stages
        const int grp = warp / kTcGroupWarps, row = tid & (kTcM - 1), oct = (tid >> 7) & 1;
        const int sl = __ldg(g.slots + mt * kTcM + row);
        const float fa = (float)(sl & 255), fb = (float)((sl >> 8) & 255);
        const float Q = g.Maa * fa * fa + g.Mbb * fb * fb;
        const int rs = 2 * g.tws;  // components per record
        const int xo = oct * 8 * rs + 2 * (sl & 255) + ((sl >> 16) & 1);
        const int yo = oct * 8 * rs + 2 * (g.offY + ((sl >> 8) & 255)) + ((sl >> 17) & 1);
        unsigned char* arow = abuf + tile_off(row, oct * 8) * 2;
        // drains: tensor-memory lanes 32 (warp & 3) .. + 31, 4-column units warp / 4 + 4 x of each block
        const int eq = warp & 3, es = warp >> 2, erow = 32 * eq + lane;
        const uint32_t tlane = (uint32_t)(32 * eq) << 16;
        const int es_slot = __ldg(g.slots + mt * kTcM + erow);
        const float ea = (float)(es_slot & 255), eb = (float)((es_slot >> 8) & 255);
        const int ca = (es_slot >> 16) & 1, cb = (es_slot >> 17) & 1;
        const int nunit = g.colw / 4, npo = g.nd * g.ncols;
        typename P::Sum S[NU][4];  // sums by sign character: two complex outputs per unit
#pragma unroll
        for (int x = 0; x < NU; ++x)
#pragma unroll
            for (int v = 0; v < 4; ++v) S[x][v] = sum_zero(typename P::Sum());
        const float eQ = g.Maa * ea * ea + g.Mbb * eb * eb;
        // the sums of a density are relative to the largest exponent of the CTA's windows, lane d density d's
        int eref = 0;
        auto of_density = [](auto v, int d) { return __shfl_sync(0xffffffffu, v, d); };
        // densities of a unit's two outputs: p = 2 un + h belongs to p mod nd, the next unit's is 8 on
        const int d00 = (2 * es) % g.nd, d01 = (2 * es + 1) % g.nd, dstep = 8 % g.nd;
        Ring b(nbuf), t(ntslots);
        int gs = 0;  // stages so far (mod 2 the group that forms it)
        bool full = false;  // every buffer used once
        for (int jw = j0; jw < j1 && ok; ++jw) {
            const int w = __ldg(wlist + jw), nst = (__ldg(g.wcnt + w) + kTcStageK - 1) / kTcStageK;
            const float cl = __ldg(g.clw + w);
            const int ew = lane < g.nd ? __ldg(g.ew + w * g.nd + lane) : P::kRefMin;
            const typename P::Cut cut(bound_exp<P>(-cl * Q));
            for (int q = 0; q < nst; ++q, ++gs, b.next(), t.next()) {
                full = full || gs >= nbuf;
                if ((gs & 1) != grp) continue;
                ok = __all_sync(0xffffffffu, mbar_wait(&sm.tfull[t.i], t.ph, abort_flag, g.spin));
                if (!ok) break;
                const typename P::Comp* tb = reinterpret_cast<const typename P::Comp*>(tring + (size_t)t.i * tslot);
                uint32_t pk[P::S][4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    uint32_t o[P::S];
                    cut.pair(P::product(tb[2 * u * rs + xo], tb[2 * u * rs + yo]),
                             P::product(tb[(2 * u + 1) * rs + xo], tb[(2 * u + 1) * rs + yo]), o);
#pragma unroll
                    for (int s = 0; s < P::S; ++s) pk[s][u] = o[s];
                }
                if (full) {
                    ok = __all_sync(0xffffffffu, mbar_wait(&sm.empty[b.i], b.ph ^ 1u, abort_flag, g.spin));
                    if (!ok) break;
                }
                unsigned char* as = arow + (size_t)b.i * P::S * kTcAsliceBytes;
#pragma unroll
                for (int s = 0; s < P::S; ++s)
                    *reinterpret_cast<uint4*>(as + (size_t)s * kTcAsliceBytes) =
                        make_uint4(pk[s][0], pk[s][1], pk[s][2], pk[s][3]);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&sm.afull[b.i]);
                    mbar_arrive(&sm.tempty[t.i]);
                }
            }
            if (!ok) break;
            // (read before the wait below, which hides it)
            if (jw == j0)
                for (int d = 0; d < g.nd; ++d) {
                    int e = INT_MIN / 2;
                    for (int k = j0 + lane; k < j1; k += 32) {
                        const int ek = __ldg(g.ew + __ldg(wlist + k) * g.nd + d);
                        if (ek != kNonFinite) e = max(e, ek);
                    }
                    e = __reduce_max_sync(0xffffffffu, e);
                    if (lane == d) eref = e;
                }
            // powers of two of this window's densities (lane d density d's), relative to the sums', 0 where they are
            // below 2^-126; then of the two outputs of each unit, as the upper halves of two floats (the crystal's pass
            // against unscaled sums: 1348 -> 1375 us; 1383 with an exponent and a remainder per output and window)
            const unsigned half = (unsigned)max(min(ew - eref, 0) + 127, 0) << 7;
            unsigned rel[NU];
            int d0 = d00, d1 = d01;
#pragma unroll
            for (int x = 0; x < NU; ++x) {
                if (x > 0 && dstep == 0) {  // 1, 2, 4 or 8 densities: every unit holds the same two
                    rel[x] = rel[0];
                    continue;
                }
                rel[x] = of_density(half, d0) | (of_density(half, d1) << 16);
                d0 += dstep;
                d1 += dstep;
                if (d0 >= g.nd) d0 -= g.nd;
                if (d1 >= g.nd) d1 -= g.nd;
            }
            if (__any_sync(0xffffffffu, ew == kNonFinite)) {
#pragma unroll
                for (int x = 0; x < NU; ++x)
#pragma unroll
                    for (int v = 0; v < 4; ++v)
                        if (of_density(ew, (2 * (es + 4 * x) + (v >> 1)) % g.nd) == kNonFinite)
                            S[x][v] = sum_nan(typename P::Sum());
            }
            // ---- drain: each block's level sums, times (-i)^{i+j} n_a^i n_b^j, into the sums by character ----
            ok = __all_sync(0xffffffffu, mbar_wait(&sm.accf, (uint32_t)((jw - j0) & 1), abort_flag, g.spin));
            if (!ok) break;
            tc_fence_after();
            const int4 wi = __ldg(g.winfo + w);
            const uint32_t nw = (uint32_t)mma_cols(wi.y, g.colw);
            const float rsc = P::row_scale(bound_exp<P>(-cl * eQ));
            for (int gb = 0; gb < wi.y; ++gb) {
                const int pr = __ldg(g.wpairs + wi.z + gb), i = pr & 7, j = pr >> 3;
                // type (ta, tb) of lane ^ mask adds to this lane's character; i^{ta - i} = i^{ca} times a real sign
                const int mask = (i & 1) | ((j & 1) << 1);
                float f = ipow(ea, i) * ipow(eb, j) * rsc;
                if ((((i >> 1) + (j >> 1) + (ca & i) + (cb & j)) & 1) != 0) f = -f;
#pragma unroll
                for (int x = 0; x < NU; ++x) {
                    const int un = es + 4 * x;
                    if (un < nunit) {
                        float T[P::ACC][4];
                        tc_ld_levels4(tmem + tlane + (uint32_t)(gb * g.colw + 4 * un), nw, T);
                        const float fu[2] = {f * __uint_as_float(rel[x] << 16), f * __uint_as_float(rel[x] & 0xffff0000u)};
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            typename P::Sum l = level_sum(T, v);
                            if (mask) l = sum_xor(l, mask);
                            S[x][v] = sum_add(S[x][v], sum_mulf(l, fu[v >> 1]));
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.acce);
        }
        // ---- partial rows: characters back to the signs of (n_a, n_b) ----
        if (ok && !*abort_flag) {
            const bool da = (es_slot >> 18) & 1, db = (es_slot >> 19) & 1, valid = (es_slot >> 20) & 1;
            const int na = da && (lane & 1) ? -(es_slot & 255) : (es_slot & 255);
            const int nb = db && (lane & 2) ? -((es_slot >> 8) & 255) : ((es_slot >> 8) & 255);
            const int* mrow = g.map + ((size_t)(na + g.nam) * (2 * g.nbm + 1) + (nb + g.nbm)) * g.ncols;
#pragma unroll
            for (int x = 0; x < NU; ++x) {
                const int un = es + 4 * x;
                if (un < nunit) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        // i^{ca + cb}, then the sign sums over the two characters of each axis
                        typename P::Sum c[2] = {S[x][2 * h], S[x][2 * h + 1]};
                        if (ca + cb == 1) {
                            const typename P::Sum t = c[0];
                            c[0] = sum_neg(c[1]);
                            c[1] = t;
                        } else if (ca + cb == 2) {
                            c[0] = sum_neg(c[0]);
                            c[1] = sum_neg(c[1]);
                        }
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            typename P::Sum o = sum_xor(c[r], 1);
                            if (da) c[r] = (lane & 1) ? sum_add(o, sum_neg(c[r])) : sum_add(c[r], o);
                            o = sum_xor(c[r], 2);
                            if (db) c[r] = (lane & 2) ? sum_add(o, sum_neg(c[r])) : sum_add(c[r], o);
                        }
                        const int p = 2 * un + h, nc = p / g.nd, d = p - nc * g.nd, er = of_density(eref, d);
                        if (valid && p < npo) {
                            int idx = __ldg(mrow + nc);
                            if (idx != INT_MIN) {
                                const bool cj = idx < 0;
                                if (cj) idx = ~idx;
                                const double re = scale_pow2(sum_double(c[0]), er), im = scale_pow2(sum_double(c[1]), er);
                                g.out[((long long)(g.d0 + d) * g.out_rows + g.out_row0 + kg) * g.ng_half + idx] =
                                    make_double2(re, cj ? -im : im);
                            }
                        }
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        if (tid == 0) atomicOr(g.err, 1);
        // NaN over the group's rows: of this CTA's points at least nobody writes them again
        for (int d = 0; d < g.nd; ++d) {
            double2* row = g.out + ((long long)(g.d0 + d) * g.out_rows + g.out_row0 + blockIdx.x) * g.ng_half;
            for (long long i = tid; i < g.ng_half; i += kTcThreadsAll) row[i] = make_double2(NAN, NAN);
        }
    }
    if (warp == kTcMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcTmemCols) : "memory");
    }
}

// c log2(e) of each record: the windows sort by it
__global__ void k_tc_width(const PairWalk* __restrict__ walk, long long npairs, float* __restrict__ cl) {
    const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < npairs) cl[r] = (float)(walk[r].c * 1.4426950408889634);
}

// Per-record factor tables in FP64, kept as double-float or double: X(0..na), Y(0..nb)
// with tws entries per record, in record order (the back-contraction's tiles)
// and in the K order (the structure-factor stages), so that a tile or a stage
// is one contiguous copy; Z(0..nc) in the K order.
template <bool F64>
__global__ void k_tc_tables(const PairWalk* __restrict__ walk, long long npairs, const int* __restrict__ kpos, int ax,
                            int bx, int cx, int nna, int nnb, int nnc, int tws, double Maa, double Mbb, double Mcc,
                            float4* __restrict__ tab, float4* __restrict__ tabk, float4* __restrict__ tabz,
                            float4* __restrict__ tabz3) {  // F64: tab, tabk, tabz as double2; Z also as triple-float
    const int tabw = nna + nnb + nnc;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= npairs * tabw) return;
    const long long r = t / tabw;
    const int e = (int)(t - r * tabw);
    const PairWalk w = walk[r];
    const double f[3] = {w.f1, w.f2, w.f3};
    double M, fr;
    int n;
    if (e < nna) {
        n = e;
        M = Maa;
        fr = f[ax];
    } else if (e < nna + nnb) {
        n = e - nna;
        M = Mbb;
        fr = f[bx];
    } else {
        n = e - nna - nnb;
        M = Mcc;
        fr = f[cx];
    }
    const double gval = exp(-w.c * M * (double)n * (double)n);
    double th = fr * (double)n;
    th -= rint(th);
    double s, c;
    sincospi(2.0 * th, &s, &c);
    float4 v;
    if (F64) {
        const double2 z = make_double2(gval * c, -gval * s);
        v = *reinterpret_cast<const float4*>(&z);
    } else {
        const df re = df_from_double(gval * c), im = df_from_double(-gval * s);
        v = make_float4(re.hi, re.lo, im.hi, im.lo);
    }
    const long long k = kpos[r];
    if (e < nna + nnb) {
        tab[r * tws + e] = v;
        tabk[k * tws + e] = v;
    } else {
        tabz[k * nnc + n] = v;
        if (F64) {
            const double z[2] = {gval * c, -gval * s};
            for (int q = 0; q < 2; ++q) {
                const float h = (float)z[q], m = (float)(z[q] - (double)h);
                tabz3[2 * (k * nnc + n) + q] = make_float4(h, m, (float)(z[q] - (double)h - (double)m), 0.f);
            }
        }
    }
}

// shared memory of one CTA with nbuf stage buffers and nts table slots (at
// least 120 KB, so that a second CTA never shares an SM: each one takes all
// 512 tensor-memory columns, and a second would wait in tcgen05.alloc)
size_t tc_smem_bytes(int slices, int npad, int tws, int nbuf, int nts) {
    const size_t need = (size_t)nbuf * slices * (kTcAsliceBytes + (size_t)npad * 32) + (size_t)nts * tab_slot_bytes(tws) +
                        sizeof(TcSmem) + 64;
    return std::max<size_t>(need, 120 * 1024);
}

int tc_alloc(ftcj_plan* P, void** ptr, size_t bytes) {
    const cudaError_t e = cudaMalloc(ptr, std::max<size_t>(bytes, 16));
    if (e != cudaSuccess) {
        cudaGetLastError();
        *ptr = nullptr;
        return fail(FTCJ_ENOMEM, std::string("cudaMalloc of ") + std::to_string(bytes) +
                                     " bytes failed: " + cudaGetErrorString(e));
    }
    P->device_bytes += std::max<size_t>(bytes, 16);
    return FTCJ_OK;
}

// The plan's host-made tables, gathered into one allocation and one copy
// (some thirty of each took a third of a small plan's set-up)
struct TcArena {
    std::vector<unsigned char> host;
    std::vector<std::pair<void**, size_t>> at;
    // n elements, of which v gives the first (the rest start at zero)
    template <class T>
    void add(T** ptr, const std::vector<T>& v, size_t n = 0) {
        const size_t off = (host.size() + 255) / 256 * 256;
        at.push_back({(void**)ptr, off});
        host.resize(off + sizeof(T) * std::max<size_t>({v.size(), n, 1}), 0);
        if (!v.empty()) std::memcpy(host.data() + off, v.data(), sizeof(T) * v.size());
    }
    int commit(ftcj_plan* P) {
        const int rc = tc_alloc(P, &P->d_tc_arena, host.size());
        if (rc) return rc;
        for (const auto& q : at) *q.first = (unsigned char*)P->d_tc_arena + q.second;
        FTCJ_CUDA(cudaMemcpy(P->d_tc_arena, host.data(), host.size(), cudaMemcpyHostToDevice));
        return FTCJ_OK;
    }
};

// Records [first, last) in the order of their widths, stable.  Positive floats
// order as their bits: one counting pass by the upper 17, then the buckets that
// hold several widths are sorted.
std::vector<int> sort_by_width(int64_t first, int64_t last, const std::vector<float>& width) {
    using Item = std::pair<uint32_t, int>;
    const auto less = [](const Item& x, const Item& y) { return x.first < y.first; };
    std::vector<Item> a((size_t)(last - first));
    const auto item = [&](int64_t r) {
        Item q{0u, (int)r};
        std::memcpy(&q.first, &width[r], 4);
        return q;
    };
    if (last - first < 4096) {  // fewer than the buckets are worth
        for (int64_t r = first; r < last; ++r) a[r - first] = item(r);
        std::stable_sort(a.begin(), a.end(), less);
    } else {
        constexpr int kShift = 15;
        std::vector<int> start((1u << (32 - kShift)) + 1, 0);
        for (int64_t r = first; r < last; ++r) ++start[(item(r).first >> kShift) + 1];
        for (size_t d = 1; d < start.size(); ++d) start[d] += start[d - 1];
        for (int64_t r = first; r < last; ++r) {
            const Item q = item(r);
            a[start[q.first >> kShift]++] = q;
        }
        for (size_t i = 0, j; i < a.size(); i = j) {
            bool sorted = true;
            for (j = i + 1; j < a.size() && (a[j].first >> kShift) == (a[i].first >> kShift); ++j)
                sorted = sorted && a[j - 1].first <= a[j].first;
            if (!sorted) std::stable_sort(a.begin() + i, a.begin() + j, less);
        }
    }
    std::vector<int> out(a.size());
    for (size_t k = 0; k < a.size(); ++k) out[k] = a[k].second;
    return out;
}

int round_up(int x, int m) { return (x + m - 1) / m * m; }


// the product kernel whose drain warps hold a block of colw columns in registers
const void* tc_rho_kernel(bool f64, int colw) {
    const int nu = (colw + 15) / 16;
    if (f64) {
        switch (nu) {
            case 1: return (const void*)k_tc_rho<Prec64, 1>;
            case 2: return (const void*)k_tc_rho<Prec64, 2>;
            case 3: return (const void*)k_tc_rho<Prec64, 3>;
            default: return (const void*)k_tc_rho<Prec64, 4>;
        }
    }
    switch (nu) {
        case 1: return (const void*)k_tc_rho<PrecRho, 1>;
        case 2: return (const void*)k_tc_rho<PrecRho, 2>;
        case 3: return (const void*)k_tc_rho<PrecRho, 3>;
        case 4: return (const void*)k_tc_rho<PrecRho, 4>;
        case 5: return (const void*)k_tc_rho<PrecRho, 5>;
        default: return (const void*)k_tc_rho<PrecRho, 6>;
    }
}

// column layout for nd densities and ncols values of n_c: real columns per
// block (a multiple of 8) and the largest block count G whose columns fit the
// MMA width; G = 0 when not even one block fits
void tc_columns(int nmax, int nd, int ncols, int* colw, int* G, int* npad) {
    *colw = round_up(2 * nd * ncols, 8);
    *G = 0;
    *npad = 0;
    for (int gg = kTcGmax; gg >= 1; --gg) {
        const int np = mma_cols(gg, *colw);
        if (np <= nmax) {
            *G = gg;
            *npad = np;
            return;
        }
    }
}

// The slots of a set of points (|n_a|, |n_b|), in groups of four lanes: the
// types (ta, tb) of one point (bit 0 ta, bit 1 tb) where both indices are
// positive; where one is zero its only type is the real part, and two such
// points share a group (the free bit says which); the origin takes one more.
// quads: the same groups for the back-contraction's operand former (bit 0:
// both indices positive, bit 1: n_b = 0, then two indices of 8 bits).
void tc_slots(const std::vector<std::pair<int, int>>& pts, std::vector<int>& slots, std::vector<int>& quads) {
    std::vector<int> axa, axb;  // n_a > 0, n_b = 0 and n_a = 0, n_b > 0
    bool origin = false;
    slots.clear();
    quads.clear();
    for (const auto& q : pts) {
        if (q.first > 0 && q.second > 0) {
            for (int t = 0; t < 4; ++t) slots.push_back(slot_pack(q.first, q.second, t & 1, t >> 1, 1, 1, 1));
            quads.push_back(1 | (q.first << 2) | (q.second << 10));
        } else if (q.first > 0) {
            axa.push_back(q.first);
        } else if (q.second > 0) {
            axb.push_back(q.second);
        } else {
            origin = true;
        }
    }
    for (size_t k = 0; k < axa.size(); k += 2) {
        const bool two = k + 1 < axa.size();
        const int n[2] = {axa[k], two ? axa[k + 1] : axa[k]};
        for (int t = 0; t < 4; ++t) slots.push_back(slot_pack(n[t >> 1], 0, t & 1, 0, 1, 0, t < 2 || two));
        quads.push_back(2 | (n[0] << 2) | (n[1] << 10));
    }
    for (size_t k = 0; k < axb.size(); k += 2) {
        const bool two = k + 1 < axb.size();
        const int n[2] = {axb[k], two ? axb[k + 1] : axb[k]};
        for (int t = 0; t < 4; ++t) slots.push_back(slot_pack(0, n[t & 1], 0, t >> 1, 0, 1, !(t & 1) || two));
        quads.push_back(0 | (n[0] << 2) | (n[1] << 10));
    }
    if (origin) {
        for (int t = 0; t < 4; ++t) slots.push_back(slot_pack(0, 0, 0, 0, 0, 0, t == 0));
        quads.push_back(0);
    }
}

// ---- the back-contraction (Alg. S1) in the same separable form -------------
//
// The walks' back-contraction sums, over the stored half sphere,
//   J'_{r,ijk} = Re sum_n (-i)^{i+j+k} n_a^i n_b^j n_c^k X_r(n_a) Y_r(n_b) Z_r(n_c) W(n).
// On the grid of (n_a, n_b) and n_c >= 0 (a stored point -n enters as conj W,
// since the conjugate of the summand at -n is the summand at n with conj W)
// this is, with the real products X_ta Y_tb of the structure-factor pass,
//   J'_{r,ijk} = Re (-i)^k sum_{n_c} n_c^k Z_r(n_c) U_ij[r, n_c],
//   U_ij[r, n_c] = sum_slots X_r,ta(|n_a|) Y_r,tb(|n_b|) V_ij[slot, n_c],
//   V_ij = i^{ta+tb} (-i)^{i+j} |n_a|^i |n_b|^j sum_{s_a,s_b} s_a^{ta+i} s_b^{tb+j} W(s_a |n_a|, s_b |n_b|, n_c),
// a matrix product with M = 128 records of one class, real A^T, K = the
// slots, N = (i, j) blocks x densities x (Re, Im) of n_c: half the
// multiply-adds and A^T entries of the complex form over signed rows.  V_ij does
// not depend on the record: it is sliced once per build (k_tc_vbound,
// k_tc_vslice) into stage tiles in global memory that bulk copies bring into
// shared memory, and only A^T is formed in the kernel, from the 128 records'
// factor tables.  Every entry of A^T has modulus <= 1 (bound 2^1 for all of
// them); each column of V_ij gets its own bound over all slots, so that entries
// far out in the sphere (where W has decayed) sit many bits below their
// column's bound (again relative to the largest of their (i, j) and density,
// which multiplies J').  Seven slices (products with s + t <= 6, 28 per k-step) keep the truncation
// below 2^-45 of the bounds.  The slots are cut into parts of at most 1024, each a work unit of its
// own: within a part, levels 0-3 are exact (the level-3 sums stay below 1024 x 14848 < 2^24 in units
// of 2^-21: |A| <= 1 bounds the leading slice of A by 32) and only levels 4-6 share the rounded fifth
// accumulator.  The tensor core's FP32 accumulation does not round to nearest, so the rounded
// accumulator's error grows with the number of MMAs that add into it and with its size; keeping level
// 3 out of it keeps that error ~2^-7 of a four-accumulator scheme's.  The level sums go straight to
// the epilogue, which forms the part's J' for k <= L - i - j in double-float and writes it as one of
// the partial FP64 sums the J -> AO map adds.

constexpr int kTcJStageM = 16;       // slots per stage: one MMA k-step
constexpr int kTcJAsliceBytes = kTcM * kTcJStageM * 2;        // 128 records x 16 K x bf16

// the (i, j) with i + j <= deg (4, for the gradient 5) in a row
__host__ __device__ constexpr int pairs_all(int deg) { return (deg + 1) * (deg + 2) / 2; }

__host__ __device__ constexpr int pair_index(int deg, int i, int j) { return i * (deg + 1) - i * (i - 1) / 2 + j; }

__device__ __forceinline__ void pair_of_index(int deg, int pr, int& i, int& j) {
    i = 0;
    while (pr > deg - i) {
        pr -= deg + 1 - i;
        ++i;
    }
    j = pr;
}

struct TcJArgs {
    const int* slots;       // the structure-factor pass's slots
    const int* quads;       // their groups of four
    const int* map;         // as in TcArgs
    const double2* W;       // potential W(G) on the half sphere, [dens][ng_half]
    const int* sched;       // [grid + 1] offsets, then unit ids grouped by CTA
    const int4* units;      // work units: class L | part << 8, first block group, block groups, first record
    const int2* groups;     // block groups: first index into ipairs, blocks
    const int* ipairs;      // (i | j << 3) of each block
    const long long* voff;  // start of each block group's V tiles in vs (elements)
    const int* vplace;      // [(i, j)][kNclass]: block group << 8 | place of the block in it, -1 none
    const void* tab;        // X(0..), Y(0..) as complex double-float or double, [tws] per record
    const void* tabz;       // Z(0..), [ncols] per record in the K order: complex double-float, or triple-float as two
                            // float4 (FP64 form)
    const int* kpos;        // position of each record in the K order of all classes
    __nv_bfloat16* vs;      // sliced V_ij: [block group][stage][slice][columns of its MMA x 16 K] stage tiles
    int* ev;                // column bounds of V_ij: [(i, j)][nd][ncols]
    int* er;                // [(i, j)][nd]: exponent that their slices are relative to, kNonFinite where a column is not
                            // finite
    double* Jp;             // partial back-contraction sums [dens][part][term] in the split form's class layout
    long long ng_half;
    long long jp_total;     // doubles per density of Jp
    long long cls_start[kNclass + 1];
    long long term_base[kNclass];
    int* err;               // device error word (bit 0: a bounded wait gave up)
    int ax, bx, cx;
    int deg;                // largest i + j + k: 4, for the gradient's sums 5
    int nam, nbm;
    int tws, offY;          // table entries per record (odd: conflict-free across records), start of Y
    int ncols, nd, d0;
    int gw;                 // real columns per density: 2 ncols rounded up to 8
    int colw;               // real columns per block: nd gw
    int npad;               // MMA N of a full unit: blocks x colw rounded up to 16
    int nslots, nstage;     // slots, stages of 16
    int nparts, spp;        // partial arrays of J' (slot parts x nsub), stages per part
    int nsub;               // a block's columns are split over this many of the four warps of a lane quadrant
    long long spin;         // clock cycles a wait between roles may take before it gives up
};

// V_ij of one slot and column, without the factor i^{ta+tb} (-i)^{i+j}: in
// double-float, or in FP64 (exact sign sums up to one rounding each)
template <class P>
__device__ __forceinline__ auto v_entry(const TcJArgs& g, int slot, int i, int j, int d, int nc) {
    constexpr bool kF64 = P::S == 8;
    cdf v{{0.f, 0.f}, {0.f, 0.f}};
    double2 v64 = make_double2(0.0, 0.0);
    const int sl = slot < g.nslots ? __ldg(g.slots + slot) : 0;
    const int na = sl & 255, nb = (sl >> 8) & 255, pa = ((sl >> 16) + i) & 1, pb = ((sl >> 17) + j) & 1;
    if ((sl >> 20) & 1) {
        for (int sa = 0; sa <= (na > 0 ? 1 : 0); ++sa)
            for (int sb = 0; sb <= (nb > 0 ? 1 : 0); ++sb) {
                const int idx = __ldg(g.map + ((size_t)((sa ? -na : na) + g.nam) * (2 * g.nbm + 1) +
                                               (sb ? -nb : nb) + g.nbm) * g.ncols + nc);
                if (idx == INT_MIN) continue;
                double2 w = __ldg(g.W + (long long)(g.d0 + d) * g.ng_half + (idx < 0 ? ~idx : idx));
                if (idx < 0) w.y = -w.y;
                const bool neg = (pa & sa) ^ (pb & sb);
                if constexpr (kF64) {
                    v64.x += neg ? -w.x : w.x;
                    v64.y += neg ? -w.y : w.y;
                } else {
                    cdf t{split_double(w.x), split_double(w.y)};
                    if (neg) t = cdf{df_neg(t.re), df_neg(t.im)};
                    v = cdf_add(v, t);
                }
            }
    }
    const float p = ipow((float)na, i) * ipow((float)nb, j);  // exact
    if constexpr (kF64) return make_double2(v64.x * (double)p, v64.y * (double)p);
    else return cdf{df_mulf(v.re, p), df_mulf(v.im, p)};
}

// the larger of |Re|, |Im| by their leading bits (an FP32 number's, the high word of an FP64 one; non-negative numbers
// order as integers, infinities and NaN on top), and the exponent e, |x| < 2^e, that they give
__device__ __forceinline__ unsigned v_top(cdf v) {
    return max(__float_as_uint(v.re.hi) & 0x7fffffffu, __float_as_uint(v.im.hi) & 0x7fffffffu);
}
__device__ __forceinline__ unsigned v_top(double2 v) {
    return max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
}
template <class P>
__device__ __forceinline__ int top_exp(unsigned top) {
    if (P::S == 8) return top >= 0x7ff00000u ? kNonFinite : (int)(top >> 20) - 1022;
    return top >= 0x7f800000u ? kNonFinite : (int)(top >> 23) - 126;
}

// column bounds: the exponent of the maximum over the slots of |Re V_ij|, |Im V_ij|
template <class P>
__global__ void __launch_bounds__(256) k_tc_vbound(TcJArgs g) {
    const int col = blockIdx.x;  // ((i, j) nd + d) ncols + n_c
    const int nc = col % g.ncols, d = (col / g.ncols) % g.nd, pr = col / (g.ncols * g.nd);
    int i, j;
    pair_of_index(g.deg, pr, i, j);
    unsigned mx = 0u;
    for (int m = threadIdx.x; m < g.nslots; m += blockDim.x) {
        mx = max(mx, v_top(v_entry<P>(g, m, i, j, d, nc)));
    }
    __shared__ unsigned red[256];
    red[threadIdx.x] = mx;
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
        if ((int)threadIdx.x < st) red[threadIdx.x] = max(red[threadIdx.x], red[threadIdx.x + st]);
        __syncthreads();
    }
    if (threadIdx.x == 0) g.ev[col] = top_exp<P>(red[0]);
}

// V_ij sliced into stage tiles: block group, stage q, slice s holds the columns
// of its blocks, d gw + 2 n_c (Re) and + 1 (Im) within a block, and K = slot;
// one thread per two slots; columns past 2 ncols are never read back.
template <class P>
__global__ void __launch_bounds__(256) k_tc_vslice(TcJArgs g) {
    constexpr int kS = P::S;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long per_pair = (long long)g.nstage * (kTcJStageM / 2) * g.nd * g.ncols;
    if (t >= pairs_all(g.deg) * per_pair) return;
    const int pr = (int)(t / per_pair);
    long long rem = t - pr * per_pair;
    const int nc = (int)(rem % g.ncols);
    rem /= g.ncols;
    const int d = (int)(rem % g.nd);
    rem /= g.nd;
    const int m2 = (int)(rem % (kTcJStageM / 2)), q = (int)(rem / (kTcJStageM / 2));
    int i, j;
    pair_of_index(g.deg, pr, i, j);
    const int* evr = g.ev + (pr * g.nd + d) * g.ncols;
    int top = evr[0];
    for (int k = 1; k < g.ncols; ++k) top = max(top, evr[k]);
    const bool finite = top != kNonFinite;
    const int er = ref_exp<P>(top), ec = col_exp<P>(evr[nc], er);
    if (nc == 0 && q == 0 && m2 == 0) g.er[pr * g.nd + d] = finite ? er : kNonFinite;
    uint32_t sr[kS], si[kS];
    if constexpr (P::S == 8) {
        unsigned long long fr[2], fi[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int slot = q * kTcJStageM + 2 * m2 + e;
            const int sl = slot < g.nslots ? __ldg(g.slots + slot) : 0;
            const double2 v = v_entry<P>(g, slot, i, j, d, nc);
            const int rot = (i + j + 8 - ((sl >> 16) & 1) - ((sl >> 17) & 1)) & 3;  // times (-i)^rot
            const double re = rot & 1 ? v.y : v.x, im = rot & 1 ? -v.x : v.y;
            fr[e] = fixed8(rot & 2 ? -re : re, finite ? er + ec : kNonFinite);
            fi[e] = fixed8(rot & 2 ? -im : im, finite ? er + ec : kNonFinite);
        }
        float w = pow2f(ec - 6);
#pragma unroll
        for (int s = 0; s < kS; ++s, w *= 0x1p-7f) {
            const int sh = 7 * (7 - s);
            auto digit = [&](unsigned long long f) {
                return (float)((int)((f >> sh) & (s == 0 ? 0xffULL : 0x7fULL)) - 64) * w;
            };
            sr[s] = pack_bf2(digit(fr[0]), digit(fr[1]));
            si[s] = pack_bf2(digit(fi[0]), digit(fi[1]));
        }
    } else {
        const typename P::Cut cut(ec);
        const float unref = pow2f(-er);
        cdf v[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int slot = q * kTcJStageM + 2 * m2 + e;
            const int sl = slot < g.nslots ? __ldg(g.slots + slot) : 0;
            const cdf t = rot_mi(v_entry<P>(g, slot, i, j, d, nc), i + j + 8 - ((sl >> 16) & 1) - ((sl >> 17) & 1));
            v[e] = cdf{{t.re.hi * unref, t.re.lo * unref}, {t.im.hi * unref, t.im.lo * unref}};
        }
        cut.pair(v[0].re, v[1].re, sr);
        cut.pair(v[0].im, v[1].im, si);
    }
    // every block group that holds (i, j), at most one per class
    for (int L = 0; L < kNclass; ++L) {
        const int pl = __ldg(g.vplace + pr * kNclass + L);
        if (pl < 0) continue;
        const int gi = pl >> 8, nw = mma_cols(__ldg(&g.groups[gi].y), g.colw);
        const int c0 = (pl & 255) * g.colw + d * g.gw + 2 * nc;
        const int o0 = tile_off(c0, 2 * m2), o1 = tile_off(c0 + 1, 2 * m2);
        __nv_bfloat16* bs = g.vs + __ldg(g.voff + gi) + (size_t)q * kS * nw * 16;
#pragma unroll
        for (int s = 0; s < kS; ++s, bs += nw * 16) {
            *reinterpret_cast<uint32_t*>(bs + o0) = sr[s];
            *reinterpret_cast<uint32_t*>(bs + o1) = si[s];
        }
    }
}

struct TcJSmem {
    uint64_t afull[kTcNbufMax], bfull[kTcNbufMax], empty[kTcNbufMax], tfull, tempty, accf, acce, done;
    uint32_t tmem;
    int abort_flag;
};

// Persistent over work units (class, slot part, 128 records), each running
// its (i, j) block groups in turn on the same staged factor tables, dealt to
// the CTAs at plan time (largest first, least loaded).  The structure-factor
// kernel's roles: warps 0-15, two groups in turn, form the A^T slices of each
// 16-slot stage, one thread per record and eight slots (two point groups: two
// 16-byte table reads and four real products each, one 16-byte core-matrix row
// per slice), lane 0 of warp 16 issues the MMAs, warp 17 brings the factor
// tables and warp 18 the V_ij stage tiles in with bulk copies; warps 0-15 then
// form J' from tensor memory (lane quadrant w & 3; (block, density) pairs,
// their columns split further where a group has fewer than four, w / 4 mod 4).
// Waits are bounded as in the structure-factor kernel.
// E = 1: the gradient's sums, one degree above the record's class.
template <class P, int E>
__global__ void __launch_bounds__(kTcThreadsAll, 1) k_tc_j(TcJArgs g, int nbuf) {
    extern __shared__ __align__(1024) unsigned char tsm[];
    const int bbytes = P::S * g.npad * 32;
    unsigned char* abuf = tsm;                                                     // [nbuf][S][4096]
    unsigned char* bbuf = abuf + (size_t)nbuf * P::S * kTcJAsliceBytes;             // [nbuf][S][npad x 32]
    float4* tabs = reinterpret_cast<float4*>(bbuf + (size_t)nbuf * bbytes);         // [128][tws]: X, Y
    TcJSmem& sm = *reinterpret_cast<TcJSmem*>(tabs + (size_t)kTcM * g.tws);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    volatile int* abort_flag = &sm.abort_flag;
    if (tid == 0) {
        for (int b = 0; b < nbuf; ++b) {
            mbar_init(&sm.afull[b], kTcGroupWarps);
            mbar_init(&sm.bfull[b], 1);
            mbar_init(&sm.empty[b], 1);
        }
        mbar_init(&sm.tfull, 1);
        mbar_init(&sm.tempty, kTcProdWarps);
        mbar_init(&sm.accf, 1);
        mbar_init(&sm.acce, kTcProdWarps);
        mbar_init(&sm.done, 1);
        sm.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // finite start: columns of B past a unit's blocks and rows of A past its records are never read into an output
    for (int i = tid; i < nbuf * bbytes / 16; i += kTcThreadsAll)
        reinterpret_cast<uint4*>(bbuf)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int i = tid; i < kTcM * g.tws; i += kTcThreadsAll) tabs[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (warp == kTcMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&sm.tmem)),
                     "r"(kTcTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tmem;
    const int j0 = __ldg(g.sched + blockIdx.x), j1 = __ldg(g.sched + blockIdx.x + 1);
    const int* ulist = g.sched + gridDim.x + 1;
    bool ok = true;

    if (warp == kTcTabWarp) {
        // the units' factor tables: consecutive records, one bulk copy each
        if (lane == 0) {
            long long nu = 0;
            for (int ju = j0; ju < j1; ++ju, ++nu) {
                const int4 un = __ldg(g.units + __ldg(ulist + ju));
                const int nv = (int)min((long long)kTcM, g.cls_start[(un.x & 255) + 1] - un.w);
                if (nu > 0 && !mbar_wait(&sm.tempty, (uint32_t)((nu - 1) & 1), abort_flag, g.spin)) break;
                const uint32_t bytes = (uint32_t)(nv * g.tws) * 16u;
                mbar_arrive_tx(&sm.tfull, bytes);
                bulk_copy(tabs, reinterpret_cast<const float4*>(g.tab) + (size_t)un.w * g.tws, bytes, &sm.tfull);
            }
            ring_settle(&sm.tfull, 1, nu);
        }
        __syncwarp();
    } else if (warp == kTcLoadWarp) {
        // the stages' V_ij tiles, one bulk copy each
        if (lane == 0) {
            Ring b(nbuf);
            long long gs = 0;
            for (int ju = j0; ju < j1 && ok; ++ju) {
                const int4 un = __ldg(g.units + __ldg(ulist + ju));
                const int q0 = (un.x >> 8) * g.spp, nst = min(g.spp, g.nstage - q0);
                for (int gi = 0; gi < un.z && ok; ++gi) {
                    const uint32_t bytes = (uint32_t)(P::S * mma_cols(__ldg(&g.groups[un.y + gi].y), g.colw) * 32);
                    const unsigned char* src = reinterpret_cast<const unsigned char*>(g.vs + __ldg(g.voff + un.y + gi)) +
                                               (size_t)q0 * bytes;
                    for (int q = 0; q < nst; ++q, ++gs, b.next()) {
                        if (gs >= nbuf && !(ok = mbar_wait(&sm.empty[b.i], b.ph ^ 1u, abort_flag, g.spin))) break;
                        mbar_arrive_tx(&sm.bfull[b.i], bytes);
                        bulk_copy(bbuf + (size_t)b.i * bbytes, src + (size_t)q * bytes, bytes, &sm.bfull[b.i]);
                    }
                }
            }
            ring_settle(sm.bfull, nbuf, gs);
        }
        __syncwarp();
    } else if (warp == kTcMmaWarp) {
        const uint32_t a0 = saddr(abuf), b0 = saddr(bbuf);
        Ring b(nbuf);
        int ng = 0;  // block groups issued
        for (int ju = j0; ju < j1 && ok; ++ju) {
            const int4 un = __ldg(g.units + __ldg(ulist + ju));
            const int nst = min(g.spp, g.nstage - (un.x >> 8) * g.spp);
            for (int gi = 0; gi < un.z && ok; ++gi, ++ng) {
                const uint32_t nw = (uint32_t)mma_cols(__ldg(&g.groups[un.y + gi].y), g.colw);
                const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTcM >> 4) << 24);
                // tensor memory drained
                if (ng > 0 && !(ok = __all_sync(0xffffffffu, mbar_wait(&sm.acce, (uint32_t)((ng - 1) & 1), abort_flag, g.spin))))
                    break;
                tc_fence_after();
                for (int q = 0; q < nst; ++q, b.next()) {
                    ok = __all_sync(0xffffffffu, mbar_wait(&sm.bfull[b.i], b.ph, abort_flag, g.spin) &&
                                                     mbar_wait(&sm.afull[b.i], b.ph, abort_flag, g.spin));
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        issue_kstep<P::S, P::ACC>(tmem, sdesc(a0 + b.i * P::S * kTcJAsliceBytes), kTcJAsliceBytes >> 4,
                                                    sdesc(b0 + b.i * bbytes), nw * 2, nw, idesc, q > 0);
                        tc_commit(&sm.empty[b.i]);
                        if (q + 1 == nst) tc_commit(&sm.accf);
                    }
                    __syncwarp();
                }
            }
        }
        // everything issued completes before tensor memory is freed
        if (elect_one()) {
            tc_commit(&sm.done);
            const long long t0 = clock64();
            while (!mbar_test(&sm.done, 0u) && clock64() - t0 < kTcSpinCycles) {
            }
        }
        __syncwarp();
    } else {
        // operand role: record rec, slots 8 oct .. 8 oct + 7 (two point groups) of its group's stages
        const int grp = warp / kTcGroupWarps, rec = tid & (kTcM - 1), oct = (tid >> 7) & 1;
        using Comp = typename P::Comp;
        using Entry = typename P::Entry;
        const Comp* trec = reinterpret_cast<const Comp*>(tabs + (size_t)rec * g.tws);  // two components per entry
        unsigned char* arow = abuf + tile_off(rec, oct * 8) * 2;
        const typename P::Cut cut(1);  // |A| <= 1 < 2^1
        // epilogue role
        const int eq = warp & 3, es = warp >> 2, erow = 32 * eq + lane;
        const uint32_t tlane = (uint32_t)(32 * eq) << 16;
        const int nquad = g.nslots / 4;
        Ring b(nbuf);
        int gs = 0, ng = 0, nu = 0;
        bool full = false;  // every buffer used once
        for (int ju = j0; ju < j1 && ok; ++ju, ++nu) {
            const int4 un = __ldg(g.units + __ldg(ulist + ju));
            const int L = un.x & 255, part = un.x >> 8, q0 = part * g.spp, nst = min(g.spp, g.nstage - q0);
            const long long r = (long long)un.w + erow;
            const bool rvalid = r < g.cls_start[L + 1];
            const long long cnt = g.cls_start[L + 1] - g.cls_start[L];
            if (!(ok = __all_sync(0xffffffffu, mbar_wait(&sm.tfull, (uint32_t)(nu & 1), abort_flag, g.spin)))) break;
            for (int gi = 0; gi < un.z && ok; ++gi, ++ng) {
                for (int q = 0; q < nst; ++q, ++gs, b.next()) {
                    full = full || gs >= nbuf;
                    if ((gs & 1) != grp) continue;
                    const int qd = (q0 + q) * 4 + oct * 2;
                    uint32_t pk[P::S][4];
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        const int info = qd + v < nquad ? __ldg(g.quads + qd + v) : 0;
                        const int n0 = (info >> 2) & 255, n1 = (info >> 10) & 255;
                        // the four products of the point group, in slot order; with one index zero its factor is 1
                        Entry a[4];
                        if (info & 1) {
                            const Comp x0 = trec[2 * n0], x1 = trec[2 * n0 + 1];
                            const Comp y0 = trec[2 * (g.offY + n1)], y1 = trec[2 * (g.offY + n1) + 1];
                            a[0] = P::product(x0, y0);
                            a[1] = P::product(x1, y0);
                            a[2] = P::product(x0, y1);
                            a[3] = P::product(x1, y1);
                        } else {
                            const int off = info & 2 ? 0 : g.offY;
                            const bool ab = info & 2;
                            const Entry x0 = P::entry(trec[2 * (off + n0)]), x1 = P::entry(trec[2 * (off + n0) + 1]);
                            const Entry y0 = P::entry(trec[2 * (off + n1)]), y1 = P::entry(trec[2 * (off + n1) + 1]);
                            a[0] = x0;
                            a[1] = ab ? x1 : y0;
                            a[2] = ab ? y0 : x1;
                            a[3] = y1;
                        }
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint32_t o[P::S];
                            cut.pair(a[2 * h], a[2 * h + 1], o);
#pragma unroll
                            for (int s = 0; s < P::S; ++s) pk[s][2 * v + h] = o[s];
                        }
                    }
                    if (full) {
                        ok = __all_sync(0xffffffffu, mbar_wait(&sm.empty[b.i], b.ph ^ 1u, abort_flag, g.spin));
                        if (!ok) break;
                    }
                    unsigned char* as = arow + (size_t)b.i * P::S * kTcJAsliceBytes;
#pragma unroll
                    for (int s = 0; s < P::S; ++s)
                        *reinterpret_cast<uint4*>(as + (size_t)s * kTcJAsliceBytes) =
                            make_uint4(pk[s][0], pk[s][1], pk[s][2], pk[s][3]);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm.afull[b.i]);
                }
                if (!ok) break;
                // the last reads of the unit's tables are done
                if (gi + 1 == un.z) {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm.tempty);
                }
                // ---- J'_{r,ijk} = Re (-i)^k sum_{n_c} n_c^k Z_r(n_c) U_ij[r, n_c] ----
                // lane l holds the l-th (block, density) of the group: (i, j) and the exponent of its sums
                const int2 gr = __ldg(g.groups + un.y + gi);
                int lpr = 0, ler = 0;
                if (lane < gr.y * g.nd) {
                    lpr = __ldg(g.ipairs + gr.x + lane / g.nd);
                    ler = __ldg(g.er + pair_index(g.deg, lpr & 7, lpr >> 3) * g.nd + lane % g.nd);
                }
                ok = __all_sync(0xffffffffu, mbar_wait(&sm.accf, (uint32_t)(ng & 1), abort_flag, g.spin));
                if (!ok) break;
                tc_fence_after();
                const uint32_t nw = (uint32_t)mma_cols(gr.y, g.colw);
                const float4* zrec =
                    reinterpret_cast<const float4*>(g.tabz) +
                    (size_t)__ldg(g.kpos + (rvalid ? r : un.w)) * g.ncols * (P::S == 8 ? 2 : 1);
                for (int ps = es; ps < gr.y * g.nd * g.nsub; ps += kTcProdWarps / 4) {
                    const int pd = ps / g.nsub, sub = ps - pd * g.nsub, gb = pd / g.nd, d = pd - gb * g.nd;
                    const int pr = __shfl_sync(0xffffffffu, lpr, pd), i = pr & 7, j = pr >> 3, nk = L + E - i - j;
                    const int er = __shfl_sync(0xffffffffu, ler, pd);
                    typename P::Sum J[5 + E];
#pragma unroll
                    for (int kk = 0; kk < 5 + E; ++kk) J[kk] = sum_zero(typename P::Sum());
                    for (int c4 = sub; c4 < g.gw / 4; c4 += g.nsub) {
                        float T[P::ACC][4];
                        typename P::Sum zr[2], zi[2];  // Z: double-float in one float4, triple-float in two
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const int nc = min(2 * c4 + u, g.ncols - 1);
                            if constexpr (P::S == 8) {
                                const float4 a = __ldg(zrec + 2 * nc), b = __ldg(zrec + 2 * nc + 1);
                                zr[u] = tf{a.x, a.y, a.z};
                                zi[u] = tf{b.x, b.y, b.z};
                            } else {
                                const float4 a = __ldg(zrec + nc);
                                zr[u] = df{a.x, a.y};
                                zi[u] = df{a.z, a.w};
                            }
                        }
                        tc_ld_levels4(tmem + tlane + (uint32_t)(gb * g.colw + d * g.gw + 4 * c4), nw, T);
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const int nc = 2 * c4 + u;
                            if (nc >= g.ncols) continue;
                            const auto vr = level_sum(T, 2 * u), vi = level_sum(T, 2 * u + 1);
                            // n_c^k exact; Re (-i)^k zu is +-Re (k even) or +-Im (k odd)
                            if constexpr (P::S == 8) {
                                const tf re = tf_add(tf_mul(zr[u], vr), tf_neg(tf_mul(zi[u], vi)));
                                J[0] = tf_add(J[0], re);
                                if (nk > 0) {
                                    const tf im = tf_add(tf_mul(zr[u], vi), tf_mul(zi[u], vr));
                                    const float x = (float)nc;
                                    J[1] = tf_add(J[1], tf_mulf(im, x));
                                    if (nk > 1) J[2] = tf_add(J[2], tf_mulf(re, x * x));
                                    if (nk > 2) J[3] = tf_add(J[3], tf_mulf(im, x * x * x));
                                    if (nk > 3) J[4] = tf_add(J[4], tf_mulf(re, x * x * x * x));
                                    if (E && nk > 4) J[4 + E] = tf_add(J[4 + E], tf_mulf(im, x * x * x * x * x));
                                }
                            } else {
                                const cdf zu = cdf_mul_u(cdf{zr[u], zi[u]}, cdf{vr, vi});
                                float pw = 1.f;
#pragma unroll
                                for (int kk = 0; kk < 5 + E; ++kk) {
                                    if (kk <= nk) J[kk] = df_add(J[kk], df_mulf_u(kk & 1 ? zu.im : zu.re, pw));
                                    pw *= (float)nc;
                                }
                            }
                        }
                    }
                    if (rvalid) {
                        const int eo = P::S == 8 ? er + 1 - 6 : er;  // with A's bound 2^1 (row_scale)
                        double* jp = g.Jp + ((long long)(g.d0 + d) * g.nparts + part * g.nsub + sub) * g.jp_total + g.term_base[L] +
                                     (r - g.cls_start[L]);
#pragma unroll
                        for (int kk = 0; kk < 5 + E; ++kk)
                            if (kk <= nk) {
                                const double v = er == kNonFinite ? NAN : scale_pow2(sum_double(J[kk]), eo);
                                jp[(long long)term_of(g.ax, g.bx, i, j, kk) * cnt] = kk == 2 || kk == 3 ? -v : v;
                            }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.acce);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        if (tid == 0) atomicOr(g.err, 1);
        // NaN over the terms of the CTA's units: what its own block groups hold nobody writes again (the bounds are read
        // anew, so that they hold no registers until here)
        const volatile int* sched = g.sched;
        const int first = sched[blockIdx.x], last = sched[blockIdx.x + 1];
        for (int ju = first; ju < last; ++ju) {
            const int4 un = __ldg(g.units + sched[gridDim.x + 1 + ju]);
            const int L = un.x & 255, part = un.x >> 8;
            const long long cnt = g.cls_start[L + 1] - g.cls_start[L], loc = un.w - g.cls_start[L];
            const int nv = (int)min((long long)kTcM, cnt - loc), nt = nterms(L + E);
            for (int i = tid; i < g.nd * g.nsub * nt * nv; i += kTcThreadsAll) {
                const int r = i % nv, t = (i / nv) % nt, sub = (i / nv / nt) % g.nsub, d = i / nv / nt / g.nsub;
                g.Jp[((long long)(g.d0 + d) * g.nparts + part * g.nsub + sub) * g.jp_total + g.term_base[L] + t * cnt + loc + r] = NAN;
            }
        }
    }
    if (warp == kTcMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcTmemCols) : "memory");
    }
}

size_t tc_j_smem_bytes(int slices, int npad, int tws, int nbuf) {
    const size_t need = (size_t)nbuf * slices * (kTcJAsliceBytes + (size_t)npad * 32) + (size_t)kTcM * tws * 16 +
                        sizeof(TcJSmem) + 64;
    return std::max<size_t>(need, 120 * 1024);
}

// the gradient's sums keep to the eight-slice form (double-float or FP64 precision)
const void* tc_j_kernel(bool f64, int extra) {
    if (extra) return (const void*)k_tc_j<Prec64, 1>;
    return f64 ? (const void*)k_tc_j<Prec64, 0> : (const void*)k_tc_j<PrecJ, 0>;
}

// work dealt to nbin bins, largest first, each to the least loaded bin (ties
// to the lower one): nbin + 1 offsets, then the item ids of each bin
std::vector<int> deal(const std::vector<double>& cost, int nbin) {
    std::vector<int> order(cost.size());
    for (size_t k = 0; k < order.size(); ++k) order[k] = (int)k;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return cost[a] > cost[b]; });
    std::vector<std::vector<int>> lists(nbin);
    using Slot = std::pair<double, int>;
    std::priority_queue<Slot, std::vector<Slot>, std::greater<Slot>> heap;
    for (int b = 0; b < nbin; ++b) heap.push({0.0, b});
    for (int k : order) {
        const Slot s = heap.top();
        heap.pop();
        lists[s.second].push_back(k);
        heap.push({s.first + cost[k], s.second});
    }
    std::vector<int> out;
    int off = 0;
    for (const auto& l : lists) {
        out.push_back(off);
        off += (int)l.size();
    }
    out.push_back(off);
    for (const auto& l : lists) out.insert(out.end(), l.begin(), l.end());
    return out;
}

}  // namespace

void release_tc(ftcj_plan* P) {
    void** owned[] = {&P->d_tc_arena, (void**)&P->d_tc_cl, &P->d_tc_tab, &P->d_tc_tabk, &P->d_tc_tabz, &P->d_tc_tabz3,
                      &P->d_tc_b, &P->tcj.vs, &P->tcg.vs};
    for (void** p : owned) {
        if (*p) cudaFree(*p);
        *p = nullptr;
    }
    // tables inside the arena; of these, callers ask for the error word and the K order
    P->d_tc_err = nullptr;
    P->d_tc_pos = nullptr;
    P->tc = P->tcj.on = P->tcg.on = false;
    P->tc_dp_total = 0;
    P->tc_passes.clear();
}

// clock-cycle budget of one wait between the kernels' roles
long long tc_spin(const ftcj_plan* P) {
    return P->params.tc_wait_log2 > 0 ? (1LL << P->params.tc_wait_log2) : kTcSpinCycles;
}

int setup_tc_j(ftcj_plan* P, int extra, TcArena& arena);

// FP64 plans and the structure factors of split walks: the finer of the two precisions
inline bool tc_eight_slices(const ftcj_plan* P) { return P->precision == FTCJ_PREC_FP64 || P->tc_rho_only; }

// Plan-time set-up of the tensor-core form: the column axis, the slots and the
// half-sphere map, the factor tables, the windows (class, block group, records
// sorted by width), their deal to CTA groups and the B tiles.
int setup_tc(ftcj_plan* P) {
    if (!P->ortho) return fail(FTCJ_EUNSUPPORTED, "the tensor-core contraction needs an orthorhombic cell");
    const bool f64 = tc_eight_slices(P);
    const int nmax = f64 ? Prec64::kNmax : PrecRho::kNmax, slices = f64 ? Prec64::S : PrecRho::S;
    const int nprod = slices * (slices + 1) / 2;
    if (P->d_rec_gcut) return fail(FTCJ_EUNSUPPORTED, "the tensor-core contraction walks the whole sphere");
    if (P->npairs >= (1 << 24)) return fail(FTCJ_EUNSUPPORTED, "more than 2^24 pair records");
    const int64_t ngh = P->ng_half;
    int64_t recs_by_class[kNclass];
    for (int L = 0; L < kNclass; ++L) recs_by_class[L] = P->class_start[L + 1] - P->class_start[L];
    // The column axis: SM cycles of both passes, per density group.  Structure factors: per 16 records and row tile
    // the slice products (A read about three times in four, 32 B per column of B, at 128 B per cycle) and the forming
    // of A, and per entry of B its forming; back-contraction: the same per 16 slots and record tile, and per (record,
    // block, n_c) the epilogue.  The per-entry costs are measured ones.
    const double kB = f64 ? 5.0 : 3.7, kE = f64 ? 5.0 : 2.9;
    struct AxisPlan {
        std::vector<int> slots, quads;
        size_t rows = 0;
        int ncols = 0, nd = 0, colw = 0, G = 0, npad = 0, nam = 0, nbm = 0;
    } best;
    int best_c = -1;
    double best_cost = 1e300;
    for (int c = 0; c < 3; ++c) {
        const int a = (c + 1) % 3, b = (c + 2) % 3;
        AxisPlan ap;
        int ncmax = 0;
        for (int64_t q = 0; q < ngh; ++q) {
            ap.nam = std::max(ap.nam, std::abs(P->gvec[3 * q + a]));
            ap.nbm = std::max(ap.nbm, std::abs(P->gvec[3 * q + b]));
            ncmax = std::max(ncmax, std::abs(P->gvec[3 * q + c]));
        }
        // (n_a, n_b) at n_c >= 0, and their absolute values
        std::vector<char> signed_seen((size_t)(2 * ap.nam + 1) * (2 * ap.nbm + 1), 0);
        std::vector<char> seen((size_t)(ap.nam + 1) * (ap.nbm + 1), 0);
        for (int64_t q = 0; q < ngh; ++q) {
            const int sg = P->gvec[3 * q + c] < 0 ? -1 : 1, na = sg * P->gvec[3 * q + a], nb = sg * P->gvec[3 * q + b];
            signed_seen[(size_t)(na + ap.nam) * (2 * ap.nbm + 1) + nb + ap.nbm] = 1;
            seen[(size_t)std::abs(na) * (ap.nbm + 1) + std::abs(nb)] = 1;
        }
        std::vector<std::pair<int, int>> pts;
        for (int na = 0; na <= ap.nam; ++na)
            for (int nb = 0; nb <= ap.nbm; ++nb)
                if (seen[(size_t)na * (ap.nbm + 1) + nb]) pts.push_back({na, nb});
        ap.rows = (size_t)std::count(signed_seen.begin(), signed_seen.end(), 1);
        ap.ncols = ncmax + 1;
        for (ap.nd = std::min(P->max_dens, kTcDensMax); ap.nd >= 1; --ap.nd) {
            tc_columns(nmax, ap.nd, ap.ncols, &ap.colw, &ap.G, &ap.npad);
            if (ap.G > 0) break;
        }
        if (ap.nd < 1 || ap.G < 1) continue;
        tc_slots(pts, ap.slots, ap.quads);
        const double mt = (double)((ap.slots.size() + kTcM - 1) / kTcM);
        const double launches = (double)((P->max_dens + ap.nd - 1) / ap.nd);
        double cost = 0.0;
        for (int L = 0; L < kNclass; ++L) {
            const int nb = (L + 1) * (L + 2) / 2;
            const double rows16 = (double)recs_by_class[L] / 16.0, nst = (double)ap.slots.size() / 16.0;
            for (int g0 = 0; g0 < nb; g0 += ap.G) {
                const double stage = 500.0 + nprod * (24.0 + 0.25 * mma_cols(std::min(ap.G, nb - g0), ap.colw));
                cost += rows16 * stage * (mt + nst / 8.0);  // a record tile of the back-contraction is 128 records
            }
            cost += (double)recs_by_class[L] * nb * ap.nd * ap.ncols * (kB + kE);
        }
        cost *= launches;
        if (cost < best_cost) {
            best_cost = cost;
            best_c = c;
            best = ap;
        }
    }
    if (best_c < 0) return fail(FTCJ_EUNSUPPORTED, "the sphere is too long on every axis for the tensor-core tile");
    const int c = best_c, a = (c + 1) % 3, b = (c + 2) % 3;
    P->tc_axis[0] = a;
    P->tc_axis[1] = b;
    P->tc_axis[2] = c;
    P->tc_ncols = best.ncols;
    P->tc_nd = best.nd;
    P->tc_colw = best.colw;
    P->tc_G = best.G;
    P->tc_npad = best.npad;
    P->tc_rows = (int)best.rows;
    P->tc_nslots = (int)best.slots.size();
    P->tc_mtiles = std::max(1, (P->tc_nslots + kTcM - 1) / kTcM);
    P->tc_nna = best.nam + 1;
    P->tc_nnb = best.nbm + 1;
    std::vector<int> slots = best.slots;
    slots.resize((size_t)P->tc_mtiles * kTcM, 0);
    // half-sphere map: (n_a, n_b) and n_c >= 0
    std::vector<int> map((size_t)(2 * best.nam + 1) * (2 * best.nbm + 1) * P->tc_ncols, INT_MIN);
    for (int64_t q = 0; q < ngh; ++q) {
        int n[3] = {P->gvec[3 * q], P->gvec[3 * q + 1], P->gvec[3 * q + 2]};
        bool cj = false;
        if (n[c] < 0) {
            for (int x = 0; x < 3; ++x) n[x] = -n[x];
            cj = true;
        }
        const size_t rix = (size_t)(n[a] + best.nam) * (2 * best.nbm + 1) + (size_t)(n[b] + best.nbm);
        map[rix * P->tc_ncols + n[c]] = cj ? ~(int)q : (int)q;
    }
    // the windows sort records by their width
    const int tws = (P->tc_nna + P->tc_nnb) | 1;
    P->tc_tws = tws;
    const size_t nrec = (size_t)std::max<int64_t>(P->npairs, 1);
    int rc;
    TcArena arena;
    arena.host.reserve(16 * nrec + 8 * map.size() + (1 << 18));
    arena.add(&P->d_tc_err, std::vector<int>(1, 0));
    if ((rc = tc_alloc(P, (void**)&P->d_tc_cl, sizeof(float) * nrec))) return rc;
    std::vector<float> clh(nrec, 0.f);
    if (P->npairs > 0) {
        k_tc_width<<<(unsigned)((P->npairs + 255) / 256), 256>>>(P->d_walk, P->npairs, P->d_tc_cl);
        FTCJ_CUDA(cudaGetLastError());
        FTCJ_CUDA(cudaMemcpy(clh.data(), P->d_tc_cl, sizeof(float) * P->npairs, cudaMemcpyDeviceToHost));
    }
    // Hermite terms in the K order: [dens][class][term][position], each class's stride a multiple of 16
    P->tc_dp_total = 0;
    for (int L = 0; L < kNclass; ++L) {
        P->tc_dp_base[L] = P->tc_dp_total;
        P->tc_dp_stride[L] = (recs_by_class[L] + 15) / 16 * 16;
        P->tc_dp_total += (long long)nterms(L) * P->tc_dp_stride[L];
    }
    // K order: the records of a class sorted by width c = 1/4p (records of similar width have entries of similar size)
    std::vector<std::vector<int>> order(kNclass);
    std::vector<int> pos(nrec, 0), kpos(nrec, 0), korder(nrec, 0);
    std::vector<float> clk(nrec, 0.f);
    for (int L = 0; L < kNclass; ++L) {
        order[L] = sort_by_width(P->class_start[L], P->class_start[L + 1], clh);
        const std::vector<int>& recs = order[L];
        for (size_t k = 0; k < recs.size(); ++k) {
            pos[recs[k]] = (int)k;
            kpos[recs[k]] = (int)(P->class_start[L] + (int64_t)k);
            clk[P->class_start[L] + k] = clh[recs[k]];
            korder[P->class_start[L] + k] = (int)(recs[k] - P->class_start[L]);
        }
    }
    // Records per window: a window costs one drain of tensor memory (~7% of a 1024-record window of 96 columns),
    // a CTA group holds at least four windows where there are enough records, so that the deal comes out even
    const int groups_max = std::max(1, P->num_sms / P->tc_mtiles);
    auto windows = [&](int wlen) {
        int64_t n = 0;
        for (int L = 0; L < kNclass; ++L) {
            const int nb = (L + 1) * (L + 2) / 2;
            n += (recs_by_class[L] + wlen - 1) / wlen * ((nb + P->tc_G - 1) / P->tc_G);
        }
        return n;
    };
    P->tc_wlen = f64 ? Prec64::kWin : PrecRho::kWin;
    while (P->tc_wlen > 128 && windows(P->tc_wlen) < 4 * (int64_t)groups_max) P->tc_wlen /= 2;
    const int wlen = P->tc_wlen;
    // windows: for each class L, its (i, j) blocks in groups of G, the class's records wlen at a time
    struct Win {
        int4 info;
        int cnt;
        double cost;
    };
    std::vector<Win> wins;
    std::vector<int> wpairs;
    for (int L = 0; L < kNclass; ++L) {
        const std::vector<int>& recs = order[L];
        if (recs.empty()) continue;
        std::vector<int> blocks;
        for (int i = 0; i <= L; ++i)
            for (int j = 0; i + j <= L; ++j) blocks.push_back(i | (j << 3));
        for (size_t g0 = 0; g0 < blocks.size(); g0 += P->tc_G) {
            const int nb = (int)std::min<size_t>(P->tc_G, blocks.size() - g0);
            const int first = (int)wpairs.size();
            wpairs.insert(wpairs.end(), blocks.begin() + g0, blocks.begin() + g0 + nb);
            for (size_t r0 = 0; r0 < recs.size(); r0 += wlen) {
                const int cnt = (int)std::min<size_t>(wlen, recs.size() - r0);
                const double nst = (double)((cnt + kTcStageK - 1) / kTcStageK);
                wins.push_back({make_int4(L, nb, first, (int)r0), cnt,
                                nst * (500.0 + nprod * (24.0 + 0.25 * mma_cols(nb, P->tc_colw))) + 70.0 * nb * P->tc_colw});
            }
        }
    }
    // Passes: the B tiles of a pass's windows fill one workspace, bounded so that a large system reuses it
    // instead of growing it, by 8 GB and by 1/32 of the memory that is free now, so that further plans and the caller
    // find theirs (each further pass costs 70 to 130 us: crystal of 1056 AOs, FP64, 2461 us in one pass, 2529 in two,
    // 2660 in four); each pass deals its windows to CTA groups, one CTA per SM over all (group, row
    // tile) pairs, so that the grid is a single wave (a partial second wave would double the pass)
    const int nwin = (int)wins.size();
    P->tc_nwin = nwin;
    size_t room = 0, all = 0;
    FTCJ_CUDA(cudaMemGetInfo(&room, &all));
    const long long work_max = std::min(kTcBWorkMax, (long long)(room / 32));
    std::vector<int4> winfo((size_t)std::max(1, nwin), make_int4(0, 0, 0, 0));
    std::vector<int> wcnt((size_t)std::max(1, nwin), 0);
    std::vector<long long> boff((size_t)std::max(1, nwin), 0);
    P->tc_passes.clear();
    P->tc_out_rows = 0;
    long long bmax = 1;
    std::vector<int> sched;
    for (int w0 = 0; w0 < nwin;) {
        long long off = 0;
        int w1 = w0;
        while (w1 < nwin) {
            const Win& w = wins[w1];
            const long long n = (long long)((w.cnt + kTcStageK - 1) / kTcStageK) * slices * mma_cols(w.info.y, P->tc_colw) * 2;
            if (w1 > w0 && (off + n) * 16 > work_max) break;
            winfo[w1] = w.info;
            wcnt[w1] = w.cnt;
            boff[w1] = off;
            off += n;
            ++w1;
        }
        bmax = std::max(bmax, off);
        const int ng = std::min(groups_max, w1 - w0);
        std::vector<double> cost;
        for (int w = w0; w < w1; ++w) cost.push_back(wins[w].cost);
        std::vector<int> s = deal(cost, ng);
        for (size_t k = (size_t)ng + 1; k < s.size(); ++k) s[k] += w0;
        P->tc_passes.push_back({w0, w1 - w0, ng, P->tc_out_rows, (int)sched.size()});
        sched.insert(sched.end(), s.begin(), s.end());
        P->tc_out_rows += ng;
        w0 = w1;
    }
    P->tc_out_rows = std::max(1, P->tc_out_rows);
    // MMA work of one pass: per window and row tile, its stages x the slice products of M = 128 rows,
    // N = the window's columns, K = 16, for every density group
    P->tc_mma_flops = 0;
    for (int d0 = 0; d0 < P->max_dens; d0 += P->tc_nd) {
        const int colw = round_up(2 * std::min(P->tc_nd, P->max_dens - d0) * P->tc_ncols, 8);
        for (const Win& w : wins)
            P->tc_mma_flops += (long long)P->tc_mtiles * ((w.cnt + kTcStageK - 1) / kTcStageK) * nprod * 2LL * kTcM *
                               mma_cols(w.info.y, colw) * 16;
    }
    // stage buffers and table slots: four buffers where at least three slots fit beside them, else fewer
    int dev = 0, optin = 0;
    FTCJ_CUDA(cudaGetDevice(&dev));
    FTCJ_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    P->tc_tslots = 0;
    for (int nbuf = kTcNbufMax; nbuf >= 2 && !P->tc_tslots; --nbuf)
        for (int nts = kTcTabSlotsMax; nts >= (nbuf > 2 ? 3 : 1) && !P->tc_tslots; --nts)
            if (tc_smem_bytes(slices, P->tc_npad, tws, nbuf, nts) <= (size_t)optin) {
                P->tc_nbuf = nbuf;
                P->tc_tslots = nts;
            }
    if (!P->tc_tslots)
        return fail(FTCJ_EUNSUPPORTED, "the G sphere is too long for the tensor-core kernel's shared-memory tables");
    arena.add(&P->d_tc_slots, slots);
    arena.add(&P->d_tc_quads, best.quads);
    arena.add(&P->d_tc_map, map);
    arena.add(&P->d_tc_wpairs, wpairs);
    arena.add(&P->d_tc_pos, pos);
    arena.add(&P->d_tc_kpos, kpos);
    if (P->precision == FTCJ_PREC_FP64) arena.add(&P->d_tc_korder, korder);
    arena.add(&P->d_tc_wcnt, wcnt);
    arena.add(&P->d_tc_boff, boff);
    arena.add(&P->d_tc_sched, sched);
    arena.add((int4**)&P->d_tc_winfo, winfo);
    arena.add(&P->d_tc_clw, std::vector<float>(), (size_t)std::max(1, nwin));
    arena.add(&P->d_tc_ew, std::vector<int>(), (size_t)std::max(1, nwin) * P->tc_nd);
    // the back-contraction's, and those of the gradient's sums where ftcj_grad takes the plan and n^5 is exact in FP32
    if (!P->tc_rho_only && (rc = setup_tc_j(P, 0, arena))) return rc;
    if (f64 && P->shard_count <= 1 && !P->rec_filter && split_grad_walk_exact(P) && (rc = setup_tc_j(P, 1, arena)))
        return rc;
    if ((rc = arena.commit(P))) return rc;
    FTCJ_CUDA(cudaMemcpy(P->d_tc_cl, clk.data(), sizeof(float) * nrec, cudaMemcpyHostToDevice));
    if ((rc = tc_alloc(P, &P->d_tc_tab, sizeof(float4) * nrec * tws))) return rc;
    if ((rc = tc_alloc(P, &P->d_tc_tabk, sizeof(float4) * nrec * tws))) return rc;
    if ((rc = tc_alloc(P, &P->d_tc_tabz, sizeof(float4) * nrec * P->tc_ncols))) return rc;
    if (f64 && (rc = tc_alloc(P, &P->d_tc_tabz3, 2 * sizeof(float4) * nrec * P->tc_ncols))) return rc;
    // the odd stride's spare entry is copied along but never read
    FTCJ_CUDA(cudaMemset(P->d_tc_tab, 0, sizeof(float4) * nrec * tws));
    FTCJ_CUDA(cudaMemset(P->d_tc_tabk, 0, sizeof(float4) * nrec * tws));
    if (P->npairs > 0) {
        const long long n = P->npairs * (long long)(P->tc_nna + P->tc_nnb + P->tc_ncols);
        auto* tables = f64 ? k_tc_tables<true> : k_tc_tables<false>;
        tables<<<(unsigned)((n + 255) / 256), 256>>>(
            P->d_walk, P->npairs, P->d_tc_kpos, a, b, c, P->tc_nna, P->tc_nnb, P->tc_ncols, tws, P->M[4 * a],
            P->M[4 * b], P->M[4 * c], reinterpret_cast<float4*>(P->d_tc_tab), reinterpret_cast<float4*>(P->d_tc_tabk),
            reinterpret_cast<float4*>(P->d_tc_tabz), reinterpret_cast<float4*>(P->d_tc_tabz3));
        FTCJ_CUDA(cudaGetLastError());
    }
    if ((rc = tc_alloc(P, &P->d_tc_b, (size_t)bmax * 16))) return rc;
    // columns between a window's blocks and the MMA's multiple of 16 are never written nor read back: finite once
    FTCJ_CUDA(cudaMemset(P->d_tc_b, 0, (size_t)bmax * 16));
    // calls with fewer densities run the instantiation of their own block width
    for (int nd = 1; nd <= P->tc_nd; ++nd)
        if ((rc = allow_dynamic_smem(tc_rho_kernel(f64, round_up(2 * nd * P->tc_ncols, 8)),
                                     tc_smem_bytes(slices, P->tc_npad, tws, P->tc_nbuf, P->tc_tslots))))
            return rc;
    return FTCJ_OK;
}

int launch_tc_rho(ftcj_plan* P, int ndens, cudaStream_t s) {
    if (P->ng_half == 0 || P->npairs == 0) {
        FTCJ_CUDA(cudaMemsetAsync(P->d_rho_part, 0, sizeof(double2) * (size_t)ndens * P->tc_out_rows * P->ng_half, s));
        return FTCJ_OK;
    }
    TcArgs g;
    g.slots = P->d_tc_slots;
    g.map = P->d_tc_map;
    g.winfo = reinterpret_cast<const int4*>(P->d_tc_winfo);
    g.wcnt = P->d_tc_wcnt;
    g.boff = P->d_tc_boff;
    g.wpairs = P->d_tc_wpairs;
    const bool f64 = tc_eight_slices(P);
    g.tabk = P->d_tc_tabk;
    g.tabz = P->d_tc_tabz;
    g.korder = P->d_tc_korder;
    g.clk = P->d_tc_cl;
    for (int cc = 0; cc < kNclass; ++cc) g.kbase[cc] = P->class_start[cc];
    g.Dp = P->d_Dp;
    const bool df_terms = P->precision == FTCJ_PREC_SPLIT;
    g.dp_total = df_terms ? P->tc_dp_total : P->total_terms;
    for (int cc = 0; cc < kNclass; ++cc) {
        g.dp_base[cc] = df_terms ? P->tc_dp_base[cc] : P->term_base[cc];
        g.dp_stride[cc] = df_terms ? P->tc_dp_stride[cc] : P->class_start[cc + 1] - P->class_start[cc];
    }
    g.bs = reinterpret_cast<uint4*>(P->d_tc_b);
    g.clw = P->d_tc_clw;
    g.ew = P->d_tc_ew;
    g.out = reinterpret_cast<double2*>(P->d_rho_part);
    g.ng_half = P->ng_half;
    g.out_rows = P->tc_out_rows;
    g.err = P->d_tc_err;
    g.Maa = (float)P->M[4 * P->tc_axis[0]];
    g.Mbb = (float)P->M[4 * P->tc_axis[1]];
    g.Mcc = (float)P->M[4 * P->tc_axis[2]];
    g.ax = P->tc_axis[0];
    g.bx = P->tc_axis[1];
    g.cx = P->tc_axis[2];
    g.nam = P->tc_nna - 1;
    g.nbm = P->tc_nnb - 1;
    g.tws = P->tc_tws;
    g.offY = P->tc_nna;
    g.ncols = P->tc_ncols;
    g.nslots = P->tc_nslots;
    g.spin = tc_spin(P);
    const size_t smem = tc_smem_bytes(f64 ? Prec64::S : PrecRho::S, P->tc_npad, g.tws, P->tc_nbuf, P->tc_tslots);
    for (int d0 = 0; d0 < ndens; d0 += P->tc_nd) {
        g.d0 = d0;
        g.nd = std::min(P->tc_nd, ndens - d0);
        // the plan's block count G is kept; a smaller density group only narrows each block
        g.colw = round_up(2 * g.nd * g.ncols, 8);
        g.npad = mma_cols(P->tc_G, g.colw);
        for (const TcPass& ps : P->tc_passes) {
            g.w0 = ps.w0;
            g.out_row0 = ps.out_row0;
            g.sched = P->d_tc_sched + ps.sched;
            if (!f64) k_tc_rho_b<PrecRho, true><<<(unsigned)ps.nwin, kTcBThreads, 0, s>>>(g);
            else if (df_terms) k_tc_rho_b<Prec64, true><<<(unsigned)ps.nwin, kTcBThreads, 0, s>>>(g);
            else k_tc_rho_b<Prec64, false><<<(unsigned)ps.nwin, kTcBThreads, 0, s>>>(g);
            FTCJ_CUDA(cudaGetLastError());
            const dim3 grid((unsigned)ps.ngroups, (unsigned)P->tc_mtiles);
            int nbuf = P->tc_nbuf, nts = P->tc_tslots;
            void* args[] = {&g, &nbuf, &nts};
            FTCJ_CUDA(cudaLaunchKernel(tc_rho_kernel(f64, g.colw), grid, dim3(kTcThreadsAll), args, smem, s));
        }
    }
    return FTCJ_OK;
}

int tc_rho_launches(const ftcj_plan* P, int nd) {
    return 2 * (int)std::max<size_t>(1, P->tc_passes.size()) * ((nd + P->tc_nd - 1) / P->tc_nd);
}

// Plan-time set-up of the tensor-core back-contraction: densities per
// launch, (i, j) blocks per group, the work units, their deal to the CTAs and
// the V_ij tile buffer.  TcBack::on stays false, and the walks run the
// back-contraction (the gradient's sums), where one density's columns exceed
// the MMA width or the factor tables exceed shared memory.
int setup_tc_j(ftcj_plan* P, int extra, TcArena& arena) {
    TcBack& B = extra ? P->tcg : P->tcj;
    B.on = false;
    B.extra = extra;
    const int deg = kNclass - 1 + extra, npairs_all = pairs_all(deg);
    const bool f64 = tc_eight_slices(P);
    const int nmax = f64 ? Prec64::kNmax : PrecJ::kNmax, slices = f64 ? Prec64::S : PrecJ::S;
    const int nprod = slices * (slices + 1) / 2, part_stages = (f64 ? Prec64::kWin : PrecJ::kWin) / kTcJStageM;
    const int gw = round_up(2 * P->tc_ncols, 8);
    int64_t tiles[kNclass];
    for (int L = 0; L < kNclass; ++L) tiles[L] = (P->class_start[L + 1] - P->class_start[L] + kTcM - 1) / kTcM;
    // densities per launch: the fewest A^T formations (tiles x block groups x launches)
    int nd_best = 0, G_best = 0;
    double cost_best = 1e300;
    for (int nd = 1; nd <= P->max_dens; ++nd) {
        const int colw = nd * gw;
        if (colw > nmax) break;
        const int G = std::min(kTcGmax, nmax / colw);
        double items = 0.0;
        for (int L = 0; L < kNclass; ++L) {
            const int nb = pairs_all(L + extra);
            items += (double)tiles[L] * ((nb + G - 1) / G);
        }
        const double cost = (double)((P->max_dens + nd - 1) / nd) * items;
        if (cost <= cost_best) {
            cost_best = cost;
            nd_best = nd;
            G_best = G;
        }
    }
    if (!nd_best) return FTCJ_OK;
    const int npad = mma_cols(G_best, nd_best * gw);
    int dev = 0, optin = 0;
    FTCJ_CUDA(cudaGetDevice(&dev));
    FTCJ_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    // as many stage buffers as fit beside the tables
    const int tws = P->tc_tws;
    int nbuf = kTcNbufMax;
    while (nbuf > 2 && tc_j_smem_bytes(slices, npad, tws, nbuf) > (size_t)optin) --nbuf;
    if (tc_j_smem_bytes(slices, npad, tws, nbuf) > (size_t)optin) return FTCJ_OK;
    B.nbuf = nbuf;
    // slot parts of one exact accumulation each (1024 slots, 512 in the FP64 form), as even as the stage count allows
    const int nstage = (P->tc_nslots + kTcJStageM - 1) / kTcJStageM;
    const int nsplit = std::max(1, (nstage + part_stages - 1) / part_stages);
    const int spp = std::max(1, (nstage + nsplit - 1) / nsplit);
    const int nparts = std::max(1, (nstage + spp - 1) / spp);  // every part holds at least one stage
    std::vector<int2> groups;
    std::vector<int> ipairs;
    std::vector<int4> units;
    std::vector<double> cost;
    std::vector<int> vplace((size_t)npairs_all * kNclass, -1);
    std::vector<long long> voff;
    long long nvs = 0;
    B.mma_flops = 0;
    // a unit holds all block groups of its class, or one group each where there are too few units to fill the GPU
    int64_t whole = 0;
    for (int L = 0; L < kNclass; ++L) whole += tiles[L] * nparts;
    const bool split_groups = whole < 4 * (int64_t)P->num_sms;
    for (int L = kNclass - 1; L >= 0; --L) {
        if (!tiles[L]) continue;
        std::vector<int> blocks;
        for (int i = 0; i <= L + extra; ++i)
            for (int j = 0; i + j <= L + extra; ++j) blocks.push_back(i | (j << 3));
        const int first = (int)groups.size();
        for (size_t g0 = 0; g0 < blocks.size(); g0 += G_best) {
            const int nb = (int)std::min<size_t>(G_best, blocks.size() - g0);
            for (int k = 0; k < nb; ++k)
                vplace[(size_t)pair_index(deg, blocks[g0 + k] & 7, blocks[g0 + k] >> 3) * kNclass + L] =
                    (int)groups.size() << 8 | k;
            voff.push_back(nvs);
            nvs += (long long)nstage * slices * mma_cols(nb, nd_best * gw) * 16;
            groups.push_back(make_int2((int)ipairs.size(), nb));
            ipairs.insert(ipairs.end(), blocks.begin() + g0, blocks.begin() + g0 + nb);
        }
        const int ngr = (int)groups.size() - first;
        for (int64_t t = 0; t < tiles[L]; ++t)
            for (int h = 0; h < nparts; ++h) {
                const int nst = std::min(spp, nstage - h * spp);
                for (int g0 = 0; g0 < ngr; g0 += split_groups ? 1 : ngr) {
                    const int n = split_groups ? 1 : ngr;
                    double cc = 2000.0;
                    for (int k = 0; k < n; ++k) {
                        const int nb = groups[first + g0 + k].y;
                        cc += nst * (nprod * (25.0 + 0.25 * mma_cols(nb, nd_best * gw)) + 500.0) + 110.0 * nb * nd_best * gw;
                        for (int d0 = 0; d0 < P->max_dens; d0 += nd_best)
                            B.mma_flops += (long long)nst * nprod * 2LL * kTcM *
                                                 mma_cols(nb, std::min(nd_best, P->max_dens - d0) * gw) * 16;
                    }
                    units.push_back(make_int4(L | (h << 8), first + g0, n, (int)(P->class_start[L] + t * kTcM)));
                    cost.push_back(cc);
                }
            }
    }
    B.nd = nd_best;
    B.gw = gw;
    B.G = G_best;
    B.npad = npad;
    B.nstage = nstage;
    B.sub = std::max(1, 4 / (G_best * nd_best));
    B.parts = nparts * B.sub;
    B.spp = spp;
    B.grid = std::max(1, std::min(P->num_sms, (int)units.size()));
    const std::vector<int> sched = deal(cost, B.grid);
    arena.add((int4**)&B.items, units);
    arena.add((int2**)&B.groups, groups);
    arena.add(&B.pairs, ipairs);
    arena.add(&B.sched, sched);
    arena.add(&B.voff, voff);
    arena.add(&B.vplace, vplace);
    arena.add(&B.ev, std::vector<int>(), (size_t)npairs_all * nd_best * P->tc_ncols);
    arena.add(&B.er, std::vector<int>(), (size_t)npairs_all * nd_best);
    int rc;
    nvs = std::max(nvs, 1LL);
    if ((rc = tc_alloc(P, &B.vs, sizeof(__nv_bfloat16) * (size_t)nvs))) return rc;
    FTCJ_CUDA(cudaMemset(B.vs, 0, sizeof(__nv_bfloat16) * (size_t)nvs));
    if ((rc = allow_dynamic_smem(tc_j_kernel(f64, extra), tc_j_smem_bytes(slices, npad, tws, nbuf)))) return rc;
    B.on = true;
    return FTCJ_OK;
}

namespace {

int launch_back(ftcj_plan* P, const TcBack& B, int ndens, const double* W, double* Jp, long long jp_total,
                const int64_t* term_base, cudaStream_t s) {
    if (P->ng_half == 0 || P->npairs == 0) {
        FTCJ_CUDA(cudaMemsetAsync(Jp, 0, sizeof(double) * (size_t)ndens * B.parts * jp_total, s));
        return FTCJ_OK;
    }
    const bool f64 = tc_eight_slices(P);
    TcJArgs g;
    g.slots = P->d_tc_slots;
    g.quads = P->d_tc_quads;
    g.map = P->d_tc_map;
    g.W = reinterpret_cast<const double2*>(W);
    g.sched = B.sched;
    g.units = reinterpret_cast<const int4*>(B.items);
    g.groups = reinterpret_cast<const int2*>(B.groups);
    g.ipairs = B.pairs;
    g.voff = B.voff;
    g.vplace = B.vplace;
    g.tab = P->d_tc_tab;
    g.tabz = f64 ? P->d_tc_tabz3 : P->d_tc_tabz;
    g.kpos = P->d_tc_kpos;
    g.vs = reinterpret_cast<__nv_bfloat16*>(B.vs);
    g.ev = B.ev;
    g.er = B.er;
    g.Jp = Jp;
    g.deg = kNclass - 1 + B.extra;
    g.ng_half = P->ng_half;
    g.jp_total = jp_total;
    for (int c = 0; c <= kNclass; ++c) g.cls_start[c] = P->class_start[c];
    for (int c = 0; c < kNclass; ++c) g.term_base[c] = term_base[c];
    g.err = P->d_tc_err;
    g.ax = P->tc_axis[0];
    g.bx = P->tc_axis[1];
    g.cx = P->tc_axis[2];
    g.nam = P->tc_nna - 1;
    g.nbm = P->tc_nnb - 1;
    g.tws = P->tc_tws;
    g.offY = P->tc_nna;
    g.ncols = P->tc_ncols;
    g.gw = B.gw;
    g.nslots = P->tc_nslots;
    g.nstage = B.nstage;
    g.nparts = B.parts;
    g.nsub = B.sub;
    g.spin = tc_spin(P);
    g.spp = B.spp;
    const size_t smem = tc_j_smem_bytes(f64 ? Prec64::S : PrecJ::S, B.npad, P->tc_tws, B.nbuf);
    for (int d0 = 0; d0 < ndens; d0 += B.nd) {
        g.d0 = d0;
        g.nd = std::min(B.nd, ndens - d0);
        // the plan's block count is kept; a smaller last density group only narrows each block
        g.colw = g.nd * g.gw;
        g.npad = mma_cols(B.G, g.colw);
        const unsigned nbound = (unsigned)(pairs_all(g.deg) * g.nd * g.ncols);
        if (f64) k_tc_vbound<Prec64><<<nbound, 256, 0, s>>>(g);
        else k_tc_vbound<PrecJ><<<nbound, 256, 0, s>>>(g);
        FTCJ_CUDA(cudaGetLastError());
        const long long nv = (long long)pairs_all(g.deg) * g.nstage * (kTcJStageM / 2) * g.nd * g.ncols;
        const unsigned nslice = (unsigned)((nv + 255) / 256);
        if (f64) k_tc_vslice<Prec64><<<nslice, 256, 0, s>>>(g);
        else k_tc_vslice<PrecJ><<<nslice, 256, 0, s>>>(g);
        FTCJ_CUDA(cudaGetLastError());
        int nbuf = B.nbuf;
        void* args[] = {&g, &nbuf};
        FTCJ_CUDA(cudaLaunchKernel(tc_j_kernel(f64, B.extra), dim3((unsigned)B.grid), dim3(kTcThreadsAll), args, smem, s));
    }
    return FTCJ_OK;
}

}  // namespace

int launch_tc_j(ftcj_plan* P, int ndens, const double* W, cudaStream_t s) {
    return launch_back(P, P->tcj, ndens, W, P->d_Jp, P->total_terms, P->term_base, s);
}

// the degree-(L+1) sums of the nuclear gradient, into d_Jg
int launch_tc_j_grad(ftcj_plan* P, int ndens, const double* W, cudaStream_t s) {
    return launch_back(P, P->tcg, ndens, W, P->d_Jg, P->total_terms_g, P->term_base_g, s);
}

int tc_j_launches(const ftcj_plan* P, int nd) { return 3 * ((nd + P->tcj.nd - 1) / P->tcj.nd); }

}  // namespace ftcj

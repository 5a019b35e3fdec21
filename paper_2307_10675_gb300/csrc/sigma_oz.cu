// FP64-accurate sigma build on the FP16 tensor cores (tcgen05), one fused
// kernel per wave of problems.
//
// GB300 runs FP64 at ~1/1800 of its 16-bit tensor rate, so the sigma builds
// that must be exact to FP64 level are emulated with integer slices (an
// Ozaki-style splitting):
//
//   W[A][B] = Wscale 2^-7 (w1 + 2^-8 w2 + ... + 2^-32 w5)    Wscale >= max|W|
//   c[K]    = dscale  2^-6 (d1 + 2^-8 d2 + ... + 2^-32 d5)    dscale > max|c|
//
// (dscale > 2 max|c| for spin-flip-symmetric c),
//
// with every slice an integer in [-128, 128], exact in FP16: c becomes the
// fixed-point integer X = round(c 2^38 / dscale), whose slices are the
// base-256 digits of X + 128 (1 + 2^8 + ... + 2^32) minus 128.  The 15 slice
// products with i + j <= 4 (0-based) go to five FP32 accumulators, one per
// scale level i + j; a level over K terms is an exact integer below
// 5 2^14 K < 2^24 (K <= 112 here).  The levels are combined in int64,
// T = sum_L 2^{8 (4 - L)} acc_L in units of 2^-45 Wscale dscale, every further
// sum is an integer sum, and each determinant is converted once.  The dropped
// terms and the slice truncation leave a relative error of order 2^-38 of
// max|W| max|c|.
//
// Spin-flip-symmetric c (C = C^T): with X_A the string matrix of E+_A and
// T_A = sum_B W[A][B] X_B C the contraction over the alpha excitations alone,
//   S = sum_A X_A T_A (alpha excitations of T) + T_A X_A (beta excitations),
//   sigma = S + S^T.
// For any other c the same S is built for C and for C^T (two passes), and
// sigma = S(C) + S(C^T)^T.
//
// Row I_a of T needs only the pairs B that I_a has an alpha excitation on:
// nexc = m (n - m + 1) of the npair = n (n + 1) / 2 pairs (48 of 171 for
// CAS(6e,18o)), the same for every I_b of the row.  So the work item of a CTA
// is one alpha string I_a, its contraction runs over K = nexc rows (rounded to
// 16), and T never leaves the SM: the epilogue adds each T element
// * to S[J_a][I_b] for the alpha excitation I_a -> J_a on its pair (one row of
//   32 consecutive I_b per warp: coalesced 64-bit reductions in L2), and
// * to S[I_a][J_b] for the beta excitation I_b -> J_b on its pair, in an int64
//   accumulator row in shared memory (two 32-bit atomics per element: 64-bit
//   ones are a compare-and-swap loop there, 23 to 43 clocks per warp against
//   2 x 3.6), added to S once per item.
// The earlier form contracted all pairs (dense K), wrote T (npair int64 per
// determinant) to HBM and read it back in a scatter kernel.
//
// Operands arrive ready for the MMA: the digit planes of c and of -c (rows of
// I_b for each J_a, written once per sigma) and the W image (rows of output
// pairs for each contracted pair) are both MN-major, so a K row of either is a
// contiguous run that cp.async places into the 128-byte-swizzled tile in
// 16-byte chunks; no thread computes on an operand.  Output pairs run in
// chunks of 48 columns: the five W slices of a chunk lie side by side
// (5 x 48 = 240 columns), so digit slice j of c multiplies slices 0..4-j in
// one MMA of N = (5 - j) 48 whose columns are the levels j..4 side by side:
// five MMAs per 16 K rows in place of fifteen, each reading its A tile once.
// Two accumulator sets (2 x 240 of the 512 TMEM columns) let the epilogue of a
// chunk overlap the MMAs of the next.
//
// Bound: per 128 x 48 tile and 16 K rows 360 tensor clocks and 332 clocks of
// shared-memory operand reads.  The epilogue is the longer side: ~25 issue
// slots per T element, of which a determinant uses 28 % (its own excitations)
// and a warp of 32 consecutive strings 90 %, and the two shared-memory
// reductions (3.4 clocks a warp).  Sixteen warps share it, twelve for the beta
// sums and four for the alpha sums; eight warps with both took 612 us.
//
// The producers' copies go out in batches of ten and eight after their row
// numbers are read: one row number and one copy at a time took a warp 240 clocks
// a copy, and the W chunks of CAS(8e,20o), reloaded for every tile, bounded it.
//
// Measured, one sigma: CAS(6e,18o) 382 us (1282 us contraction + 254 us scatter
// before), CAS(8e,20o) 17.0 ms (96.0 + 9.8 ms in three waves of 16 GB, now 0.7 GB
// at once; 29.4 ms with the copies one at a time).
#include <cuda_fp16.h>

#include <algorithm>

#include "fold.cuh"
#include "fp64int.cuh"
#include "sigma.cuh"
#include "tcgen05.cuh"

namespace ifci {

namespace {

using namespace tc;

constexpr int kS = 5;                       // slices per operand
constexpr int kNC = 48;                     // output pairs per chunk
constexpr int kTBuf = kS * kNC;             // TMEM columns of one accumulator set
constexpr int kOzTmemCols = 512;
constexpr int kMaxK = 112;                  // contracted pairs of one string, rounded to 16
constexpr int kMaxNp = 304;                 // pairs (norb <= 24)
constexpr int kMaxStrings = 32767;          // 16-bit map entries (sign << 15 | J), 0xFFFF = none
// Longest lists of the narrow epilogue.  A digit is at most 128, the top one of c
// at most 65, so a level over K rows is at most K (65 + 4 128) 128: below 2^22 up
// to K = 56, as is a row sum of K 26-bit words below 2^32 and of K T's below 2^57.
// Lists of 54 to 56 entries: 1 to 8 % off a sigma against the wide form (6e,20o:
// 1044 us, 973 us).  A third form for up to 72, with four levels narrow, gave 1 %.
constexpr int kNarrowK = 56;
constexpr int kMaxW = 8;                    // W chunk buffers
constexpr int kBetaWarps = 12, kAlphaWarps = 4, kAWarps = 4, kWWarps = 2;
constexpr int kEpiWarps = kBetaWarps + kAlphaWarps;
constexpr int kOzThreads = 32 * (kEpiWarps + kAWarps + kWWarps + 1);
constexpr int kSmemLimit = 232448 - 3696 - 1024;   // dynamic part: 227 KB less static (3.6 KB) and alignment
constexpr long long kDigitBias = 128ll * 0x0101010101ll;      // 128 in each of the five digits
constexpr uint32_t kNoMap = 0xFFFFu, kNone = 0xFFFFFFFFu;
constexpr uint32_t kMagic = 0x4B400000u;     // FP32 1.5 2^23: kMagic + i are the bits of 1.5 2^23 + i, |i| < 2^22
constexpr int kLowBits = 26;

__host__ __device__ inline int np_pad(int np) { return round_up(np, 16); }
__host__ __device__ inline int row_ld(int nstr) { return (nstr + 7) / 8 * 8; }   // digit plane row (halves)

// slice a value in [-1, 1] into kS integers in [-128, 128]: x = 2^-7 sum_i 2^{-8i} s_i
__device__ __forceinline__ void slice5(double x, float (&sl)[kS]) {
    double r = x * 128.0;
#pragma unroll
    for (int i = 0; i < kS; i++) {
        double q = rint(r);
        sl[i] = (float)q;
        r = (r - q) * 256.0;
    }
}

// The same for w / 2^e, |w| < 2^e, on the integer pipe (an FP64 instruction
// takes a sub-partition 64 to 104 clk, a division 564): w 2^(59 - e) with a
// sticky lowest bit, its digits rounded to nearest even one by one as rint does.
__device__ __forceinline__ void slice5_pow2(double w, int e, float (&sl)[kS]) {
    const int f = dexp_field(w);
    const long long mant = (dbits(w) & 0xFFFFFFFFFFFFFll) | (f ? 1ll << 52 : 0ll);
    const int sh = (f ? f : 1) - 1075 - e + 59;   // <= 6
    long long x = sh >= 0 ? mant << sh : sh > -63 ? (mant >> -sh) | ((mant & ((1ll << -sh) - 1)) != 0) : mant != 0;
    if (dbits(w) < 0) x = -x;
#pragma unroll
    for (int i = 0; i < kS; i++) {
        const int b = 52 - 8 * i;
        const long long half = 1ll << (b - 1), q = (x + half - 1 + (x >> b & 1)) >> b;
        sl[i] = (float)(int)q;
        x -= q << b;
    }
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    __half a = __float2half_rn(lo), b = __float2half_rn(hi);   // exact: |lo|, |hi| <= 128, integers
    return (uint32_t)__half_as_ushort(a) | ((uint32_t)__half_as_ushort(b) << 16);
}

// FP16 pair (u0 - 128, u1 - 128) of byte D of a and of b: the byte permute
// puts u into the low mantissa bits of the FP16 number 1024 (0x6400), which
// then reads 1024 + u exactly, and one packed subtraction of 1152 leaves
// u - 128 in [-128, 127] (exact).
__device__ __forceinline__ uint32_t digit_pair_f16(uint32_t a, uint32_t b, int D) {
    const uint32_t sel = D | (D << 4) | ((D + 4) << 8) | ((D + 4) << 12);   // a compile-time constant once unrolled
    const uint32_t t = (__byte_perm(a, b, sel) & 0x00FF00FFu) | 0x64006400u;
    __half2 v = *reinterpret_cast<const __half2 *>(&t);
    const __half2 off = __halves2half2(__ushort_as_half((unsigned short)0x6480), __ushort_as_half((unsigned short)0x6480));
    v = __hsub2(v, off);
    return *reinterpret_cast<uint32_t *>(&v);
}

__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
    return r != 0;
}

// tcgen05 shared-memory descriptor of an MN-major operand, 128-byte swizzle:
// atoms of 64 MN elements x 8 K rows (1024 B); `lbo` bytes between MN atoms,
// 1024 B between groups of 8 K rows.
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t addr, uint32_t lbo) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | (uint64_t)(lbo >> 4) << 16 | (uint64_t)(1024 >> 4) << 32 |
           (uint64_t)1 << 46 | (uint64_t)2 << 61;
}

// kind::f16, FP16 x FP16 -> FP32, A and B MN-major
__device__ __forceinline__ uint32_t idesc_f16_mn(int M, int N) { return idesc_f16(M, N) | (1u << 15) | (1u << 16); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool live) {
    const int bytes = live ? 16 : 0;   // 0: the 16 bytes are zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
// own copies landed and visible to the tensor core's proxy
__device__ __forceinline__ void cp_async_done() {
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void named_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}

__device__ __forceinline__ uint32_t tmem_ld1(uint32_t taddr) {
    uint32_t r;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr));
    return r;
}
// (x, y) = (x sx, y sy) + (c, c)
__device__ __forceinline__ void fma2(uint32_t &x, uint32_t &y, uint32_t sx, uint32_t sy, uint32_t c) {
    asm("{\n\t.reg .b64 a, b, d;\n\t"
        "mov.b64 a, {%0, %1};\n\t"
        "mov.b64 b, {%2, %3};\n\t"
        "mov.b64 d, {%4, %4};\n\t"
        "fma.rn.f32x2 a, a, b, d;\n\t"
        "mov.b64 {%0, %1}, a;\n\t}"
        : "+r"(x), "+r"(y)
        : "r"(sx), "r"(sy), "r"(c));
}
__device__ __forceinline__ unsigned long long mad_wide(uint32_t a, uint32_t b, unsigned long long c) {
    unsigned long long d;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// Row sum in two 32-bit words of shared memory where the map entry m names a
// string.  Narrow: the caller's words are T's low 26 bits and T >> 26, which
// need no carry.  Wide: T's halves, the carry taken from the low word's old
// value.  Predicated, so that the columns of an unrolled loop interleave.
__device__ __forceinline__ void row_add_narrow(uint32_t m, uint32_t lo, uint32_t hi, uint32_t x, uint32_t y) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %0, 65535;\n\t"
        "@p red.shared.add.u32 [%1], %3;\n\t"
        "@p red.shared.add.u32 [%2], %4;\n\t}" ::"r"(m),
        "r"(lo), "r"(hi), "r"(x), "r"(y));
}
__device__ __forceinline__ void row_add_wide(uint32_t m, uint32_t lo, uint32_t hi, uint32_t x, uint32_t y) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .u32 o, c;\n\t"
        "setp.ne.u32 p, %0, 65535;\n\t"
        "mov.u32 o, 0;\n\t"
        "@p atom.shared.add.u32 o, [%1], %3;\n\t"
        "add.u32 o, o, %3;\n\t"
        "setp.lt.u32 q, o, %3;\n\t"
        "selp.u32 c, 1, 0, q;\n\t"
        "add.u32 c, c, %4;\n\t"
        "@p red.shared.add.u32 [%2], c;\n\t}" ::"r"(m),
        "r"(lo), "r"(hi), "r"(x), "r"(y));
}

// *dst += v in L2 where `on`
__device__ __forceinline__ void red_add_if(bool on, unsigned long long *dst, unsigned long long v) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %0, 0;\n\t"
        "@p red.global.add.u64 [%1], %2;\n\t}" ::"r"((uint32_t)on),
        "l"(dst), "l"(v)
        : "memory");
}

struct OzGeom {
    int nA, nW;      // stages of c tiles, chunk buffers of W
    int kmax;        // K rows a buffer holds
    int rows;        // strings the shared accumulator row holds; 0: the row is added to S in L2 directly
    uint32_t m8, m16, m24;   // 2^8, 2^16, 2^24, in registers: one multiply-add per level instead of a shift and two adds
};

// T of levels that may reach 2^24; levels 0 and 1 (at most two products of 2^14 a
// row) stay below 2^22 and take the biased form.
static_assert(2 * (1 << 14) * kMaxK < (1 << 22), "levels 0 and 1 of the wide form");
__device__ __forceinline__ unsigned long long wide_sum(float sg, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                       uint32_t a4) {
    const uint32_t h = __float_as_uint(fmaf(sg, __uint_as_float(a0), 12582912.0f)) - kMagic;
    const uint32_t l = __float_as_uint(fmaf(sg, __uint_as_float(a1), 12582912.0f)) - kMagic;
    long long T = __float2int_rn(sg * __uint_as_float(a4));
    T += (long long)__float2int_rn(sg * __uint_as_float(a3)) * 256;
    T += (long long)__float2int_rn(sg * __uint_as_float(a2)) * 65536;
    T += (long long)(int)l * 16777216;
    return (unsigned long long)T + ((unsigned long long)h << 32);
}
// The biased value of T from its level sums: each level as kMagic + acc, so
// T + kBias = sum_L (kMagic + acc_L) 2^{8 (4 - L)} needs no sign handling.
constexpr unsigned long long kBias = (unsigned long long)kMagic * 0x0101010101ull;
__device__ __forceinline__ unsigned long long biased(const uint32_t (&b)[kS], const OzGeom &g) {
    unsigned long long t = mad_wide(b[3], g.m8, b[4]);
    t = mad_wide(b[2], g.m16, t);
    t = mad_wide(b[1], g.m24, t);
    return t + ((unsigned long long)b[0] << 32);
}

// The K rows of item (prob, ka): excitations e of string ka whose pair is
// contracted, in list order.  out[k] = digit plane row (ROWS) or row of the W
// image; returns their number.  NT threads with named barrier `id`.
template <int NT, bool ROWS, typename TL>
__device__ __forceinline__ int build_list(const SigmaProb &p, int ka, int tid, int id, TL *out, uint32_t *msk) {
    constexpr int NWARP = NT / 32, R = (kMaxK + NT - 1) / NT;
    const int lane = tid & 31, wi = tid >> 5, nexc = p.nexc, nstr = p.nstr;
    const int32_t *row = p.exc + (size_t)ka * nexc;
    const int16_t *pinv = p.pinv;
    int val[R];
    uint32_t bal[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int e = r * NT + tid;
        int idx = -1, v = 0;
        if (e < nexc) {
            const int32_t x = row[e];
            idx = pinv ? pinv[exc_pair(x)] : exc_pair(x);
            v = ROWS ? exc_J(x) + ((x & 1) ? kS * nstr : 0) : idx;
        }
        val[r] = v;
        bal[r] = __ballot_sync(0xffffffffu, idx >= 0);
    }
    named_sync(id, NT);   // the previous list is no longer read
#pragma unroll
    for (int r = 0; r < R; r++)
        if (lane == 0) msk[r * NWARP + wi] = bal[r];
    named_sync(id, NT);
    int total = 0;
#pragma unroll
    for (int r = 0; r < R; r++) {
        int at = 0;
        for (int w = 0; w < R * NWARP; w++)
            if (w < r * NWARP + wi) at += __popc(msk[w]);
        at += __popc(bal[r] & ((1u << lane) - 1u));
        if (bal[r] >> lane & 1u) out[at] = (TL)val[r];
    }
    for (int w = 0; w < R * NWARP; w++) total += __popc(msk[w]);
    named_sync(id, NT);
    return total;
}

// One item = alpha string tile.start of pass tile.sub (0: C, 1: C^T) of problem
// tile.prob.  WIDE: items with more than kNarrowK excitations per string; ROW: the
// item's row of S is summed in shared memory (always, unless WIDE).
template <bool WIDE, bool ROW>
__global__ void __launch_bounds__(kOzThreads, 1)
oz_sigma_kernel(const SigmaProb *__restrict__ probs, const WorkItem *__restrict__ items, int nitem,
                const __half *__restrict__ Q, long long *__restrict__ S, int *__restrict__ err, OzGeom g) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t b_fullA[2], b_emptyA[2], b_fullW[kMaxW], b_emptyW[kMaxW], b_tfull[2], b_tempty[2],
        b_epi, b_drain;
    __shared__ uint32_t tmem_slot;
    __shared__ int kp_of[2], okA[2], okW[2], lstA[kMaxK];
    __shared__ uint16_t lstW[kMaxK];
    __shared__ uint32_t mskA[4], mskW[4];
    // the alpha excitations of the item's string, in column order, one copy per alpha warp:
    // output pair, and J nstr | sign << 31 (element offset of row J of S)
    __shared__ uint32_t s_aofs[kAlphaWarps][kMaxK];
    __shared__ uint16_t s_acol[kAlphaWarps][kMaxK];
    uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t stageA = (uint32_t)kS * g.kmax * 256, stageW = (uint32_t)g.kmax * 512;
    uint8_t *Asm = base, *Wsm = base + g.nA * stageA;
    uint32_t *rlo = (uint32_t *)(Wsm + g.nW * stageW), *rhi = rlo + g.rows;
    // the warp index through a shuffle: uniform for the compiler, so that tensor
    // addresses and descriptors stay in uniform registers (the instructions take
    // no others; from a divergent value each operand is moved over, ~200 clocks an MMA)
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(kOzTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < 2; i++) {
            mbar_init(smem_u32(&b_fullA[i]), 32 * kAWarps);
            mbar_init(smem_u32(&b_emptyA[i]), 1);
            mbar_init(smem_u32(&b_tfull[i]), 1);
            mbar_init(smem_u32(&b_tempty[i]), kEpiWarps);
        }
        for (int i = 0; i < kMaxW; i++) {
            mbar_init(smem_u32(&b_fullW[i]), 32 * kWWarps);
            mbar_init(smem_u32(&b_emptyW[i]), 1);
        }
        mbar_init(smem_u32(&b_epi), 32 * kBetaWarps);
        mbar_init(smem_u32(&b_drain), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < 2 * g.rows; i += kOzThreads) rlo[i] = 0u;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    bool ok = true;

    if (warp < kBetaWarps) {
        // ---- beta excitations: every T element to the item's row of S
        const int q = warp & 3, part = warp >> 2;   // TMEM lane quarter, share of the columns
        const uint32_t lane_base = (uint32_t)(q * 32) << 16, row_lo = smem_u32(rlo), row_hi = row_lo + 4u * (uint32_t)g.rows;
        uint32_t tn = 0, ep = 0;
        auto epi_sync = [&]() {   // bounded: a role that gave up must not hang the others
            mbar_arrive(smem_u32(&b_epi));
            const bool r = mbar_wait(smem_u32(&b_epi), ep & 1);
            ep++;
            return __all_sync(0xffffffffu, r) != 0;
        };
        for (int it = blockIdx.x; it < nitem && ok; it += gridDim.x) {
            const WorkItem item = items[it];
            const SigmaProb &p = probs[item.prob];
            if (p.active && !*p.active) continue;
            const int nstr = p.nstr, npad = np_pad(p.act ? p.npc : p.np), ldj = p.ldj, ka = (int)item.start;
            long long *Srow = S + p.doff + (item.sub ? p.ndet : 0) + (long long)ka * nstr;
            const uint2 *jmap = reinterpret_cast<const uint2 *>(p.jmap);
            for (int mt = 0; mt * kTM < nstr && ok; mt++) {
                const int ib0 = mt * kTM + q * 32;
                const bool wlive = ib0 < nstr;
                // map entries of four output pairs of this determinant's string
                const uint2 *jcol = jmap + ib0 + lane;
                for (int c0 = 0; c0 < npad; c0 += kNC, tn++) {
                    const int w = min(kNC, npad - c0);
                    const uint32_t buf = tn & 1;
                    constexpr int kStep = kBetaWarps;   // columns between two groups of a warp
                    auto map_of = [&](int cc) {
                        return wlive && cc < w ? jcol[(size_t)((c0 + cc) >> 2) * ldj] : make_uint2(kNone, kNone);
                    };
                    uint2 jn[2] = {map_of(4 * part), map_of(4 * part + kStep)};
                    if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&b_tfull[buf]), (tn >> 1) & 1))) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    for (int cc = 4 * part; cc < w && wlive; cc += 2 * kStep) {
                        // two groups of four columns, all levels
                        uint32_t v[2][kS][4];
#pragma unroll
                        for (int h = 0; h < 2; h++)
#pragma unroll
                            for (int L = 0; L < kS; L++)
                                tmem_ld4(tmem + lane_base + buf * kTBuf + (uint32_t)(L * w + min(cc + kStep * h, w - 4)), v[h][L]);
                        const uint2 jm[2] = {jn[0], jn[1]};
                        jn[0] = map_of(cc + 2 * kStep);
                        jn[1] = map_of(cc + 3 * kStep);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int h = 0; h < 2; h++)
#pragma unroll
                            for (int k = 0; k < 2; k++) {
                                const uint32_t mw = k ? jm[h].y : jm[h].x;   // kNone past the last column
                                const uint32_t s0 = 0x3F800000u | (mw << 16 & 0x80000000u), s1 = 0x3F800000u | (mw & 0x80000000u);
                                if (!WIDE) {
                                    // |acc| < 2^22: 1.5 2^23 +- acc is exact and holds it in its low bits
#pragma unroll
                                    for (int L = 0; L < kS; L++) fma2(v[h][L][2 * k], v[h][L][2 * k + 1], s0, s1, kMagic);
                                }
#pragma unroll
                                for (int e = 2 * k; e < 2 * k + 2; e++) {
                                    const uint32_t m = e & 1 ? mw >> 16 : mw & 0xFFFFu, j4 = (m & 0x7FFFu) * 4u;
                                    if (WIDE) {
                                        const unsigned long long T = wide_sum(__uint_as_float(e & 1 ? s1 : s0), v[h][0][e], v[h][1][e],
                                                                              v[h][2][e], v[h][3][e], v[h][4][e]);
                                        if (ROW) row_add_wide(m, row_lo + j4, row_hi + j4, (uint32_t)T, (uint32_t)(T >> 32));
                                        else red_add_if(m != kNoMap, reinterpret_cast<unsigned long long *>(Srow) + (m & 0x7FFFu), T);
                                    } else {
                                        const uint32_t b[kS] = {v[h][0][e], v[h][1][e], v[h][2][e], v[h][3][e], v[h][4][e]};
                                        const unsigned long long T = biased(b, g);
                                        row_add_narrow(m, row_lo + j4, row_hi + j4, (uint32_t)T & ((1u << kLowBits) - 1u),
                                                       __funnelshift_r((uint32_t)T, (uint32_t)(T >> 32), kLowBits));
                                    }
                                }
                            }
                    }
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&b_tempty[buf]));
                }
            }
            if (!ok) break;
            if (ROW) {
                ok = epi_sync();   // every beta excitation of the row is in
                for (int i = tid; i < nstr && ok; i += 32 * kBetaWarps) {
                    const uint32_t lo = rlo[i], hi = rhi[i];
                    rlo[i] = 0u;
                    rhi[i] = 0u;
                    unsigned long long v;
                    if (WIDE) {
                        v = (unsigned long long)hi << 32 | lo;
                    } else {
                        // less the bias of every term; |row sum| < 2^57, so its low 58 bits are enough
                        v = ((unsigned long long)hi << kLowBits) + lo;
                        v -= (unsigned long long)(p.kcnt ? p.kcnt[i] : p.nexc) * kBias;
                        v = (unsigned long long)((long long)(v << (32 - kLowBits)) >> (32 - kLowBits));
                    }
                    red_add_if(v != 0, reinterpret_cast<unsigned long long *>(Srow) + i, v);
                }
                ok = epi_sync() && ok;   // the row is clear again
            }
        }
    } else if (warp < kEpiWarps) {
        // ---- alpha excitations of the item's string: some columns, the same for every lane
        const int q = warp & 3;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        uint32_t *aofs = s_aofs[q];
        uint16_t *acol = s_acol[q];
        uint32_t tn = 0;
        for (int it = blockIdx.x; it < nitem && ok; it += gridDim.x) {
            const WorkItem item = items[it];
            const SigmaProb &p = probs[item.prob];
            if (p.active && !*p.active) continue;
            const int nstr = p.nstr, npad = np_pad(p.act ? p.npc : p.np), ldj = p.ldj, ka = (int)item.start;
            unsigned long long *Sp = reinterpret_cast<unsigned long long *>(S) + p.doff + (item.sub ? p.ndet : 0);
            int na = 0;
            for (int A0 = 0; A0 < npad; A0 += 32) {
                const int A = A0 + lane;
                const uint32_t m = A < npad ? p.jmap[((size_t)(A >> 2) * ldj + ka) * 4 + (A & 3)] : kNoMap;
                const uint32_t bal = __ballot_sync(0xffffffffu, m != kNoMap);
                if (m != kNoMap) {
                    const int at = na + __popc(bal & ((1u << lane) - 1u));
                    acol[at] = (uint16_t)A;
                    aofs[at] = (m & 0x7FFFu) * (uint32_t)nstr | (m >> 15) << 31;
                }
                na += __popc(bal);
            }
            __syncwarp();
            for (int mt = 0; mt * kTM < nstr && ok; mt++) {
                const int ib0 = mt * kTM + q * 32, ib = ib0 + lane;
                int i = 0;
                for (int c0 = 0; c0 < npad; c0 += kNC, tn++) {
                    const int w = min(kNC, npad - c0);
                    const uint32_t buf = tn & 1, tcol = tmem + lane_base + buf * kTBuf - (uint32_t)c0;
                    if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&b_tfull[buf]), (tn >> 1) & 1))) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    // four columns of the list at a time
                    while (i < na && acol[i] < c0 + w) {
                        uint32_t v[4][kS], of[4];
                        int n = 0;
#pragma unroll
                        for (int u = 0; u < 4; u++) {
                            const int k = min(i + u, na - 1);
                            const uint32_t col = min((uint32_t)acol[k], (uint32_t)(c0 + w - 1));
                            n += i + u < na && acol[k] < c0 + w;
                            of[u] = aofs[k];
#pragma unroll
                            for (int L = 0; L < kS; L++) v[u][L] = tmem_ld1(tcol + (uint32_t)(L * w) + col);
                        }
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int u = 0; u < 4; u++) {
                            const float sg = __uint_as_float(0x3F800000u | (of[u] & 0x80000000u));
                            unsigned long long T;
                            if (WIDE) {
                                T = wide_sum(sg, v[u][0], v[u][1], v[u][2], v[u][3], v[u][4]);
                            } else {
#pragma unroll
                                for (int L = 0; L < kS; L++)
                                    v[u][L] = __float_as_uint(fmaf(sg, __uint_as_float(v[u][L]), 12582912.0f));
                                T = biased(v[u], g) - kBias;
                            }
                            red_add_if(u < n && ib < nstr, Sp + (of[u] & 0x7FFFFFFFu) + ib, T);
                        }
                        i += n;
                    }
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&b_tempty[buf]));
                }
            }
        }
    } else if (warp < kEpiWarps + kAWarps) {
        // ---- digit tiles of c: K rows J_a, 128 determinants of each
        const int t = tid - 32 * kEpiWarps;
        uint32_t an = 0;
        for (int it = blockIdx.x; it < nitem && ok; it += gridDim.x) {
            const WorkItem item = items[it];
            const SigmaProb &p = probs[item.prob];
            if (p.active && !*p.active) continue;
            const int nstr = p.nstr, ldq = row_ld(nstr);
            const __half *src = Q + p.qoff + (item.sub ? (size_t)2 * kS * nstr * ldq : 0);
            const int kc = build_list<32 * kAWarps, true>(p, (int)item.start, t, 1, lstA, mskA), Kp = round_up(kc, 16);
            const int ch = t & 15;
            for (int mt = 0; mt * kTM < nstr; mt++, an++) {
                const uint32_t slot = an % g.nA;
                if (t == 0) okA[an & 1] = mbar_wait(smem_u32(&b_emptyA[slot]), ((an / g.nA) & 1) ^ 1);
                named_sync(1, 32 * kAWarps);
                if (!okA[an & 1]) { ok = false; break; }
                const uint32_t dst = smem_u32(Asm) + slot * stageA + (ch >> 3) * (uint32_t)Kp * 128;
                const int col = mt * kTM + ch * 8;
                // two K rows (of this thread's Kp / 8, an even number) and all digits at a time
                const size_t plane = (size_t)nstr * ldq;
                const bool in = col < nstr;
                for (int k0 = t >> 4; k0 < Kp; k0 += 4 * kAWarps) {
                    const int k1 = k0 + 2 * kAWarps, r0 = lstA[k0], r1 = lstA[k1];
                    const bool lv0 = in && k0 < kc, lv1 = in && k1 < kc;
                    const __half *s0 = lv0 ? src + (size_t)r0 * ldq + col : Q, *s1 = lv1 ? src + (size_t)r1 * ldq + col : Q;
                    const size_t p0 = lv0 ? plane : 0, p1 = lv1 ? plane : 0;
                    const uint32_t d0 = dst + (uint32_t)(k0 * 128 + (((ch & 7) ^ (k0 & 7)) << 4));
                    const uint32_t d1 = dst + (uint32_t)(k1 * 128 + (((ch & 7) ^ (k1 & 7)) << 4));
#pragma unroll
                    for (int j = 0; j < kS; j++) {
                        cp_async16(d0 + (uint32_t)(j * Kp * 256), s0 + j * p0, lv0);
                        cp_async16(d1 + (uint32_t)(j * Kp * 256), s1 + j * p1, lv1);
                    }
                }
                if (t == 0) kp_of[slot] = Kp;
                cp_async_done();
                mbar_arrive(smem_u32(&b_fullA[slot]));
            }
        }
        cp_async_done();
    } else if (warp < kEpiWarps + kAWarps + kWWarps) {
        // ---- W chunks: K rows = contracted pairs, 5 slices x w output pairs of each
        const int t = tid - 32 * (kEpiWarps + kAWarps), wi = t >> 5;
        uint32_t wn = 0;
        for (int it = blockIdx.x; it < nitem && ok; it += gridDim.x) {
            const WorkItem item = items[it];
            const SigmaProb &p = probs[item.prob];
            if (p.active && !*p.active) continue;
            const int nstr = p.nstr, npc = p.act ? p.npc : p.np, npad = np_pad(npc), nch = (npad + kNC - 1) / kNC;
            const uint8_t *img = (const uint8_t *)p.Woz;
            const int kc = build_list<32 * kWWarps, false>(p, (int)item.start, t, 2, lstW, mskW), Kp = round_up(kc, 16);
            const int reps = nch <= g.nW ? 1 : (nstr + kTM - 1) / kTM;   // resident chunks are loaded once per item
            for (int r = 0; r < reps && ok; r++)
                for (int c0 = 0; c0 < npad; c0 += kNC, wn++) {
                    const int w = min(kNC, npad - c0);
                    const uint32_t slot = wn % g.nW;
                    if (t == 0) okW[wn & 1] = mbar_wait(smem_u32(&b_emptyW[slot]), ((wn / g.nW) & 1) ^ 1);
                    named_sync(2, 32 * kWWarps);
                    if (!okW[wn & 1]) { ok = false; break; }
                    const uint8_t *cimg = img + (size_t)npc * 10 * c0;
                    const int n8 = lane;                       // 16-byte chunk of a row (5 w / 8 <= 30 of them)
                    const uint32_t dst = smem_u32(Wsm) + slot * stageW + (uint32_t)(n8 >> 3) * Kp * 128;
                    if (n8 < kS * w / 8)
                        for (int k0 = wi; k0 < Kp; k0 += 8 * kWWarps) {   // Kp / 2 rows a warp, a multiple of 8
                            int b[8];
#pragma unroll
                            for (int u = 0; u < 8; u++) b[u] = lstW[k0 + u * kWWarps];
#pragma unroll
                            for (int u = 0; u < 8; u++) {
                                const int k = k0 + u * kWWarps;
                                const bool lv = k < kc;
                                cp_async16(dst + (uint32_t)(k * 128 + (((n8 & 7) ^ (k & 7)) << 4)),
                                           lv ? cimg + (uint32_t)(b[u] * 10 * w) + n8 * 16 : img, lv);
                            }
                        }
                    cp_async_done();
                    mbar_arrive(smem_u32(&b_fullW[slot]));
                }
        }
        cp_async_done();
    } else {
        // ---- the MMAs: the warp runs the loop together, one elected lane issues
        const bool lead = elect_one();
        const uint32_t idesc0 = idesc_f16_mn(kTM, 0);
        uint32_t an = 0, wn = 0, tn = 0;
        for (int it = blockIdx.x; it < nitem && ok; it += gridDim.x) {
            const WorkItem item = items[it];
            const SigmaProb &p = probs[item.prob];
            if (p.active && !*p.active) continue;
            const int nstr = p.nstr, npad = np_pad(p.act ? p.npc : p.np), nch = (npad + kNC - 1) / kNC;
            const int nmt = (nstr + kTM - 1) / kTM;
            const bool res = nch <= g.nW;
            const uint32_t w0 = wn;
            for (int mt = 0; mt < nmt && ok; mt++, an++) {
                const uint32_t sa = an % g.nA;
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&b_fullA[sa]), (an / g.nA) & 1));
                if (!ok) break;
                const int Kp = __shfl_sync(0xffffffffu, kp_of[sa], 0), ns = Kp / 16;
                const uint32_t lbo = (uint32_t)Kp * 128;
                const uint64_t ad0 = smem_desc_mn(smem_u32(Asm) + sa * stageA, lbo);
                for (int c = 0; c < nch; c++, tn++) {
                    const int w = min(kNC, npad - c * kNC);
                    uint32_t sw = (w0 + c) % g.nW;
                    if (!res || mt == 0) {
                        sw = wn % g.nW;
                        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&b_fullW[sw]), (wn / g.nW) & 1));
                        if (!ok) break;
                        wn++;
                    }
                    const uint32_t tb = tn & 1;
                    ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&b_tempty[tb]), ((tn >> 1) & 1) ^ 1));
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    if (lead) {
                        const uint64_t wd = smem_desc_mn(smem_u32(Wsm) + sw * stageW, lbo);
#pragma unroll
                        for (int j = 0; j < kS; j++) {
                            const uint32_t idesc = idesc0 | (uint32_t)((kS - j) * w >> 3) << 17;
                            const uint32_t td = tmem + tb * kTBuf + (uint32_t)(j * w);
                            const uint64_t aj = ad0 + (uint64_t)(j * Kp * 16);
                            mma_f16(td, aj, wd, idesc, j > 0 ? 1u : 0u);
                            for (int s = 1; s < ns; s++)
                                mma_f16(td, aj + (uint64_t)(s * 128), wd + (uint64_t)(s * 128), idesc, 1u);
                        }
                        mma_commit(smem_u32(&b_tfull[tb]));
                        if (!res || mt + 1 == nmt) mma_commit(smem_u32(&b_emptyW[sw]));
                        if (c + 1 == nch) mma_commit(smem_u32(&b_emptyA[sa]));
                    }
                    __syncwarp();
                }
            }
        }
        if (!ok) {   // MMAs may still be in flight: wait for them (bounded) before the buffers go
            if (lead) mma_commit(smem_u32(&b_drain));
            __syncwarp();
            mbar_wait(smem_u32(&b_drain), 0);
        }
    }
    __syncwarp();
    if (!ok && lane == 0) atomicExch(err, 1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kOzTmemCols)
                     : "memory");
}

// Digit planes of a problem's input vector: plane (sign s, digit j) of pass t
// at [(t 2 + s) kS + j][nstr][row_ld] holds digit j (0 = most significant) of
// +-round(c 2^38 / dscale); pass 1 (only without spin-flip symmetry) is C^T.
// Clears the problem's S as well.
__device__ __forceinline__ void quantise_one(const SigmaProb &p, long long I, double dscale, __half *__restrict__ Q,
                                             long long *__restrict__ S) {
    const int nstr = p.nstr, ldq = row_ld(nstr);
    const int ka = (int)(I / nstr), kb = (int)(I % nstr);
    const double *c = p.cbase + (p.cslot ? (long long)*p.cslot : 0ll) * p.stride;
    // 2^38 / dscale: exact on the integer pipe while both are normal powers of two
    const int f = dexp_field(dscale);
    const double sc = f > 38 && f < 2047 ? __hiloint2double((2046 + 38 - f) << 20, 0) : 274877906944.0 / dscale;
    const size_t plane = (size_t)nstr * ldq;
    unsigned short *out = reinterpret_cast<unsigned short *>(Q) + p.qoff + (size_t)ka * ldq + kb;
    for (int t = 0; t < (p.sym ? 1 : 2); t++) {
        const long long x = __double2ll_rn((t ? c[(long long)kb * nstr + ka] : c[I]) * sc);
        const unsigned long long u = (unsigned long long)(x + kDigitBias), v = (unsigned long long)(-x + kDigitBias);
#pragma unroll
        for (int j = 0; j < kS; j++) {
            const uint32_t h = j == 0 ? digit_pair_f16((uint32_t)(u >> 32), (uint32_t)(v >> 32), 0)
                                      : digit_pair_f16((uint32_t)u, (uint32_t)v, kS - 1 - j);
            out[(size_t)j * plane] = (unsigned short)(h & 0xFFFF);
            out[(size_t)(kS + j) * plane] = (unsigned short)(h >> 16);
        }
        out += 2 * kS * plane;
        S[p.doff + (t ? p.ndet : 0) + I] = 0;
    }
}

__global__ void __launch_bounds__(kGatherChunk)
oz_quantise_kernel(const SigmaProb *__restrict__ probs, const WorkItem *__restrict__ items, __half *__restrict__ Q,
                   long long *__restrict__ S) {
    const WorkItem it = items[blockIdx.x];
    const SigmaProb &p = probs[it.prob];
    if (p.active && !*p.active) return;
    const long long I = it.start + threadIdx.x;
    if (I < p.ndet) quantise_one(p, I, p.dscale, Q, S);
}

// sigma = S + S^T (spin-flip-symmetric) or S(C) + S(C^T)^T, converted from the
// integer units; one 32 x 32 tile of strings and its transpose per block.
__global__ void __launch_bounds__(256)
oz_finish_kernel(const SigmaProb *__restrict__ probs, const WorkItem *__restrict__ items, const long long *__restrict__ S) {
    const WorkItem it = items[blockIdx.x];
    const SigmaProb &p = probs[it.prob];
    if (p.active && !*p.active) return;
    __shared__ double sh[2][32][33];
    const int n = p.nstr, r0 = (int)it.start * 32, c0 = it.sub * 32, x = threadIdx.x & 31, y0 = threadIdx.x >> 5;
    const double f = p.Wexp[0] * p.dscale * 0x1p-45;
    const long long *S1 = S + p.doff, *S2 = p.sym ? S1 : S1 + p.ndet;
    double *s = p.sbase + (p.sslot ? (long long)*p.sslot : 0ll) * p.stride;
    for (int y = y0; y < 32; y += 8) {
        const int r = r0 + y, c = c0 + y;   // rows of the tile and of its transpose
        sh[0][y][x] = c < n && r0 + x < n ? (double)S2[(long long)c * n + r0 + x] * f : 0.0;
        sh[1][y][x] = !p.sym && r < n && c0 + x < n ? (double)S2[(long long)r * n + c0 + x] * f : 0.0;
    }
    __syncthreads();
    double v[4], u[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int y = y0 + 8 * k, r = r0 + y, c = c0 + y;
        v[k] = r < n && c0 + x < n ? (double)S1[(long long)r * n + c0 + x] * f + sh[0][x][y] : 0.0;
        u[k] = !p.sym && c < n && r0 + x < n ? (double)S1[(long long)c * n + r0 + x] * f + sh[1][x][y] : 0.0;
    }
    __syncthreads();
    if (p.sym)
#pragma unroll
        for (int k = 0; k < 4; k++) sh[0][y0 + 8 * k][x] = v[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int y = y0 + 8 * k, r = r0 + y, c = c0 + y;
        if (r < n && c0 + x < n) s[(long long)r * n + c0 + x] = v[k];
        if (c < n && r0 + x < n) s[(long long)c * n + r0 + x] = p.sym ? sh[0][x][y] : u[k];
    }
}

// one exponent per problem: max |W| over the contracted pairs <= 2^e (Wexp[0])
__global__ void __launch_bounds__(512) oz_wmax_kernel(const SigmaProb *__restrict__ probs) {
    const SigmaProb &p = probs[blockIdx.x];
    const int np = p.act ? p.npc : p.np, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t *act = p.act;
    __shared__ double red[16];
    double mx = 0.0;
    for (int r = warp; r < np; r += 16)
        for (int c = lane; c < np; c += 32)
            mx = fmax(mx, fabs(p.W[(act ? act[r] : r) * (long long)p.ld + (act ? act[c] : c)]));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 16; w++) mx = fmax(mx, red[w]);
        int e = 0;
        if (mx > 0.0) frexp(mx, &e);          // max = f 2^e, f in [0.5, 1)
        p.Wexp[0] = ldexp(1.0, e);
    }
}

// Sliced image of W, MN-major: for each chunk of w = 48 output pairs (the last
// one narrower, a multiple of 16) [contracted pair b][slice i][output pair of
// the chunk] FP16, zeros beyond npair.  A sectored space packs its active
// pairs only, in compact order.  Group t of 8 output pairs; scale = 2^e > max |W|.
__device__ __forceinline__ void pack_group(const SigmaProb &p, int t, double scale) {
    const int np = p.act ? p.npc : p.np, npad = np_pad(np), n8 = npad / 8;
    const int32_t *act = p.act;
    uint8_t *img = (uint8_t *)const_cast<void *>(p.Woz);
    const int b = t / n8, a0 = t % n8 * 8, c0 = a0 / kNC * kNC, w = min(kNC, npad - c0);
    const int kb = act ? act[b] : b, f = dexp_field(scale);
    float sl[8][kS];
    for (int e = 0; e < 8; e++) {
        const int a = a0 + e;
        const double x = a < np ? p.W[(long long)(act ? act[a] : a) * p.ld + kb] : 0.0;
        if (f > 0 && f < 2047 && dexp_field(x) < 2047) slice5_pow2(x, f - 1023, sl[e]);
        else slice5(x / scale, sl[e]);
    }
    for (int i = 0; i < kS; i++)
        *(uint4 *)(img + (size_t)np * 10 * c0 + ((size_t)b * kS * w + i * w + (a0 - c0)) * 2) =
            make_uint4(pack2(sl[0][i], sl[1][i]), pack2(sl[2][i], sl[3][i]), pack2(sl[4][i], sl[5][i]),
                       pack2(sl[6][i], sl[7][i]));
}

// Blocks (problem, part).
__global__ void __launch_bounds__(256) oz_pack_w_kernel(const SigmaProb *__restrict__ probs) {
    const SigmaProb &p = probs[blockIdx.x];
    const int np = p.act ? p.npc : p.np;
    for (int t = blockIdx.y * 256 + threadIdx.x; t < np * (np_pad(np) / 8); t += gridDim.y * 256) pack_group(p, t, p.Wexp[0]);
}

// Excitation map of a string class: entry of output pair A and string I at
// [A / 4][I][A % 4] (one 8-byte load per thread and four columns), sign << 15 | J
// of E+_A |I> = +-|J>, kNoMap where there is none, beyond np and beyond nstr
// (ldj strings, np_pad(np) pairs).  kMapRows strings, built in shared memory so
// that the table is read and the map written in whole lines (220 strings of 30
// entries: 11.4 us with one thread walking each list).
constexpr int kMapRows = 32;

__device__ __forceinline__ void map_rows(int I0, int nstr, int nexc, int np, int ldj, const int32_t *__restrict__ exc,
                                         uint16_t *__restrict__ jmap, uint16_t (*tile)[kMaxNp + 2]) {
    const int npad = np_pad(np), rows = min(kMapRows, nstr - I0);
    for (int t = threadIdx.x; t < kMapRows * (npad / 2); t += 256)
        *reinterpret_cast<uint32_t *>(&tile[t / (npad / 2)][2 * (t % (npad / 2))]) = kNoMap << 16 | kNoMap;
    __syncthreads();
    for (int t = threadIdx.x; t < rows * nexc; t += 256) {
        const int32_t x = exc[(size_t)I0 * nexc + t];
        tile[t / nexc][exc_pair(x)] = (uint16_t)((uint32_t)exc_J(x) | (uint32_t)(x & 1) << 15);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < kMapRows * (npad / 4); t += 256) {
        const int g = t / kMapRows, i = t % kMapRows;
        const uint32_t *v = reinterpret_cast<const uint32_t *>(&tile[i][4 * g]);
        reinterpret_cast<uint2 *>(jmap)[(size_t)g * ldj + I0 + i] = make_uint2(v[0], v[1]);
    }
}

__global__ void __launch_bounds__(256) oz_map_kernel(int nstr, int nexc, int np, int ldj, const int32_t *__restrict__ exc,
                                                     uint16_t *__restrict__ jmap) {
    __shared__ __align__(8) uint16_t tile[kMapRows][kMaxNp + 2];
    map_rows(blockIdx.x * kMapRows, nstr, nexc, np, ldj, exc, jmap, tile);
}

// maps of the sectored units: their class's map restricted to the active pairs
__global__ void __launch_bounds__(256) oz_compact_maps_kernel(const OzMapDesc *__restrict__ desc, int n) {
    for (int u = blockIdx.x; u < n; u += gridDim.x) {
        const OzMapDesc d = desc[u];
        for (int t = threadIdx.x; t < np_pad(d.npc) / 4 * d.ldj; t += 256) {
            const int g = t / d.ldj, I = t % d.ldj;
            uint32_t v[4];
            for (int k = 0; k < 4; k++) {
                const int A = 4 * g + k < d.npc ? d.act[4 * g + k] : -1;
                v[k] = A >= 0 ? d.map[((size_t)(A >> 2) * d.ldj + I) * 4 + (A & 3)] : kNoMap;
            }
            reinterpret_cast<uint2 *>(d.out)[t] = make_uint2(v[0] | v[1] << 16, v[2] | v[3] << 16);
        }
        // contracted pairs of each string
        for (int I = threadIdx.x; I < d.nstr; I += 256) {
            int k = 0;
            for (int c = 0; c < d.npc; c++)
                k += d.map[((size_t)(d.act[c] >> 2) * d.ldj + I) * 4 + (d.act[c] & 3)] != kNoMap;
            d.kcnt[I] = (uint8_t)k;
        }
    }
}

// A single problem is prepared in two launches around its two maxima: CAS(4e,12o)
// takes 37 us a call (41 us with the plan's arrays copied one by one), 92 us with
// one launch per step (fold, max W, pack, map, max c, scale, quantise: 62 us of
// device time before the contraction).

// Largest |x| of the block's values to *out (as ordered bits; NaN left out).
__device__ __forceinline__ void block_max_bits(long long m, unsigned long long *out) {
    __shared__ long long red[8];
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; w++) m = max(m, red[w]);
        if (m > 0) atomicMax(out, (unsigned long long)m);
    }
}
__device__ __forceinline__ long long number_mag(double x) { return dmag(x) <= 0x7FF0000000000000ll ? dmag(x) : 0ll; }

// smallest power of two > m (1 for 0)
__device__ __forceinline__ double pow2_above(double m) {
    int e = 0;
    if (m > 0.0) frexp(m, &e);   // m = f 2^e, f in [0.5, 1)
    return ldexp(1.0, e);
}

// Blocks [0, nfold): W and max |W| (mx[0]); [nfold, nfold + nabs): max |c|
// (mx[1]); the others: kMapRows strings each of the excitation map.
__global__ void __launch_bounds__(256) oz_prepare_one_kernel(FoldDesc d, int nfold, const double *__restrict__ c, long long n,
                                                             int nabs, unsigned long long *__restrict__ mx, int nstr, int nexc,
                                                             int ldj, const int32_t *__restrict__ exc,
                                                             uint16_t *__restrict__ jmap) {
    __shared__ __align__(8) uint16_t tile[kMapRows][kMaxNp + 2];
    const int np = d.n * (d.n + 1) / 2;
    int blk = blockIdx.x;
    long long m = 0;
    if (blk < nfold) {
        double *kpair = reinterpret_cast<double *>(&tile[0][0]);   // np <= kMaxNp
        for (int A = threadIdx.x; A < np; A += 256) kpair[A] = fold_pair(d, A);
        __syncthreads();
        const double invN = d.nelec > 0 ? 1.0 / (double)d.nelec : 0.0;
        for (int t = blk * 256 + threadIdx.x; t < np * np; t += nfold * 256) {
            const int A = t / np, B = t % np;
            const double w = fold_element(d, kpair, invN, A, B);
            d.W[(long long)A * d.ld + B] = w;
            m = max(m, number_mag(w));
        }
        block_max_bits(m, mx);
    } else if ((blk -= nfold) < nabs) {
        for (long long i = blk * 256ll + threadIdx.x; i < n; i += nabs * 256ll) m = max(m, number_mag(c[i]));
        block_max_bits(m, mx + 1);
    } else {
        map_rows((blk - nabs) * kMapRows, nstr, nexc, np, ldj, exc, jmap, tile);
    }
}

// Blocks [0, nquant): the digit planes of c, the others the image of W, both
// scaled by the maxima.  dscale of a caller's vector: the smallest power of two
// above 2 max|c| with spin-flip symmetry, above max|c| without (two passes, each
// with its own rounding: half the scale keeps their sum below the error of one
// pass over alpha and beta sums; the top digit stays below 65).
__global__ void __launch_bounds__(kGatherChunk)
oz_quantise_pack_one_kernel(SigmaProb *probs, int nquant, const unsigned long long *__restrict__ mx, __half *__restrict__ Q,
                            long long *__restrict__ S) {
    const SigmaProb &p = probs[0];
    const int blk = blockIdx.x;
    if (blk < nquant) {
        const double dscale = pow2_above((p.sym ? 2.0 : 1.0) * __longlong_as_double((long long)mx[1]));
        if (blk == 0 && threadIdx.x == 0) probs[0].dscale = dscale;   // for the finish
        const long long I = (long long)blk * kGatherChunk + threadIdx.x;
        if (I < p.ndet) quantise_one(p, I, dscale, Q, S);
    } else {
        const double scale = pow2_above(__longlong_as_double((long long)mx[0]));
        const int t = (blk - nquant) * kGatherChunk + threadIdx.x;
        if (t == 0) p.Wexp[0] = scale;
        if (t < p.np * (np_pad(p.np) / 8)) pack_group(p, t, scale);
    }
}

int contracted_pairs(const SigmaProb &p) { return p.act ? p.npc : p.np; }

// Buffers for items of at most k contracted pairs per string, nch chunks and
// nstr strings: the accumulator row in shared memory if anything can be had
// with it (its atomics are ~5 times cheaper there than in L2), then two c
// stages before more than two W buffers, then as many W buffers as there are
// chunks (resident for the whole item).
bool choose_geom(int k, int nch, int nstr, OzGeom &g) {
    g.kmax = round_up(k, 16);
    if (g.kmax > kMaxK) return false;
    const int sa = kS * g.kmax * 256, sw = g.kmax * 512;
    for (int row = 1; row >= 0; row--)
        for (int nA = 2; nA >= 1; nA--)
            for (int nW = std::min(kMaxW, std::max(nch, 2)); nW >= (row || nA > 1 ? 2 : 1); nW--)
                if (nA * sa + nW * sw + row * 8 * nstr <= kSmemLimit) {
                    g.nA = nA;
                    g.nW = nW;
                    g.rows = row * nstr;
                    return true;
                }
    return false;
}

}  // namespace

int oz_operand_bytes(int np) { return np * np_pad(np) * 2 * kS + 256; }
int oz_map_ld(int nstr) { return round_up(nstr, kTM); }
size_t oz_map_elems(int np, int nstr) { return (size_t)np_pad(np) * oz_map_ld(nstr); }
long long oz_plane_elems(int nstr, bool sym) { return (sym ? 2ll : 4ll) * kS * nstr * row_ld(nstr); }
bool oz_supported(int np, int nstr, int nexc) { return np <= kMaxNp && nstr <= kMaxStrings && nexc <= kMaxK; }
bool oz_wide(int nexc) { return nexc > kNarrowK; }

int launch_oz_map(ifci_handle_t h, int nstr, int nexc, int np, const int32_t *exc, uint16_t *jmap, cudaStream_t s) {
    const int ldj = oz_map_ld(nstr);
    oz_map_kernel<<<ldj / kMapRows, 256, 0, s>>>(nstr, nexc, np, ldj, exc, jmap);
    IFCI_LAUNCH_CHECK(h);
    return IFCI_OK;
}

int launch_oz_compact_maps(ifci_handle_t h, int n, const OzMapDesc *d_desc, cudaStream_t s) {
    if (n <= 0) return IFCI_OK;
    oz_compact_maps_kernel<<<stride_grid(h->device, n, 8), 256, 0, s>>>(d_desc, n);
    IFCI_LAUNCH_CHECK(h);
    return IFCI_OK;
}

int launch_oz_pack_w(ifci_handle_t h, int nprob, const SigmaProb *d_probs, int max_np, cudaStream_t s) {
    if (nprob <= 0) return IFCI_OK;
    oz_wmax_kernel<<<nprob, 512, 0, s>>>(d_probs);
    IFCI_LAUNCH_CHECK(h);
    // one 8-pair group per thread while there are few problems
    const int parts = (max_np * np_pad(max_np) / 8 + 255) / 256;
    const int room = std::max(1, 16 * device_sm_count(h->device) / nprob);
    oz_pack_w_kernel<<<dim3(nprob, std::max(1, std::min(parts, room))), 256, 0, s>>>(d_probs);
    IFCI_LAUNCH_CHECK(h);
    return IFCI_OK;
}

static int contract_oz(ifci_handle_t h, const SigmaPlan &plan, const SigmaWave &w, __half *Q, long long *S, cudaStream_t s) {
    static SmemOptIn opt_n, opt_w, opt_g;
    for (int wide = 0; wide < 2; wide++) {
        const int i0 = wide ? w.tc0 + w.ntc : w.tc0, ni = wide ? w.nwide : w.ntc;
        if (ni == 0) continue;
        int k = 0, nch = 0, nstr = 0;
        for (int i = w.prob0; i < w.prob0 + w.nprob; i++) {
            const SigmaProb &p = plan.probs[i];
            if (oz_wide(p.nexc) != (wide != 0)) continue;
            k = std::max(k, std::min(p.nexc, contracted_pairs(p)));
            nch = std::max(nch, (np_pad(contracted_pairs(p)) + kNC - 1) / kNC);
            nstr = std::max(nstr, p.nstr);
        }
        OzGeom g{};
        g.m8 = 1u << 8;
        g.m16 = 1u << 16;
        g.m24 = 1u << 24;
        if (!choose_geom(k, nch, nstr, g) || (!wide && !g.rows)) return set_error(h, IFCI_ERR_UNSUPPORTED, "FP64E: %d excitations per string", k);
        const size_t smem = 1024 + (size_t)g.nA * kS * g.kmax * 256 + (size_t)g.nW * g.kmax * 512 + (size_t)g.rows * 8;
        const int grid = std::min(ni, device_sm_count(h->device));
        ProfScope ps(h, s, PK_CONTRACT_HI);
        auto launch = [&](auto kernel, SmemOptIn &opt) {
            const cudaError_t e = ensure_smem(opt, h->device, kernel, (int)smem);
            if (e == cudaSuccess)
                kernel<<<grid, kOzThreads, smem, s>>>(plan.d_probs, plan.d_tctiles + i0, ni, Q, S, h->d_err, g);
            return e;
        };
        IFCI_CUDA_TRY(h, !wide ? launch(oz_sigma_kernel<false, true>, opt_n)
                         : g.rows ? launch(oz_sigma_kernel<true, true>, opt_w) : launch(oz_sigma_kernel<true, false>, opt_g));
        IFCI_LAUNCH_CHECK(h);
    }
    ProfScope ps(h, s, PK_SCATTER);
    oz_finish_kernel<<<w.nfin, 256, 0, s>>>(plan.d_probs, plan.d_tiles + w.tile0, S);
    IFCI_LAUNCH_CHECK(h);
    return IFCI_OK;
}

int run_sigma_oz(ifci_handle_t h, const SigmaPlan &plan, const SigmaWave &w, void *D, void *G, cudaStream_t s) {
    if (!h->d_err) return set_error(h, IFCI_ERR_INVALID_ARG, "FP64E: no error flag");
    auto *Q = static_cast<__half *>(D);
    auto *S = static_cast<long long *>(G);
    {
        ProfScope ps(h, s, PK_GATHER);
        oz_quantise_kernel<<<w.nitem, kGatherChunk, 0, s>>>(plan.d_probs, plan.d_items + w.item0, Q, S);
        IFCI_LAUNCH_CHECK(h);
    }
    return contract_oz(h, plan, w, Q, S, s);
}

int run_sigma_oz_one(ifci_handle_t h, const SigmaPlan &plan, const FoldDesc &f, const double *c, uint16_t *jmap,
                     unsigned long long *mx, void *D, void *G, cudaStream_t s) {
    if (!h->d_err) return set_error(h, IFCI_ERR_INVALID_ARG, "FP64E: no error flag");
    const SigmaProb &p = plan.probs[0];
    auto *Q = static_cast<__half *>(D);
    auto *S = static_cast<long long *>(G);
    {
        ProfScope ps(h, s, PK_GATHER);
        IFCI_CUDA_TRY(h, cudaMemsetAsync(mx, 0, 2 * sizeof(*mx), s));
        const int nfold = (p.np * p.np + 511) / 512;   // two elements a thread
        const int nabs = (int)std::min<long long>(2 * device_sm_count(h->device), (p.ndet + 511) / 512);
        oz_prepare_one_kernel<<<nfold + nabs + p.ldj / kMapRows, 256, 0, s>>>(f, nfold, c, p.ndet, nabs, mx, p.nstr, p.nexc,
                                                                              p.ldj, p.exc, jmap);
        IFCI_LAUNCH_CHECK(h);
        const int nquant = (int)((p.ndet + kGatherChunk - 1) / kGatherChunk);
        const int npack = (p.np * (np_pad(p.np) / 8) + kGatherChunk - 1) / kGatherChunk;
        oz_quantise_pack_one_kernel<<<nquant + npack, kGatherChunk, 0, s>>>(plan.d_probs, nquant, mx, Q, S);
        IFCI_LAUNCH_CHECK(h);
    }
    return contract_oz(h, plan, plan.waves[0], Q, S, s);
}

}  // namespace ifci

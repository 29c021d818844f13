// Split-precision TSMTTSM on the 5th-generation tensor cores (tcgen05).
//
// G = X^T Y for real tall & skinny X (K x P) and Y (K x Q) in binary64 --
// complex A^T B / A^H B are the real product of the interleaved (re, im)
// columns, recombined at the end -- computed with error-free splitting after
// Ozaki, Ogita, Oishi, Rump (Numer. Algorithms 59, 2012), shown here for
// S = 6 slices (the kernel is templated on S in [4, 6]):
//
//   x = 2^e * sum_s alpha_s * 2^(-7 - 8s),  s = 0..5, alpha_s integer, |alpha_s| <= 128
//
// where e is a running maximum exponent of x's column (|x| < 2^e), so every
// alpha_s is exact in fp16 (11-bit significand).  Then, per accumulation tile
// of at most 256 rows in which no column exponent changes,
//
//   sum_k x_kp y_kq = 2^(e_p + e_q - 14) * sum_d 2^(-8d) P_d[p][q],
//   P_d = sum_k sum_{s+t=d} alpha_s beta_t,  d = 0..5 (pairs with s+t > 5 dropped),
//
// and each P_d is a sum of at most 6 * 256 products of magnitude <= 2^14:
// exact in FP32 for d <= 3 (<= 2^24), and within a few FP32 units for
// d = 4, 5 whose weight is below 2^-46.  (Steps with a value above 2^e, whose
// top digit may reach 255, shorten the tile: such a step costs 3 of a
// tile's 32, the others 2, which keeps the same bounds.)  The tensor cores
// form all P_d in tensor memory; the epilogue converts them to one exact
// 64-bit integer W = sum_d P_d 2^(8(5-d)) per entry and sums W exactly in
// 64-bit integers across tiles, moving the sum to binary64 only when an
// exponent of its row or column grows, when it would overflow, and at the
// end.  Partials of all CTAs are reduced in a fixed order.
//
// CTA organisation (one or two CTAs per SM, as tensor memory and shared
// memory allow; each persistent over a contiguous K range and a chunk of Y's
// columns):
//   converter warps  take units (16 columns of a 16-row step) in turn, write
//                    the S fp16 slices, 16 bytes per slice and lane, into a
//                    ring of digit stages in the canonical K-major
//                    core-matrix layout of the MMA operands, and pass the
//                    columns' running exponents from step to step.  As many
//                    warps as the register file holds: a unit is a chain of
//                    a global load, the exponent, about 200 integer
//                    instructions, a proxy fence and an arrival, and only
//                    other warps hide its latency;
//   MMA warp         allocates tensor memory, issues tcgen05.mma and decides
//                    the tile boundaries (a step at which an exponent grew,
//                    or the tile's budget); it copies the tile's exponents
//                    for the epilogue;
//   epilogue warps   8 (two per tensor-memory lane quarter, each on half
//                    of the columns) or, with two CTAs per SM, 4:
//                    drain tensor memory after each tile (tcgen05.ld) and
//                    accumulate.
// MMA operand A (M = 128 rows): X slices, 4, 2 or 1 to a 128-row block
// (P <= 32, 64, 128).  Operand B (N rows): the six Y slices stacked, Qp rows
// each.  Accumulator column block j holds the slice pairs whose weight index
// is d = j in the rows of a block's first slice, d = j + h in those of its
// h-th.
//
// What bounds it (complex 64 x 64, S = 6, ncu): the integer pipe is 54 % busy
// and 58 % of the issue slots are taken: 12 units a step at about 83 cycles of
// the integer pipe each are 1000 cycles of the 2450 a step takes, against
// 1260 for the step's MMAs and operand reads; the rest is the chain above
// (no loads, no digits and no drain leave 700 cycles of waits) and the drain
// (460).  Measured before and after this organisation (one warp per 16
// columns in lock step with the MMA, exponents that ended a tile at every
// new maximum; 2^22 rows): complex 64 x 64 6.07 / 4.65 ms (uniform
// data) and 11.8 / 5.4 ms (normal data); real 24 x 40, S = 5, 10^6 rows 0.54 /
// 0.32 ms.
//
// Every wait on an mbarrier is bounded by a clock budget; on expiry the
// kernel records an error word, stops issuing work, drains its own MMAs,
// frees tensor memory and exits; the combine kernel then writes NaN.
#include <algorithm>
#include <cstdint>
#include <cstdio>

#include <cuda_fp16.h>

#include <type_traits>

#include "tsm_internal.h"
#include "tsm_split.h"

namespace tsm {
namespace split {

constexpr int KSTEP = 16;           // rows per MMA (16-bit inputs: K = 16)
constexpr int TILE_BUDGET = 32;     // per accumulation tile: a step costs 2, one with values above 2^e costs 3
constexpr int SOFT_STEPS = 4;       // steps in which a column may exceed 2^e before e is raised
constexpr int PRE_STEPS = 8;        // steps scanned for the first exponents (128 rows)
constexpr int NSLICE_MAX = 6;       // 8-bit slices per input: S in [4, 6], a template parameter
constexpr int NDIG_MAX = 12;        // digit stages (converters -> MMA): as many as fit, up to this
constexpr int MAX_GROUPS = 16;      // column groups (converter units per step) of 16: P + Q <= 256
constexpr int MAX_RANGES = 2;       // exponent ranges of a CTA that start from scanned exponents
constexpr int NEXP = 4;             // exponent snapshot ring (MMA warp -> epilogue)
constexpr int NEPI_MAX = 8;         // epilogue warps: 8 (two per lane quarter) or 4
constexpr int TMEM_COLS_MAX = 512;
// Words of the stream workspace's ticket array used here: the status that
// tsm_split_status reads, the error word of the launch in progress (zero
// between launches) and the combine kernel's ticket.
constexpr int kStatusWord = 32, kErrWord = 33, kTicketWord = 34;
constexpr int E_NONE = -4000;       // running exponent before any value
constexpr long long kDefaultTimeout = 4000000000ll;  // SM cycles (~2 s)
// Threads per SM: 64 registers each fill the register file.
constexpr int kThreadsPerSM = 1024;

struct Params {
    const double* X;
    int64_t ldx;  // doubles
    const double* Y;
    int64_t ldy;
    int P, Q;     // real column counts of X and Y
    int64_t K;
    int n_kr, n_qc;
    int q0[2], qw[2];
    int64_t steps_per_kr;
    int64_t steps_per_range;  // the column exponents restart after so many steps
    int stack;    // slices of X per 128-row operand block: 4 (P <= 32), 2 (P <= 64) or 1
    int Qp;       // padded chunk width (multiple of 16)
    int ncg;      // column groups of 16: converter units per step
    int nconv;    // converter warps; the MMA warp and the epilogue warps follow
    int nepi;     // epilogue warps: 8 (two per lane quarter, half the columns each) or 4
    int tmem_cols;  // tensor-memory columns allocated: a power of two >= S * Qp
    int smem_budget;  // bytes of shared memory the layout may use (several CTAs per SM share 228 KB)
    int smem_floor;   // minimum dynamic shared memory: keeps more CTAs than planned off an SM
    double* ws;     // [n_kr][P][Q]
    double* flush;  // [CTA][Qp][128]: binary64 totals of the epilogue lanes
    int* err;
    long long timeout;
};

// ------------------------------------------------------------ PTX helpers

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: false if the phase did not complete within `timeout` SM
// cycles (the error word is then set to `code`), or if another warp raised
// the CTA's abort flag meanwhile (`abort_flag` may be null: wait regardless).
// mbarrier.try_wait itself suspends the warp until the phase completes or a
// hardware time limit passes, so the loop wakes as soon as the barrier
// flips; only waits longer than 2^16 cycles (never in steady state) add a
// sleep to leave issue slots to the working warps.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, long long timeout, int* err,
                                          int code, const volatile int* abort_flag) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if (abort_flag && *abort_flag) return false;
        const long long dt = clock64() - t0;
        if (dt > timeout) {
            atomicCAS(err, 0, code);
            return false;
        }
        if (dt > 65536) __nanosleep(256);
    }
}
// Waits until the shared counter at `seq` reaches `s`: bounded, warp-uniform.
__device__ __forceinline__ bool seq_wait(uint32_t seq, int s, long long timeout, int* err, int code,
                                         const volatile int* abort_flag) {
    auto at = [&]() {
        int v;
        asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(seq) : "memory");
        return v == s;
    };
    if (__all_sync(0xffffffffu, at())) return true;
    const long long t0 = clock64();
    bool ok = true;
    while (!at()) {
        if (*abort_flag) {
            ok = false;
            break;
        }
        if (clock64() - t0 > timeout) {
            atomicCAS(err, 0, code);
            ok = false;
            break;
        }
    }
    return __all_sync(0xffffffffu, ok);
}
// The same wait taken by every lane of a warp: warp-uniform result.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, long long timeout, int* err, int code,
                                          const volatile int* abort_flag) {
    const bool ok = mbar_try_wait(bar, parity);
    if (__all_sync(0xffffffffu, ok)) return true;
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, timeout, err, code, abort_flag));
}
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared-memory matrix descriptor, no swizzle, K-major canonical layout:
// core matrices of 8 rows x 16 bytes (128 contiguous bytes); 128 is the byte
// distance between core matrices adjacent along K, 256 between those
// adjacent along M/N.  Bits 46-48 hold the fixed value 0b001.  The high word
// is the same for every operand.
constexpr uint32_t kDescHi = (256u >> 4) | (1u << 14);
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return ((addr >> 4) & 0x3FFFu) | ((128u >> 4) << 16); }
// Instruction descriptor of kind::f16: D = F32, A = B = F16 (format code 0),
// both K-major, M = 128, N as given.
__device__ __forceinline__ uint32_t instr_desc(int n) {
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
// (`lead`: one lane of the warp; a predicate instead of a branch, so that the
// control flow stays uniform and the operands need no per-MMA move)
__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc,
                                         uint32_t accumulate, uint32_t lead) {
    asm volatile(
        "{\n.reg .pred p, q;\n.reg .b64 a, b;\nsetp.ne.b32 p, %5, 0;\nsetp.ne.b32 q, %6, 0;\n"
        "mov.b64 a, {%1, %3};\nmov.b64 b, {%2, %3};\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, p;\n}\n" ::"r"(d_tmem),
        "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate), "r"(lead));
}
__device__ __forceinline__ void mma_commit(uint32_t bar, uint32_t lead) {
    asm volatile(
        "{\n.reg .pred q;\nsetp.ne.b32 q, %1, 0;\n"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar),
        "r"(lead)
        : "memory");
}
// The MMAs of one step: for every 128-row block of X's slices the Y slices
// t with s + t < S, as many per MMA as fit in N <= 256.  All shapes are
// constants, so an MMA costs its issue and no descriptor arithmetic.
// `fresh`: the step starts its tile, whose accumulators row block 0 covers.
template <int S, int STACK, int QP>
__device__ __forceinline__ void issue_step(uint32_t tm, uint32_t a0, uint32_t b0, bool fresh, uint32_t lead) {
    constexpr int MAXS = 256 / QP, NRB = (S + STACK - 1) / STACK;
#pragma unroll
    for (int rb = 0; rb < NRB; ++rb)
#pragma unroll
        for (int t0 = 0; t0 < S - rb * STACK; t0 += MAXS) {
            const int cnt = S - rb * STACK - t0 < MAXS ? S - rb * STACK - t0 : MAXS;
            mma_f16(tm + (uint32_t)((rb * STACK + t0) * QP), a0 + (uint32_t)(rb * 256), b0 + (uint32_t)(t0 * QP * 2),
                    kDescHi, instr_desc(cnt * QP), rb > 0 || !fresh, lead);
        }
}
template <int S, int STACK>
__device__ __forceinline__ void issue_step_qp(int Qp, uint32_t tm, uint32_t a0, uint32_t b0, bool fresh,
                                              uint32_t lead) {
    switch (Qp) {
        case 16: issue_step<S, STACK, 16>(tm, a0, b0, fresh, lead); break;
        case 32: issue_step<S, STACK, 32>(tm, a0, b0, fresh, lead); break;
        case 48: issue_step<S, STACK, 48>(tm, a0, b0, fresh, lead); break;
        case 64: issue_step<S, STACK, 64>(tm, a0, b0, fresh, lead); break;
        case 80: issue_step<S, STACK, 80>(tm, a0, b0, fresh, lead); break;
        case 96:
            if (S <= 5) issue_step<S, STACK, 96>(tm, a0, b0, fresh, lead);
            break;
        case 112:
            if (S <= 4) issue_step<S, STACK, 112>(tm, a0, b0, fresh, lead);
            break;
        default:
            if (S <= 4) issue_step<S, STACK, 128>(tm, a0, b0, fresh, lead);
            break;
    }
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t* v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// One lane of a converged warp (the same lane every time: the lowest).
__device__ __forceinline__ bool elect_one() {
    uint32_t pred = 0;
    asm volatile("{\n.reg .pred P;\nelect.sync _|P, 0xffffffff;\nselp.u32 %0, 1, 0, P;\n}\n" : "=r"(pred));
    return pred != 0;
}

// ------------------------------------------------------------ shared layout

struct Layout {
    int nrb;            // 128-row blocks of operand A per step
    int ndig;           // digit stages
    int ne;             // exponent entries: P + Qp
    uint32_t a_bytes;   // operand A bytes per step
    uint32_t b_bytes;   // operand B bytes per step
    uint32_t stage;     // digit stage bytes (1024-aligned)
    uint32_t dig_off;   // offset of digit stage 0
    uint32_t acc_off;   // 64-bit integer accumulators [Qp][128]
    uint32_t exps_off;  // per-stage column exponents [ndig][ne]
    uint32_t snap_off;  // per-tile exponent snapshots [NEXP][ne]
    uint32_t col_off;   // column exponents [ne], overflow counts [ne], the ranges' first exponents [MAX_RANGES][ne]
    uint32_t misc_off;  // barriers, flags, tmem slot
    uint32_t total;
};

constexpr uint32_t kSmemBudget = 227u * 1024u;  // one CTA per SM
constexpr uint32_t kSmemPerSM = 228u * 1024u;   // shared by the CTAs of an SM, 1 KB reserved per CTA
constexpr uint32_t kMiscBytes = 512u;

__host__ __device__ inline Layout make_layout(int P, int Qp, int stack, uint32_t budget, uint32_t floor_bytes,
                                              int S) {
    Layout L;
    L.nrb = (S + stack - 1) / stack;
    L.ne = P + Qp;
    L.a_bytes = (uint32_t)L.nrb * 4096u;
    L.b_bytes = (uint32_t)S * Qp * 32u;
    L.stage = ((L.a_bytes + L.b_bytes) + 1023u) & ~1023u;
    const uint32_t acc = (uint32_t)Qp * 128u * 8u;
    const uint32_t exps = (uint32_t)L.ne * 4u;
    const uint32_t fixed = acc + (NEXP + 2 + MAX_RANGES) * exps + kMiscBytes + 256u;  // + alignment slack
    int ndig = budget > fixed ? (int)((budget - fixed) / (L.stage + exps)) : 0;
    if (ndig > NDIG_MAX) ndig = NDIG_MAX;
    L.ndig = ndig;  // the host rejects fewer than 2
    L.dig_off = 0;
    L.acc_off = L.dig_off + (uint32_t)ndig * L.stage;
    L.exps_off = L.acc_off + acc;
    L.snap_off = L.exps_off + (uint32_t)ndig * exps;
    L.col_off = L.snap_off + NEXP * exps;
    L.misc_off = (L.col_off + (2 + MAX_RANGES) * exps + 127u) & ~127u;
    L.total = L.misc_off + kMiscBytes;
    if (L.total < floor_bytes) L.total = floor_bytes;  // no more CTAs per SM than tensor memory was split for
    return L;
}

// misc area: byte offsets of the barriers and flags
enum {
    M_DIG_FULL = 0,     // NDIG_MAX x 8
    M_DIG_EMPTY = 96,   // NDIG_MAX x 8
    M_EXP_EMPTY = 192,  // NEXP x 8
    M_TILE_FULL = 224,
    M_TMEM_EMPTY = 232,
    M_MMA_DONE = 240,
    M_TMEM_SLOT = 248,
    M_SOFT = 256,       // NDIG_MAX ints: last step that held values above its column's 2^e
    M_CHG = 304,        // NDIG_MAX ints: last step at which a column exponent grew
    M_SEQ = 352,        // MAX_GROUPS ints: step whose exponents are next, per column group
    M_ABORT = 416,
    M_TILE_INFO = 420,  // slot | last << 8 | empty << 9 | exponents changed << 10
};
static_assert(M_SEQ + 4 * MAX_GROUPS <= M_ABORT && M_TILE_INFO + 4 <= (int)kMiscBytes, "misc area");

// ------------------------------------------------------------ digit maths

// With 4 slices, whose results are good to about 1e-9, digits are truncated
// and the exponents are the plain running maxima of their range: any other
// choice moves the results by as much as their error.  With 5 and 6 slices
// digits are rounded, the exponents start from a scan of the range's first
// rows (at most a bit above the first step's), and a column may exceed its
// 2^e a few times; the error against 64 bits over 60 shapes of 10^3 .. 6 10^4
// rows, eight inputs each, is 0.78 of that of truncated digits and running
// maxima in the geometric mean, 1.05 at most.
template <int S>
constexpr bool plain_digits() {
    return S == 4;
}

// |x| as a fixed-point integer with 8S - 1 bits below 2^e (rounded to
// nearest, or truncated: plain_digits), plus the S - 1 low bytes biased by 0x80 so that they read back as
// balanced digits: returns Y = X + 0x80...80 where X = round(|x| 2^(8S-1-e)).
// The S base-256 digits of X = sum_s d_s 2^(8(S-1-s)) are d_0 = byte S-1 of Y,
// in [0, 128] for |x| < 2^e and below 256 for a value that exceeds 2^e by
// less than a bit, and d_s = byte (S-1-s) of Y - 128 in [-128, 127] for
// s >= 1.  The rounding bit is added with the bias, at twice the scale.
// Subnormals are exact (no implicit bit); values below the column's range
// give 0 (the shift is clamped to 63).
template <int S>
constexpr unsigned long long digit_bias() {  // 0x80...80; twice that, and the rounding bit, where digits are rounded
    return ((1ull << (8 * (S - 1))) - 1) / 255 * (plain_digits<S>() ? 0x80 : 0x100) + (plain_digits<S>() ? 0 : 1);
}
// the shift drops one bit fewer than the digits keep where they are rounded
template <int S>
constexpr int digit_shift() {
    return (plain_digits<S>() ? 1076 : 1075) - 8 * S;
}
template <int S>
__device__ __forceinline__ unsigned long long fixed_digits(double x, int e) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const uint32_t hi = (uint32_t)(bits >> 32);
    const int ef = (int)((hi >> 20) & 0x7FFu);
    const uint32_t mhi = (hi & 0xFFFFFu) | (ef ? 0x100000u : 0u);
    const unsigned long long mant = ((unsigned long long)mhi << 32) | (uint32_t)bits;
    const int sh = min(e + digit_shift<S>() - max(ef, 1), 63);
    const unsigned long long y = (mant >> sh) + digit_bias<S>();
    return plain_digits<S>() ? y : y >> 1;
}

// fixed_digits for columns whose running exponent e exceeds -960, with
// Eb = ((e + digit_shift) << 20) + 0xFFFFF precomputed per column: the shift
// e + digit_shift - ef is then one subtraction of the magnitude's high word and
// one shift (the low 20 bits never borrow).  The implicit bit is set
// unconditionally, which changes nothing here, since a zero or subnormal x
// (exponent field 0) then shifts by at least 63 and gives 0, as its exact
// value (|x| < 2^-1022, so |x| 2^(8S-1-e) < 2^-15) does; PTX shifts clamp
// amounts above 63 to a result of 0.
template <int S>
__device__ __forceinline__ unsigned long long fixed_digits_fast(double x, uint32_t Eb) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const uint32_t hi = (uint32_t)(bits >> 32);
    const uint32_t sh = (Eb - (hi & 0x7FFFFFFFu)) >> 20;
    const unsigned long long mant = ((unsigned long long)((hi & 0xFFFFFu) | 0x100000u) << 32) | (uint32_t)bits;
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(mant), "r"(sh));
    r += digit_bias<S>();
    return plain_digits<S>() ? r : r >> 1;
}

// The S fp16 slices of two values a (row r) and b (row r + 1) of one
// column, packed per slice as (a, b) in one 32-bit word, sign applied.  A
// digit byte placed under the fp16 exponent of 1024 (0x64XX) is 1024 + byte
// exactly.  Byte permutes gather the digit bytes of both values two slices at
// a time and place them under 0x64; one packed fused multiply-add then forms
// sign * (1024 + byte) - sign * bias, bias = 1024 for the top digit and 1152
// (1024 + 128) for the balanced low digits: exact, since every result is a
// small integer.  Slice s is byte S - 1 - s of Y.  The integer pipe (64
// lanes a cycle) bounds the converters, so the signed biases come from two
// packed multiplies of the signs, on the other pipe.
// FAST: `eb` is the Eb of fixed_digits_fast instead of the exponent.
template <int S, bool FAST>
__device__ __forceinline__ void split_pair(double xa, double xb, int eb, uint32_t* w) {
    const unsigned long long ya = FAST ? fixed_digits_fast<S>(xa, (uint32_t)eb) : fixed_digits<S>(xa, eb);
    const unsigned long long yb = FAST ? fixed_digits_fast<S>(xb, (uint32_t)eb) : fixed_digits<S>(xb, eb);
    const uint32_t alo = (uint32_t)ya, ahi = (uint32_t)(ya >> 32);
    const uint32_t blo = (uint32_t)yb, bhi = (uint32_t)(yb >> 32);
    const uint32_t k64 = 0x64646464u;
    // high halves of a and b: their signs in bits 15 and 31
    const uint32_t top = __byte_perm((uint32_t)__double2hiint(xa), (uint32_t)__double2hiint(xb), 0x7632);
    const uint32_t mulw = (top & 0x80008000u) | 0x3C003C00u;  // (+-1.0, +-1.0)
    const __half2 mul = *reinterpret_cast<const __half2*>(&mulw);
    const __half2 c_top = __hmul2(mul, __half2half2(__ushort_as_half(0xE400)));  // -1024 * sign
    const __half2 c_low = __hmul2(mul, __half2half2(__ushort_as_half(0xE480)));  // -1152 * sign
    // [b5 a5 b4 a4], [b3 a3 b2 a2], [b1 a1 b0 a0] (byte n of Y written an, bn)
    const uint32_t m45 = __byte_perm(ahi, bhi, 0x5140);
    const uint32_t m23 = __byte_perm(alo, blo, 0x7362);
    const uint32_t m01 = __byte_perm(alo, blo, 0x5140);
    auto fin = [&](uint32_t pair, uint32_t sel, __half2 add) {
        uint32_t u = __byte_perm(pair, k64, sel);  // [0x64 b 0x64 a]
        __half2 h = __hfma2(*reinterpret_cast<__half2*>(&u), mul, add);
        return *reinterpret_cast<uint32_t*>(&h);
    };
#pragma unroll
    for (int sl = 0; sl < S; ++sl) {
        const int y = S - 1 - sl;  // byte of Y
        const uint32_t pair = y >= 4 ? m45 : (y >= 2 ? m23 : m01);
        w[sl] = fin(pair, (y & 1) ? 0x4342u : 0x4140u, sl == 0 ? c_top : c_low);
    }
}

// W = sum_d P_d 2^(8(S-1-d)) for accumulator entry qq of the S blocks v[j]
// (tensor-memory words, FP32 integers): block j holds weight d = j + H (rows
// of the H-th stacked slice; weights from S on are dropped).  The terms
// shifted by 32 or more bits (P_0 2^8 + P_1 for S = 6, P_0 for S = 5) are
// summed in 32 bits (|P_0| < 2^22.9, |P_1| < 2^24), the rest are exact 64-bit
// multiply-adds.
template <int H, int S>
__device__ __forceinline__ long long combine_w(const uint32_t (&v)[S][4], int qq) {
    int pd[S];
#pragma unroll
    for (int d = 0; d < S; ++d) pd[d] = d >= H ? __float2int_rn(__uint_as_float(v[d - H][qq])) : 0;
    long long lo = 0;
    int hi = 0;
#pragma unroll
    for (int d = 0; d < S; ++d) {
        const int sh = 8 * (S - 1 - d);
        if (sh >= 32)
            hi += pd[d] * (1 << (sh - 32));
        else
            lo += (long long)pd[d] * (1ll << sh);
    }
    return (long long)((unsigned long long)lo + ((unsigned long long)(unsigned int)hi << 32));
}

// Exponent from the largest magnitude high word of a column: |x| < 2^e for
// every x of the column (zero and subnormal columns give the subnormal bound).
__device__ __forceinline__ int exp_from_hi(uint32_t hmax) {
    const int ef = (int)(hmax >> 20);
    return (ef > 0 ? ef : 1) - 1022;
}

// Byte offset of element (row r, k-group g) inside a K-major operand block
// (core matrices of 8 rows x 16 bytes; LBO = 128, SBO = 256).
__device__ __forceinline__ uint32_t kmajor_off(int r, int g) {
    return (uint32_t)((r >> 3) * 256 + g * 128 + (r & 7) * 16);
}

// ------------------------------------------------------------ the kernel

template <int S>
__global__ void __launch_bounds__(kThreadsPerSM, 1) k_split(const Params prm) {
    constexpr int R = 8;  // rows of a converter unit
    extern __shared__ __align__(1024) unsigned char smem[];
    const int P = prm.P;
    const int kr = blockIdx.x / prm.n_qc, qc = blockIdx.x - kr * prm.n_qc;
    // (selects, not an indexed load: indexing the parameter arrays would
    // copy the whole parameter block to local memory)
    const int q0 = qc ? prm.q0[1] : prm.q0[0];
    const int Qw = qc ? prm.qw[1] : prm.qw[0];
    const int Qp = prm.Qp;
    const int64_t Ktot = prm.K;
    const int stack = prm.stack, Pp = 128 / stack;  // slices per 128-row block, rows of each
    const Layout L = make_layout(P, Qp, stack, (uint32_t)prm.smem_budget, (uint32_t)prm.smem_floor, S);
    const int NE = L.ne, ndig = L.ndig;
    unsigned char* dig = smem + L.dig_off;
    long long* iacc = reinterpret_cast<long long*>(smem + L.acc_off);
    int* exps = reinterpret_cast<int*>(smem + L.exps_off);
    int* snap = reinterpret_cast<int*>(smem + L.snap_off);
    int* col_e = reinterpret_cast<int*>(smem + L.col_off);
    int* col_soft = col_e + NE;
    int* col_e0 = col_soft + NE;
    unsigned char* misc = smem + L.misc_off;
    const uint32_t misc_a = smem_addr(misc);
    auto bar = [&](int off) { return misc_a + (uint32_t)off; };
    volatile int* soft_step = reinterpret_cast<volatile int*>(misc + M_SOFT);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + M_ABORT);
    volatile int* chg_step = reinterpret_cast<volatile int*>(misc + M_CHG);
    volatile int* tile_info = reinterpret_cast<volatile int*>(misc + M_TILE_INFO);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long tmo = prm.timeout;
    const int ncg = prm.ncg;
    const int NCONV_WARPS = prm.nconv;
    const int MMA_WARP = NCONV_WARPS;
    const int NTHREADS = blockDim.x;

    // K range of this CTA, in 16-row steps
    const int64_t steps_total = (Ktot + KSTEP - 1) / KSTEP;
    const int64_t s_begin = (int64_t)kr * prm.steps_per_kr;
    int64_t s_end = s_begin + prm.steps_per_kr;
    if (s_end > steps_total) s_end = steps_total;
    const int nsteps = s_end > s_begin ? (int)(s_end - s_begin) : 0;  // (2^31 steps a CTA are 40 TB of a column)

    // ---- set-up: accumulators and exponent records to zero; barriers.  The
    // operand stages stay as they are: rows past P and columns past Qw only
    // reach accumulator entries that nothing reads.
    for (uint32_t i = L.acc_off + threadIdx.x * 16u; i < L.misc_off + kMiscBytes; i += NTHREADS * 16u)
        *reinterpret_cast<uint4*>(smem + i) = make_uint4(0, 0, 0, 0);
    __syncthreads();
    for (int i = threadIdx.x; i < NE; i += NTHREADS) {
        col_e[i] = E_NONE;
        for (int j = 0; j < MAX_RANGES; ++j) col_e0[j * NE + i] = E_NONE;
    }
    if (threadIdx.x == 0) {
        for (int i = 0; i < ndig; ++i) {
            mbar_init(bar(M_DIG_FULL + 8 * i), ncg);
            mbar_init(bar(M_DIG_EMPTY + 8 * i), 1);
            soft_step[i] = chg_step[i] = -1;
        }
        for (int i = 0; i < NEXP; ++i) mbar_init(bar(M_EXP_EMPTY + 8 * i), prm.nepi);
        mbar_init(bar(M_TILE_FULL), 2);  // the MMAs' commit and the issuer's tile record
        mbar_init(bar(M_TMEM_EMPTY), prm.nepi);
        mbar_init(bar(M_MMA_DONE), 1);
        fence_mbar_init();
    }
    if (warp == MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         bar(M_TMEM_SLOT)),
                     "r"(prm.tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(misc + M_TMEM_SLOT);

    if (warp < NCONV_WARPS) {
        // ================================================= converters
        // Unit (s, cg) is step s of column slots 16 cg .. 16 cg + 15; the
        // warps take the units of the step order in turn.  Lane l holds
        // rows 8 (l / 16) .. + 7 of slot 16 cg + l % 16, whose 8 digits of
        // one slice are the 16 contiguous bytes of one K-major core-matrix
        // row, written with a single 16-byte store; a warp's store covers
        // 512 contiguous bytes (four core matrices), free of bank conflicts.
        // Slots [0, P) are X's columns, [P, P + Qw) this chunk's Y columns;
        // the rest are idle.
        const int g = lane >> 4;
        int cg = warp % ncg;
        int s = warp / ncg;
        const int dcg = NCONV_WARPS % ncg, ds = NCONV_WARPS / ncg;
        // loads of step s (zero beyond this CTA's steps and beyond row K);
        // whole units inside the matrix skip the per-row bounds checks
        auto load_unit = [&](double(&v)[R], int st, int grp) {
            const int slot = 16 * grp + (lane & 15);
            const bool is_x = slot < P;
            const char* src = reinterpret_cast<const char*>(is_x ? prm.X + slot : prm.Y + q0 + (slot - P));
            const int64_t ldb = (is_x ? prm.ldx : prm.ldy) * 8;  // row stride in bytes
            const int64_t k = (s_begin + st) * KSTEP + 8 * g;
            const bool live = slot < P + Qw && st < nsteps;
            const int64_t left = live ? Ktot - k : 0;
            if (left >= R) {
                const char* p = src + k * ldb;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    v[r] = __ldg(reinterpret_cast<const double*>(p));
                    p += ldb;
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r)
                    v[r] = left > r ? __ldg(reinterpret_cast<const double*>(src + (k + r) * ldb)) : 0.0;
            }
        };
        auto high_max = [&](const double(&v)[R]) {
            uint32_t hm = 0;
#pragma unroll
            for (int r = 0; r < R; ++r) hm = max(hm, (uint32_t)__double2hiint(v[r]) & 0x7FFFFFFFu);
            return max(hm, __shfl_xor_sync(0xffffffffu, hm, 16));
        };
        double v[R];
        // The column exponents of a range start at the maximum over its
        // first PRE_STEPS steps, if that is at most a bit above the first
        // step's: rounding then costs the first rows no more than truncation
        // at the running maximum did.  Columns that grow faster start at the
        // first step's, so that small rows before large ones keep their
        // bits.  Without the scan every new maximum of a column's first rows
        // ends an accumulation tile, at about 10 us of the CTA (normal data:
        // real 24 x 40, S = 5, 10^6 rows 569 us against 370, complex 64 x 64,
        // 10^5 rows 404 against 231; with the whole scan's maximum 352 and 191).
        const int srange = (int)min(prm.steps_per_range, (int64_t)nsteps + 1);
        if (!plain_digits<S>()) {
            int* first = exps;  // not in use yet: the ranges' first steps' exponents [MAX_RANGES][NE], ndig >= MAX_RANGES
            for (int j = 0; j < MAX_RANGES && j * srange < nsteps; ++j) {
                const int pre = min(min(nsteps - j * srange, srange), PRE_STEPS) * ncg;
                for (int u = warp; u < pre; u += NCONV_WARPS) {
                    const int grp = u % ncg, slot = 16 * grp + (lane & 15);
                    load_unit(v, j * srange + u / ncg, grp);
                    const uint32_t hm = high_max(v);
                    if (slot < P + Qw && g == 0) {
                        atomicMax(&col_e0[j * NE + slot], exp_from_hi(hm));
                        if (u < ncg) first[j * NE + slot] = exp_from_hi(hm);
                    }
                }
            }
            asm volatile("bar.sync 1, %0;" ::"r"(NCONV_WARPS * 32) : "memory");
#pragma unroll 1
            for (int i = threadIdx.x; i < MAX_RANGES * NE; i += NCONV_WARPS * 32) {
                int e = col_e0[i];
                if (e > first[i] + 1) col_e0[i] = e = first[i];
                if (i < NE) col_e[i] = e;
            }
            asm volatile("bar.sync 1, %0;" ::"r"(NCONV_WARPS * 32) : "memory");
        }
        int rs = s % srange;  // step within its range
        int d = s % ndig;
        uint32_t phase = (uint32_t)(s / ndig) & 1u;
        load_unit(v, s, cg);
        while (s < nsteps) {
            const int slot = 16 * cg + (lane & 15);
            const bool is_x = slot < P, valid = slot < P + Qw;
            // slice j of X: operand-A block j / stack, rows (j % stack) Pp + slot
            const uint32_t off0 = is_x ? kmajor_off(slot, g) : L.a_bytes + kmajor_off(slot - P, g);
            const uint32_t dsl = is_x ? 4096u / (uint32_t)stack : (uint32_t)Qp * 32u;
            const uint32_t hm = high_max(v);
            // The column's exponent, passed on from step to step in order, so
            // that it depends on the data alone.  It restarts with every
            // range.  With 5 or 6 slices a value may exceed 2^e by one bit
            // (not quite: its top digit has to stay below 256) in up to
            // SOFT_STEPS steps of a column; after that, or beyond it, e is
            // raised, which ends the tile.  The digits of such a step keep
            // the unit 2^(e + 1 - 8S).
            if (!seq_wait(bar(M_SEQ + 4 * cg), s, tmo, prm.err, 9, abort_flag)) {
                *abort_flag = 1;
                break;
            }
            const int was = valid ? *reinterpret_cast<volatile int*>(&col_e[slot]) : 0;
            int e = was;
            if (rs == 0 && s > 0 && valid) e = plain_digits<S>() ? E_NONE : col_e0[NE + slot];
            const uint32_t lim = e == E_NONE ? 0u : (uint32_t)(e + 1023) << 20;
            const bool over = valid && hm >= lim;
            bool soft = false;
            if (__any_sync(0xffffffffu, over)) {
                int n = 0;
                if (!plain_digits<S>() && over) n = *reinterpret_cast<volatile int*>(&col_soft[slot]);
                soft = over && !plain_digits<S>() && hm < lim + 0xFE000u && n < SOFT_STEPS;
                if (over && !soft) e = exp_from_hi(hm);
                __syncwarp();  // both lanes of a column have read
                if (soft && g == 0) *reinterpret_cast<volatile int*>(&col_soft[slot]) = n + 1;
                soft = __any_sync(0xffffffffu, soft);
            }
            const bool grew = __any_sync(0xffffffffu, e != was);
            if (grew && valid && g == 0) *reinterpret_cast<volatile int*>(&col_e[slot]) = e;
            __syncwarp();
            if (lane == 0)
                asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(bar(M_SEQ + 4 * cg)), "r"(s + 1)
                             : "memory");
            // the stage must be free
            if (!warp_wait(bar(M_DIG_EMPTY + 8 * d), phase ^ 1u, tmo, prm.err, 2, abort_flag)) {
                *abort_flag = 1;
                break;
            }
            if (lane == 0) {
                if (soft) soft_step[d] = s;
                if (grew) chg_step[d] = s;
            }
            const bool fast = !__any_sync(0xffffffffu, valid && e <= -960);
            if (valid && g == 0) exps[d * NE + slot] = e;
            uint32_t w[S][R / 2];
            if (fast) {  // warp-uniform
                const int eb = (int)(((uint32_t)(e + digit_shift<S>()) << 20) + 0xFFFFFu);
#pragma unroll
                for (int r = 0; r < R; r += 2) {
                    uint32_t wp[S];
                    split_pair<S, true>(v[r], v[r + 1], eb, wp);
#pragma unroll
                    for (int sl = 0; sl < S; ++sl) w[sl][r >> 1] = wp[sl];
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; r += 2) {
                    uint32_t wp[S];
                    split_pair<S, false>(v[r], v[r + 1], e, wp);
#pragma unroll
                    for (int sl = 0; sl < S; ++sl) w[sl][r >> 1] = wp[sl];
                }
            }
            if (valid) {
                unsigned char* out = dig + d * L.stage + off0;
#pragma unroll
                for (int sl = 0; sl < S; ++sl)
                    *reinterpret_cast<uint4*>(out + sl * dsl) = make_uint4(w[sl][0], w[sl][1], w[sl][2], w[sl][3]);
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(M_DIG_FULL + 8 * d));
            // the next unit's loads come after the arrival, which as a
            // release would wait for them; the other warps hide their latency
            int step = ds;
            cg += dcg;
            if (cg >= ncg) {
                cg -= ncg;
                ++step;
            }
            s += step;
            d += step;
            if (d >= ndig) {
                d -= ndig;
                phase ^= 1u;
            }
            rs += step;
            while (rs >= srange) rs -= srange;
            load_unit(v, s, cg);
        }
    } else if (warp == MMA_WARP) {
        // ================================================= MMA issuer
        // The whole warp runs the loop, with uniform control flow; one lane
        // issues the tcgen05 operations.
        int64_t tile = -1;
        int used = 0, cur_slot = 0, cur_chg = 0;
        bool failed = false;
        uint32_t phase = 0;
        int d = 0;
        const uint32_t dig_a = smem_addr(dig);
        // (shuffles, so that the compiler knows these to be warp-uniform)
        const uint32_t a_lo = __shfl_sync(0xffffffffu, desc_lo(dig_a), 0);
        const uint32_t b_lo = __shfl_sync(0xffffffffu, desc_lo(dig_a + L.a_bytes), 0);
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
        auto wait = [&](uint32_t b, uint32_t par, int code) {
            return warp_wait(b, par, tmo, prm.err, code, abort_flag);
        };
        // hands the finished tile to the epilogue: its record, and the
        // completion of its MMAs, on the same barrier
        auto hand_over = [&](int info) {
            if (lane == 0) {
                *tile_info = info;
                tc_fence_before();
                mbar_arrive(bar(M_TILE_FULL));
            }
            __syncwarp();
            mma_commit(bar(M_TILE_FULL), elect_one());
        };
        for (int s = 0; s < nsteps; ++s) {
            if (!wait(bar(M_DIG_FULL + 8 * d), phase, 3)) {
                failed = true;
                break;
            }
            tc_fence_after();
            const bool chg = chg_step[d] == s;
            const int cost = soft_step[d] == s ? 3 : 2;
            const int* ex = exps + d * NE;
            const bool new_tile = tile < 0 || chg || used + cost > TILE_BUDGET;
            if (new_tile) {
                if (tile >= 0) {
                    hand_over(cur_slot | (cur_chg << 10));
                    if (!wait(bar(M_TMEM_EMPTY), (uint32_t)(tile & 1), 5)) {
                        failed = true;
                        break;
                    }
                    tc_fence_after();
                }
                ++tile;
                used = 0;
                cur_slot = (int)(tile % NEXP);
                cur_chg = chg ? 1 : 0;
                if (!wait(bar(M_EXP_EMPTY + 8 * cur_slot), (uint32_t)(((tile / NEXP) & 1) ^ 1), 8)) {
                    failed = true;
                    break;
                }
                int* sn = snap + cur_slot * NE;
                for (int i = lane; i < NE; i += 32) sn[i] = ex[i];
                __syncwarp();
            }
            used += cost;
            // stage d's operands: the same descriptors moved by d stages (the
            // address field counts 16-byte units and stays below 2^14)
            const uint32_t so = ((uint32_t)d * L.stage) >> 4, lead = elect_one();
            if (stack == 1)
                issue_step_qp<S, 1>(Qp, tm, a_lo + so, b_lo + so, new_tile, lead);
            else if (stack == 2)
                issue_step_qp<S, 2>(Qp, tm, a_lo + so, b_lo + so, new_tile, lead);
            else
                issue_step_qp<S, 4>(Qp, tm, a_lo + so, b_lo + so, new_tile, lead);
            mma_commit(bar(M_DIG_EMPTY + 8 * d), lead);
            if (++d == ndig) {
                d = 0;
                phase ^= 1u;
            }
        }
        // last tile (or drain after a failure): no MMA may be in flight at exit
        if (!failed && tile >= 0) hand_over(cur_slot | (1 << 8) | (cur_chg << 10));
        if (!failed && tile < 0) hand_over(1 << 9);  // empty range: nothing to drain
        mma_commit(bar(M_MMA_DONE), elect_one());
        __syncwarp();
        if (lane == 0) {
            const bool drained = mbar_wait(bar(M_MMA_DONE), 0, kDefaultTimeout, prm.err, 6, nullptr);
            if (failed || !drained) *abort_flag = 1;  // the epilogue stops waiting
        }
        __syncwarp();
    } else {
        // ================================================= epilogue
        // Per (lane, column): an exact 64-bit integer sum of the tiles' W in
        // shared memory, at the scale of the current column exponents.  It
        // moves to binary64 (`flush`, this thread's own entries in global
        // memory) only when an exponent of its row or column grows, when
        // the integer sum would overflow, and at the end -- not once per tile.
        const int lane_base = 32 * (warp & 3);
        const int row = lane_base + lane;  // TMEM lane = accumulator row
        const int p = row & (Pp - 1), half = row / Pp;  // column of X, stacked slice (warp-uniform: Pp >= 32)
        const bool prow = p < P;
        // 8 warps: warps w and w + 4 share a lane quarter and split the columns
        const int ew = warp - MMA_WARP - 1;
        const int qh = prm.nepi == 8 ? Qp / 2 : Qp;  // a multiple of 8
        const int qlo = (ew >> 2) * qh, qhi = min(qlo + qh, Qw);
        double* flush = prm.flush + (int64_t)blockIdx.x * Qp * 128 + row;
        long long* acc = iacc + row;
        for (int q = qlo; q < qhi; ++q) flush[q * 128] = 0.0;
        auto scaled = [](long long a, int E) {
            return (E >= -1022 && E <= 1023) ? (double)a * __longlong_as_double((long long)(E + 1023) << 52)
                                             : scalbn((double)a, E);
        };
        // sums that carry a scale which has grown
        auto flush_changed = [&](const int* was, const int* now) {
            if (!prow) return;
            const bool pc = was[p] != now[p];
            // eight columns at a time: the binary64 totals are in global memory
            for (int qb = qlo; qb < qhi; qb += 8) {
                double f[8];
                uint32_t m = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int q = qb + i;
                    f[i] = 0.0;
                    if (q >= qhi || (!pc && was[P + q] == now[P + q])) continue;
                    m |= 1u << i;
                    f[i] = flush[q * 128];
                }
                if (!m) continue;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int q = qb + i;
                    if (!(m >> i & 1u)) continue;
                    flush[q * 128] = f[i] + scaled(acc[q * 128], was[p] + was[P + q] - (8 * S + 6));
                    acc[q * 128] = 0;
                }
            }
        };
        int prev_slot = -1;
        for (int64_t tile = 0;; ++tile) {
            int w_ok = 1;
            if (lane == 0) w_ok = mbar_wait(bar(M_TILE_FULL), (uint32_t)(tile & 1), tmo, prm.err, 7, abort_flag);
            if (!__shfl_sync(0xffffffffu, w_ok, 0)) break;
            tc_fence_after();
            const int info = *tile_info;
            if (info & (1 << 9)) break;
            const int slot = info & 0xFF;
            const int* ex = snap + slot * NE;
            const int ep = prow ? ex[p] : 0;
            if (prev_slot >= 0) {
                if ((info >> 10) & 1) flush_changed(snap + prev_slot * NE, ex);
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(M_EXP_EMPTY + 8 * prev_slot));
            }
            // the weight offset of a warp's rows is warp-uniform: one loop per
            // value.  The next four columns are read while these are summed.
            auto drain = [&](auto half_tag) {
                constexpr int H = decltype(half_tag)::value;
                if (qlo >= qhi) return;
                uint32_t v[S][4];
                auto issue = [&](int qb) {
#pragma unroll
                    for (int j = 0; j < S - H; ++j)
                        tmem_ld4(tmem + ((uint32_t)lane_base << 16) + (uint32_t)(j * Qp + qb), v[j]);
                };
                issue(qlo);
                for (int qb = qlo; qb < qhi; qb += 4) {
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < S - H; ++j)  // no use of v moves above the wait
#pragma unroll
                        for (int i = 0; i < 4; ++i) asm volatile("" : "+r"(v[j][i]));
                    long long W[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) W[i] = combine_w<H, S>(v, i);
                    if (qb + 4 < qhi) issue(qb + 4);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        // (rows past P and columns past Qw sum what nothing reads)
                        const int q = qb + i;
                        const long long a = acc[q * 128];
                        long long sum = (long long)((unsigned long long)a + (unsigned long long)W[i]);
                        if (((a ^ sum) & (W[i] ^ sum)) < 0) {  // would overflow: move a to binary64
                            if (prow && q < qhi) flush[q * 128] += scaled(a, ep + ex[P + q] - (8 * S + 6));
                            sum = W[i];
                        }
                        acc[q * 128] = sum;
                    }
                }
            };
            if (half == 0)
                drain(std::integral_constant<int, 0>());
            else if (half == 1)
                drain(std::integral_constant<int, 1>());
            else if (half == 2)
                drain(std::integral_constant<int, 2>());
            else
                drain(std::integral_constant<int, 3>());
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(M_TMEM_EMPTY));
            prev_slot = slot;
            if (info & (1 << 8)) {
                // this lane's totals, as binary64 in the accumulators' place
                if (prow)
                    for (int qb = qlo; qb < qhi; qb += 4) {
                        double f[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) f[i] = qb + i < qhi ? flush[(qb + i) * 128] : 0.0;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int q = qb + i;
                            if (q >= qhi) continue;
                            const double t = f[i] + scaled(acc[q * 128], ep + ex[P + q] - (8 * S + 6));
                            acc[q * 128] = __double_as_longlong(t);
                        }
                    }
                break;
            }
        }
    }

    __syncthreads();
    // CTA partial: G[p][q0 + q] for this K range
    double* out = prm.ws + (int64_t)kr * P * prm.Q;
    const double* tot = reinterpret_cast<const double*>(iacc);
    for (int i = threadIdx.x; i < P * Qw; i += NTHREADS) {
        const int pp = i / Qw, q = i - pp * Qw;
        double t = tot[q * 128 + pp];
        for (int h = 1; h < stack; ++h) t += tot[q * 128 + h * Pp + pp];
        out[(int64_t)pp * prm.Q + q0 + q] = t;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == MMA_WARP) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(prm.tmem_cols));
    }
}

// Sums the per-range partials and applies alpha / beta; for complex data G
// holds the real products of interleaved columns:
// A^T B = (RR - II) + i (RI + IR), A^H B = (RR + II) + i (RI - IR).
// Eight threads share an entry (thread s takes ranges s, s + 8, ... in
// order; their sums are combined by a fixed pairwise tree): one thread alone
// would wait for n_kr partials in a row, which set the time of short
// products (complex 64 x 64 at 3000 rows: 129 us before, 37 us with this and
// the set-up that no longer clears the operand stages).  The last CTA moves the
// launch's error word to the status word and clears it.
constexpr int kCombSlices = 8;
__global__ void __launch_bounds__(32 * kCombSlices) k_split_combine(const double* ws, int n_kr, int P, int Q, int M,
                                                                    int N, int cplx, int conj, double ar, double ai,
                                                                    double br, double bi, int beta_zero, double* C,
                                                                    int64_t ldc, int* words) {
    __shared__ double red[4][kCombSlices][32];
    const int c = threadIdx.x & 31, s = threadIdx.x >> 5;
    const int o = blockIdx.x * 32 + c;
    const bool mine = o < M * N;
    const int m = mine ? o / N : 0, n = mine ? o - m * N : 0;
    const bool bad = *reinterpret_cast<volatile int*>(words + kErrWord) != 0;
    const int nc = cplx ? 4 : 1;
    const int64_t PQ = (int64_t)P * Q;
    if (!cplx) {
        const double* p = ws + (int64_t)m * Q + n;
        double t = 0.0;
#pragma unroll 8
        for (int r = s; r < n_kr; r += kCombSlices) t += p[r * PQ];
        red[0][s][c] = t;
    } else {
        // entries (2m, 2n), (2m, 2n + 1) and (2m + 1, ...): P and Q are even,
        // so pairs are 16-byte aligned
        const double* p = ws + (int64_t)(2 * m) * Q + 2 * n;
        double2 u = make_double2(0.0, 0.0), v = make_double2(0.0, 0.0);
#pragma unroll 4
        for (int r = s; r < n_kr; r += kCombSlices) {
            const double2 a = *reinterpret_cast<const double2*>(p + r * PQ);
            const double2 b = *reinterpret_cast<const double2*>(p + r * PQ + Q);
            u.x += a.x;
            u.y += a.y;
            v.x += b.x;
            v.y += b.y;
        }
        red[0][s][c] = u.x;
        red[1][s][c] = u.y;
        red[2][s][c] = v.x;
        red[3][s][c] = v.y;
    }
    __syncthreads();
    for (int h = kCombSlices / 2; h >= 1; h >>= 1) {
        if (s < h)
            for (int k = 0; k < nc; ++k) red[k][s][c] += red[k][s + h][c];
        __syncthreads();
    }
    if (s == 0 && mine) {
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        if (!cplx) {
            double v = ar * red[0][0][c];
            double* out = C + (int64_t)m * ldc + n;
            if (!beta_zero) v = fma(br, *out, v);
            *out = bad ? nan : v;
        } else {
            const double rr = red[0][0][c], ri = red[1][0][c], ir = red[2][0][c], ii = red[3][0][c];
            const double gr = conj ? rr + ii : rr - ii;
            const double gi = conj ? ri - ir : ri + ir;
            double vr = ar * gr - ai * gi, vi = ar * gi + ai * gr;
            double* out = C + ((int64_t)m * ldc + n) * 2;
            if (!beta_zero) {
                const double orr = out[0], oi = out[1];
                vr += br * orr - bi * oi;
                vi += br * oi + bi * orr;
            }
            out[0] = bad ? nan : vr;
            out[1] = bad ? nan : vi;
        }
    }
    // every thread of the CTA has read the error word (barriers above)
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(reinterpret_cast<unsigned*>(words + kTicketWord), 1u) == gridDim.x - 1) {
            words[kStatusWord] = atomicExch(words + kErrWord, 0);
            words[kTicketWord] = 0;
        }
    }
}

long long g_timeout = kDefaultTimeout;

}  // namespace split

tsm_status validate_common(int dtype, int M, int N, int64_t K, const double* alpha, const double* beta);

}  // namespace tsm

using namespace tsm;

namespace tsm {
namespace split {

// Everything about a launch that depends on the shape only.
struct Plan {
    Params prm;     // shape fields filled; pointers, workspace and timeout are the caller's
    Layout L;
    int S = 6;      // slices per input
    int cps = 0;    // CTAs per SM
    int threads = 0;
    const void* fn = nullptr;
};

const void* kernel_for(int S) {
    return S == 4 ? (const void*)k_split<4> : S == 5 ? (const void*)k_split<5> : (const void*)k_split<6>;
}

// Ranges of K per SM after which the column exponents restart: 1 to 4.  The
// finer they are, the closer the digits' unit follows the data, and with 4
// slices the results show it (at 1e-9), so the number is part of what a
// shape's result means and does not follow the kernel's launch shape.  It is
// the number of CTAs an SM could hold of a kernel with one warp per 8 (up to
// 128 columns) or 16 columns, 5 more warps, 28 (24) warps and 3 stages of
// digits with two slices of X to a block.
int ranges_per_sm(int P, int qmax, int Qp, int S, int tcols) {
    const int cols = P + qmax, ne = P + Qp;
    const int conv = cols <= 128 ? (cols + 7) / 8 : (cols + 15) / 16, warps = cols <= 128 ? 28 : 24;
    const int blocks = P <= 64 ? (S + 1) / 2 : S;
    const int stage = (blocks * 4096 + S * Qp * 32 + 1023) / 1024 * 1024;
    for (int r = min(TMEM_COLS_MAX / tcols, 4); r > 1; --r) {
        const int room = (int)((kSmemPerSM / r - 1024u) & ~127u) - (Qp * 1024 + 16 * ne + 512);
        if (warps / (conv + 5) >= r && room / (stage + 4 * ne) >= 3) return r;
    }
    return 1;
}

tsm_status make_plan(int cplx, int M, int N, int64_t K, int S, Plan* pl) {
    if (S < 4 || S > NSLICE_MAX) return TSM_ERR_NOT_SUPPORTED;
    pl->S = S;
    const DeviceInfo& di = device_info();
    Params& prm = pl->prm;
    const int c = cplx ? 2 : 1;
    const int P = M * c, Q = N * c;
    prm.P = P;
    prm.Q = Q;
    prm.K = K;
    prm.stack = P <= 32 ? 4 : (P <= 64 ? 2 : 1);
    // Y column chunks: one if S slices of it fit tensor memory (512
    // columns) and its column groups fit the converter warps, else two
    // chunks split on an even column
    prm.q0[0] = prm.q0[1] = prm.qw[1] = 0;
    if (((Q + 15) & ~15) * S <= TMEM_COLS_MAX && (P + Q + 15) / 16 <= 13) {
        prm.n_qc = 1;
        prm.qw[0] = Q;
    } else {
        const int q1 = ((Q / 2) + 1) & ~1;
        prm.n_qc = 2;
        prm.qw[0] = q1;
        prm.q0[1] = q1;
        prm.qw[1] = Q - q1;
    }
    const int qmax = prm.qw[0] > prm.qw[1] ? prm.qw[0] : prm.qw[1];
    prm.Qp = (qmax + 15) & ~15;

    // CTA shape.  Accumulators take S * Qp tensor-memory columns; the
    // allocation is the next power of two, so chunks of up to 256 columns
    // leave room for a second CTA per SM, whose conversion then overlaps the
    // first one's drains.  Shared memory is split between them and padded so
    // that no more CTAs than planned share an SM (a further one would block
    // in its tensor-memory allocation).
    int tcols = 32;
    while (tcols < S * prm.Qp) tcols <<= 1;
    prm.tmem_cols = tcols;
    prm.ncg = (P + qmax + 15) / 16;
    pl->fn = kernel_for(S);
    pl->cps = 0;
    int ranges = ranges_per_sm(P, qmax, prm.Qp, S, tcols);
    const int cc_max = 2 * tcols <= TMEM_COLS_MAX && (S > 4 || ranges % 2 == 0) ? 2 : 1;
    for (int cc = cc_max; cc >= 1 && !pl->cps; --cc) {
        // several CTAs per SM share the drains: 4 epilogue warps each; alone, 8
        prm.nepi = cc > 1 ? 4 : NEPI_MAX;
        const int warps = kThreadsPerSM / cc / 32 - 1 - prm.nepi;
        const uint32_t budget = cc == 1 ? kSmemBudget : ((kSmemPerSM / cc - 1024u) & ~127u);
        const uint32_t floor_b = kSmemPerSM / (cc + 1);
        const Layout L = make_layout(P, prm.Qp, prm.stack, budget, floor_b, S);
        if (L.ndig < (cc > 1 ? 3 : 2) || L.total > (uint32_t)di.smem_optin) continue;
        // as many warps as fit, but at most a ring's worth of units: a warp
        // is never more than one use of a stage ahead (the barrier's parity
        // tells no more apart)
        prm.nconv = min(warps, (L.ndig - 1) * prm.ncg);
        pl->cps = cc;
        pl->threads = 32 * (prm.nconv + 1 + prm.nepi);
        pl->L = L;
        prm.smem_budget = (int)budget;
        prm.smem_floor = (int)floor_b;
    }
    if (!pl->cps) return TSM_ERR_NOT_SUPPORTED;
    // (the occupancy query reports one CTA for this kernel although two
    // measurably run together: the plan counts registers, threads, tensor
    // and shared memory itself)
    if (cudaFuncSetAttribute(pl->fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100) != cudaSuccess ||
        cudaFuncSetAttribute(pl->fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget) != cudaSuccess)
        return TSM_ERR_LAUNCH;

    // K in exponent ranges, and those, in order, in equal numbers to the
    // resident CTAs.  With more than 4 slices the ranges may be finer, so
    // that every CTA has as many.
    if (S > 4) ranges = (ranges + pl->cps - 1) / pl->cps * pl->cps;
    const int64_t steps = (K + KSTEP - 1) / KSTEP;
    int64_t n_range = std::min<int64_t>(ranges * di.sm_count / prm.n_qc, steps);
    if (n_range < 1) n_range = 1;
    prm.steps_per_range = std::max<int64_t>((steps + n_range - 1) / n_range, 1);
    n_range = std::max<int64_t>((steps + prm.steps_per_range - 1) / prm.steps_per_range, 1);
    const int64_t n_cta = std::max(pl->cps * di.sm_count / prm.n_qc, 1);
    const int64_t per_cta = (n_range + n_cta - 1) / n_cta;
    prm.steps_per_kr = per_cta * prm.steps_per_range;
    prm.n_kr = (int)((n_range + per_cta - 1) / per_cta);
    return TSM_OK;
}

}  // namespace split
}  // namespace tsm

namespace tsm {
namespace split {

tsm_status run(tsm_op opA, tsm_dtype dtype, int M, int N, int64_t K, const double* alpha, const void* A,
               int64_t lda, const void* B, int64_t ldb, const double* beta, void* C, int64_t ldc, int kind,
               int slices, tsm_stream_t stream) {
    tsm_status st = validate_common(dtype, M, N, K, alpha, beta);
    if (st != TSM_OK) return st;
    if (kind != TSM_SPLIT_DIGITS_F16) return TSM_ERR_INVALID_VALUE;
    if (slices < 4 || slices > NSLICE_MAX) return TSM_ERR_NOT_SUPPORTED;
    if (opA != TSM_OP_T && opA != TSM_OP_C) return TSM_ERR_INVALID_VALUE;
    if (lda < M || ldb < N || ldc < N || !C) return TSM_ERR_INVALID_VALUE;
    const int cplx = dtype == TSM_C64;
    const bool alpha0 = alpha[0] == 0.0 && (!cplx || alpha[1] == 0.0);
    if (K > 0 && !alpha0 && (!A || !B)) return TSM_ERR_INVALID_VALUE;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return TSM_ERR_NO_DEVICE;
    const DeviceInfo& di = device_info();
    if (di.cc_major != 10 || di.cc_minor != 3) return TSM_ERR_NO_DEVICE;
    const int beta_zero = beta[0] == 0.0 && (!cplx || beta[1] == 0.0);
    cudaStream_t s = (cudaStream_t)stream;
    if (K == 0 || alpha0) {
        return launch_scale_small((double*)C, M, N, ldc, cplx, beta[0], cplx ? beta[1] : 0.0, beta_zero, s) ==
                       cudaSuccess
                   ? TSM_OK
                   : TSM_ERR_LAUNCH;
    }
    Plan pl;
    if ((st = make_plan(cplx, M, N, K, slices, &pl)) != TSM_OK) return st;
    Params& prm = pl.prm;
    const int c = cplx ? 2 : 1;
    prm.X = (const double*)A;
    prm.ldx = lda * c;
    prm.Y = (const double*)B;
    prm.ldy = ldb * c;
    prm.timeout = g_timeout;
    const int n_kr = prm.n_kr, P = prm.P, Q = prm.Q;

    Workspace* ws = nullptr;
    const size_t part = (size_t)n_kr * P * Q * sizeof(double);
    const size_t flush = (size_t)n_kr * prm.n_qc * prm.Qp * 128 * sizeof(double);
    if ((st = workspace_get(s, part + flush + 256, 1, &ws)) != TSM_OK) return st;
    prm.ws = ws->partials;
    prm.flush = ws->partials + (size_t)n_kr * P * Q;
    int* words = reinterpret_cast<int*>(ws->tickets);
    prm.err = words + kErrWord;
    void* args[] = {&prm};
    if (cudaLaunchKernel(pl.fn, dim3(n_kr * prm.n_qc), dim3(pl.threads), args, pl.L.total, s) != cudaSuccess)
        return TSM_ERR_LAUNCH;
    const int outs = M * N;
    k_split_combine<<<(outs + 31) / 32, 32 * kCombSlices, 0, s>>>(
        ws->partials, n_kr, P, Q, M, N, cplx, (cplx && opA == TSM_OP_C) ? 1 : 0, alpha[0], cplx ? alpha[1] : 0.0,
        beta[0], cplx ? beta[1] : 0.0, beta_zero, (double*)C, ldc, words);
    if (cudaGetLastError() != cudaSuccess) return TSM_ERR_LAUNCH;
    return TSM_OK;
}

}  // namespace split
}  // namespace tsm

extern "C" tsm_status tsm_tsmttsm_split(tsm_op opA, tsm_dtype dtype, int M, int N, int64_t K,
                                        const double* alpha, const void* A, int64_t lda, const void* B,
                                        int64_t ldb, const double* beta, void* C, int64_t ldc,
                                        tsm_stream_t stream) {
    return split::run(opA, dtype, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, TSM_SPLIT_DIGITS_F16, 6, stream);
}

extern "C" tsm_status tsm_tsmttsm_split_ex(tsm_op opA, tsm_dtype dtype, int M, int N, int64_t K,
                                           const double* alpha, const void* A, int64_t lda, const void* B,
                                           int64_t ldb, const double* beta, void* C, int64_t ldc,
                                           tsm_split_kind kind, int slices, tsm_stream_t stream) {
    return split::run(opA, dtype, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, kind, slices, stream);
}

extern "C" tsm_status tsm_split_plan_ex(tsm_dtype dtype, int M, int N, int64_t K, int slices,
                                        tsm_split_plan_info* info) {
    if (!info || (dtype != TSM_R64 && dtype != TSM_C64) || K < 1) return TSM_ERR_INVALID_VALUE;
    if (M < 1 || N < 1 || M > 64 || N > 64 || slices < 4 || slices > split::NSLICE_MAX)
        return TSM_ERR_NOT_SUPPORTED;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return TSM_ERR_NO_DEVICE;
    const DeviceInfo& di = device_info();
    if (di.cc_major != 10 || di.cc_minor != 3) return TSM_ERR_NO_DEVICE;
    split::Plan pl;
    const tsm_status st = split::make_plan(dtype == TSM_C64, M, N, K, slices, &pl);
    if (st != TSM_OK) return st;
    info->ctas = pl.prm.n_kr * pl.prm.n_qc;
    info->ctas_per_sm = pl.cps;
    info->column_chunks = pl.prm.n_qc;
    info->converter_threads = 32 * pl.prm.nconv;
    info->epilogue_warps = pl.prm.nepi;
    info->threads_per_cta = pl.threads;
    info->digit_stages = pl.L.ndig;
    info->tmem_columns = pl.prm.tmem_cols;
    info->smem_bytes = (int)pl.L.total;
    return TSM_OK;
}

extern "C" tsm_status tsm_split_plan(tsm_dtype dtype, int M, int N, int64_t K, tsm_split_plan_info* info) {
    return tsm_split_plan_ex(dtype, M, N, K, 6, info);
}

extern "C" tsm_status tsm_split_status(tsm_stream_t stream) {
    cudaStream_t s = (cudaStream_t)stream;
    Workspace* ws = nullptr;
    tsm_status st = workspace_get(s, 256, 1, &ws);
    if (st != TSM_OK) return st;
    if (cudaStreamSynchronize(s) != cudaSuccess) return TSM_ERR_LAUNCH;
    int err = 0;
    int* p = reinterpret_cast<int*>(ws->tickets) + split::kStatusWord;
    if (cudaMemcpy(&err, p, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return TSM_ERR_LAUNCH;
    if (err) return zero_now(p, sizeof(int)) == cudaSuccess ? TSM_ERR_TIMEOUT : TSM_ERR_LAUNCH;
    return TSM_OK;
}

extern "C" tsm_status tsm_split_set_timeout(int64_t timeout_cycles) {
    split::g_timeout = timeout_cycles > 0 ? (long long)timeout_cycles : split::kDefaultTimeout;
    return TSM_OK;
}

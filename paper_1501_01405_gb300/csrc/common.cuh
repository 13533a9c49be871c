// Shared device helpers of the MRIP engine: the Philox4x32-10 stream, the
// 53-bit uniform and exponential variates, launch plumbing and the library's
// error state.  Written for sm_103a (GB300).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include <nvtx3/nvToolsExt.h>

#include "../../include/mrip.h"

namespace mrip {

// A named NVTX range for the lifetime of the object (host timeline; profilers
// can attribute and filter the kernels a call launches by it).
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

// ---------------------------------------------------------------------------
// Bounds checks of a debug build (-DMRIP_DEBUG).
//
// MRIP_CHECK(cond, site, index) guards one access: in a release build it is
// the constant true and the compiler drops it; in a debug build a false
// cond records (site, index) in this translation unit's record -- the first
// failure since the record was last read wins -- and evaluates to false, so
// the caller skips (or clamps) the access.  Nothing traps, asserts or waits.
// Sites are numbered per file (forest fire 1xx, queues 2xx, walk 3xx,
// network 4xx, control variate 5xx, area walk 6xx, statistics 7xx); the
// host reads and clears the records with mrip_debug_checks.
// ---------------------------------------------------------------------------
#ifdef MRIP_DEBUG
static __device__ unsigned long long g_check_first;

__device__ __forceinline__ bool check_record(bool ok, unsigned site, long long index) {
    if (!ok) {
        const unsigned long long rec =
            (static_cast<unsigned long long>(site) << 40) | (static_cast<unsigned long long>(index) & ((1ull << 40) - 1));
        atomicCAS(&g_check_first, 0ull, rec);
    }
    return ok;
}

#define MRIP_CHECK(cond, site, index) \
    (::mrip::check_record(static_cast<bool>(cond), (site), static_cast<long long>(index)))

// The host half of a unit's record: read it and put it back to zero.
#define MRIP_DEBUG_UNIT(name)                                                       \
    namespace mrip {                                                                \
    mrip_status debug_take_##name(unsigned long long* rec) {                        \
        const unsigned long long zero = 0;                                          \
        cudaError_t e = cudaMemcpyFromSymbol(rec, g_check_first, sizeof(*rec));     \
        if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_check_first, &zero, sizeof(zero)); \
        return e == cudaSuccess ? MRIP_OK : cuda_status(e, "debug checks: " #name); \
    }                                                                               \
    }
#else
#define MRIP_CHECK(cond, site, index) true
#define MRIP_DEBUG_UNIT(name)
#endif

// Bytes of dynamic shared memory this launch was given (the PTX special
// register), for the debug checks of dynamically sized shared arrays.
__device__ __forceinline__ unsigned dynamic_smem_bytes() {
    unsigned r;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(r));
    return r;
}

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11).  The ten round keys are
// fixed per seed, so the host expands them once and every kernel reads them
// from its parameter bank (uniform across the grid, no registers).
// ---------------------------------------------------------------------------
struct RoundKeys {
    uint32_t k0[10];
    uint32_t k1[10];
};

inline RoundKeys expand_key(uint64_t seed) {
    RoundKeys rk;
    uint32_t a = static_cast<uint32_t>(seed);
    uint32_t b = static_cast<uint32_t>(seed >> 32);
    for (int r = 0; r < 10; ++r) {
        rk.k0[r] = a;
        rk.k1[r] = b;
        a += 0x9E3779B9u;  // Weyl increments of the key schedule
        b += 0xBB67AE85u;
    }
    return rk;
}

// The full 64-bit product of two 32-bit words as one widening multiply
// (mul.wide.u32), both halves from one instruction.
__host__ __device__ __forceinline__ void mul_wide_u32(uint32_t a, uint32_t b, uint32_t& hi, uint32_t& lo) {
#ifdef __CUDA_ARCH__
    unsigned long long r;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
#else
    const uint64_t r = static_cast<uint64_t>(a) * b;
#endif
    hi = static_cast<uint32_t>(r >> 32);
    lo = static_cast<uint32_t>(r);
}

// One Philox4x32 round: products of (0xD2511F53, x0) and (0xCD9E8D57, x2);
// high halves xored with the other words and the round key; low halves
// moved to positions 1 and 3.
__host__ __device__ __forceinline__ void philox_round(uint32_t& x0, uint32_t& x1, uint32_t& x2,
                                                      uint32_t& x3, uint32_t ka, uint32_t kb) {
#ifdef __CUDA_ARCH__
    uint32_t p0_lo, p0_hi, p1_lo, p1_hi;
    mul_wide_u32(0xD2511F53u, x0, p0_hi, p0_lo);
    mul_wide_u32(0xCD9E8D57u, x2, p1_hi, p1_lo);
#else
    const uint64_t p0 = static_cast<uint64_t>(0xD2511F53u) * x0;
    const uint64_t p1 = static_cast<uint64_t>(0xCD9E8D57u) * x2;
    const uint32_t p0_lo = static_cast<uint32_t>(p0), p0_hi = static_cast<uint32_t>(p0 >> 32);
    const uint32_t p1_lo = static_cast<uint32_t>(p1), p1_hi = static_cast<uint32_t>(p1 >> 32);
#endif
    x0 = p1_hi ^ x1 ^ ka;
    x1 = p1_lo;
    x2 = p0_hi ^ x3 ^ kb;
    x3 = p0_lo;
}

__host__ __device__ __forceinline__ uint4 philox(uint32_t c0, uint32_t c1, uint32_t c2,
                                                 uint32_t c3, const RoundKeys& rk) {
#pragma unroll
    for (int r = 0; r < 10; ++r) philox_round(c0, c1, c2, c3, rk.k0[r], rk.k1[r]);
    return make_uint4(c0, c1, c2, c3);
}

// Counter word 3: stream tag in the top byte, design point below.
__host__ __device__ __forceinline__ uint32_t stream_word(uint32_t tag, uint32_t dp) {
    return (tag << 24) | dp;
}

// u = (top 53 bits of hi:lo) * 2^-53, exact in double.
__device__ __forceinline__ double u53(uint32_t lo, uint32_t hi) {
    const unsigned long long bits = (static_cast<unsigned long long>(hi) << 32) | lo;
    return __ull2double_rn(bits >> 11) * 0x1p-53;
}

// Counters (c0, c1, rep, c3) of one replication with a small c0 and a running
// c1 (the queues' clients, the walks' and pi's blocks).  Three of the first six
// products do not depend on c1: round 1's products (of c0 <= 1, whose high
// half is 0, and of rep), round 2's product of word 2 and round 3's product of
// word 0.  RowKey holds what they leave, once per replication: 16 (c0 = 0) or
// 31 (the pair c0 = 0, 1, which shares round 2's product) products per client
// remain of 20 or 40, same words.  (With the recurrences' sums and
// maxima as carry chains and sign masks: M/M/1 65,536 x 1,000 clients 0.604 ->
// 0.569 ms, tandem 4,096 x 256 x 10,000 clients 123.7 -> 122.7 ms; part of it
// the compiler had already hoisted.)
struct RowKey {
    uint32_t h;     // word 0 after round 1, without c1
    uint32_t u;     // word 1 after round 2, with round 3's key
    uint32_t t, l;  // round 3's product of word 0: high half with its key, low half
};

__device__ __forceinline__ RowKey row_key(uint32_t rep, uint32_t c3, const RoundKeys& rk) {
    RowKey r;
    uint32_t hi, lo, w0;
    mul_wide_u32(0xCD9E8D57u, rep, hi, lo);
    r.h = hi ^ rk.k0[0];
    w0 = lo ^ rk.k0[1];
    mul_wide_u32(0xCD9E8D57u, c3 ^ rk.k1[0], hi, lo);
    w0 ^= hi;
    r.u = lo ^ rk.k0[2];
    mul_wide_u32(0xD2511F53u, w0, hi, lo);
    r.t = hi ^ rk.k1[2];
    r.l = lo;
    return r;
}

// Rounds 3 to 10 of block (kC0, c1), c0 = kC0 = 0 or 1; (p_hi, p_lo) is round
// 2's product 0xD2511F53 * (r.h ^ c1), the same for both.
template <uint32_t kC0>
__device__ __forceinline__ uint4 row_rounds(const RowKey& r, uint32_t p_hi, uint32_t p_lo, const RoundKeys& rk) {
    static_assert(kC0 <= 1, "0xD2511F53 * c0 must fit its low half");
    uint32_t x0, x1, x2, x3, hi;
    mul_wide_u32(0xCD9E8D57u, p_hi ^ (kC0 * 0xD2511F53u) ^ rk.k1[1], hi, x1);
    x0 = hi ^ r.u;
    x2 = r.t ^ p_lo;
    x3 = r.l;
#pragma unroll
    for (int i = 3; i < 10; ++i) philox_round(x0, x1, x2, x3, rk.k0[i], rk.k1[i]);
    return make_uint4(x0, x1, x2, x3);
}

// philox(0, c1, rep, c3) from the replication's row key.
__device__ __forceinline__ uint4 philox_row(const RowKey& r, uint32_t c1, const RoundKeys& rk) {
    uint32_t hi, lo;
    mul_wide_u32(0xD2511F53u, r.h ^ c1, hi, lo);
    return row_rounds<0>(r, hi, lo, rk);
}

// philox(0, c1, rep, c3) and philox(1, c1, rep, c3).
__device__ __forceinline__ void philox_row2(const RowKey& r, uint32_t c1, const RoundKeys& rk, uint4& b0, uint4& b1) {
    uint32_t hi, lo;
    mul_wide_u32(0xD2511F53u, r.h ^ c1, hi, lo);
    b0 = row_rounds<0>(r, hi, lo, rk);
    b1 = row_rounds<1>(r, hi, lo, rk);
}

// ---------------------------------------------------------------------------
// Exponential variates without the FP64 log.
//
// GB300's FP64 pipe retires about 2 FMAs per SM per clock, its integer pipes
// over 40 multiplies, so -log(1 - u) is evaluated in 64-bit fixed point
// (Tang's table-driven reduction, ACM TOMS 16(4), 1990, carried out in
// integers).  With 1 - u = K 2^-53, K in [1, 2^53], K = 2^e M, M in [1, 2):
//   -log(1 - u) = (53 - e) ln 2 - ln M,
//   ln M = -ln w_j + log1p(r),  r = w_j M - 1,  |r| <= 2^-14,
// w_j a 27-bit approximation of 1/c_j, c_j the centre of the j-th of 8192
// slices of [1, 2) (j = the 13 bits after the leading one).
//
// The kernels that draw variates are bound by instruction issue, so the
// scales are chosen for the fewest instructions:
//  - w_j has 27 bits and M 2^63 is a two-word integer, so V = w_j M 2^58 takes
//    one high and one wide multiply and no shift: it enters the result as it
//    is, and its bits 13..44 are r 2^45 as a signed word (1 2^45 vanishes
//    modulo 2^32);
//  - |r| <= 2^-14 leaves log1p(r) = r - r^2/2 + r^3/3 - r^4/4: r^2 to 2^-58 is
//    one 32-bit high multiply; the last two terms (below 2^-42) are FP32, on
//    the half of the FMA pipe that integer multiplies cannot use, and rounded
//    to an integer by an added 1.5 2^23;
//  - n ln 2 and 2^58 + ln w_j come rounded from tables, so four 64-bit terms
//    are added once, at 2^-58 (the largest result, 53 ln 2, still fits).
// w_j is taken among the candidates near 1/c_j whose logarithm lies closest to
// a multiple of 2^-58 (Gal's accurate tables); the table also carries the
// truncations' mean.  Absolute error against 113-bit arithmetic, in units of
// 2^-58: 0.58 rms and 2.04 at most over uniform u, slice edges and every
// exponent (6 million draws each); the earlier 4,096-slice form, rounded to
// 2^-57, had 0.83 and 2.2.
//
// Measured against that form: 157 instead of 235 warp instructions per M/M/1
// client (two variates); M/M/1 65,536 replications x 1,000 clients 0.795 ->
// 0.604 ms, tandem 4,096 x 256 replications x 10,000 clients 178.3 -> 123.7
// ms, 16 x 100,000 clients (CTA) 0.611 -> 0.449 ms, skip-sampled 128 x 128
// forest fire 2.89 -> 2.52 ms.  That moved the limit to the FMA-heavy pipe (78 %
// busy on the tandem); the FP32 tail, n ln 2 from shared memory (no 64-bit
// address multiply) and carry-chain adds (on the other pipe) take the M/M/1
// row on from 0.569 to 0.531 ms and the tandem's from 121.2 to 119.0.
// ---------------------------------------------------------------------------
constexpr int kLogSliceBits = 13;
constexpr int kLogSlices = 1 << kLogSliceBits;

struct __align__(16) LogSlice {
    unsigned long long lnw;  // 2^58 + ln(w_j) 2^58, rounded
    uint32_t w;              // w_j 2^27
    uint32_t pad;
};

struct LogTable {
    // entry kLogSlices + j is slice j (the leading one need not be masked off),
    // the entries before are zero
    const ulonglong2* slice;
    const unsigned long long* nln2;  // [s] = round((s + 1) ln 2 2^58), s = 0..63; [64] see neg_log_q58
    uint32_t nln2_shared;            // the same table in the CTA's shared memory (stage_nln2)
};
constexpr int kLogExponents = 65;
// coefficients of the FP32 tail in a = r 2^45, result in half units of 2^-58
constexpr float kLogR3 = -0x1p-76f / 3.0f, kLogR4 = 0x1p-123f, kLogMagic = 12582912.0f;  // 1.5 2^23
constexpr uint32_t kLogMagicBits = 0x4B400000u;

// Table for the current device (built and uploaded on first use; call it
// outside stream capture before the first launch that needs it).
mrip_status log_table(LogTable* out);

// The CTA's copy of the n ln 2 table, for neg_log_q58<true> (every thread calls;
// ends with a barrier).
__device__ __forceinline__ void stage_nln2(LogTable& tab, unsigned long long (&buf)[kLogExponents]) {
    for (int i = threadIdx.x; i < kLogExponents; i += blockDim.x) buf[i] = tab.nln2[i];
    tab.nln2_shared = static_cast<uint32_t>(__cvta_generic_to_shared(buf));
    __syncthreads();
}

// hi:lo + c as an explicit carry chain (both adds on the integer ALU; a plain
// 64-bit add may be put on the multiply pipe).
__device__ __forceinline__ unsigned long long add_carry(uint32_t lo, uint32_t hi, uint32_t c) {
    asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(lo), "+r"(hi) : "r"(c));
    return (static_cast<unsigned long long>(hi) << 32) | lo;
}

// a b >> 32 plus c.
__device__ __forceinline__ uint32_t mad_hi_u32(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("mad.hi.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}

// -log(1 - u) * 2^58, u = top 53 bits of hi:lo times 2^-53.  kShared: n ln 2
// from the copy stage_nln2 made.  kRare: takes every u; otherwise *top is negative
// for the 2^-32 of the words it does not (their result is meaningless, the
// look-ups stay within the tables: s held to 64, any 14 bits).
template <bool kShared, bool kRare>
__device__ __forceinline__ unsigned long long neg_log_impl(uint32_t lo, uint32_t hi, const LogTable& tab, uint32_t* top) {
    // K 2^11 = 2^64 - (hi:lo without its 11 lowest bits); 0 stands for K = 2^53
    const unsigned long long K = 0ull - ((static_cast<unsigned long long>(hi) << 32) | (lo & 0xFFFFF800u));
    const uint32_t kh = static_cast<uint32_t>(K >> 32), kl = static_cast<uint32_t>(K);
    uint32_t s, ml;
    asm("bfind.shiftamt.u32 %0, %1;" : "=r"(s) : "r"(kh));
    uint32_t mh = __funnelshift_lc(kl, kh, s);
    asm("shl.b32 %0, %1, %2;" : "=r"(ml) : "r"(kl), "r"(s));  // 0 for s >= 32
    if constexpr (kRare) {
        while (static_cast<int>(s) < 0) {  // kh = 0 (s = 2^32 - 1), once in 2^32 draws: one turn
            s = 32u + static_cast<uint32_t>(__clz(kl));
            mh = kl ? kl << (s & 31u) : 0x80000000u;  // K = 2^53: M = 1, s = 64
            ml = 0u;
        }
    } else {
        *top = s;
    }
    const ulonglong2 e = __ldg(tab.slice + (mh >> (31 - kLogSliceBits)));
    unsigned long long nln2;
    if constexpr (kShared)
        asm volatile("ld.shared.u64 %0, [%1];"
                     : "=l"(nln2)
                     : "r"(tab.nln2_shared + 8u * (kRare ? s : min(s, 64u)))
                     : "memory");  // (after stage_nln2's barrier)
    else
        nln2 = __ldg(tab.nln2 + (kRare ? s : min(s, 64u)));
    const uint32_t w = static_cast<uint32_t>(e.y);
    uint32_t v_hi, v_lo;
    mul_wide_u32(mh, w, v_hi, v_lo);
    const unsigned long long V = add_carry(v_lo, v_hi, __umulhi(ml, w));  // (1 + r) 2^58
    const int a = static_cast<int>(static_cast<uint32_t>(V >> 13));       // r 2^45
    const uint32_t r2 = static_cast<uint32_t>(__mulhi(a, a));             // r^2 2^58
    const float f = __int2float_rn(a);
    const float tail = __fmaf_rn(f * f * f, __fmaf_rn(f, kLogR4, kLogR3), kLogMagic);  // -2 r^3/3 + r^4/2
    return nln2 + e.x - V + ((r2 + (__float_as_uint(tail) - kLogMagicBits)) >> 1);
}

template <bool kShared>
__device__ __forceinline__ unsigned long long neg_log_q58(uint32_t lo, uint32_t hi, const LogTable& tab) {
    return neg_log_impl<kShared, true>(lo, hi, tab, nullptr);
}

// kN logarithms with one branch for the rare words of all: y[i] from words
// (lo[i], hi[i]); kShared: n ln 2 from the copy stage_nln2 made.  It saves a branch with
// its reconvergence, a compare and moves per logarithm, and keeps the words
// alive: 65,536 M/M/1 replications x 1,000 clients 500 -> 475 us (eight at a
// time).  The tandem's kernels, short of registers and bound by the multiply
// pipe, gain nothing (119 ms) or lose 4 % (a replication per CTA).  s is held to 64
// rather than the copy moved up by an entry for s = -1: any offset there cost the
// tandem 0.3 % (this kernel 472 us).
template <int kN, bool kShared>
__device__ __forceinline__ void neg_log_many(const uint32_t (&lo)[kN], const uint32_t (&hi)[kN], const LogTable& tab,
                                             unsigned long long (&y)[kN]) {
    uint32_t rare = 0u;
#pragma unroll
    for (int i = 0; i < kN; ++i) {
        uint32_t top;
        y[i] = neg_log_impl<kShared, false>(lo[i], hi[i], tab, &top);
        rare |= top;
    }
    if (__builtin_expect(static_cast<int>(rare) < 0, 0)) {
#pragma unroll
        for (int i = 0; i < kN; ++i) y[i] = neg_log_q58<kShared>(lo[i], hi[i], tab);
    }
}

// Exponential variate from words (lo, hi): -log(1 - u) * inv_rate_q58 where
// inv_rate_q58 = 2^-58 / rate.
template <bool kShared>
__device__ __forceinline__ double expo_fast(uint32_t lo, uint32_t hi, const LogTable& tab,
                                            double inv_rate_q58) {
    return __ull2double_rn(neg_log_q58<kShared>(lo, hi, tab)) * inv_rate_q58;
}

// Bernoulli threshold floor(p 2^32) for p in [0, 1) -- exact in double.
// Values outside [0, 1) (or NaN) are clamped to the nearest end.
__host__ __device__ __forceinline__ uint32_t threshold32(double p) {
    if (!(p > 0.0)) return 0u;
    if (p >= 1.0) return 0xFFFFFFFFu;
    return static_cast<uint32_t>(floor(p * 4294967296.0));
}

// ---------------------------------------------------------------------------
// Host-side error plumbing
// ---------------------------------------------------------------------------
void set_error(const std::string& msg);
mrip_status fail(mrip_status code, const std::string& msg);
mrip_status cuda_status(cudaError_t e, const char* what);
mrip_status launch_status(const char* what);

// Scratch memory shared by the stage entry points of one device: grows on
// demand, never shrinks, freed at exit.
void* scratch(size_t bytes, int slot);
int* device_error_flags();
int sm_count();

inline unsigned ceil_div_u(long long a, long long b) {
    return static_cast<unsigned>((a + b - 1) / b);
}

}  // namespace mrip

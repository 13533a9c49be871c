// Queueing models of the MRIP engine: the M/M/1 queue of the paper
// (Section 5.1, second model) and a 3-station tandem of M/M/1 stations.
//
// Mappings (paper, Section 3):
//   THREAD      one replication per thread (TLP);
//   WARP_1LANE  one replication per warp, lane 0 works, 31 lanes idle (WLP);
//   WARP_COOP   one replication per warp, the clients split into 32
//               contiguous segments.  The Lindley step W -> max(0, W + S - A)
//               composes to maps W -> max(c, W + d); lanes compose their
//               segment's map, a warp scan of the maps gives each segment's
//               entry wait, and each lane then replays its segment with the
//               plain recurrence.  The tandem does the same with 3-station
//               max-plus maps (lower-triangular 3x3 matrix plus constants).
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace mrip {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// ---------------------------------------------------------------------------
// Times in 64-bit fixed point.  GB300 retires about two FP64 operations per
// SM-clock and over forty 32-bit integer multiplies, so the queue recurrences
// (additions, subtractions and maxima only) run on integers: a time t is held
// as round(t 2^48).  A variate is E / rate with E = y58 2^-58 from the
// fixed-point log, i.e. round(y58 * (2^-10 / rate)), the factor stored as a
// 64-bit multiplier cm = round(2^56 / rate) (2^-10 / rate = cm 2^-66).  A
// variate then carries the multiplier's relative error (2^-53, as an FP64
// division would) plus at most one unit (2^-48), and every recurrence step is
// exact, where FP64 rounds each addition; the outputs agree with
// FP64 evaluation far inside 1e-12 as long as the variates are not tiny
// against 2^-48: rates are limited to [2^-6, 2^4] (mean variate >= 1/16).
// A variate is then below 36.8 * 64 < 2^11.3 time units (E <= 53 ln 2);
// while the largest state stays below 2^12 (2^60 units) one more step stays
// below 2^61.5, so nothing overflows.  Design points with other rates run the
// FP64 recurrence, and a replication whose sojourn time reaches 2^12
// restarts in FP64.  Means of single variates (the early-window features)
// are summed in FP64 from the same log values, where a variate's relative
// precision matters.
// ---------------------------------------------------------------------------
constexpr long long kFixGuard = 1LL << 60;
constexpr long long kFixNegInf = -(1LL << 62);  // "empty" state: v - A stays above -2^63

// 2^-10 / rate as cm 2^-66 (cm in [2^52, 2^62] for the rates above: at least
// 53 significant bits), so that round(y58 2^-10 / rate) = (hi(y58 cm) + 2) >> 2.
// Of the four partial products of hi(y58 cm) the lowest is dropped and the two
// middle ones enter by their high halves only, 0 to 3 units short in all, so
// 3 is added instead of 2: the variate is then within one unit (2^-48) of
// y58 2^-10 / rate.  cm < 2^62 keeps the sum of the middle halves (below
// 1.15 2^31 + 2^30 + 4) in 32 bits, so the first additions ride on the multiplies.
//
// This rounding, not the logarithm, is the M/M/1 outputs' error.  With cl the low
// word of cm, 1 + cl 2^-33 units are missing on average (a half where cl is 0), so a
// variate is (1/2 - cl 2^-33)/4 of a unit too large on average, 1/4 where cl is 0 (mu = 1),
// and S - A drifts by the difference within a busy period.  The error of one rate
// therefore depends on the bits of its multiplier: mean waits of 400 random rates x
// 32 replications x 1,000 clients are off by 3.3e-15 rms (relative, against 64-bit mantissas),
// 3.2e-15 when a variate was (hi(y57 cm) + 3) >> 2 with cm = round(2^57 / rate); single
// rates differ by a factor of two either way.
__device__ __forceinline__ bool fix_rate_ok(double rate) { return rate >= 0x1p-6 && rate <= 0x1p4; }

__device__ __forceinline__ unsigned long long fix_scale(double rate) {
    return static_cast<unsigned long long>(0x1p56 / rate + 0.5);
}

__device__ __forceinline__ long long to_fix(unsigned long long y58, unsigned long long cm) {
    const uint32_t yh = static_cast<uint32_t>(y58 >> 32), yl = static_cast<uint32_t>(y58);
    const uint32_t ch = static_cast<uint32_t>(cm >> 32), cl = static_cast<uint32_t>(cm);
    const uint32_t mid = mad_hi_u32(yl, ch, mad_hi_u32(yh, cl, 3u));
    uint32_t p_hi, p_lo;
    mul_wide_u32(yh, ch, p_hi, p_lo);
    return static_cast<long long>(add_carry(p_lo, p_hi, mid) >> 2);
}

// Sum of up to 2^32 values below 2^61: 96 bits (one carry chain of three adds).
struct U96 {
    unsigned long long lo = 0;
    uint32_t hi = 0;
    __device__ __forceinline__ void add(unsigned long long v) { add(v, 0u); }
    __device__ __forceinline__ void add(unsigned long long v, uint32_t v_hi) {
        uint32_t l0 = static_cast<uint32_t>(lo), l1 = static_cast<uint32_t>(lo >> 32);
        // (the low words wait in registers of the statement's own: %0 and %1 may not
        // change before every input has been read)
        asm("{\n .reg .u32 a, b;\n add.cc.u32 a, %0, %3;\n addc.cc.u32 b, %1, %4;\n addc.u32 %2, %2, %5;\n"
            " mov.u32 %0, a;\n mov.u32 %1, b;\n}"
            : "+r"(l0), "+r"(l1), "+r"(hi)
            : "r"(static_cast<uint32_t>(v)), "r"(static_cast<uint32_t>(v >> 32)), "r"(v_hi));
        lo = (static_cast<unsigned long long>(l1) << 32) | l0;
    }
    __device__ __forceinline__ double to_double() const {  // value 2^-48
        return static_cast<double>(hi) * 0x1p16 + static_cast<double>(lo) * 0x1p-48;
    }
};

// max(x, 0) from the sign alone.
__device__ __forceinline__ long long relu64(long long x) { return x & ~(x >> 63); }

constexpr long long kSat = 1LL << 61;

__device__ __forceinline__ long long sat61(long long x) { return x > kSat ? kSat : (x < -kSat ? -kSat : x); }

__device__ __forceinline__ U96 shfl_down_u96(const U96& x, int off) {
    U96 r;
    r.lo = __shfl_down_sync(kFull, x.lo, off);
    r.hi = __shfl_down_sync(kFull, x.hi, off);
    return r;
}
__device__ __forceinline__ void add_u96(U96& a, const U96& b) { a.add(b.lo, b.hi); }

struct Mm1Out {
    double* wait;
    double* idle;
    double* system;
};

// Client n of a replication: service S_n from words (0,1), gap A_{n+1} from (2,3).
// inv_mu, inv_lam are 2^-58 / rate (see expo_fast).
template <bool kShared>
__device__ __forceinline__ void mm1_client(uint32_t n, const RowKey& row, double inv_lam,
                                           double inv_mu, const RoundKeys& rk, const LogTable& tab,
                                           double& s, double& a) {
    const uint4 b = philox_row(row, n, rk);
    s = expo_fast<kShared>(b.x, b.y, tab, inv_mu);
    a = expo_fast<kShared>(b.z, b.w, tab, inv_lam);
}

// Clients n .. n + kCount - 1 in FP64, their logarithms with one branch for the rare words.
template <int kCount>
__device__ __forceinline__ void mm1_clients(uint32_t n, const RowKey& row, double inv_lam, double inv_mu,
                                            const RoundKeys& rk, const LogTable& tab, double (&s)[kCount],
                                            double (&a)[kCount]) {
    uint32_t lo[2 * kCount], hi[2 * kCount];
    unsigned long long y[2 * kCount];
#pragma unroll
    for (int i = 0; i < kCount; ++i) {
        const uint4 b = philox_row(row, n + i, rk);
        lo[2 * i] = b.x;
        hi[2 * i] = b.y;
        lo[2 * i + 1] = b.z;
        hi[2 * i + 1] = b.w;
    }
    neg_log_many<2 * kCount, false>(lo, hi, tab, y);
#pragma unroll
    for (int i = 0; i < kCount; ++i) {
        s[i] = __ull2double_rn(y[2 * i]) * inv_mu;
        a[i] = __ull2double_rn(y[2 * i + 1]) * inv_lam;
    }
}

// Clients whose variates are drawn together: a thread per replication gives an SM too
// few warps (13.5 at 2^16 replications) to hide one client's chain of Philox rounds and
// logarithms behind other warps.  2^16 x 1,000 clients at 1, 2, 3 and 4 clients: 561, 526,
// 504, 500 us, and 475 with one branch for the rare words of a group's eight
// logarithms (128 registers: a minimum of three CTAs per SM leaves them).  The choice holds
// over the range: 1,000, 16,384, 65,536, 262,144, 10^6 replications x 400 clients take 80, 80,
// 198, 648, 2,350 us, with two clients and four CTAs 82, 82, 200, 647, 2,344, with one and six
// 116, 115, 220, 672, 2,392.
constexpr uint32_t kMm1Group = 4;

template <bool kLane0Only>
__global__ void __launch_bounds__(128, 3) mm1_serial_kernel(const double* __restrict__ dps, long long n_items,
                                  long long n_reps, long long rep0, long long n_clients,
                                  const __grid_constant__ RoundKeys rk, LogTable tab, Mm1Out out) {
    __shared__ unsigned long long nln2[kLogExponents];
    stage_nln2(tab, nln2);
    long long item;
    if (kLane0Only) {
        if ((threadIdx.x & 31) != 0) return;
        item = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) >> 5;
    } else {
        item = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    }
    if (item >= n_items) return;
    const uint32_t dp = static_cast<uint32_t>(item / n_reps);
    const uint32_t rep = static_cast<uint32_t>(rep0 + item % n_reps);
    const double lam = dps[2 * dp], mu = dps[2 * dp + 1];
    const double inv = static_cast<double>(n_clients);
    const RowKey row = row_key(rep, stream_word(0u, dp), rk);
    if (fix_rate_ok(lam) && fix_rate_ok(mu)) {  // 48-bit fixed-point times
        const unsigned long long cl = fix_scale(lam), cmu = fix_scale(mu);
        long long wf = 0;
        U96 sw, si, sv;
        bool overflow = false;
        // (client indices are 32-bit: n_clients < 2^32, the counter word c1)
        const uint32_t nc = static_cast<uint32_t>(n_clients);
        // kMm1Group clients' variates at a time: their Philox rounds and
        // logarithms are independent chains, the Lindley steps follow.  The
        // guard is tested per group: a wait below 2^60 grows by less than 2^59.3
        // a client, so nothing overflows before the test.
        auto clients = [&](uint32_t n, auto count) {
            constexpr int kCount = decltype(count)::value;
            long long s_[kCount], a_[kCount];
            uint32_t lo[2 * kCount], hi[2 * kCount];
            unsigned long long y[2 * kCount];
#pragma unroll
            for (int i = 0; i < kCount; ++i) {
                const uint4 b = philox_row(row, n + i, rk);
                lo[2 * i] = b.x;
                hi[2 * i] = b.y;
                lo[2 * i + 1] = b.z;
                hi[2 * i + 1] = b.w;
            }
            neg_log_many<2 * kCount, true>(lo, hi, tab, y);
#pragma unroll
            for (int i = 0; i < kCount; ++i) {
                s_[i] = to_fix(y[2 * i], cmu);
                a_[i] = to_fix(y[2 * i + 1], cl);
            }
            long long any = 0;
#pragma unroll
            for (int i = 0; i < kCount; ++i) {
                sw.add(wf);
                const long long v = wf + s_[i];
                sv.add(v);
                const long long t = v - a_[i];
                wf = relu64(t);
                si.add(wf - t);  // max(0, -t)
                any |= wf;
            }
            return any < kFixGuard;
        };
        uint32_t n = 0;
        for (; nc - n >= kMm1Group && !overflow; n += kMm1Group)
            overflow = !clients(n, std::integral_constant<int, kMm1Group>{});
        for (; n < nc && !overflow; ++n) overflow = !clients(n, std::integral_constant<int, 1>{});
        if (!overflow) {
            if (out.wait) out.wait[item] = sw.to_double() / inv;
            if (out.idle) out.idle[item] = si.to_double() / inv;
            if (out.system) out.system[item] = sv.to_double() / inv;
            return;
        }
    }
    const double inv_lam = 0x1p-58 / lam, inv_mu = 0x1p-58 / mu;
    double w = 0.0, sum_w = 0.0, sum_i = 0.0, sum_v = 0.0;
    for (long long n = 0; n < n_clients; ++n) {
        double s, a;
        mm1_client<true>(static_cast<uint32_t>(n), row, inv_lam, inv_mu, rk, tab, s, a);
        sum_w += w;
        const double v = w + s;
        sum_v += v;
        const double t = v - a;
        sum_i += (t < 0.0) ? -t : 0.0;
        w = (t > 0.0) ? t : 0.0;
    }
    if (out.wait) out.wait[item] = sum_w / inv;
    if (out.idle) out.idle[item] = sum_i / inv;
    if (out.system) out.system[item] = sum_v / inv;
}

// Max-plus map W -> max(c, W + d).  compose(first, then).
struct MaxPlus {
    double c, d;
};
__device__ __forceinline__ MaxPlus compose(MaxPlus f, MaxPlus g) {
    // g(f(W)) = max(g.c, max(f.c, W + f.d) + g.d) = max(max(g.c, f.c + g.d), W + (f.d + g.d))
    MaxPlus r;
    const double cc = f.c + g.d;
    r.c = (g.c > cc) ? g.c : cc;
    r.d = f.d + g.d;
    return r;
}

// One warp per replication; clients staged in shared memory when kStage.  What bounds
// it is the latency of a client's chain (few warps per SM, and the staged slices leave
// its L1 little room for the logarithm's 128 KB table), so kMm1WarpGroup clients are
// drawn together: 500 x 1,000 clients 46.0 -> 41.2 us, 32 x 1,000 43.4 -> 39.2, 150 x 5,000
// 185 -> 169 (four together 43.2, 39.2, 165, but 1,500 x 150 20.6 instead of 18.6).
constexpr int kMm1WarpGroup = 2;

template <bool kStage>
__global__ void mm1_warp_coop_kernel(const double* __restrict__ dps, long long n_items,
                                     long long n_reps, long long rep0, long long n_clients,
                                     const __grid_constant__ RoundKeys rk, LogTable tab, Mm1Out out) {
    extern __shared__ double stage[];  // per warp: S[seg_cap*32], A[seg_cap*32]
    const int lane = threadIdx.x & 31;
    const int warp_in_cta = threadIdx.x >> 5;
    const long long item = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) >> 5;
    if (item >= n_items) return;  // warp-uniform
    const uint32_t dp = static_cast<uint32_t>(item / n_reps);
    const uint32_t rep = static_cast<uint32_t>(rep0 + item % n_reps);
    const double inv_lam = 0x1p-58 / dps[2 * dp], inv_mu = 0x1p-58 / dps[2 * dp + 1];
    const RowKey row = row_key(rep, stream_word(0u, dp), rk);
    const long long seg = (n_clients + 31) / 32;
    const long long lo = lane * seg;
    const long long hi = (lo + seg < n_clients) ? lo + seg : n_clients;
    double* s_buf = stage + static_cast<size_t>(warp_in_cta) * 2 * seg * 32;
    double* a_buf = s_buf + seg * 32;
    // staged only where the warp's slice fits the launch's shared memory
    // (always, unless the host sized it wrong: then the debug build records
    // it and the variates are recomputed instead)
    const bool staged =
        kStage && MRIP_CHECK((warp_in_cta + 1ull) * 2 * seg * 32 * sizeof(double) <= dynamic_smem_bytes(), 201, seg);

    auto for_clients = [&](long long from, long long to, auto use) {
        long long n = from;
        for (; n + kMm1WarpGroup <= to; n += kMm1WarpGroup) {
            double s[kMm1WarpGroup], a[kMm1WarpGroup];
            mm1_clients<kMm1WarpGroup>(static_cast<uint32_t>(n), row, inv_lam, inv_mu, rk, tab, s, a);
#pragma unroll
            for (int i = 0; i < kMm1WarpGroup; ++i) use(n + i, s[i], a[i]);
        }
        for (; n < to; ++n) {
            double s, a;
            mm1_client<false>(static_cast<uint32_t>(n), row, inv_lam, inv_mu, rk, tab, s, a);
            use(n, s, a);
        }
    };

    // pass 1: the segment's composed map
    MaxPlus f{-INFINITY, 0.0};
    auto map = [&](long long n, double s, double a) {
        if (staged) {
            s_buf[(n - lo) * 32 + lane] = s;
            a_buf[(n - lo) * 32 + lane] = a;
        }
        f = compose(f, MaxPlus{0.0, s - a});
    };
    for_clients(lo, hi, map);
    // inclusive scan of maps over lanes (earlier lanes first), then shift
    MaxPlus acc = f;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        MaxPlus prev;
        prev.c = __shfl_up_sync(kFull, acc.c, off);
        prev.d = __shfl_up_sync(kFull, acc.d, off);
        if (lane >= off) acc = compose(prev, acc);
    }
    MaxPlus excl;
    excl.c = __shfl_up_sync(kFull, acc.c, 1);
    excl.d = __shfl_up_sync(kFull, acc.d, 1);
    double w = 0.0;
    if (lane > 0) w = (excl.c > excl.d) ? excl.c : excl.d;  // entry wait = map(0)

    // pass 2: replay the segment with the plain recurrence
    double sum_w = 0.0, sum_i = 0.0, sum_v = 0.0;
    auto replay = [&](long long, double s, double a) {
        sum_w += w;
        const double v = w + s;
        sum_v += v;
        const double t = v - a;
        sum_i += (t < 0.0) ? -t : 0.0;
        w = (t > 0.0) ? t : 0.0;
    };
    if (staged) {
        for (long long n = lo; n < hi; ++n) replay(n, s_buf[(n - lo) * 32 + lane], a_buf[(n - lo) * 32 + lane]);
    } else {
        for_clients(lo, hi, replay);
    }
    // fixed-order (lane-ordered tree) reduction of the three sums
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double ow = __shfl_down_sync(kFull, sum_w, off);
        const double oi = __shfl_down_sync(kFull, sum_i, off);
        const double ov = __shfl_down_sync(kFull, sum_v, off);
        if ((lane & (2 * off - 1)) == 0) {
            sum_w += ow;
            sum_i += oi;
            sum_v += ov;
        }
    }
    if (lane == 0) {
        const double inv = static_cast<double>(n_clients);
        if (out.wait) out.wait[item] = sum_w / inv;
        if (out.idle) out.idle[item] = sum_i / inv;
        if (out.system) out.system[item] = sum_v / inv;
    }
}

// ---------------------------------------------------------------------------
// Tandem: V_{n,j} = max(V_{n-1,j} - A_n, V_{n,j-1}) + S_{n,j}
// ---------------------------------------------------------------------------
struct TandemOut {
    double* y;
    double* feat;     // 8 planes of n_items (may be null)
    long long plane;  // plane stride = n_items
};

// One client in fixed point: v_j <- max(v_j - a, v'_{j-1}) + s_j (v'_0 = 0), the
// maximum as v'_{j-1} + max(v_j - a - v'_{j-1}, 0): three-input adds and a sign
// mask instead of a two-word compare and two selects.  Every state is at
// least kFixNegInf and below 2^62, so no difference overflows.
__device__ __forceinline__ void tandem_step(long long& v1, long long& v2, long long& v3, long long a, long long s1,
                                            long long s2, long long s3) {
    v1 = relu64(v1 - a) + s1;
    v2 = v1 + s2 + relu64(v2 - a - v1);
    v3 = v2 + s3 + relu64(v3 - a - v2);
}

// Five CTAs per SM (96 registers, nothing spilled): 121.2 ms for 4,096 x 256
// replications of 10,000 clients against 124.1, 122.2, 122.1 and 122.7 at 4, 6, 7 and
// 8 (104 bytes spilled).
template <bool kLane0Only>
__global__ void __launch_bounds__(128, 5) tandem3_serial_kernel(const double* __restrict__ dps, long long n_items,
                                      long long n_reps, long long rep0, long long n_clients,
                                      long long window, uint32_t tag,
                                      const __grid_constant__ RoundKeys rk, LogTable tab,
                                      TandemOut out) {
    __shared__ unsigned long long nln2[kLogExponents];
    stage_nln2(tab, nln2);
    long long item;
    if (kLane0Only) {
        if ((threadIdx.x & 31) != 0) return;
        item = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) >> 5;
    } else {
        item = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    }
    if (item >= n_items) return;
    const uint32_t dp = static_cast<uint32_t>(item / n_reps);
    const uint32_t rep = static_cast<uint32_t>(rep0 + item % n_reps);
    const double lam = dps[4 * dp], mu1 = dps[4 * dp + 1], mu2 = dps[4 * dp + 2],
                 mu3 = dps[4 * dp + 3];
    const double i_lam = 0x1p-58 / lam, i_mu1 = 0x1p-58 / mu1, i_mu2 = 0x1p-58 / mu2,
                 i_mu3 = 0x1p-58 / mu3;
    const RowKey row = row_key(rep, stream_word(tag, dp), rk);
    const long long w_len = (n_clients < window) ? n_clients : window;
    double sum_y = 0.0, sum_a = 0.0, sum_1 = 0.0, sum_2 = 0.0, sum_3 = 0.0;
    bool fixed_done = false;
    if (fix_rate_ok(lam) && fix_rate_ok(mu1) && fix_rate_ok(mu2) && fix_rate_ok(mu3)) {
        const unsigned long long fl = fix_scale(lam), f1 = fix_scale(mu1), f2 = fix_scale(mu2),
                                 f3 = fix_scale(mu3);
        long long v1 = kFixNegInf, v2 = kFixNegInf, v3 = kFixNegInf;
        U96 sy;
        double wa = 0.0, w1 = 0.0, w2 = 0.0, w3 = 0.0;
        bool overflow = false;
        // client n's four log values; then one step of the recurrence
        auto logs = [&](uint32_t n, unsigned long long& ya, unsigned long long& y1, unsigned long long& y2,
                        unsigned long long& y3) {
            uint4 b0, b1;
            philox_row2(row, n, rk, b0, b1);
            ya = neg_log_q58<true>(b0.x, b0.y, tab);
            y1 = neg_log_q58<true>(b0.z, b0.w, tab);
            y2 = neg_log_q58<true>(b1.x, b1.y, tab);
            y3 = neg_log_q58<true>(b1.z, b1.w, tab);
        };
        auto step = [&](unsigned long long ya, unsigned long long y1, unsigned long long y2,
                        unsigned long long y3) {
            tandem_step(v1, v2, v3, to_fix(ya, fl), to_fix(y1, f1), to_fix(y2, f2), to_fix(y3, f3));
            sy.add(v3);
            return v3 < kFixGuard;
        };
        // the early window also sums the same variates as doubles (expo_fast);
        // the loop after it carries none of that state.  Client indices are
        // 32-bit (n_clients < 2^32, the counter word c1).
        const uint32_t nc = static_cast<uint32_t>(n_clients), nw = static_cast<uint32_t>(w_len);
        uint32_t n = 0;
        for (; n < nw; ++n) {
            unsigned long long ya, y1, y2, y3;
            logs(n, ya, y1, y2, y3);
            wa += __ull2double_rn(ya) * i_lam;
            w1 += __ull2double_rn(y1) * i_mu1;
            w2 += __ull2double_rn(y2) * i_mu2;
            w3 += __ull2double_rn(y3) * i_mu3;
            if (!step(ya, y1, y2, y3)) {
                overflow = true;
                break;
            }
        }
        for (; !overflow && n < nc; ++n) {
            unsigned long long ya, y1, y2, y3;
            logs(n, ya, y1, y2, y3);
            if (!step(ya, y1, y2, y3)) overflow = true;
        }
        if (!overflow) {
            fixed_done = true;
            sum_y = sy.to_double();
            sum_a = wa;
            sum_1 = w1;
            sum_2 = w2;
            sum_3 = w3;
        }
    }
    double v1 = -INFINITY, v2 = -INFINITY, v3 = -INFINITY;
    for (long long n = 0; !fixed_done && n < n_clients; ++n) {
        uint4 b0, b1;
        philox_row2(row, static_cast<uint32_t>(n), rk, b0, b1);
        const double a = expo_fast<true>(b0.x, b0.y, tab, i_lam);
        const double s1 = expo_fast<true>(b0.z, b0.w, tab, i_mu1);
        const double s2 = expo_fast<true>(b1.x, b1.y, tab, i_mu2);
        const double s3 = expo_fast<true>(b1.z, b1.w, tab, i_mu3);
        double q = v1 - a;
        v1 = ((q > 0.0) ? q : 0.0) + s1;
        q = v2 - a;
        v2 = ((q > v1) ? q : v1) + s2;
        q = v3 - a;
        v3 = ((q > v2) ? q : v2) + s3;
        sum_y += v3;
        if (n < w_len) {
            sum_a += a;
            sum_1 += s1;
            sum_2 += s2;
            sum_3 += s3;
        }
    }
    out.y[item] = sum_y / static_cast<double>(n_clients);
    if (out.feat) {
        const double wl = static_cast<double>(w_len);
        double* f = out.feat + item;
        const long long p = out.plane;
        f[0] = lam;
        f[p] = mu1;
        f[2 * p] = mu2;
        f[3 * p] = mu3;
        f[4 * p] = sum_a / wl;
        f[5 * p] = sum_1 / wl;
        f[6 * p] = sum_2 / wl;
        f[7 * p] = sum_3 / wl;
    }
}

// Tandem, one warp per replication.  One client maps the arrival-relative
// state v = (v1, v2, v3) to v'_j = max(v_j - A, v'_{j-1}) + S_j (v'_0 = 0),
// a max-plus affine map with a lower-triangular matrix:
//   v'_j = max(c_j, max_{k <= j} (v_k + d_jk)).
// Maps compose (TMap below), so a warp scan over the lanes' segment maps gives
// each segment's entry state (the composed map applied to the empty state,
// i.e. its constant terms c); every lane then replays its segment with the
// plain recurrence, as the serial kernel does.
struct TMap {
    double c1, c2, c3, d11, d21, d22, d31, d32, d33;
};

__device__ __forceinline__ TMap tmap_identity() {
    return TMap{-INFINITY, -INFINITY, -INFINITY, 0.0, -INFINITY, 0.0, -INFINITY, -INFINITY, 0.0};
}

__device__ __forceinline__ double dmax(double x, double y) { return x > y ? x : y; }

// f followed by one client (a, s1, s2, s3)
__device__ __forceinline__ TMap tmap_push(const TMap& f, double a, double s1, double s2, double s3) {
    const double e1 = s1 - a, e2 = s2 - a, e3 = s3 - a;
    TMap r;
    r.c1 = dmax(s1, f.c1 + e1);
    r.d11 = f.d11 + e1;
    r.c2 = dmax(f.c2 + e2, r.c1 + s2);
    r.d21 = dmax(f.d21 + e2, r.d11 + s2);
    r.d22 = f.d22 + e2;
    r.c3 = dmax(f.c3 + e3, r.c2 + s3);
    r.d31 = dmax(f.d31 + e3, r.d21 + s3);
    r.d32 = dmax(f.d32 + e3, r.d22 + s3);
    r.d33 = f.d33 + e3;
    return r;
}

// g after f
__device__ __forceinline__ TMap tmap_compose(const TMap& f, const TMap& g) {
    TMap h;
    h.c1 = dmax(g.c1, f.c1 + g.d11);
    h.c2 = dmax(g.c2, dmax(f.c1 + g.d21, f.c2 + g.d22));
    h.c3 = dmax(g.c3, dmax(f.c1 + g.d31, dmax(f.c2 + g.d32, f.c3 + g.d33)));
    h.d11 = f.d11 + g.d11;
    h.d21 = dmax(f.d11 + g.d21, f.d21 + g.d22);
    h.d22 = f.d22 + g.d22;
    h.d31 = dmax(f.d11 + g.d31, dmax(f.d21 + g.d32, f.d31 + g.d33));
    h.d32 = dmax(f.d22 + g.d32, f.d32 + g.d33);
    h.d33 = f.d33 + g.d33;
    return h;
}

__device__ __forceinline__ TMap tmap_shfl_up(const TMap& m, int off) {
    TMap r;
    r.c1 = __shfl_up_sync(kFull, m.c1, off);
    r.c2 = __shfl_up_sync(kFull, m.c2, off);
    r.c3 = __shfl_up_sync(kFull, m.c3, off);
    r.d11 = __shfl_up_sync(kFull, m.d11, off);
    r.d21 = __shfl_up_sync(kFull, m.d21, off);
    r.d22 = __shfl_up_sync(kFull, m.d22, off);
    r.d31 = __shfl_up_sync(kFull, m.d31, off);
    r.d32 = __shfl_up_sync(kFull, m.d32, off);
    r.d33 = __shfl_up_sync(kFull, m.d33, off);
    return r;
}

struct TandemClient {
    double a, s1, s2, s3;
};

__device__ __forceinline__ TandemClient tandem_client(uint32_t n, const RowKey& row, const RoundKeys& rk, const LogTable& tab,
                                                      double i_lam, double i_mu1, double i_mu2,
                                                      double i_mu3) {
    uint4 b0, b1;
    philox_row2(row, n, rk, b0, b1);
    return TandemClient{expo_fast<false>(b0.x, b0.y, tab, i_lam), expo_fast<false>(b0.z, b0.w, tab, i_mu1),
                        expo_fast<false>(b1.x, b1.y, tab, i_mu2), expo_fast<false>(b1.z, b1.w, tab, i_mu3)};
}

// The same maps in 48-bit fixed point, every sum saturated at +-2^61 (the
// empty state's -inf is -2^61).  After one client every constant is positive,
// so a term pushed down to -2^61 never decides a maximum for states in
// [0, 2^60]; a state or constant past 2^60 sends the replication to FP64.
struct FTMap {
    long long c1, c2, c3, d11, d21, d22, d31, d32, d33;
};

__device__ __forceinline__ FTMap ftmap_identity() {
    return FTMap{-kSat, -kSat, -kSat, 0, -kSat, 0, -kSat, -kSat, 0};
}

__device__ __forceinline__ long long lmax(long long x, long long y) { return x > y ? x : y; }

// f followed by one client, without saturation: each of the nine grows or
// shrinks by less than four variates.
__device__ __forceinline__ FTMap ftmap_push(const FTMap& f, long long a, long long s1, long long s2, long long s3) {
    const long long e1 = s1 - a, e2 = s2 - a, e3 = s3 - a;
    FTMap r;
    r.c1 = lmax(s1, f.c1 + e1);
    r.d11 = f.d11 + e1;
    r.c2 = lmax(f.c2 + e2, r.c1 + s2);
    r.d21 = lmax(f.d21 + e2, r.d11 + s2);
    r.d22 = f.d22 + e2;
    r.c3 = lmax(f.c3 + e3, r.c2 + s3);
    r.d31 = lmax(f.d31 + e3, r.d21 + s3);
    r.d32 = lmax(f.d32 + e3, r.d22 + s3);
    r.d33 = f.d33 + e3;
    return r;
}

__device__ __forceinline__ void ftmap_saturate(FTMap& f) {
    f.c1 = sat61(f.c1);
    f.c2 = sat61(f.c2);
    f.c3 = sat61(f.c3);
    f.d11 = sat61(f.d11);
    f.d21 = sat61(f.d21);
    f.d22 = sat61(f.d22);
    f.d31 = sat61(f.d31);
    f.d32 = sat61(f.d32);
    f.d33 = sat61(f.d33);
}

// Clients between two saturations.  A variate is below 36.8 / rate time units:
// for rates of at least 1/4 that is 2^55.3 units of 2^-48, so 8 clients move a
// saturated map by less than 2^60.3 and nothing leaves 63 bits; for the
// slowest rates (2^-6) it is 2^59.3 and every client saturates.  (16 replications x
// 100,000 clients on 64 SMs: 134.8 us, 143.7 when every client saturates.)
__device__ __forceinline__ uint32_t saturation_mask(double r0, double r1, double r2, double r3) {
    return fmin(fmin(r0, r1), fmin(r2, r3)) >= 0.25 ? 7u : 0u;
}

// State after the clients of f, from state v.
__device__ __forceinline__ void ftmap_apply(const FTMap& f, long long& v1, long long& v2, long long& v3) {
    const long long w1 = lmax(f.c1, sat61(v1 + f.d11));
    const long long w2 = lmax(f.c2, sat61(lmax(v1 + f.d21, v2 + f.d22)));
    const long long w3 = lmax(f.c3, sat61(lmax(v1 + f.d31, lmax(v2 + f.d32, v3 + f.d33))));
    v1 = w1;
    v2 = w2;
    v3 = w3;
}

__device__ __forceinline__ FTMap ftmap_compose(const FTMap& f, const FTMap& g) {  // g after f
    FTMap h;
    h.c1 = lmax(g.c1, sat61(f.c1 + g.d11));
    h.c2 = lmax(g.c2, sat61(lmax(f.c1 + g.d21, f.c2 + g.d22)));
    h.c3 = lmax(g.c3, sat61(lmax(f.c1 + g.d31, lmax(f.c2 + g.d32, f.c3 + g.d33))));
    h.d11 = sat61(f.d11 + g.d11);
    h.d21 = sat61(lmax(f.d11 + g.d21, f.d21 + g.d22));
    h.d22 = sat61(f.d22 + g.d22);
    h.d31 = sat61(lmax(f.d11 + g.d31, lmax(f.d21 + g.d32, f.d31 + g.d33)));
    h.d32 = sat61(lmax(f.d22 + g.d32, f.d32 + g.d33));
    h.d33 = sat61(f.d33 + g.d33);
    return h;
}

__device__ __forceinline__ FTMap ftmap_shfl_up(const FTMap& m, int off) {
    FTMap r;
    r.c1 = __shfl_up_sync(kFull, m.c1, off);
    r.c2 = __shfl_up_sync(kFull, m.c2, off);
    r.c3 = __shfl_up_sync(kFull, m.c3, off);
    r.d11 = __shfl_up_sync(kFull, m.d11, off);
    r.d21 = __shfl_up_sync(kFull, m.d21, off);
    r.d22 = __shfl_up_sync(kFull, m.d22, off);
    r.d31 = __shfl_up_sync(kFull, m.d31, off);
    r.d32 = __shfl_up_sync(kFull, m.d32, off);
    r.d33 = __shfl_up_sync(kFull, m.d33, off);
    return r;
}

// FP64 warp scan of one replication (the fallback of the fixed-point paths):
// lane l takes the l-th of 32 contiguous client segments.
__device__ void tandem_coop_fp64(long long item, double lam, double mu1, double mu2,
                                 double mu3, long long n_clients, long long window, const RowKey& row,
                                 const RoundKeys& rk, const LogTable& tab, const TandemOut& out) {
        const int lane = threadIdx.x & 31;
    const double i_lam = 0x1p-58 / lam, i_mu1 = 0x1p-58 / mu1, i_mu2 = 0x1p-58 / mu2, i_mu3 = 0x1p-58 / mu3;
    const long long w_len = (n_clients < window) ? n_clients : window;
    const long long seg = (n_clients + 31) / 32;
    const long long lo = min(lane * seg, n_clients);
    const long long hi = min(lo + seg, n_clients);
    // pass 1: this segment's map
    TMap f = tmap_identity();
    for (long long n = lo; n < hi; ++n) {
        const TandemClient k = tandem_client(static_cast<uint32_t>(n), row, rk, tab, i_lam, i_mu1, i_mu2, i_mu3);
        f = tmap_push(f, k.a, k.s1, k.s2, k.s3);
    }
    // inclusive scan over lanes, then the previous lane's prefix is the entry map
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const TMap prev = tmap_shfl_up(f, off);
        if (lane >= off) f = tmap_compose(prev, f);
    }
    const TMap excl = tmap_shfl_up(f, 1);
    double v1 = -INFINITY, v2 = -INFINITY, v3 = -INFINITY;
    if (lane > 0) {
        v1 = excl.c1;
        v2 = excl.c2;
        v3 = excl.c3;
    }

    // pass 2: replay the segment with the plain recurrence
    double sum_y = 0.0, sum_a = 0.0, sum_1 = 0.0, sum_2 = 0.0, sum_3 = 0.0;
    for (long long n = lo; n < hi; ++n) {
        const TandemClient k = tandem_client(static_cast<uint32_t>(n), row, rk, tab, i_lam, i_mu1, i_mu2, i_mu3);
        double q = v1 - k.a;
        v1 = ((q > 0.0) ? q : 0.0) + k.s1;
        q = v2 - k.a;
        v2 = ((q > v1) ? q : v1) + k.s2;
        q = v3 - k.a;
        v3 = ((q > v2) ? q : v2) + k.s3;
        sum_y += v3;
        if (n < w_len) {
            sum_a += k.a;
            sum_1 += k.s1;
            sum_2 += k.s2;
            sum_3 += k.s3;
        }
    }
    // fixed-order (lane-ordered tree) reduction
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double oy = __shfl_down_sync(kFull, sum_y, off);
        const double oa = __shfl_down_sync(kFull, sum_a, off);
        const double o1 = __shfl_down_sync(kFull, sum_1, off);
        const double o2 = __shfl_down_sync(kFull, sum_2, off);
        const double o3 = __shfl_down_sync(kFull, sum_3, off);
        if ((lane & (2 * off - 1)) == 0) {
            sum_y += oy;
            sum_a += oa;
            sum_1 += o1;
            sum_2 += o2;
            sum_3 += o3;
        }
    }
    if (lane != 0) return;
    out.y[item] = sum_y / static_cast<double>(n_clients);
    if (out.feat) {
        const double wl = static_cast<double>(w_len);
        double* fo = out.feat + item;
        const long long p = out.plane;
        fo[0] = lam;
        fo[p] = mu1;
        fo[2 * p] = mu2;
        fo[3 * p] = mu3;
        fo[4 * p] = sum_a / wl;
        fo[5 * p] = sum_1 / wl;
        fo[6 * p] = sum_2 / wl;
        fo[7 * p] = sum_3 / wl;
    }
}

__global__ void __launch_bounds__(128) tandem3_warp_coop_kernel(
    const double* __restrict__ dps, long long n_items, long long n_reps, long long rep0,
    long long n_clients, long long window, uint32_t tag, const __grid_constant__ RoundKeys rk,
    LogTable tab, TandemOut out) {
    const int lane = threadIdx.x & 31;
    const long long item = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) >> 5;
    if (item >= n_items) return;  // warp-uniform
    const uint32_t dp = static_cast<uint32_t>(item / n_reps);
    const uint32_t rep = static_cast<uint32_t>(rep0 + item % n_reps);
    const double lam = dps[4 * dp], mu1 = dps[4 * dp + 1], mu2 = dps[4 * dp + 2], mu3 = dps[4 * dp + 3];
    const double i_lam = 0x1p-58 / lam, i_mu1 = 0x1p-58 / mu1, i_mu2 = 0x1p-58 / mu2,
                 i_mu3 = 0x1p-58 / mu3;
    const RowKey row = row_key(rep, stream_word(tag, dp), rk);
    const long long w_len = (n_clients < window) ? n_clients : window;
    const long long seg = (n_clients + 31) / 32;
    const long long lo = min(lane * seg, n_clients);
    const long long hi = min(lo + seg, n_clients);

    if (fix_rate_ok(lam) && fix_rate_ok(mu1) && fix_rate_ok(mu2) && fix_rate_ok(mu3)) {
        const unsigned long long cl = fix_scale(lam), c1 = fix_scale(mu1), c2 = fix_scale(mu2),
                                 c3f = fix_scale(mu3);
        FTMap f = ftmap_identity();
        const uint32_t every = saturation_mask(lam, mu1, mu2, mu3);
        for (long long n = lo; n < hi; ++n) {
            uint4 b0, b1;
            philox_row2(row, static_cast<uint32_t>(n), rk, b0, b1);
            f = ftmap_push(f, to_fix(neg_log_q58<false>(b0.x, b0.y, tab), cl),
                           to_fix(neg_log_q58<false>(b0.z, b0.w, tab), c1),
                           to_fix(neg_log_q58<false>(b1.x, b1.y, tab), c2),
                           to_fix(neg_log_q58<false>(b1.z, b1.w, tab), c3f));
            if ((static_cast<uint32_t>(n - lo) & every) == every) ftmap_saturate(f);
        }
        ftmap_saturate(f);
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const FTMap prev = ftmap_shfl_up(f, off);
            if (lane >= off) f = ftmap_compose(prev, f);
        }
        const FTMap excl = ftmap_shfl_up(f, 1);
        long long v1 = kFixNegInf, v2 = kFixNegInf, v3 = kFixNegInf;
        if (lane > 0) {
            v1 = excl.c1;
            v2 = excl.c2;
            v3 = excl.c3;
        }
        bool bad = v3 >= kFixGuard;
        U96 sy;
        double wa = 0.0, w1 = 0.0, w2 = 0.0, w3 = 0.0;
        for (long long n = lo; n < hi && !bad; ++n) {
            uint4 b0, b1;
            philox_row2(row, static_cast<uint32_t>(n), rk, b0, b1);
            const unsigned long long ya = neg_log_q58<false>(b0.x, b0.y, tab);
            const unsigned long long y1 = neg_log_q58<false>(b0.z, b0.w, tab);
            const unsigned long long y2 = neg_log_q58<false>(b1.x, b1.y, tab);
            const unsigned long long y3 = neg_log_q58<false>(b1.z, b1.w, tab);
            tandem_step(v1, v2, v3, to_fix(ya, cl), to_fix(y1, c1), to_fix(y2, c2), to_fix(y3, c3f));
            sy.add(v3);
            if (n < w_len) {
                wa += __ull2double_rn(ya) * i_lam;
                w1 += __ull2double_rn(y1) * i_mu1;
                w2 += __ull2double_rn(y2) * i_mu2;
                w3 += __ull2double_rn(y3) * i_mu3;
            }
            bad = v3 >= kFixGuard;
        }
        if (!__any_sync(kFull, bad)) {
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {  // lane-ordered tree (integers: exact)
                const U96 oy = shfl_down_u96(sy, off);
                const double oa = __shfl_down_sync(kFull, wa, off);
                const double o1 = __shfl_down_sync(kFull, w1, off);
                const double o2 = __shfl_down_sync(kFull, w2, off);
                const double o3 = __shfl_down_sync(kFull, w3, off);
                if ((lane & (2 * off - 1)) == 0) {
                    add_u96(sy, oy);
                    wa += oa;
                    w1 += o1;
                    w2 += o2;
                    w3 += o3;
                }
            }
            if (lane != 0) return;
            out.y[item] = sy.to_double() / static_cast<double>(n_clients);
            if (out.feat) {
                const double wl = static_cast<double>(w_len);
                double* fo = out.feat + item;
                const long long p = out.plane;
                fo[0] = lam;
                fo[p] = mu1;
                fo[2 * p] = mu2;
                fo[3 * p] = mu3;
                fo[4 * p] = wa / wl;
                fo[5 * p] = w1 / wl;
                fo[6 * p] = w2 / wl;
                fo[7 * p] = w3 / wl;
            }
            return;
        }
    }

    // FP64
    tandem_coop_fp64(item, lam, mu1, mu2, mu3, n_clients, window, row, rk, tab, out);
}

// ---------------------------------------------------------------------------
// M/M/1, one replication per CTA or cluster of CTAs (few replications of a
// latency-bound length; cta_shape): thread i takes the contiguous clients
// [i k, (i+1) k).  Pass 1
// composes each thread's Lindley maps W -> max(c, W + d); a block scan (warp
// shuffles, then the warp totals in shared memory) gives every thread the
// map of all clients before it, whose value at W_0 = 0 is its entry wait;
// in a cluster the maps of the earlier CTAs, read over distributed shared
// memory, carry W_0 = 0 to the CTA's first client (14 replications x 100,003
// clients 201 -> 41 us, 32 x 10,000 36 -> 14.5 us);
// pass 2 replays the thread's clients with the plain recurrence.  Times run
// in the 48-bit fixed point of the tandem, so composition is exact and the
// sums are exact integers (order-free); c and d saturate at +-2^61, which
// changes no map value for waits in [0, 2^60] unless a wait passes 2^60 --
// then, or for rates outside [2^-6, 2^4], the CTA redoes the replication in
// FP64 with the same structure (maps with -inf, sums in a fixed tree).
// ---------------------------------------------------------------------------

struct FixMap {
    long long c, d;
};
__device__ __forceinline__ FixMap fcompose(const FixMap& f, const FixMap& g) {  // g after f
    const long long cc = sat61(f.c + g.d);
    return FixMap{g.c > cc ? g.c : cc, sat61(f.d + g.d)};
}
struct DblMap {
    double c, d;
};
__device__ __forceinline__ DblMap dcompose(const DblMap& f, const DblMap& g) {
    const double cc = f.c + g.d;
    return DblMap{g.c > cc ? g.c : cc, f.d + g.d};
}

template <class Map>
__device__ __forceinline__ Map shfl_up_map(const Map& m, int off) {
    return Map{__shfl_up_sync(kFull, m.c, off), __shfl_up_sync(kFull, m.d, off)};
}

// Exclusive block scan of per-thread maps (thread order); `identity` for
// thread 0.  smem: one Map per warp.  *total (by the last thread): all of them.
template <class Map, class Compose>
__device__ Map block_exclusive_map(Map f, Map identity, Map* smem, Map* total, Compose compose) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Map incl = f;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const Map prev = shfl_up_map(incl, off);
        if (lane >= off) incl = compose(prev, incl);
    }
    if (lane == 31) smem[warp] = incl;
    __syncthreads();
    Map before = identity;  // maps of the earlier warps, composed in order
    for (int w = 0; w < warp; ++w) before = compose(before, smem[w]);
    if (threadIdx.x == blockDim.x - 1) *total = compose(before, incl);
    Map excl = shfl_up_map(incl, 1);
    if (lane == 0) excl = identity;
    __syncthreads();  // smem reusable
    return compose(before, excl);
}

struct Mm1Sums {
    U96 w, i, v;
};


// Clients whose variates are drawn together, before the two multipliers of the
// rates are needed (FP64 divisions on a slow pipe: two lanes of the last warp,
// which has the fewest clients, compute them meanwhile for all), and the most
// threads per CTA.  32 x 10,000 clients 20.9 -> 14.5 us, 1,024 x 1,000 26.7 -> 20.6, 14
// x 100,003 47.2 -> 41.1; one client at a time 18.3, 22.0, 43.1; up to 1,024 threads
// 18.4, 20.6, 42.8; 256 14.5, 20.6, 53.1.
constexpr int kMm1CtaGroup = 2, kMm1CtaThreads = 512;

template <bool kCluster>
__global__ void __launch_bounds__(kMm1CtaThreads) mm1_cta_kernel(
    const double* __restrict__ dps, long long n_reps, long long rep0, long long n_clients, bool staged,
    const __grid_constant__ RoundKeys rk, LogTable tab, Mm1Out out) {
    namespace cg = cooperative_groups;
    extern __shared__ long long fix_stage[];  // [client - lo][thread] x (S, A) when staged
    __shared__ FixMap fmaps[32];
    __shared__ DblMap dmaps[32];
    __shared__ U96 part[3][32];
    __shared__ double dpart[3][32];
    __shared__ DblMap dtotal;
    __shared__ unsigned long long scale[2];
    __shared__ struct {
        FixMap map;  // all clients of this CTA
        U96 sum[3];
        int bad;
    } mine;
    cg::cluster_group cluster = cg::this_cluster();
    const int ctas = kCluster ? static_cast<int>(cluster.num_blocks()) : 1;
    const int rank = kCluster ? static_cast<int>(cluster.block_rank()) : 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const long long item = blockIdx.x / ctas;
    const uint32_t dp = static_cast<uint32_t>(item / n_reps);
    const uint32_t rep = static_cast<uint32_t>(rep0 + item % n_reps);
    const double lam = dps[2 * dp], mu = dps[2 * dp + 1];
    const RowKey row = row_key(rep, stream_word(0u, dp), rk);
    const long long threads = static_cast<long long>(ctas) * blockDim.x;
    const long long k = (n_clients + threads - 1) / threads;
    long long lo = min((static_cast<long long>(rank) * blockDim.x + threadIdx.x) * k, n_clients);
    long long hi = min(lo + k, n_clients);
    const double inv_n = static_cast<double>(n_clients);
    // (debug build: a stage larger than the launch's shared memory is
    // recorded and the variates recomputed)
    staged = staged && MRIP_CHECK(2ull * k * blockDim.x * sizeof(long long) <= dynamic_smem_bytes(), 202, k);

    bool fixed_ok = fix_rate_ok(lam) && fix_rate_ok(mu);
    if (fixed_ok) {
        FixMap f{-kSat, 0};
        long long* st_s = fix_stage + threadIdx.x;
        long long* st_a = fix_stage + k * blockDim.x + threadIdx.x;
        unsigned long long cl = 0, cmu = 0, ys[kMm1CtaGroup], ya[kMm1CtaGroup];
        auto draw = [&](long long n0) {
#pragma unroll
            for (int g = 0; g < kMm1CtaGroup; ++g) {
                const uint4 b = philox_row(row, static_cast<uint32_t>(n0 + g), rk);
                ys[g] = neg_log_q58<false>(b.x, b.y, tab);
                ya[g] = neg_log_q58<false>(b.z, b.w, tab);
            }
        };
        auto use = [&](long long n, unsigned long long s58, unsigned long long a58) {
            const long long sv = to_fix(s58, cmu);
            const long long av = to_fix(a58, cl);
            if (staged) {
                st_s[(n - lo) * blockDim.x] = sv;
                st_a[(n - lo) * blockDim.x] = av;
            }
            f = fcompose(f, FixMap{0, sv - av});
        };
        const bool whole = lo + kMm1CtaGroup <= hi;
        if (warp == nwarp - 1 && lane < 2) scale[lane] = fix_scale(lane == 0 ? lam : mu);
        if (whole) draw(lo);
        __syncthreads();
        cl = scale[0];
        cmu = scale[1];
        long long n0 = lo;
        if (whole) {
#pragma unroll
            for (int g = 0; g < kMm1CtaGroup; ++g) use(lo + g, ys[g], ya[g]);
            n0 += kMm1CtaGroup;
            for (; n0 + kMm1CtaGroup <= hi; n0 += kMm1CtaGroup) {
                draw(n0);
#pragma unroll
                for (int g = 0; g < kMm1CtaGroup; ++g) use(n0 + g, ys[g], ya[g]);
            }
        }
        for (; n0 < hi; ++n0) {
            const uint4 b = philox_row(row, static_cast<uint32_t>(n0), rk);
            use(n0, neg_log_q58<false>(b.x, b.y, tab), neg_log_q58<false>(b.z, b.w, tab));
        }
        const FixMap pre = block_exclusive_map(f, FixMap{-kSat, 0}, fmaps, &mine.map, fcompose);
        long long w = 0;  // W_0
        if constexpr (kCluster) {
            cluster.sync();
            for (int r = 0; r < rank; ++r) {
                const FixMap e = *cluster.map_shared_rank(&mine.map, r);
                w = max(e.c, sat61(w + e.d));
            }
        }
        if (threadIdx.x > 0) w = max(pre.c, sat61(w + pre.d));
        bool bad = w >= kFixGuard;
        Mm1Sums sm;
        for (long long n = lo; n < hi && !bad; ++n) {
            long long sv, av;
            if (staged) {
                sv = st_s[(n - lo) * blockDim.x];
                av = st_a[(n - lo) * blockDim.x];
            } else {
                const uint4 b = philox_row(row, static_cast<uint32_t>(n), rk);
                sv = to_fix(neg_log_q58<false>(b.x, b.y, tab), cmu);
                av = to_fix(neg_log_q58<false>(b.z, b.w, tab), cl);
            }
            sm.w.add(w);
            const long long v = w + sv;
            sm.v.add(v);
            const long long t = v - av;
            w = relu64(t);
            sm.i.add(w - t);  // max(0, -t)
            bad = w >= kFixGuard;
        }
        const bool cta_bad = __syncthreads_or(bad) != 0;
        fixed_ok = !cta_bad;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            add_u96(sm.w, shfl_down_u96(sm.w, off));
            add_u96(sm.i, shfl_down_u96(sm.i, off));
            add_u96(sm.v, shfl_down_u96(sm.v, off));
        }
        if (lane == 0) {
            part[0][warp] = sm.w;
            part[1][warp] = sm.i;
            part[2][warp] = sm.v;
        }
        __syncthreads();
        U96 tot;
        if (threadIdx.x < 3)
            for (int x = 0; x < nwarp; ++x) add_u96(tot, part[threadIdx.x][x]);
        if constexpr (kCluster) {
            if (threadIdx.x < 3) mine.sum[threadIdx.x] = tot;
            if (threadIdx.x == 0) mine.bad = cta_bad ? 1 : 0;
            cluster.sync();
            if (rank == 0) {
                for (int r = 1; r < ctas; ++r) {
                    fixed_ok = fixed_ok && *cluster.map_shared_rank(&mine.bad, r) == 0;
                    if (threadIdx.x < 3) add_u96(tot, cluster.map_shared_rank(&mine.sum[0], r)[threadIdx.x]);
                }
            }
            cluster.sync();  // the first CTA has read the others' shared memory
        }
        if (rank != 0) return;
        if (fixed_ok) {
            if (threadIdx.x < 3) {
                double* dst = threadIdx.x == 0 ? out.wait : threadIdx.x == 1 ? out.idle : out.system;
                if (dst) dst[item] = tot.to_double() / inv_n;
            }
            return;
        }
    }
    if (rank != 0) return;
    // FP64: the same passes with doubles, by the first CTA alone
    const long long k1 = (n_clients + blockDim.x - 1) / blockDim.x;
    lo = min(static_cast<long long>(threadIdx.x) * k1, n_clients);
    hi = min(lo + k1, n_clients);
    const double inv_lam = 0x1p-58 / lam, inv_mu = 0x1p-58 / mu;
    DblMap f{-INFINITY, 0.0};
    for (long long n = lo; n < hi; ++n) {
        double sv, av;
        mm1_client<false>(static_cast<uint32_t>(n), row, inv_lam, inv_mu, rk, tab, sv, av);
        f = dcompose(f, DblMap{0.0, sv - av});
    }
    const DblMap pre = block_exclusive_map(f, DblMap{-INFINITY, 0.0}, dmaps, &dtotal, dcompose);
    double w = pre.c > pre.d ? pre.c : pre.d;
    if (threadIdx.x == 0) w = 0.0;
    double sw = 0.0, si = 0.0, sv_sum = 0.0;
    for (long long n = lo; n < hi; ++n) {
        double sv, av;
        mm1_client<false>(static_cast<uint32_t>(n), row, inv_lam, inv_mu, rk, tab, sv, av);
        sw += w;
        const double v = w + sv;
        sv_sum += v;
        const double t = v - av;
        si += (t < 0.0) ? -t : 0.0;
        w = (t > 0.0) ? t : 0.0;
    }
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {  // lane-ordered tree
        const double ow = __shfl_down_sync(kFull, sw, off);
        const double oi = __shfl_down_sync(kFull, si, off);
        const double ov = __shfl_down_sync(kFull, sv_sum, off);
        if ((lane & (2 * off - 1)) == 0) {
            sw += ow;
            si += oi;
            sv_sum += ov;
        }
    }
    if (lane == 0) {
        dpart[0][warp] = sw;
        dpart[1][warp] = si;
        dpart[2][warp] = sv_sum;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double tot = 0.0;
        for (int x = 0; x < nwarp; ++x) tot += dpart[threadIdx.x][x];
        double* dst = threadIdx.x == 0 ? out.wait : threadIdx.x == 1 ? out.idle : out.system;
        if (dst) dst[item] = tot / inv_n;
    }
}

// ---------------------------------------------------------------------------
// Tandem, one replication per CTA or cluster of CTAs (few replications of a
// long horizon): thread i of the cluster takes the contiguous clients
// [i k, (i+1) k); its fixed-point max-plus map (FTMap) is composed in pass 1, a
// block scan (warp shuffles, then the warp totals in order) gives every thread
// the map of the CTA's clients before it, the maps of the earlier CTAs (read
// over distributed shared memory) applied to the empty state give the CTA's
// entry state, and pass 2 replays the thread's clients from there.  Sojourn
// sums are exact integers; the early-window sums FP64 in a fixed order.  Rates
// outside the fixed-point range or a sojourn past 2^12 hand the replication to
// the FP64 warp scan (the first CTA's warp 0).
//
// One CTA per replication leaves the SMs without one idle, so few replications
// are split over clusters of up to 8 CTAs (cta_shape): 16 x 100,000 clients run on
// 96 SMs instead of 16, 439 -> 102 us.  FP64 is kept to the warps that need it
// (its pipe takes a warp instruction every 16 cycles, however few lanes are
// active): the four multipliers by four lanes for the CTA, the reciprocals and
// the sums of the early window only in the warps that hold its clients: 90 us.
// At most 512 threads per CTA (16 x 100,000 at 512, 768 and 1,024 threads: 90, 98, 111;
// 33 replications x 50,021 clients 76, 84, 96: the scan grows with the warps); 256 where
// there are more replications than SMs and 128 where more than twice as many,
// so that several CTAs share one (333 x 5,021 clients at 128, 256, 384 threads: 85, 88,
// 109 us; 1,400 x 2,000: 115, 136, 221).  Two clients drawn together gain nothing
// (96 us: 16 warps of 128 registers hide the chains).
constexpr int kTandemThreads = 512;
template <bool kCluster>
__global__ void __launch_bounds__(kTandemThreads) tandem3_cta_kernel(const double* __restrict__ dps, long long n_reps,
                                                           long long rep0, long long n_clients, long long window,
                                                           uint32_t tag, const __grid_constant__ RoundKeys rk,
                                                           LogTable tab, TandemOut out) {
    namespace cg = cooperative_groups;
    __shared__ FTMap wmap[32];
    __shared__ U96 wy[32];
    __shared__ double wsum[4][32];
    __shared__ unsigned long long scale[4];
    __shared__ struct {
        FTMap map;     // all clients of this CTA
        U96 y;
        double sum[4];
        int bad;
    } mine;
    cg::cluster_group cluster = cg::this_cluster();
    const int ctas = kCluster ? static_cast<int>(cluster.num_blocks()) : 1;
    const int rank = kCluster ? static_cast<int>(cluster.block_rank()) : 0;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nwarp = blockDim.x >> 5;
    const long long item = blockIdx.x / ctas;
    const uint32_t dp = static_cast<uint32_t>(item / n_reps);
    const uint32_t rep = static_cast<uint32_t>(rep0 + item % n_reps);
    const double lam = dps[4 * dp], mu1 = dps[4 * dp + 1], mu2 = dps[4 * dp + 2], mu3 = dps[4 * dp + 3];
    const RowKey row = row_key(rep, stream_word(tag, dp), rk);
    const long long w_len = (n_clients < window) ? n_clients : window;
    const long long threads = static_cast<long long>(ctas) * blockDim.x;
    const long long k = (n_clients + threads - 1) / threads;
    const long long lo = min((static_cast<long long>(rank) * blockDim.x + t) * k, n_clients);
    const long long hi = min(lo + k, n_clients);

    if (fix_rate_ok(lam) && fix_rate_ok(mu1) && fix_rate_ok(mu2) && fix_rate_ok(mu3)) {
        // every thread needs the same four multipliers: one division each in
        // four lanes (FP64 is a slow pipe, and a warp occupies it as long as one lane)
        if (t < 4) scale[t] = fix_scale(t == 0 ? lam : t == 1 ? mu1 : t == 2 ? mu2 : mu3);
        __syncthreads();
        const unsigned long long cl = scale[0], c1 = scale[1], c2 = scale[2], c3f = scale[3];
        struct Draw {
            unsigned long long a, s1, s2, s3;
        };
        auto draw = [&](long long n) {
            uint4 b0, b1;
            philox_row2(row, static_cast<uint32_t>(n), rk, b0, b1);
            return Draw{neg_log_q58<false>(b0.x, b0.y, tab), neg_log_q58<false>(b0.z, b0.w, tab),
                        neg_log_q58<false>(b1.x, b1.y, tab), neg_log_q58<false>(b1.z, b1.w, tab)};
        };
        FTMap f = ftmap_identity();
        const uint32_t every = saturation_mask(lam, mu1, mu2, mu3);
        auto push = [&](long long n, const Draw& d) {
            f = ftmap_push(f, to_fix(d.a, cl), to_fix(d.s1, c1), to_fix(d.s2, c2), to_fix(d.s3, c3f));
            if ((static_cast<uint32_t>(n - lo) & every) == every) ftmap_saturate(f);
        };
        for (long long n = lo; n < hi; ++n) push(n, draw(n));
        ftmap_saturate(f);
        // block exclusive scan of the maps
        FTMap incl = f;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const FTMap prev = ftmap_shfl_up(incl, off);
            if (lane >= off) incl = ftmap_compose(prev, incl);
        }
        if (lane == 31) wmap[warp] = incl;
        __syncthreads();
        FTMap pre = ftmap_identity();
        for (int w = 0; w < warp; ++w) pre = ftmap_compose(pre, wmap[w]);
        if (kCluster && t == blockDim.x - 1) mine.map = ftmap_compose(pre, incl);
        FTMap excl = ftmap_shfl_up(incl, 1);
        if (lane == 0) excl = ftmap_identity();
        pre = ftmap_compose(pre, excl);
        long long v1 = -kSat, v2 = -kSat, v3 = -kSat;  // empty
        if constexpr (kCluster) {
            cluster.sync();
            for (int r = 0; r < rank; ++r) ftmap_apply(*cluster.map_shared_rank(&mine.map, r), v1, v2, v3);
        }
        ftmap_apply(pre, v1, v2, v3);
        bool bad = v3 >= kFixGuard;
        U96 sy;
        double wa = 0.0, w1 = 0.0, w2 = 0.0, w3 = 0.0;
        double i_lam = 0.0, i_mu1 = 0.0, i_mu2 = 0.0, i_mu3 = 0.0;
        const bool early = __any_sync(kFull, lo < w_len);  // the warp has clients of the early window
        if (early) {
            i_lam = 0x1p-58 / lam;
            i_mu1 = 0x1p-58 / mu1;
            i_mu2 = 0x1p-58 / mu2;
            i_mu3 = 0x1p-58 / mu3;
        }
        auto step = [&](long long n, const Draw& d) {
            tandem_step(v1, v2, v3, to_fix(d.a, cl), to_fix(d.s1, c1), to_fix(d.s2, c2), to_fix(d.s3, c3f));
            sy.add(v3);
            if (n < w_len) {
                wa += __ull2double_rn(d.a) * i_lam;
                w1 += __ull2double_rn(d.s1) * i_mu1;
                w2 += __ull2double_rn(d.s2) * i_mu2;
                w3 += __ull2double_rn(d.s3) * i_mu3;
            }
            bad = v3 >= kFixGuard;
        };
        for (long long n = lo; n < hi && !bad; ++n) step(n, draw(n));
        const bool cta_bad = __syncthreads_or(bad) != 0;
        bool any_bad = cta_bad;
        if (!cta_bad) {
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {  // lane-ordered tree (integers: exact)
                const U96 oy = shfl_down_u96(sy, off);
                if ((lane & (2 * off - 1)) == 0) add_u96(sy, oy);
            }
            if (early) {
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const double oa = __shfl_down_sync(kFull, wa, off);
                    const double o1 = __shfl_down_sync(kFull, w1, off);
                    const double o2 = __shfl_down_sync(kFull, w2, off);
                    const double o3 = __shfl_down_sync(kFull, w3, off);
                    if ((lane & (2 * off - 1)) == 0) {
                        wa += oa;
                        w1 += o1;
                        w2 += o2;
                        w3 += o3;
                    }
                }
            }
            if (lane == 0) {
                wy[warp] = sy;
                wsum[0][warp] = wa;
                wsum[1][warp] = w1;
                wsum[2][warp] = w2;
                wsum[3][warp] = w3;
            }
        }
        __syncthreads();
        if (t == 0) {
            U96 ty;
            double sum[4] = {0.0, 0.0, 0.0, 0.0};
            if (!cta_bad) {
                for (int w = 0; w < nwarp; ++w) {
                    add_u96(ty, wy[w]);
                    for (int q = 0; q < 4; ++q) sum[q] += wsum[q][w];
                }
            }
            mine.y = ty;
            for (int q = 0; q < 4; ++q) mine.sum[q] = sum[q];
            mine.bad = cta_bad ? 1 : 0;
        }
        if constexpr (kCluster) {
            cluster.sync();
            if (rank == 0)
                for (int r = 1; r < ctas; ++r) any_bad = any_bad || *cluster.map_shared_rank(&mine.bad, r) != 0;
        }
        if (rank == 0 && t == 0 && !any_bad) {
            U96 ty = mine.y;
            double sum[4] = {mine.sum[0], mine.sum[1], mine.sum[2], mine.sum[3]};
            for (int r = 1; r < ctas; ++r) {
                add_u96(ty, *cluster.map_shared_rank(&mine.y, r));
                for (int q = 0; q < 4; ++q) sum[q] += cluster.map_shared_rank(&mine.sum[0], r)[q];
            }
            out.y[item] = ty.to_double() / static_cast<double>(n_clients);
            if (out.feat) {
                const double wl = static_cast<double>(w_len);
                double* fo = out.feat + item;
                const long long p = out.plane;
                fo[0] = lam;
                fo[p] = mu1;
                fo[2 * p] = mu2;
                fo[3 * p] = mu3;
                for (int q = 0; q < 4; ++q) fo[(4 + q) * p] = sum[q] / wl;
            }
        }
        if constexpr (kCluster) cluster.sync();  // the first CTA has read the others' shared memory
        if (!any_bad) return;
    }
    if (rank == 0 && warp == 0)
        tandem_coop_fp64(item, lam, mu1, mu2, mu3, n_clients, window, row, rk, tab, out);
}

}  // namespace
}  // namespace mrip

namespace mrip {
namespace {

// Launch shape of a CTA-mapped queue kernel: CTAs per replication (a cluster),
// threads per CTA, dynamic shared memory.
struct CtaShape {
    unsigned ctas = 1, threads = 32;
    size_t smem = 0;
    bool staged = false;
};

void cluster_config(long long n_items, const CtaShape& s, cudaStream_t st, cudaLaunchConfig_t* cfg,
                    cudaLaunchAttribute* attr) {
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3(static_cast<unsigned>(n_items * s.ctas));
    cfg->blockDim = dim3(s.threads);
    cfg->dynamicSmemBytes = s.smem;
    cfg->stream = st;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = s.ctas;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg->attrs = attr;
    cfg->numAttrs = s.ctas > 1 ? 1 : 0;
}

// About 4 clients per thread, 32 .. `most` threads per CTA.  Where one CTA would
// leave its threads more than 4, the clients are split over the largest
// cluster of 2 .. 8 CTAs per replication that still leaves every replication
// running at once (the driver says how many clusters fit: on 152 SMs 36 of four
// CTAs with an SM each, 15 of eight).  stage: the
// variates of the first pass are kept in shared memory when they fit 96 KiB.
template <class Kernel>
mrip_status cta_shape(Kernel one, Kernel many, long long n_items, long long n_clients, int most, bool stage, CtaShape* out) {
    auto shape_of = [&](unsigned ctas) {
        CtaShape s;
        s.ctas = ctas;
        const long long part = (n_clients + ctas - 1) / ctas;
        const long long threads = ((part + 3) / 4 + 31) / 32 * 32;
        s.threads = static_cast<unsigned>(threads < 32 ? 32 : (threads > most ? most : threads));
        const long long all = static_cast<long long>(s.threads) * ctas;
        const size_t bytes = static_cast<size_t>(s.threads * ((n_clients + all - 1) / all)) * 2 * sizeof(long long);
        s.staged = stage && bytes <= 96 * 1024;
        s.smem = s.staged ? bytes : 0;
        return s;
    };
    *out = shape_of(1);
    const long long sms = sm_count();
    const long long wanted = std::min<long long>(8, (n_clients + 4ll * most - 1) / (4ll * most));
    for (unsigned ctas = static_cast<unsigned>(wanted); ctas > 1; --ctas) {
        if (n_items * ctas > sms) continue;
        const CtaShape s = shape_of(ctas);
        if (s.smem > 40 * 1024) {
            cudaError_t e = cudaFuncSetAttribute(many, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
            if (e != cudaSuccess) return cuda_status(e, "queues: shared memory attribute");
        }
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr;
        cluster_config(n_items, s, nullptr, &cfg, &attr);
        int fit = 0;
        if (cudaOccupancyMaxActiveClusters(&fit, many, &cfg) != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        if (fit >= n_items) {
            *out = s;
            return MRIP_OK;
        }
    }
    if (out->smem > 40 * 1024) {  // plus ~3.3 KB of static shared memory
        cudaError_t e = cudaFuncSetAttribute(one, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
        if (e != cudaSuccess) return cuda_status(e, "queues: shared memory attribute");
    }
    return MRIP_OK;
}

template <class... P, class... A>
mrip_status launch_ctas(void (*kernel)(P...), long long n_items, const CtaShape& s, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    cluster_config(n_items, s, st, &cfg, &attr);
    return cuda_status(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...), "queues: launch");
}

}  // namespace
}  // namespace mrip

using namespace mrip;

extern "C" mrip_status mrip_mm1_simulate(const double* d_dps, int32_t n_dp, int64_t rep0, int64_t n_reps,
                                         int64_t n_clients, uint64_t seed, int mapping,
                                         double* d_wait, double* d_idle, double* d_system,
                                         void* stream) {
    if (n_dp < 0 || n_reps < 0 || rep0 < 0 || n_clients < 1)
        return fail(MRIP_EINVAL, "mrip_mm1_simulate: need n_dp, n_reps, rep0 >= 0 and n_clients >= 1");
    if (n_dp >= (1 << 24) || rep0 + n_reps > 0x100000000ll || n_clients > 0xFFFFFFFFll)
        return fail(MRIP_EINVAL, "mrip_mm1_simulate: n_dp < 2^24, replication indices < 2^32, n_clients <= 2^32-1");
    const long long n_items = static_cast<long long>(n_dp) * n_reps;
    if (n_items == 0) return MRIP_OK;
    if (!d_dps) return fail(MRIP_EINVAL, "mrip_mm1_simulate: null design points");
    const RoundKeys rk = expand_key(seed);
    LogTable tab;
    mrip_status ts = log_table(&tab);
    if (ts != MRIP_OK) return ts;
    Mm1Out out{d_wait, d_idle, d_system};
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (mapping == MRIP_MAP_AUTO || mapping == MRIP_MAP_THREAD) {
        mm1_serial_kernel<false><<<ceil_div_u(n_items, 128), 128, 0, st>>>(
            d_dps, n_items, n_reps, rep0, n_clients, rk, tab, out);
    } else if (mapping == MRIP_MAP_WARP_1LANE) {
        mm1_serial_kernel<true><<<ceil_div_u(n_items * 32, 128), 128, 0, st>>>(
            d_dps, n_items, n_reps, rep0, n_clients, rk, tab, out);
    } else if (mapping == MRIP_MAP_CTA) {
        if (n_items > 0x7FFFFFFFll) return fail(MRIP_EINVAL, "mrip_mm1_simulate: too many replications for CTA");
        CtaShape shape;
        mrip_status cs = cta_shape(mm1_cta_kernel<false>, mm1_cta_kernel<true>, n_items, n_clients, kMm1CtaThreads,
                                   true, &shape);
        if (cs != MRIP_OK) return cs;
        cs = launch_ctas(shape.ctas > 1 ? mm1_cta_kernel<true> : mm1_cta_kernel<false>, n_items, shape, st, d_dps, static_cast<long long>(n_reps),
                         static_cast<long long>(rep0), static_cast<long long>(n_clients), shape.staged, rk, tab, out);
        if (cs != MRIP_OK) return cs;
    } else if (mapping == MRIP_MAP_WARP_COOP) {
        const long long seg = (n_clients + 31) / 32;
        const size_t per_warp = static_cast<size_t>(seg) * 32 * 2 * sizeof(double);
        // Staged where the slices leave an SM enough warps (24 KB: nine) or all of its
        // replications fit it at once; else the second pass draws again.  Staged and not:
        // 1,500 x 5,000 clients 742 and 307 us, 500 x 5,000 304 and 181, 5,000 x 2,000 484 and
        // 381; 1,500 x 1,000 67 and 80, 700 x 2,000 80 and 105.
        const int warps = 1;
        const long long per_sm = (n_items + sm_count() - 1) / sm_count();
        if (per_warp <= 24 * 1024 || (per_warp <= 96 * 1024 && per_warp * per_sm <= 220 * 1024)) {
            const size_t smem = per_warp * warps;
            if (smem > 48 * 1024)
                cudaFuncSetAttribute(mm1_warp_coop_kernel<true>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(smem));
            mm1_warp_coop_kernel<true><<<ceil_div_u(n_items, warps), 32 * warps, smem, st>>>(
                d_dps, n_items, n_reps, rep0, n_clients, rk, tab, out);
        } else {
            mm1_warp_coop_kernel<false><<<ceil_div_u(n_items, 4), 128, 0, st>>>(
                d_dps, n_items, n_reps, rep0, n_clients, rk, tab, out);
        }
    } else {
        return fail(MRIP_EINVAL, "mrip_mm1_simulate: mapping must be THREAD, WARP_1LANE, WARP_COOP or CTA");
    }
    return launch_status("mrip_mm1_simulate");
}

extern "C" mrip_status mrip_tandem3_simulate(const double* d_dps, int32_t n_dp, int64_t rep0,
                                             int64_t n_reps, int64_t n_clients, int64_t window,
                                             uint64_t seed, uint32_t tag, int mapping,
                                             double* d_y, double* d_feat, void* stream) {
    if (n_dp < 0 || n_reps < 0 || rep0 < 0 || n_clients < 1 || window < 1)
        return fail(MRIP_EINVAL,
                    "mrip_tandem3_simulate: need n_dp, n_reps, rep0 >= 0 and n_clients, window >= 1");
    if (n_dp >= (1 << 24) || rep0 + n_reps > 0x100000000ll || n_clients > 0xFFFFFFFFll || tag > 255)
        return fail(MRIP_EINVAL,
                    "mrip_tandem3_simulate: n_dp < 2^24, replication indices < 2^32, tag < 256");
    const long long n_items = static_cast<long long>(n_dp) * n_reps;
    if (n_items == 0) return MRIP_OK;
    if (!d_dps || !d_y) return fail(MRIP_EINVAL, "mrip_tandem3_simulate: null pointer");
    const RoundKeys rk = expand_key(seed);
    LogTable tab;
    mrip_status ts = log_table(&tab);
    if (ts != MRIP_OK) return ts;
    TandemOut out{d_y, d_feat, n_items};
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (mapping == MRIP_MAP_AUTO || mapping == MRIP_MAP_THREAD) {
        tandem3_serial_kernel<false><<<ceil_div_u(n_items, 128), 128, 0, st>>>(
            d_dps, n_items, n_reps, rep0, n_clients, window, tag, rk, tab, out);
    } else if (mapping == MRIP_MAP_WARP_1LANE) {
        tandem3_serial_kernel<true><<<ceil_div_u(n_items * 32, 128), 128, 0, st>>>(
            d_dps, n_items, n_reps, rep0, n_clients, window, tag, rk, tab, out);
    } else if (mapping == MRIP_MAP_WARP_COOP) {
        tandem3_warp_coop_kernel<<<ceil_div_u(n_items * 32, 128), 128, 0, st>>>(
            d_dps, n_items, n_reps, rep0, n_clients, window, tag, rk, tab, out);
    } else if (mapping == MRIP_MAP_CTA) {
        if (n_items > 0x7FFFFFFFll) return fail(MRIP_EINVAL, "mrip_tandem3_simulate: too many replications for CTA");
        CtaShape shape;
        const long long sms = sm_count();
        const int most = n_items > 2 * sms ? kTandemThreads / 4 : n_items > sms ? kTandemThreads / 2 : kTandemThreads;
        mrip_status cs = cta_shape(tandem3_cta_kernel<false>, tandem3_cta_kernel<true>, n_items, n_clients, most, false,
                                   &shape);
        if (cs != MRIP_OK) return cs;
        cs = launch_ctas(shape.ctas > 1 ? tandem3_cta_kernel<true> : tandem3_cta_kernel<false>, n_items, shape, st, d_dps, static_cast<long long>(n_reps),
                         static_cast<long long>(rep0), static_cast<long long>(n_clients),
                         static_cast<long long>(window), tag, rk, tab, out);
        if (cs != MRIP_OK) return cs;
    } else {
        return fail(MRIP_EINVAL, "mrip_tandem3_simulate: mapping must be THREAD, WARP_1LANE, WARP_COOP or CTA");
    }
    return launch_status("mrip_tandem3_simulate");
}

MRIP_DEBUG_UNIT(queues)

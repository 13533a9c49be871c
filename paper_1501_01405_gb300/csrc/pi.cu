// Monte Carlo pi (paper, Section 5.1, first model): points in the unit
// square counted when they fall in the quarter disc.  Draw k of replication
// `rep` uses words 2(k mod 2), 2(k mod 2)+1 of Philox block (c0 = 0,
// c1 = k div 2) as integer coordinates x, y in [0, 2^32); it is inside iff
// x^2 + y^2 < 2^64, tested exactly as the absence of a carry out of 64 bits.
//
// Draws are independent, so a replication is split over CTAs of up to 2^16
// draws, fewer (down to 2^12) while that leaves fewer than eight CTAs per SM: a
// 10^7-draw replication fills the whole GPU by itself; each CTA reduces its count (warp reduction, then
// shared memory) and adds it to the replication's counter with one 64-bit
// atomic -- integer addition, so the result does not depend on the order.
#include <algorithm>

#include "common.cuh"

namespace mrip {
namespace {

constexpr int kPiThreads = 256;
constexpr long long kPiChunk = 1LL << 16, kPiLeast = 1LL << 12;  // most and least draws per CTA (even)
constexpr long long kPiFew = 768;

// outside += 1 if x^2 + y^2 >= 2^64: the carry out of the 64-bit sum, taken by
// the multiply that adds y^2 to x^2 (two multiplies and an add; comparing x^2
// with the complement of y^2 took four instructions more).
__device__ __forceinline__ void add_outside(uint32_t x, uint32_t y, uint32_t& outside) {
    uint32_t hi, lo;
    mul_wide_u32(x, x, hi, lo);
    asm("{\n .reg .u32 sum;\n mad.lo.cc.u32 sum, %1, %1, %2;\n madc.hi.cc.u32 sum, %1, %1, %3;\n addc.u32 %0, %0, 0;\n}"
        : "+r"(outside)
        : "r"(y), "r"(lo), "r"(hi));
}

// What bounds it is the FMA-heavy pipe (16 widening multiplies of Philox per
// block of two draws and 4 of the squares, 4.2 cycles each: 84 of the 87 cycles a
// warp takes).  Measured, 64 replications x 10^7 draws: 0.921 -> 0.700 ms (row keys
// alone 0.809); one replication 29.0 -> 17.7 us, 3 x 200,001 draws 23 -> 9.8 us.  The
// test in FP32 with an exact second look needs two multiplies less but four
// conversions more: 0.717 ms.
// kFew: any number of threads up to kPiThreads.
template <bool kFew>
__global__ void __launch_bounds__(kPiThreads) pi_kernel(long long n_draws, long long chunk, long long chunks, long long rep0,
                                                        const __grid_constant__ RoundKeys rk,
                                                        unsigned long long* __restrict__ hits) {
    __shared__ uint32_t part[kPiThreads / 32];
    const uint32_t threads = kFew ? blockDim.x : kPiThreads;
    const long long rep = blockIdx.x / chunks;
    const long long start = (blockIdx.x - rep * chunks) * chunk;
    const uint32_t draws = static_cast<uint32_t>(min(chunk, n_draws - start));
    const RowKey row = row_key(static_cast<uint32_t>(rep0 + rep), stream_word(0u, 0u), rk);
    const uint32_t first = static_cast<uint32_t>(start / 2), pairs = draws / 2;  // whole blocks
    uint32_t outside = 0;
#pragma unroll 2
    for (uint32_t b = threadIdx.x; b < pairs; b += threads) {
        const uint4 w = philox_row(row, first + b, rk);
        add_outside(w.x, w.y, outside);
        add_outside(w.z, w.w, outside);
    }
    if ((draws & 1u) && threadIdx.x == 0) {  // the last draw of an odd number
        const uint4 w = philox_row(row, first + pairs, rk);
        add_outside(w.x, w.y, outside);
    }
    outside = __reduce_add_sync(0xFFFFFFFFu, outside);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = outside;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t tot = 0;
        for (uint32_t i = 0; i < threads / 32; ++i) tot += part[i];
        atomicAdd(hits + rep, static_cast<unsigned long long>(draws - tot));
    }
}

}  // namespace
}  // namespace mrip

using namespace mrip;

extern "C" mrip_status mrip_pi_simulate(int64_t rep0, int64_t n_reps, int64_t n_draws, uint64_t seed,
                                        int64_t* d_hits, void* stream) {
    if (rep0 < 0 || n_reps < 0 || n_draws < 0) return fail(MRIP_EINVAL, "mrip_pi_simulate: negative size");
    if (rep0 + n_reps > 0x100000000ll || n_draws > (1LL << 33))
        return fail(MRIP_EINVAL, "mrip_pi_simulate: replication indices < 2^32, n_draws <= 2^33");
    if (n_reps == 0) return MRIP_OK;
    if (!d_hits) return fail(MRIP_EINVAL, "mrip_pi_simulate: null output");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemsetAsync(d_hits, 0, static_cast<size_t>(n_reps) * sizeof(int64_t), st);
    if (e != cudaSuccess) return cuda_status(e, "mrip_pi_simulate: clear");
    if (n_draws == 0) return MRIP_OK;
    long long chunk = kPiChunk;
    auto ctas = [&]() { return (n_draws + chunk - 1) / chunk; };
    while (chunk > kPiLeast && ctas() * n_reps < 8ll * sm_count()) chunk /= 2;
    const long long chunks = ctas();
    if (chunks * n_reps > 0x7FFFFFFFll) return fail(MRIP_EINVAL, "mrip_pi_simulate: too many draws in total");
    // Replications of fewer than kPiFew draws spread them evenly over as many threads
    // as one or two rounds need: 100,000 replications of 1, 100, 300, 600 draws take 57, 57,
    // 107, 148 us so and 86, 96, 120, 164 with 256 threads; of 1,000 (the loop's stride is no
    // constant here) 226 and 205.
    const long long pairs = std::max<long long>(1, n_draws / 2), rounds = (pairs + kPiThreads - 1) / kPiThreads;
    const bool few = n_draws < kPiFew;
    const unsigned threads = few ? static_cast<unsigned>(((pairs + rounds - 1) / rounds + 31) / 32 * 32) : kPiThreads;
    auto* kernel = few ? pi_kernel<true> : pi_kernel<false>;
    kernel<<<static_cast<unsigned>(chunks * n_reps), threads, 0, st>>>(
        n_draws, chunk, chunks, rep0, expand_key(seed), reinterpret_cast<unsigned long long*>(d_hits));
    return launch_status("mrip_pi_simulate");
}

// Area walk: the paper's random-walk model (Section 5.1, third model) and
// the experiment it uses to compare one replication per warp (WLP) with one
// per thread (TLP) (Section 5.3).  A walker moves on a 60 x 50 periodic map
// split into 30 areas of 10 x 10 cells (area x/10 + 6 (y/10)), starting at
// (30, 25); move m reads field m mod 64 of Philox block (c0 = 0,
// c1 = m div 64) (0:+x 1:-x 2:+y 3:-y); after every move the visit count of
// the walker's area grows by one.  Outputs: final area and 30 visit counts.
//
// Mappings:
//   THREAD      one replication per thread; one histogram per thread
//               ([area][thread]: the per-move scatter never conflicts on a bank)
//               and, from 64 moves, a table of every cell's four successors in
//               shared memory;
//   WARP_1LANE  one replication per warp, lane 0 only (the paper's WLP);
//   WARP_COOP   one replication per warp: a round covers 512 moves, lane l
//               takes moves 16l .. 16l+15, a warp scan of the 16-move
//               displacements (popcounts) gives each lane's start, and the
//               lanes add their visits to one warp histogram.
#include "common.cuh"

namespace mrip {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr uint32_t kEven = 0x55555555u;
constexpr int kW = 60, kH = 50, kCell = 10, kAreas = 30, kThreads = 128;

__device__ __forceinline__ int area_of(int x, int y) { return x / kCell + (kW / kCell) * (y / kCell); }

__device__ __forceinline__ void move(uint32_t f, int& x, int& y) {
    if (f & 2u) {
        y += (f & 1u) ? kH - 1 : 1;
        if (y >= kH) y -= kH;
    } else {
        x += (f & 1u) ? kW - 1 : 1;
        if (x >= kW) x -= kW;
    }
}

// THREAD and WARP_1LANE, walks of fewer than kTableMoves moves: two coordinates,
// and the area by division.  The table below costs a CTA 3,000 entries and 61 KB before
// its first move, which short walks do not earn back.  300,000 replications x 1,
// 10, 30, 63 moves: 8.5, 9.8, 16.4, 26.8 us here, 18.6, 20.6, 24.7, 30.8 with the
// table; x 64 28 and 24.  16,384 replications by one lane per warp x 1, 30, 63 moves: 8.7,
// 24.4, 41.2 and 30.9, 39.1, 49.3; x 64 45 and 37.
constexpr int kTableMoves = 64;

template <bool kLane0Only>
__global__ void __launch_bounds__(kThreads) area_walk_short_kernel(long long rep0, long long n_reps, int n_steps,
                                                                   const __grid_constant__ RoundKeys rk,
                                                                   int32_t* __restrict__ final_area,
                                                                   int32_t* __restrict__ visits) {
    constexpr int kWalkers = kLane0Only ? kThreads / 32 : kThreads;
    static_assert(kTableMoves <= 64, "the moves of one Philox block");
    __shared__ uint32_t hist[kAreas][kWalkers];
    if (kLane0Only && (threadIdx.x & 31) != 0) return;
    const int slot = kLane0Only ? threadIdx.x >> 5 : threadIdx.x;
    const long long item = blockIdx.x * static_cast<long long>(kWalkers) + slot;
    if (item >= n_reps) return;
    for (int a = 0; a < kAreas; ++a) hist[a][slot] = 0u;
    int x = kW / 2, y = kH / 2;
    const uint4 b = philox(0u, 0u, static_cast<uint32_t>(rep0 + item), stream_word(0u, 0u), rk);
    const uint32_t words[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t w = words[k];
        for (int s = 16 * k; s < min(16 * k + 16, n_steps); ++s, w >>= 2) {
            move(w & 3u, x, y);
            const int a = area_of(x, y);
            if (MRIP_CHECK(a >= 0 && a < kAreas, 604, a)) hist[a][slot] += 1u;
        }
    }
    final_area[item] = area_of(x, y);
    if (visits)
        for (int a = 0; a < kAreas; ++a) visits[a * n_reps + item] = static_cast<int32_t>(hist[a][slot]);
}

// THREAD and WARP_1LANE.  A move is one table look-up: cell c of area a has the
// code 128 a + c, and next[code] holds the codes (times 8) of its four
// successors, so the walker's state is e = 8 code, 16 bits; e | 2 f is the byte
// address of the successor by move f, and with 256 threads per CTA the
// histogram row of its area starts at byte e & 0xFC00.  Five instructions a
// move: a shift, two logic operations, the look-up and the counter's addition in
// shared memory (two coordinates with wrap-around and two divisions by 10 took
// 38).  What bounds it is shared memory: the look-ups of 32 walkers conflict
// on about 3.4 banks.  The counter's own column makes the addition race-free, but
// the one-way atomic beats a load, an add and a store (53 us).  Measured, 65,536
// replications x 1,000 moves: 102.7 -> 43.2 us, x 100 14.4 -> 10.4; 300,000 x 300 112 ->
// 55.5; 16,384 x 1,000 by one lane per warp 596 -> 152.
constexpr int kSerialThreads = 256;
constexpr int kCodes = 128 * kAreas;
static_assert(4 * kSerialThreads == 1024, "a histogram row is 1 << 10 bytes: the area bits of e");

__device__ __forceinline__ uint32_t code8(int x, int y) {
    return 8u * static_cast<uint32_t>(128 * area_of(x, y) + (x % kCell) + kCell * (y % kCell));
}

struct SerialSmem {
    uint32_t hist[kAreas][kSerialThreads];
    ushort4 next[kCodes];  // codes with c >= 100 are never reached
};

template <bool kLane0Only>
__global__ void __launch_bounds__(kSerialThreads) area_walk_serial_kernel(long long rep0, long long n_reps, int n_steps,
                                                                          const __grid_constant__ RoundKeys rk,
                                                                          int32_t* __restrict__ final_area,
                                                                          int32_t* __restrict__ visits) {
    extern __shared__ __align__(16) unsigned char area_smem[];
    SerialSmem& S = *reinterpret_cast<SerialSmem*>(area_smem);
    if (!MRIP_CHECK(sizeof(SerialSmem) <= dynamic_smem_bytes(), 603, sizeof(SerialSmem))) return;  // CTA-uniform
    for (int c = threadIdx.x; c < kW * kH; c += kSerialThreads) {
        const int x = c % kW, y = c / kW;
        const int e = x + 1 < kW ? x + 1 : 0, w = x > 0 ? x - 1 : kW - 1;
        const int n = y + 1 < kH ? y + 1 : 0, s = y > 0 ? y - 1 : kH - 1;
        S.next[code8(x, y) >> 3] =
            make_ushort4(static_cast<unsigned short>(code8(e, y)), static_cast<unsigned short>(code8(w, y)),
                         static_cast<unsigned short>(code8(x, n)), static_cast<unsigned short>(code8(x, s)));
    }
    for (int a = 0; a < kAreas; ++a) S.hist[a][threadIdx.x] = 0u;
    __syncthreads();
    const long long thread = blockIdx.x * static_cast<long long>(kSerialThreads) + threadIdx.x;
    if (kLane0Only && (threadIdx.x & 31) != 0) return;
    const long long item = kLane0Only ? thread >> 5 : thread;
    if (item >= n_reps) return;
    const RowKey row = row_key(static_cast<uint32_t>(rep0 + item), stream_word(0u, 0u), rk);
    const unsigned char* next = reinterpret_cast<const unsigned char*>(S.next);
    unsigned char* hist = reinterpret_cast<unsigned char*>(&S.hist[0][0]);
    const uint32_t column = 4u * threadIdx.x;
    uint32_t e = code8(kW / 2, kH / 2);
    auto step = [&](uint32_t f2) {  // f2: bits 1 and 2 are the move
        e = *reinterpret_cast<const unsigned short*>(next + (e | (f2 & 6u)));
        if (MRIP_CHECK(e < 8u * kCodes, 601, e))
            atomicAdd(reinterpret_cast<uint32_t*>(hist + ((e & 0xFC00u) | column)), 1u);
    };
    for (int m0 = 0; m0 < n_steps; m0 += 64) {
        const uint4 b = philox_row(row, static_cast<uint32_t>(m0 >> 6), rk);
        const uint32_t words[4] = {b.x, b.y, b.z, b.w};
        if (n_steps - m0 >= 64) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                step(words[k] << 1);
#pragma unroll
                for (int s = 1; s < 16; ++s) step(words[k] >> (2 * s - 1));
            }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                uint32_t w = words[k];
                for (int s = m0 + 16 * k; s < min(m0 + 16 * k + 16, n_steps); ++s, w >>= 2) step(w << 1);
            }
        }
    }
    final_area[item] = static_cast<int32_t>(e >> 10);
    if (visits)
        for (int a = 0; a < kAreas; ++a) visits[a * n_reps + item] = static_cast<int32_t>(S.hist[a][threadIdx.x]);
}

__device__ __forceinline__ int wrap(int v, int n) {
    v %= n;
    return v < 0 ? v + n : v;
}

__global__ void __launch_bounds__(kThreads) area_walk_coop_kernel(long long rep0, long long n_reps, int n_steps,
                                                                  const __grid_constant__ RoundKeys rk,
                                                                  int32_t* __restrict__ final_area,
                                                                  int32_t* __restrict__ visits) {
    __shared__ uint32_t hist[kThreads / 32][kAreas];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long item = (blockIdx.x * static_cast<long long>(kThreads) + threadIdx.x) >> 5;
    if (item >= n_reps) return;  // warp-uniform
    if (lane < kAreas) hist[warp][lane] = 0u;
    __syncwarp();
    const RowKey row = row_key(static_cast<uint32_t>(rep0 + item), stream_word(0u, 0u), rk);
    int px = kW / 2, py = kH / 2;  // warp-uniform position before the round
    for (int m0 = 0; m0 < n_steps; m0 += 512) {
        const uint4 b = philox_row(row, static_cast<uint32_t>((m0 >> 6) + (lane >> 2)), rk);
        const int sel = lane & 3;
        const uint32_t w = sel == 0 ? b.x : sel == 1 ? b.y : sel == 2 ? b.z : b.w;
        const int first = m0 + 16 * lane;
        const int cnt = max(0, min(16, n_steps - first));
        // displacement of this lane's moves (only the ones that exist)
        const uint32_t valid = cnt == 16 ? 0xFFFFFFFFu : ((1u << (2 * cnt)) - 1u);
        const uint32_t sgn = w & kEven & valid;
        const uint32_t axis = (w >> 1) & kEven & valid;
        const uint32_t used = kEven & valid;
        const int nx = __popc(~axis & used);
        const int dx = nx - 2 * __popc(~axis & sgn);
        const int dy = (cnt - nx) - 2 * __popc(axis & sgn);
        int sx = dx, sy = dy;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int ox = __shfl_up_sync(kFull, sx, off);
            const int oy = __shfl_up_sync(kFull, sy, off);
            if (lane >= off) {
                sx += ox;
                sy += oy;
            }
        }
        int x = wrap(px + sx - dx, kW), y = wrap(py + sy - dy, kH);
        for (int s = 0; s < cnt; ++s) {
            move((w >> (2 * s)) & 3u, x, y);
            const int a = area_of(x, y);
            if (MRIP_CHECK(a >= 0 && a < kAreas, 602, a)) atomicAdd(&hist[warp][a], 1u);
        }
        px = wrap(px + __shfl_sync(kFull, sx, 31), kW);
        py = wrap(py + __shfl_sync(kFull, sy, 31), kH);
    }
    __syncwarp();
    if (lane == 0) final_area[item] = area_of(px, py);
    if (visits && lane < kAreas) visits[lane * n_reps + item] = static_cast<int32_t>(hist[warp][lane]);
}

template <bool kLane0Only>
mrip_status launch_serial(int64_t rep0, int64_t n_reps, int32_t n_steps, const RoundKeys& rk, int32_t* d_final_area,
                          int32_t* d_visits, cudaStream_t st) {
    const int64_t threads = kLane0Only ? n_reps * 32 : n_reps;
    if (n_steps < kTableMoves) {
        area_walk_short_kernel<kLane0Only><<<ceil_div_u(threads, kThreads), kThreads, 0, st>>>(rep0, n_reps, n_steps, rk,
                                                                                             d_final_area, d_visits);
        return MRIP_OK;
    }
    cudaError_t e = cudaFuncSetAttribute(area_walk_serial_kernel<kLane0Only>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(sizeof(SerialSmem)));
    if (e != cudaSuccess) return cuda_status(e, "mrip_area_walk_simulate: shared memory attribute");
    area_walk_serial_kernel<kLane0Only><<<ceil_div_u(threads, kSerialThreads), kSerialThreads, sizeof(SerialSmem), st>>>(
        rep0, n_reps, n_steps, rk, d_final_area, d_visits);
    return MRIP_OK;
}

}  // namespace
}  // namespace mrip

using namespace mrip;

extern "C" mrip_status mrip_area_walk_simulate(int64_t rep0, int64_t n_reps, int32_t n_steps, uint64_t seed,
                                               int mapping, int32_t* d_final_area, int32_t* d_visits,
                                               void* stream) {
    if (rep0 < 0 || n_reps < 0 || n_steps < 0) return fail(MRIP_EINVAL, "mrip_area_walk_simulate: negative size");
    if (rep0 + n_reps > 0x100000000ll)
        return fail(MRIP_EINVAL, "mrip_area_walk_simulate: replication indices < 2^32");
    if (n_steps > (1 << 30)) return fail(MRIP_EINVAL, "mrip_area_walk_simulate: n_steps <= 2^30");
    if (n_reps == 0) return MRIP_OK;
    if (!d_final_area) return fail(MRIP_EINVAL, "mrip_area_walk_simulate: null output");
    const RoundKeys rk = expand_key(seed);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (mapping == MRIP_MAP_AUTO || mapping == MRIP_MAP_THREAD) {
        const mrip_status s = launch_serial<false>(rep0, n_reps, n_steps, rk, d_final_area, d_visits, st);
        if (s != MRIP_OK) return s;
    } else if (mapping == MRIP_MAP_WARP_1LANE) {
        const mrip_status s = launch_serial<true>(rep0, n_reps, n_steps, rk, d_final_area, d_visits, st);
        if (s != MRIP_OK) return s;
    } else if (mapping == MRIP_MAP_WARP_COOP) {
        area_walk_coop_kernel<<<ceil_div_u(n_reps * 32, kThreads), kThreads, 0, st>>>(rep0, n_reps, n_steps, rk,
                                                                                     d_final_area, d_visits);
    } else {
        return fail(MRIP_EINVAL, "mrip_area_walk_simulate: mapping must be THREAD, WARP_1LANE or WARP_COOP");
    }
    return launch_status("mrip_area_walk_simulate");
}

MRIP_DEBUG_UNIT(area_walk)

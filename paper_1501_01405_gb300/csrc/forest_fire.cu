// Stochastic forest-fire cellular automaton (Drossel-Schwabl rules), one
// replication per CTA, the lattice held in shared memory and registers.
//
// Layout: the L x L lattice (L = 32 W) is two bit planes, "tree" and
// "burning", one 32-bit word per 32 cells of a row (bit m of word j is cell
// x = 32 j + m).  Thread y of the CTA (L threads) owns row y, or thread y + L h
// the h-th half of it (2 L threads, for few replications): its words are read and
// written as 16-byte vectors, east and west neighbours are funnel
// shifts within the thread's own words, and only the burning plane, which the
// rows above and below read, is double-buffered in shared memory (one barrier
// per step).  A plane keeps vector q of all rows together (ff_word), so that
// neighbouring threads touch neighbouring 16-byte slots and no access
// conflicts on a bank.  The new state of 32 cells is a few bitwise operations:
//   ignite = burning neighbour | lightning,
//   burning' = tree & ignite,
//   tree'    = (tree & ~ignite) | (empty & grow).
// (With the words dealt out to the threads in turn, every one with its own
// address arithmetic and eight scalar accesses, 128 x 128 took 10.31 instead of
// 10.11 ms, and the skip-sampled variant spent a third of its time on it.)
// The burning count of each step is a popcount, a warp reduction and a
// shared-memory atomic; counts are flushed to global memory every 64 steps
// (coalesced, 16-byte stores where aligned) from a double-buffered slot array.
//
// The random word of cell i = y L + x at step t is word (i mod 4) of Philox
// block (c0 = i div 4, c1 = t); lattice word k = y W + j uses blocks c0 = 8k ..
// 8k+7.  The kernel is bound by Philox's 32x32->64 multiplies, which GB300
// retires at under one warp instruction per SM-clock.  Of a block's 20
// products, those of rounds 1 and 2 with words 0 and 2 and round 3's with
// word 0 depend on the step alone or on the cell alone.  The words do not
// depend on the lattice, so a thread draws several steps of a word at once
// (ff_draw): the step's products are shared by all blocks of a row, the cell's
// by all steps of the batch, and 15 + 2/NT products remain per block (NT steps;
// 17.1 when each step was drawn by itself); the growth masks wait in shared
// memory, one word per step, read back by the thread that wrote them, and the
// rare lightning masks in local memory behind a flag bit.
// Measured, against one step at a time on words dealt out in turn: 128 x 128, 1,024
// replications x 1,000 steps 11.28 -> 9.85 ms; 256 x 256, 2,048 replications x 400
// steps 34.5 -> 30.5 ms; 512 x 512, 308 x 122 9.09 -> 8.46 ms.  The FMA-heavy pipe is
// 79 % busy, the ALU 61 %.
#include <type_traits>

#include "common.cuh"
#include "model.cuh"

namespace mrip {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// bits |= bit if w < t, as a compare and a predicated OR.  With constant bits the
// multiply pipe carries 165 instructions per word and step (ncu's pipe counter), with
// variable ones 136, but those are 6 % slower (128 x 128: 9.84 and 10.48 ms): the ALU and
// the issue slots are as near their limits.
__device__ __forceinline__ void or_if_below(uint32_t& bits, uint32_t w, uint32_t t, uint32_t bit) {
    asm("{\n .reg .pred p;\n setp.lt.u32 p, %1, %2;\n @p or.b32 %0, %0, %3;\n}\n"
        : "+r"(bits)
        : "r"(w), "r"(t), "r"(bit));
}

// Flush the n_slot (<= 64) burning counts of one 64-step chunk from the
// shared slot array to dst (skipped when null) and add them to my_sum,
// clearing the slots when asked.  Where dst is 16-byte aligned and n_slot a
// multiple of 4 (every chunk when n_steps is), a thread moves four counts
// with one 16-byte store.
template <int TPB>
__device__ __forceinline__ void ff_flush(int* slot, int n_slot, int32_t* dst, bool clear, long long& my_sum) {
    if (dst && (reinterpret_cast<uintptr_t>(dst) & 15u) == 0 && (n_slot & 3) == 0) {
        for (int s4 = threadIdx.x; s4 < (n_slot >> 2); s4 += TPB) {
            int4* src = reinterpret_cast<int4*>(slot) + s4;
            const int4 v = *src;
            if (clear) *src = make_int4(0, 0, 0, 0);
            my_sum += static_cast<long long>(v.x) + v.y + v.z + v.w;
            reinterpret_cast<int4*>(dst)[s4] = v;
        }
    } else {
        for (int s = threadIdx.x; s < n_slot; s += TPB) {
            const int v = slot[s];
            if (clear) slot[s] = 0;
            my_sum += v;
            if (dst) dst[s] = v;
        }
    }
}


// ---------------------------------------------------------------------------
// Rows and planes
// ---------------------------------------------------------------------------
// Threads per CTA for a lattice of W words per row: one per row.
template <int W>
constexpr int ff_threads() {
    return 32 * W;
}

// Index of word j of row y in a plane of L W words.
template <int W>
__device__ __forceinline__ int ff_word(int y, int j) {
    constexpr int V = W < 4 ? W : 4;
    return ((j / V) * 32 * W + y) * V + j % V;
}

// Words j0 .. j0 + N - 1 of row y (N divides W, j0 a multiple of N).
template <int W, int N>
__device__ __forceinline__ void row_load(const uint32_t* plane, int y, int j0, uint32_t (&w)[N]) {
    if constexpr (N == 1) {
        w[0] = plane[ff_word<W>(y, j0)];
    } else if constexpr (N == 2) {
        const uint2 v = *reinterpret_cast<const uint2*>(plane + ff_word<W>(y, j0));
        w[0] = v.x;
        w[1] = v.y;
    } else {
#pragma unroll
        for (int q = 0; q < N / 4; ++q) {
            const uint4 v = *reinterpret_cast<const uint4*>(plane + ff_word<W>(y, j0 + 4 * q));
            w[4 * q] = v.x;
            w[4 * q + 1] = v.y;
            w[4 * q + 2] = v.z;
            w[4 * q + 3] = v.w;
        }
    }
}

template <int W, int N>
__device__ __forceinline__ void row_store(uint32_t* plane, int y, int j0, const uint32_t (&w)[N]) {
    if constexpr (N == 1) {
        plane[ff_word<W>(y, j0)] = w[0];
    } else if constexpr (N == 2) {
        *reinterpret_cast<uint2*>(plane + ff_word<W>(y, j0)) = make_uint2(w[0], w[1]);
    } else {
#pragma unroll
        for (int q = 0; q < N / 4; ++q)
            *reinterpret_cast<uint4*>(plane + ff_word<W>(y, j0 + 4 * q)) =
                make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
    }
}

// One step of words j0 .. j0 + N - 1 of row y: their tree and burning words from
// the burning plane `cur`, the growth words g and the lightning words l; the
// new burning words go to `nxt`.  Returns their burning cells.
template <int W, int N>
__device__ __forceinline__ int row_step(uint32_t (&t)[N], uint32_t (&b)[N], const uint32_t* cur, uint32_t* nxt, int y,
                                        int j0, const uint32_t (&g)[N], const uint32_t (&l)[N]) {
    constexpr int L = 32 * W;
    uint32_t up[N], dn[N], nb[N];
    row_load<W, N>(cur, (y + L - 1) & (L - 1), j0, up);
    row_load<W, N>(cur, (y + 1) & (L - 1), j0, dn);
    // the words beside them: the thread's own where it has the whole row
    const uint32_t before = N == W ? b[N - 1] : cur[ff_word<W>(y, (j0 + W - 1) % W)];
    const uint32_t after = N == W ? b[0] : cur[ff_word<W>(y, (j0 + N) % W)];
    int c = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const uint32_t west = __funnelshift_l(j > 0 ? b[j > 0 ? j - 1 : 0] : before, b[j], 1);
        const uint32_t east = __funnelshift_r(b[j], j + 1 < N ? b[j + 1 < N ? j + 1 : j] : after, 1);
        const uint32_t ignite = up[j] | dn[j] | west | east | l[j];
        nb[j] = t[j] & ignite;
        t[j] = (t[j] & ~ignite) | (~(t[j] | b[j]) & g[j]);
        c += __popc(nb[j]);
    }
#pragma unroll
    for (int j = 0; j < N; ++j) b[j] = nb[j];
    row_store<W, N>(nxt, y, j0, b);
    return c;
}

// Initial state into the planes: from `init` (one byte per cell, 0 empty, 1
// tree, 2 burning) or from tag 1 (tree iff word < t_dens).
template <int W, int TPB>
__device__ void ff_load_initial(uint32_t* tree, uint32_t* burning, const uint8_t* __restrict__ init, long long item,
                                uint32_t t_dens, uint32_t rep, uint32_t dp, const RoundKeys& rk) {
    constexpr int L = 32 * W;
    constexpr int NWORD = L * W;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(init + item * static_cast<long long>(L) * L);
    const uint32_t c3i = stream_word(1u, dp);
    for (int k = threadIdx.x; k < NWORD; k += TPB) {
        uint32_t tw = 0, bw = 0;
        if (init) {
            for (int r = 0; r < 8; ++r) {
                const uint32_t v = src[8 * k + r];
                for (int q = 0; q < 4; ++q) {
                    const uint32_t s = (v >> (8 * q)) & 0xFFu;
                    tw |= (s == 1u ? 1u : 0u) << (4 * r + q);
                    bw |= (s == 2u ? 1u : 0u) << (4 * r + q);
                }
            }
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint4 b = philox(8u * k + q, 0u, rep, c3i, rk);
                tw |= (b.x < t_dens) ? (1u << (4 * q)) : 0u;
                tw |= (b.y < t_dens) ? (1u << (4 * q + 1)) : 0u;
                tw |= (b.z < t_dens) ? (1u << (4 * q + 2)) : 0u;
                tw |= (b.w < t_dens) ? (1u << (4 * q + 3)) : 0u;
            }
        }
        const int at = ff_word<W>(k / W, k % W);
        tree[at] = tw;
        burning[at] = bw;
    }
}

// The planes back to one byte per cell.
template <int W, int TPB>
__device__ void ff_store_final(const uint32_t* tree, const uint32_t* burning, uint8_t* __restrict__ final_state,
                               long long item) {
    constexpr int L = 32 * W;
    constexpr int NWORD = L * W;
    uint32_t* dst = reinterpret_cast<uint32_t*>(final_state + item * static_cast<long long>(L) * L);
    for (int k = threadIdx.x; k < NWORD; k += TPB) {
        const int at = ff_word<W>(k / W, k % W);
        const uint32_t tw = tree[at], bw = burning[at];
        for (int r = 0; r < 8; ++r) {
            uint32_t v = 0;
            for (int q = 0; q < 4; ++q) {
                const int m = 4 * r + q;
                const uint32_t s = ((tw >> m) & 1u) ? 1u : (((bw >> m) & 1u) ? 2u : 0u);
                v |= s << (8 * q);
            }
            dst[8 * k + r] = v;
        }
    }
}

// Per-replication scalar: the mean burning fraction (block reduction of the
// threads' step sums).
template <int NWARP>
__device__ void ff_store_scalar(long long my_sum, long long* red, double* scalar, long long item, int n_steps,
                                int L) {
    long long s = my_sum;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(kFull, s, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long tot = 0;
        for (int w = 0; w < NWARP; ++w) tot += red[w];
        scalar[item] = static_cast<double>(tot) / (static_cast<double>(n_steps) * static_cast<double>(L) * L);
    }
}

// Step t is done (the CTA has met): flush the 64-step chunk it ends.
template <int TPB>
__device__ __forceinline__ void ff_end_step(int (*cnt)[64], int t, int n_steps, int32_t* counts, long long item,
                                            long long& my_sum) {
    if ((t & 63) == 0 || t == n_steps) {
        const int chunk = (t - 1) >> 6;
        const int n_slot = t - chunk * 64;
        if (MRIP_CHECK(n_slot >= 1 && n_slot <= 64 && chunk * 64 + n_slot <= n_steps, 102, t))
            ff_flush<TPB>(cnt[chunk & 1], n_slot, counts ? counts + item * n_steps + chunk * 64 : nullptr, true,
                          my_sum);
    }
}

// ---------------------------------------------------------------------------
// The per-cell kernel
// ---------------------------------------------------------------------------
// Steps drawn together: eight, or four where the masks of eight would not fit in
// shared memory (L = 512: 224 KB with four).  A batch is also the number of
// independent Philox chains a thread interleaves.  128 x 128 at 2, 4, 6, 8, 12 and
// 16 steps: 11.0, 10.1, 10.0, 9.94, 9.97, 10.5 ms; 256 x 256 at 4, 5, 6, 7, 8: 31.7,
// 31.2, 31.1, 30.9, 30.8; 512 x 512 at 2 and 4: 8.91, 8.44.
template <int W>
constexpr int ff_batch() {
    return W == 16 ? 4 : 8;
}

// What the counters (c0, t, rep, c3) of the steps t0 .. t0 + NS - 1 of one
// replication share: word 1 after round 1 and, per step, round 2's product of
// word 0 (each with a round key).
template <int NS>
struct StepKeys {
    uint32_t x1;
    uint32_t p_hi[NS], p_lo[NS];
};

template <int NS>
__device__ __forceinline__ StepKeys<NS> step_keys(uint32_t t0, uint32_t rep, const RoundKeys& rk) {
    StepKeys<NS> s;
    uint32_t h1, x1;
    mul_wide_u32(0xCD9E8D57u, rep, h1, x1);
    s.x1 = x1 ^ rk.k0[1];
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        uint32_t hi, lo;
        mul_wide_u32(0xD2511F53u, h1 ^ (t0 + i) ^ rk.k0[0], hi, lo);
        s.p_hi[i] = hi ^ rk.k1[1];
        s.p_lo[i] = lo ^ rk.k1[2];
    }
    return s;
}

// Philox4x32-10 of counter (c0, t0 + i, rep, c3) for i < NS, from a = 0xD2511F53
// c0: the two products that do not depend on the step, then rounds 3 to 10.
template <int NS>
__device__ __forceinline__ void step_blocks(uint32_t a_hi, uint32_t a_lo, uint32_t c3, const StepKeys<NS>& sk,
                                            const RoundKeys& rk, uint4 (&b)[NS]) {
    uint32_t hi, u, r_hi, r_lo;
    mul_wide_u32(0xCD9E8D57u, a_hi ^ c3 ^ rk.k1[0], hi, u);
    u ^= rk.k0[2];
    mul_wide_u32(0xD2511F53u, hi ^ sk.x1, r_hi, r_lo);
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        uint32_t x0, x1, x2, x3;
        mul_wide_u32(0xCD9E8D57u, sk.p_hi[i] ^ a_lo, hi, x1);
        x0 = hi ^ u;
        x2 = r_hi ^ sk.p_lo[i];
        x3 = r_lo;
#pragma unroll
        for (int r = 3; r < 10; ++r) philox_round(x0, x1, x2, x3, rk.k0[r], rk.k1[r]);
        b[i] = make_uint4(x0, x1, x2, x3);
    }
}

// Growth and lightning masks of lattice word k for NS steps.  Lightning is
// rare: its masks are formed only where a word of a block, over kTest steps of the
// batch, is below its threshold.
template <int NS, int kUnroll, int kTest>
__device__ __forceinline__ void ff_draw(uint32_t k, uint32_t c3, const StepKeys<NS>& sk, const RoundKeys& rk,
                                        uint32_t t_grow, uint32_t t_light, uint32_t (&g)[NS], uint32_t (&l)[NS]) {
    uint32_t a_hi, a_lo;
    mul_wide_u32(0xD2511F53u, 8u * k, a_hi, a_lo);
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        g[i] = 0u;
        l[i] = 0u;
    }
#pragma unroll kUnroll
    for (int q = 0; q < 8; ++q) {
        uint4 b[NS];
        step_blocks<NS>(a_hi, a_lo, c3, sk, rk, b);
#pragma unroll
        for (int i0 = 0; i0 < NS; i0 += kTest) {
            bool any = false;
#pragma unroll
            for (int i = i0; i < i0 + kTest; ++i) {
                g[i] >>= 4;
                or_if_below(g[i], b[i].x, t_grow, 1u << 28);
                or_if_below(g[i], b[i].y, t_grow, 1u << 29);
                or_if_below(g[i], b[i].z, t_grow, 1u << 30);
                or_if_below(g[i], b[i].w, t_grow, 1u << 31);
                any = any || b[i].x < t_light || b[i].y < t_light || b[i].z < t_light || b[i].w < t_light;
            }
            if (__builtin_expect(any, 0)) {
#pragma unroll
                for (int i = i0; i < i0 + kTest; ++i) {
                    uint32_t nib = 0u;
                    or_if_below(nib, b[i].x, t_light, 1u);
                    or_if_below(nib, b[i].y, t_light, 2u);
                    or_if_below(nib, b[i].z, t_light, 4u);
                    or_if_below(nib, b[i].w, t_light, 8u);
                    l[i] |= nib << (4 * q);
                }
            }
        }
        asm("add.cc.u32 %0, %0, 0xD2511F53;\n\taddc.u32 %1, %1, 0;" : "+r"(a_lo), "+r"(a_hi));
    }
}

// R threads share a row, each N = W / R of its words.
// Register budget: 512 threads per SM, 128 registers each (128 x 128 with 512, 640
// and 384 threads: 9.96, 10.13, 9.94 ms).
template <int W, int R>
constexpr int ff_min_blocks() {
    return 512 / (32 * W * R);
}

template <int W, int R>
__global__ void __launch_bounds__(R * ff_threads<W>(), ff_min_blocks<W, R>()) forest_fire_kernel(
    const double* __restrict__ dps, long long n_reps, long long rep0, int n_steps, uint32_t t_dens,
    const __grid_constant__ RoundKeys rk, const uint8_t* __restrict__ init,
    int32_t* __restrict__ counts, double* __restrict__ scalar, uint8_t* __restrict__ final_state) {
    constexpr int L = 32 * W;
    constexpr int NWORD = L * W;  // words per plane
    constexpr int TPB = R * ff_threads<W>();
    constexpr int NWARP = TPB / 32;
    constexpr int NT = ff_batch<W>();
    constexpr int N = W / R;  // words per thread
    static_assert(N * R == W && N * NT <= 64, "one flag bit per word and step");
    extern __shared__ __align__(16) uint32_t ff_smem[];
    uint32_t* burning = ff_smem;             // [2][NWORD], by step parity
    uint32_t* tree = ff_smem + 2 * NWORD;    // [NWORD], each row private to its thread
    uint32_t* grow = ff_smem + 3 * NWORD;    // [NT][NWORD], likewise
    __shared__ __align__(16) int cnt[2][64];
    __shared__ long long red[NWARP];

    const int y = threadIdx.x % L, j0 = (threadIdx.x / L) * N, lane = threadIdx.x & 31;
    const long long item = blockIdx.x;
    if (!MRIP_CHECK((3u + NT) * NWORD * sizeof(uint32_t) <= dynamic_smem_bytes(), 101, NWORD)) return;  // CTA-uniform
    const uint32_t dp = static_cast<uint32_t>(item / n_reps);
    const uint32_t rep = static_cast<uint32_t>(rep0 + item % n_reps);
    const uint32_t t_grow = threshold32(dps[2 * dp]);
    const uint32_t t_light = threshold32(dps[2 * dp + 1]);
    const uint32_t c3 = stream_word(0u, dp);

    ff_load_initial<W, TPB>(tree, burning, init, item, t_dens, rep, dp, rk);
    for (int i = threadIdx.x; i < 128; i += TPB) (&cnt[0][0])[i] = 0;
    __syncthreads();

    long long my_sum = 0;
    uint32_t light[N * NT];  // [j][s], written and read only where flagged (local memory)
    for (int t0 = 1; t0 <= n_steps; t0 += NT) {
        unsigned long long flags = 0;  // bit NT j + s: word j has lightning at step t0 + s
        const int ns = min(NT, n_steps + 1 - t0);
        // masks of steps t0 + s .. t0 + s + K - 1 (L = 32 tests a batch for lightning by halves:
        // at p_lightning = 10^-3 most warps find some in a whole one.  1,000 replications x 100
        // steps 105 -> 101 us there, 92.5 at 10^-5 either way; 128 x 128 loses 0.7 % at 10^-5)
        auto draw = [&](int s, auto steps, auto unroll) {
            constexpr int K = decltype(steps)::value;
            const StepKeys<K> sk = step_keys<K>(static_cast<uint32_t>(t0 + s), rep, rk);
#pragma unroll 1
            for (int j = 0; j < N; ++j) {
                uint32_t g[K], l[K];
                ff_draw<K, decltype(unroll)::value, (W == 1 && K > 4 ? K / 2 : K)>(static_cast<uint32_t>(y * W + j0 + j), c3, sk, rk, t_grow, t_light, g, l);
                const int at = ff_word<W>(y, j0 + j);
#pragma unroll
                for (int i = 0; i < K; ++i) {
                    grow[(s + i) * NWORD + at] = g[i];
                    if (__builtin_expect(l[i] != 0u, 0)) {
                        light[j * NT + s + i] = l[i];
                        flags |= 1ull << (j * NT + s + i);
                    }
                }
            }
        };
        if (__builtin_expect(ns == NT, 1)) {
            draw(0, std::integral_constant<int, NT>{}, std::integral_constant<int, 1>{});
        } else {
            // The last n_steps mod NT steps, two at a time: one at a time, as fast as before
            // the batches at best, cost up to 14 % more where a run has fewer steps than a batch
            // (256 x 256, 600 replications x 7 steps 218 us, 202 so, 208 before them; 32 x 32,
            // 1,000 x 7 14.4, 12.4, 12.4).
            int s = 0;
#pragma unroll 1
            for (; s + 2 <= ns; s += 2) draw(s, std::integral_constant<int, 2>{}, std::integral_constant<int, 4>{});
            if (s < ns) draw(s, std::integral_constant<int, 1>{}, std::integral_constant<int, 8>{});
        }
        uint32_t t_row[N], b_row[N];
        row_load<W, N>(tree, y, j0, t_row);
        row_load<W, N>(burning + ((t0 - 1) & 1) * NWORD, y, j0, b_row);
#pragma unroll 1
        for (int s = 0; s < ns; ++s) {
            const int t = t0 + s;
            uint32_t g[N], l[N];
            row_load<W, N>(grow + s * NWORD, y, j0, g);
#pragma unroll
            for (int j = 0; j < N; ++j) l[j] = 0u;
            if (__builtin_expect(flags != 0ull, 0)) {
#pragma unroll
                for (int j = 0; j < N; ++j)
                    if ((flags >> (j * NT + s)) & 1ull) l[j] = light[j * NT + s];
            }
            int c = row_step<W, N>(t_row, b_row, burning + ((t - 1) & 1) * NWORD, burning + (t & 1) * NWORD, y, j0, g, l);
            c = __reduce_add_sync(kFull, c);
            if (lane == 0) atomicAdd(&cnt[((t - 1) >> 6) & 1][(t - 1) & 63], c);
            __syncthreads();
            ff_end_step<TPB>(cnt, t, n_steps, counts, item, my_sum);
        }
        row_store<W, N>(tree, y, j0, t_row);
    }

    if (scalar) ff_store_scalar<NWARP>(my_sum, red, scalar, item, n_steps, L);
    if (final_state) {
        __syncthreads();  // every row's trees
        ff_store_final<W, TPB>(tree, burning + (n_steps & 1) * NWORD, final_state, item);
    }
}

template <int W, int R>
mrip_status launch_ff(const double* dps, long long n_items, long long n_reps, long long rep0, int n_steps,
                      uint32_t t_dens, const RoundKeys& rk, const uint8_t* init, int32_t* counts,
                      double* scalar, uint8_t* final_state, cudaStream_t st) {
    const size_t smem = (3 + ff_batch<W>()) * static_cast<size_t>(32 * W) * W * sizeof(uint32_t);
    if (smem > 40 * 1024) {  // beside about 1 KB of static shared memory
        cudaError_t e = cudaFuncSetAttribute(forest_fire_kernel<W, R>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(smem));
        if (e != cudaSuccess) return cuda_status(e, "forest fire: shared memory attribute");
    }
    forest_fire_kernel<W, R><<<static_cast<unsigned>(n_items), R * ff_threads<W>(), smem, st>>>(
        dps, n_reps, rep0, n_steps, t_dens, rk, init, counts, scalar, final_state);
    return MRIP_OK;
}

// ---------------------------------------------------------------------------
// Skip-sampled variant: the same automaton, but each step's growth and
// lightning events are drawn as gaps between successes over the cells
// i = 0 .. L^2 - 1 (gap j: K_j = floor(E_j / mu), mu = -log1p(-p), E_j the
// exponential variate of words 2(j mod 2), 2(j mod 2)+1 of block
// (c0 = j div 2, c1 = t) under tag 5 (growth) or 6 (lightning)).  Work per
// step is p L^2 variates instead of L^2 words.
//
// The event sets do not depend on the lattice, so several steps are drawn at
// once, each by its own warps (group g of a CTA's kSlots groups draws step
// t0 + g), and the CTA then updates the lattice kSlots times, a barrier per
// step.  A warp draws 64 gaps per round (lane l takes one block, i.e. two
// gaps), a warp scan of the lanes' (2 + K_2l + K_2l+1) places the events (a
// group of several warps adds the warps' totals, met in shared memory behind
// the group's own named barrier), and each event sets its bit in the step's
// event plane (atomicOr); the update reads and clears the plane row by row.
// The lightning set is empty at most steps, which one compare of its first
// gap tells: lane l tests step t0 + l for 32 steps at once.
//
// The floor is decided in FP32 (MUFU.LG2) where the error bound leaves no
// doubt, else by the fixed-point logarithm (gap_fast); same integers.
// Measured against one set drawn per step by all warps, fixed-point floors and
// scalar updates: 128 x 128, 1,024 replications x 1,000 steps 2.52 -> 1.44 ms; 256 x
// 256, 2,048 x 400 11.3 -> 6.3 ms; 512 x 512, 183 x 65 1.80 -> 1.09 ms; 64 x 64, 2,155 x
// 333 1.75 -> 0.74 ms; 32 x 32, 7,155 x 334 1.57 -> 0.83 ms.
// ---------------------------------------------------------------------------
// K = floor(E / mu) without the FP64 pipe: E = y58 2^-58 (the fixed-point
// log), 2^-58 / mu = dm 2^-shift with dm a 64-bit integer (dm = the double's
// significand scaled to [2^63, 2^64)), so K = (y58 dm) >> shift on the
// 128-bit product, saturated at n_cells.  It differs from floor of the FP64
// quotient only when that quotient is within a few ulps of an integer.
struct GapScale {
    unsigned long long dm;
    int shift;  // >= 0; >= 128 means every gap is 0 (p >= 1)
};

__device__ __forceinline__ GapScale gap_scale(double p) {
    GapScale g{0ull, 128};
    if (p >= 1.0) return g;
    const double d = 0x1p-58 / -log1p(-p);  // p in (0, 1)
    if (!(d < 0x1p64)) {                     // mu below 2^-122: every positive E saturates
        g.dm = ~0ull;
        g.shift = 0;
        return g;
    }
    int ex;
    const double mant = frexp(d, &ex);  // d = mant 2^ex, mant in [0.5, 1), ex <= 64
    g.dm = static_cast<unsigned long long>(ldexp(mant, 64));
    g.shift = 64 - ex;  // >= 128: d < 2^-64, so y58 d < 1 and every gap is 0
    return g;
}

__device__ __forceinline__ int gap_cells(unsigned long long y58, const GapScale& g, int n_cells) {
    if (g.shift >= 128) return 0;
    const unsigned long long hi = __umul64hi(y58, g.dm);
    unsigned long long k;
    if (g.shift >= 64) {
        k = hi >> (g.shift - 64);
    } else {
        const unsigned long long lo = y58 * g.dm;
        if (g.shift == 0)
            k = hi ? ~0ull : lo;
        else
            k = (hi >> g.shift) ? ~0ull : ((hi << (64 - g.shift)) | (lo >> g.shift));
    }
    return k >= static_cast<unsigned long long>(n_cells) ? n_cells : static_cast<int>(k);
}

// The FP32 side of a gap: E / mu = q within q 2^-20 + c, where q = -log2(x)
// scale from x = 1 - u rounded: v = the complement of u's top 32 bits, x = (v +
// 1/2) 2^-32, is off by at most 2^-21 relative (v >= 2^20) plus 2^-23 of
// rounding, log2 by 2^-22 absolute or relative (CUDA's bound for __log2f), in
// all below 2^-20 / mu plus a relative 2^-21; 2^-22 more covers the roundings
// of the interval's ends.
struct GapFast {
    float scale;  // ln 2 / mu
    float c;
};

__device__ __forceinline__ GapFast gap_fast_scale(double p) {
    if (p >= 1.0) return GapFast{0.0f, 0x1p-22f};
    const double inv_mu = 1.0 / -log1p(-p);
    return GapFast{static_cast<float>(fmin(0.69314718055994531 * inv_mu, 1e30)),
                   static_cast<float>(fmin(0x1p-20 * inv_mu + 0x1p-22, 1e30))};
}

// K of words (lo, hi) if FP32 decides it, else -1.  RN(y - 1/2) at the
// magnitude of 1.5 2^23 is floor(y) or, at an integer y, one less: where both
// ends of the interval give the same k, the value between them is in [k, k + 1).
__device__ __forceinline__ int gap_try(uint32_t hi, const GapFast& f, int n_cells) {
    const uint32_t v = ~hi;
    const float x = __fmaf_rn(__uint2float_rn(v), 0x1p-32f, 0x1p-33f);
    const float q = fminf(-__log2f(x) * f.scale, 0x1p20f);  // past every lattice
    const float a = __fmaf_rn(q, 1.0f - 0x1p-20f, -0.5f - f.c) + 12582912.0f;
    const float b = __fmaf_rn(q, 1.0f + 0x1p-20f, -0.5f + f.c) + 12582912.0f;
    const int k = static_cast<int>(__float_as_uint(a) - 0x4B400000u);
    return (a == b && v >= (1u << 20)) ? min(k, n_cells) : -1;
}

// Both gaps of a block.
__device__ __forceinline__ void block_gaps(const uint4& b, const GapFast& f, const GapScale& gs, int n_cells,
                                           const LogTable& tab, int& k0, int& k1) {
    k0 = gap_try(b.y, f, n_cells);
    k1 = gap_try(b.w, f, n_cells);
    if (__builtin_expect((k0 | k1) < 0, 0)) {
        k0 = gap_cells(neg_log_q58<false>(b.x, b.y, tab), gs, n_cells);
        k1 = gap_cells(neg_log_q58<false>(b.z, b.w, tab), gs, n_cells);
    }
}

// Smallest 53-bit u (as an integer) for which the first gap of a set of
// probability p passes n cells: u >= 1 - (1 - p)^n, i.e. -log(1 - u) >= n mu.
// At least 1 (u = 0 gives the gap 0) and at most 2^53 (never, for p >= 1).
// At the boundary this and the gap's own floor can disagree only where
// E / mu is within a few ulps of n, which the oracle reports as a near tie.
__device__ __forceinline__ unsigned long long first_gap_none(double p, int n) {
    if (p >= 1.0) return 1ull << 53;
    const double q = -expm1(static_cast<double>(n) * log1p(-p));  // 1 - (1 - p)^n
    const double t = ceil(q * 0x1p53);
    if (!(t >= 1.0)) return 1ull;
    return t >= 0x1p53 ? (1ull << 53) : static_cast<unsigned long long>(t);
}

// Event sets drawn together (and so warps per set): one per warp up to four.
// 256 x 256 at two, four and eight sets (4, 2 and 1 warps each; the planes of eight
// leave one CTA per SM): 7.2, 6.3, 8.0 ms; 128 x 128 at two and four: 2.09, 1.65.  L = 512
// has room for two.
template <int W>
constexpr int skip_slots() {
    return W == 16 ? 2 : W < 4 ? W : 4;
}
template <int W>
constexpr int skip_warps() {
    return W / skip_slots<W>();
}

// Draw the set of step t under (rep, c3) into the plane ev, by kWarps warps (sub
// the index of this one; tot their shared totals, `bar` their named barrier).
// Call only for p > 0.
template <int W, int kWarps>
__device__ __forceinline__ void draw_events(uint32_t* __restrict__ ev, const GapFast& gf, const GapScale& gs,
                                            uint32_t t, uint32_t rep, uint32_t c3, const RoundKeys& rk,
                                            const LogTable& tab, int sub, int (*tot)[kWarps], int bar) {
    constexpr int L = 32 * W, n_cells = L * L;
    const int lane = threadIdx.x & 31;
    const StepKeys<1> sk = step_keys<1>(t, rep, rk);
    int pos = -1;  // last event so far (the same in every warp of the group)
    for (int r = 0; pos + 1 < n_cells; ++r) {
        uint32_t a_hi, a_lo;
        mul_wide_u32(0xD2511F53u, static_cast<uint32_t>((r * kWarps + sub) * 32 + lane), a_hi, a_lo);
        uint4 b[1];
        step_blocks<1>(a_hi, a_lo, c3, sk, rk, b);
        int k0, k1;
        block_gaps(b[0], gf, gs, n_cells, tab, k0, k1);
        const int span = 2 + k0 + k1;
        int incl = span;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int v = __shfl_up_sync(kFull, incl, off);
            if (lane >= off) incl += v;
        }
        int before = 0, total;
        if constexpr (kWarps > 1) {
            int* tt = tot[r & 1];
            if (lane == 31) tt[sub] = incl;
            asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(32 * kWarps) : "memory");
            total = 0;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const int v = tt[w];
                before += w < sub ? v : 0;
                total += v;
            }
        } else {
            total = __shfl_sync(kFull, incl, 31);
        }
        const int p0 = pos + before + (incl - span) + 1 + k0;
        const int p1 = p0 + 1 + k1;
        if (p0 < n_cells && MRIP_CHECK(p0 >= 0, 103, p0))
            atomicOr(ev + ff_word<W>(p0 / L, (p0 % L) / 32), 1u << (p0 & 31));
        if (p1 < n_cells && MRIP_CHECK(p1 > p0, 104, p1))
            atomicOr(ev + ff_word<W>(p1 / L, (p1 % L) / 32), 1u << (p1 & 31));
        pos += total;
    }
}

// Resident CTAs asked for at L = 128: seven (72 registers) are a compromise over the
// replications.  200 steps of 100, 800, 1,024, 2,000, 10,000 replications take 148, 264, 300, 557,
// 2,421 us with seven, 144, 255, 352, 565, 2,447 with the compiler's six (85 registers), 150,
// 267, 302, 547, 2,368 with eight: six are 3 % faster while they hold every replication and
// 15 % slower just beyond.  L = 64 and 32 take the compiler's choice: sixteen CTAs of 64 x
// 64 gain 2 % from 4,000 replications (12 % where 2,000 just need them) and lose 2 to 6 %
// below, more of 32 x 32 lose 3 to 5 % throughout.  From L = 256 shared memory holds two.
template <int W>
constexpr int skip_min_blocks() {
    return W == 4 ? 7 : 1;
}

template <int W>
__global__ void __launch_bounds__(ff_threads<W>(), skip_min_blocks<W>()) forest_fire_skip_kernel(
    const double* __restrict__ dps, long long n_reps, long long rep0, int n_steps, uint32_t t_dens,
    const __grid_constant__ RoundKeys rk, LogTable tab, const uint8_t* __restrict__ init,
    int32_t* __restrict__ counts, double* __restrict__ scalar, uint8_t* __restrict__ final_state) {
    constexpr int L = 32 * W;
    constexpr int NWORD = L * W;
    constexpr int TPB = ff_threads<W>();
    constexpr int NWARP = TPB / 32;
    constexpr int NS = skip_slots<W>();
    constexpr int GW = skip_warps<W>();
    static_assert(32 % NS == 0 && NWARP == NS * GW, "32 steps are whole batches");
    extern __shared__ __align__(16) uint32_t ff_smem[];
    uint32_t* burning = ff_smem;                        // [2][NWORD], by step parity
    uint32_t* ev_grow = ff_smem + 2 * NWORD;            // [NS][NWORD]
    uint32_t* ev_light = ff_smem + (2 + NS) * NWORD;    // [NS][NWORD]
    __shared__ __align__(16) int cnt[2][64];
    __shared__ long long red[NWARP];
    __shared__ int tot[NS][2][GW];

    const int y = threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int slot = warp / GW, sub = warp % GW;
    const long long item = blockIdx.x;
    if (!MRIP_CHECK((2u + 2u * NS) * NWORD * sizeof(uint32_t) <= dynamic_smem_bytes(), 107, NWORD)) return;
    const uint32_t dp = static_cast<uint32_t>(item / n_reps);
    const uint32_t rep = static_cast<uint32_t>(rep0 + item % n_reps);
    // The scales of both sets by lanes 0 and 1 of the first warp and the lightning's
    // threshold by the last one: logarithms and divisions in FP64, whose pipe a warp
    // occupies as long as one lane does.  (By every thread for itself, 300 replications
    // of 1 step took 130 us at L = 512, 53.5 at 256 and 26 at 128, and take 74, 24.7 and 14.4;
    // 1,024 of 128 x 128 x 1,000 1.446 -> 1.406 ms.)  A CTA of one warp computes them in every
    // lane: it has nothing to share out, and its rounds are up to 8 % faster so.
    __shared__ GapScale gs[2];
    __shared__ GapFast gf[2];
    __shared__ unsigned long long none_from;
    const double p_grow = dps[2 * dp], p_light = dps[2 * dp + 1];
    const bool any_grow = p_grow > 0.0, any_light = p_light > 0.0;
    if (W > 1 && warp == 0 && lane < 2) {
        const double p = lane == 0 ? p_grow : p_light;
        gs[lane] = p > 0.0 ? gap_scale(p) : GapScale{0ull, 128};
        gf[lane] = gap_fast_scale(p > 0.0 ? p : 1.0);
    }
    if (W > 1 && warp == NWARP - 1 && lane == 0) none_from = any_light ? first_gap_none(p_light, L * L) : 0ull;
    const uint32_t c3_grow = stream_word(5u, dp), c3_light = stream_word(6u, dp);

    ff_load_initial<W, TPB>(ev_grow, burning, init, item, t_dens, rep, dp, rk);
    for (int i = threadIdx.x; i < 128; i += TPB) (&cnt[0][0])[i] = 0;
    __syncthreads();
    GapScale gs_grow, gs_light;
    GapFast gf_grow, gf_light;
    unsigned long long light_none;
    if constexpr (W == 1) {
        gs_grow = any_grow ? gap_scale(p_grow) : GapScale{0ull, 128};
        gs_light = any_light ? gap_scale(p_light) : GapScale{0ull, 128};
        gf_grow = gap_fast_scale(any_grow ? p_grow : 1.0);
        gf_light = gap_fast_scale(any_light ? p_light : 1.0);
        light_none = any_light ? first_gap_none(p_light, L * L) : 0ull;
    } else {
        gs_grow = gs[0], gs_light = gs[1], gf_grow = gf[0], gf_light = gf[1], light_none = none_from;
    }
    uint32_t t_row[W], b_row[W];
    row_load<W, W>(ev_grow, y, 0, t_row);
    row_load<W, W>(burning, y, 0, b_row);
    __syncthreads();  // every row has its trees: the event planes start empty
    for (int k = threadIdx.x; k < 2 * NS * NWORD; k += TPB) ev_grow[k] = 0u;
    __syncthreads();

    long long my_sum = 0;
    unsigned none = 0u;  // bit i: no lightning at step 32 floor((t0 - 1) / 32) + 1 + i
    for (int t0 = 1; t0 <= n_steps; t0 += NS) {
        if (((t0 - 1) & 31) == 0) {
            const uint4 b = philox(0u, static_cast<uint32_t>(t0 + lane), rep, c3_light, rk);
            none = __ballot_sync(kFull, (((static_cast<unsigned long long>(b.y) << 32) | b.x) >> 11) >= light_none);
        }
        const int ns = min(NS, n_steps + 1 - t0);
        if (slot < ns) {
            const int t = t0 + slot;
            if (any_grow)
                draw_events<W, GW>(ev_grow + slot * NWORD, gf_grow, gs_grow, static_cast<uint32_t>(t), rep, c3_grow,
                                   rk, tab, sub, tot[slot], 1 + slot);
            if (sub == GW - 1 && !((none >> ((t - 1) & 31)) & 1u))
                draw_events<W, 1>(ev_light + slot * NWORD, gf_light, gs_light, static_cast<uint32_t>(t), rep, c3_light,
                                  rk, tab, 0, nullptr, 0);
        }
        __syncthreads();
#pragma unroll 1
        for (int s = 0; s < ns; ++s) {
            const int t = t0 + s;
            uint32_t g[W], l[W], zero[W];
#pragma unroll
            for (int j = 0; j < W; ++j) zero[j] = l[j] = 0u;
            row_load<W, W>(ev_grow + s * NWORD, y, 0, g);
            row_store<W, W>(ev_grow + s * NWORD, y, 0, zero);
            if (!((none >> ((t - 1) & 31)) & 1u)) {
                row_load<W, W>(ev_light + s * NWORD, y, 0, l);
                row_store<W, W>(ev_light + s * NWORD, y, 0, zero);
            }
            int c = row_step<W, W>(t_row, b_row, burning + ((t - 1) & 1) * NWORD, burning + (t & 1) * NWORD, y, 0, g, l);
            c = __reduce_add_sync(kFull, c);
            if (lane == 0) atomicAdd(&cnt[((t - 1) >> 6) & 1][(t - 1) & 63], c);
            __syncthreads();
            ff_end_step<TPB>(cnt, t, n_steps, counts, item, my_sum);
        }
    }
    if (scalar) ff_store_scalar<NWARP>(my_sum, red, scalar, item, n_steps, L);
    if (final_state) {
        row_store<W, W>(ev_grow, y, 0, t_row);
        __syncthreads();
        ff_store_final<W, TPB>(ev_grow, burning + (n_steps & 1) * NWORD, final_state, item);
    }
}

template <int W>
mrip_status launch_ff_skip(const double* dps, long long n_items, long long n_reps, long long rep0, int n_steps,
                           uint32_t t_dens, const RoundKeys& rk, const LogTable& tab, const uint8_t* init,
                           int32_t* counts, double* scalar, uint8_t* final_state, cudaStream_t st) {
    const size_t smem = (2 + 2 * skip_slots<W>()) * static_cast<size_t>(32 * W) * W * sizeof(uint32_t);
    if (smem > 40 * 1024) {  // beside about 1 KB of static shared memory
        cudaError_t e = cudaFuncSetAttribute(forest_fire_skip_kernel<W>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(smem));
        if (e != cudaSuccess) return cuda_status(e, "forest fire (skip): shared memory attribute");
    }
    forest_fire_skip_kernel<W><<<static_cast<unsigned>(n_items), ff_threads<W>(), smem, st>>>(
        dps, n_reps, rep0, n_steps, t_dens, rk, tab, init, counts, scalar, final_state);
    return MRIP_OK;
}

}  // namespace
}  // namespace mrip

using namespace mrip;

namespace mrip {
mrip_status forest_fire_launch(const double* d_dps, int32_t n_dp, int64_t rep0, int64_t n_reps, int32_t L,
                               int32_t n_steps, double density, uint64_t seed, const uint8_t* d_init,
                               int32_t* d_counts, double* d_scalar, uint8_t* d_final, cudaStream_t st) {
    if (n_dp < 0 || n_reps < 0 || n_steps < 0 || rep0 < 0)
        return fail(MRIP_EINVAL, "mrip_forest_fire_simulate: negative size");
    if (L < 32 || L > 512 || L % 32 != 0 || (L & (L - 1)) != 0)
        return fail(MRIP_EINVAL, "mrip_forest_fire_simulate: L must be 32, 64, 128, 256 or 512");
    if (!(density >= 0.0 && density < 1.0))
        return fail(MRIP_EINVAL, "mrip_forest_fire_simulate: density must be in [0, 1)");
    if (n_dp >= (1 << 24) || rep0 + n_reps > 0x100000000ll)
        return fail(MRIP_EINVAL, "mrip_forest_fire_simulate: n_dp < 2^24 and replication indices < 2^32");
    const long long n_items = static_cast<long long>(n_dp) * n_reps;
    if (n_items == 0) return MRIP_OK;
    if (n_items > 0x7FFFFFFFll) return fail(MRIP_EINVAL, "mrip_forest_fire_simulate: too many replications");
    if (!d_dps) return fail(MRIP_EINVAL, "mrip_forest_fire_simulate: null design points");
    if ((d_init && (reinterpret_cast<uintptr_t>(d_init) & 15u)) ||
        (d_final && (reinterpret_cast<uintptr_t>(d_final) & 15u)))
        return fail(MRIP_EINVAL, "mrip_forest_fire_simulate: state buffers need 16-byte alignment");
    const RoundKeys rk = expand_key(seed);
    const uint32_t t_dens = threshold32(density);
    // Two threads per lattice row where one per row would leave the SMs with at
    // most 256 of the 512 threads the register budget allows: 100 replications
    // of 128 x 128 x 999 steps take 1.63 ms with two and 2.07 with one, 101 of 256 x
    // 256 x 502 2.84 and 2.97.  On a full GPU one is faster (1,024 of 128 x 128: 9.95
    // against 10.16 ms, 2,048 of 256 x 256: 30.8 against 31.6); four per row gain
    // nothing over two (1.66 ms).
    const bool wide = n_items * L <= 256ll * sm_count();
    auto launch = [&](auto* f) {
        return f(d_dps, n_items, n_reps, rep0, n_steps, t_dens, rk, d_init, d_counts, d_scalar, d_final, st);
    };
    mrip_status rc = MRIP_OK;
    switch (L) {
        case 32: rc = launch(launch_ff<1, 1>); break;
        case 64: rc = wide ? launch(launch_ff<2, 2>) : launch(launch_ff<2, 1>); break;
        case 128: rc = wide ? launch(launch_ff<4, 2>) : launch(launch_ff<4, 1>); break;
        case 256: rc = wide ? launch(launch_ff<8, 2>) : launch(launch_ff<8, 1>); break;
        case 512: rc = launch(launch_ff<16, 1>); break;
    }
    if (rc != MRIP_OK) return rc;
    return launch_status("mrip_forest_fire_simulate");
}
}  // namespace mrip

extern "C" mrip_status mrip_forest_fire_skip_simulate(const double* d_dps, int32_t n_dp, int64_t rep0, int64_t n_reps,
                                                      int32_t L, int32_t n_steps, double density,
                                                      uint64_t seed, const uint8_t* d_init,
                                                      int32_t* d_counts, double* d_scalar,
                                                      uint8_t* d_final, void* stream) {
    if (n_dp < 0 || n_reps < 0 || n_steps < 0 || rep0 < 0)
        return fail(MRIP_EINVAL, "mrip_forest_fire_skip_simulate: negative size");
    if (L < 32 || L > 512 || L % 32 != 0 || (L & (L - 1)) != 0)
        return fail(MRIP_EINVAL, "mrip_forest_fire_skip_simulate: L must be 32, 64, 128, 256 or 512");
    if (!(density >= 0.0 && density < 1.0))
        return fail(MRIP_EINVAL, "mrip_forest_fire_skip_simulate: density must be in [0, 1)");
    if (n_dp >= (1 << 24) || rep0 + n_reps > 0x100000000ll)
        return fail(MRIP_EINVAL, "mrip_forest_fire_skip_simulate: n_dp < 2^24 and replication indices < 2^32");
    const long long n_items = static_cast<long long>(n_dp) * n_reps;
    if (n_items == 0) return MRIP_OK;
    if (n_items > 0x7FFFFFFFll) return fail(MRIP_EINVAL, "mrip_forest_fire_skip_simulate: too many replications");
    if (!d_dps) return fail(MRIP_EINVAL, "mrip_forest_fire_skip_simulate: null design points");
    if ((d_init && (reinterpret_cast<uintptr_t>(d_init) & 15u)) ||
        (d_final && (reinterpret_cast<uintptr_t>(d_final) & 15u)))
        return fail(MRIP_EINVAL, "mrip_forest_fire_skip_simulate: state buffers need 16-byte alignment");
    LogTable tab;
    mrip_status rc = log_table(&tab);
    if (rc != MRIP_OK) return rc;
    const RoundKeys rk = expand_key(seed);
    const uint32_t t_dens = threshold32(density);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    switch (L) {
        case 32: rc = launch_ff_skip<1>(d_dps, n_items, n_reps, rep0, n_steps, t_dens, rk, tab, d_init, d_counts, d_scalar, d_final, st); break;
        case 64: rc = launch_ff_skip<2>(d_dps, n_items, n_reps, rep0, n_steps, t_dens, rk, tab, d_init, d_counts, d_scalar, d_final, st); break;
        case 128: rc = launch_ff_skip<4>(d_dps, n_items, n_reps, rep0, n_steps, t_dens, rk, tab, d_init, d_counts, d_scalar, d_final, st); break;
        case 256: rc = launch_ff_skip<8>(d_dps, n_items, n_reps, rep0, n_steps, t_dens, rk, tab, d_init, d_counts, d_scalar, d_final, st); break;
        case 512: rc = launch_ff_skip<16>(d_dps, n_items, n_reps, rep0, n_steps, t_dens, rk, tab, d_init, d_counts, d_scalar, d_final, st); break;
    }
    if (rc != MRIP_OK) return rc;
    return launch_status("mrip_forest_fire_skip_simulate");
}

extern "C" mrip_status mrip_forest_fire_simulate(const double* d_dps, int32_t n_dp, int64_t rep0, int64_t n_reps,
                                                 int32_t L, int32_t n_steps, double density,
                                                 uint64_t seed, const uint8_t* d_init,
                                                 int32_t* d_counts, double* d_scalar,
                                                 uint8_t* d_final, void* stream) {
    return forest_fire_launch(d_dps, n_dp, rep0, n_reps, L, n_steps, density, seed, d_init, d_counts,
                              d_scalar, d_final, static_cast<cudaStream_t>(stream));
}

MRIP_DEBUG_UNIT(forest_fire)

// Library runtime: thread-local error state, per-device scratch memory,
// device error flags, and the random-stream stage entry points
// (mrip_philox, mrip_expo).
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "common.cuh"

namespace mrip {

namespace {
thread_local std::string g_last_error;

struct DeviceScratch {
    void* ptr[8] = {nullptr};
    size_t bytes[8] = {0};
    int* flags = nullptr;
    int sms = 0;
    LogSlice* log_slices = nullptr;
};
std::mutex g_scratch_mutex;
std::vector<DeviceScratch> g_scratch;

DeviceScratch& dev_scratch() {
    int dev = 0;
    cudaGetDevice(&dev);
    if (static_cast<int>(g_scratch.size()) <= dev) g_scratch.resize(dev + 1);
    return g_scratch[dev];
}
}  // namespace

void set_error(const std::string& msg) { g_last_error = msg; }

mrip_status fail(mrip_status code, const std::string& msg) {
    g_last_error = msg;
    return code;
}

mrip_status cuda_status(cudaError_t e, const char* what) {
    if (e == cudaSuccess) return MRIP_OK;
    return fail(MRIP_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

mrip_status launch_status(const char* what) { return cuda_status(cudaGetLastError(), what); }

void* scratch(size_t bytes, int slot) {
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    DeviceScratch& d = dev_scratch();
    if (d.bytes[slot] >= bytes && d.ptr[slot]) return d.ptr[slot];
    if (d.ptr[slot]) {
        cudaDeviceSynchronize();  // the old buffer may still be in use
        cudaFree(d.ptr[slot]);
        d.ptr[slot] = nullptr;
        d.bytes[slot] = 0;
    }
    size_t want = bytes < 256 ? 256 : bytes;
    if (cudaMalloc(&d.ptr[slot], want) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    d.bytes[slot] = want;
    return d.ptr[slot];
}

int* device_error_flags() {
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    DeviceScratch& d = dev_scratch();
    if (!d.flags) {
        if (cudaMalloc(&d.flags, 16 * sizeof(int)) != cudaSuccess) {
            cudaGetLastError();
            d.flags = nullptr;
            return nullptr;
        }
        cudaMemset(d.flags, 0, 16 * sizeof(int));
    }
    return d.flags;
}

namespace {
// neg_log_q58's 64-bit sum without the n ln 2 term, for the mantissa mh:ml of
// slice e.
unsigned long long log_core(uint32_t mh, uint32_t ml, const LogSlice& e) {
    auto hi_u = [](uint32_t a, uint32_t b) { return static_cast<uint32_t>((static_cast<uint64_t>(a) * b) >> 32); };
    auto hi_s = [](int32_t a, int32_t b) { return static_cast<int32_t>((static_cast<int64_t>(a) * b) >> 32); };
    const uint64_t V = static_cast<uint64_t>(mh) * e.w + hi_u(ml, e.w);
    const int32_t a = static_cast<int32_t>(static_cast<uint32_t>(V >> 13));
    const uint32_t r2 = static_cast<uint32_t>(hi_s(a, a));
    const float f = static_cast<float>(a);
    const float tail = std::fma(f * f * f, std::fma(f, kLogR4, kLogR3), kLogMagic);
    uint32_t bits;
    std::memcpy(&bits, &tail, sizeof(bits));
    return e.lnw - V + ((r2 + (bits - kLogMagicBits)) >> 1);
}

// The slices' w_j and ln w_j from the host's long-double logarithm (64-bit or
// wider mantissa).  w_j keeps |r| <= 2^-14 over its slice; among up to 49 such
// 27-bit values around 1/c_j the one whose logarithm's rounding to 2^-58, about
// the mean 0.05 of the truncations, is smallest.
void build_log_slices(std::vector<LogSlice>& t) {
    constexpr long double kMean = 0.05L;
    t.resize(kLogSlices);
    for (int j = 0; j < kLogSlices; ++j) {
        const long double from = 1.0L + static_cast<long double>(j) / kLogSlices;
        const long double to = 1.0L + static_cast<long double>(j + 1) / kLogSlices;
        const long long lo = static_cast<long long>(ceill(ldexpl((1.0L - 0x1p-14L) / from, 27)));
        const long long hi = static_cast<long long>(floorl(ldexpl((1.0L + 0x1p-14L) / to, 27)));
        const long long mid = static_cast<long long>(ldexpl(2.0L / (from + to), 27) + 0.5L);
        long double best = 2.0L;
        for (long long w = mid - 24; w <= mid + 24; ++w) {
            if (w < lo || w > hi) continue;
            const long double x = ldexpl(logl(ldexpl(static_cast<long double>(w), -27)), 58) + kMean;
            const long double r = floorl(x + 0.5L);
            if (fabsl(x - r) < best) {
                best = fabsl(x - r);
                t[j].w = static_cast<uint32_t>(w);
                t[j].lnw = (1ull << 58) - static_cast<unsigned long long>(-r);
                t[j].pad = 0;
            }
        }
    }
}
}  // namespace

mrip_status log_table(LogTable* out) {
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    DeviceScratch& d = dev_scratch();
    if (!d.log_slices) {
        std::vector<LogSlice> t;
        build_log_slices(t);
        // n ln2 2^58 rounded, from the 128-bit product n * round(ln2 2^64);
        // entry 64 makes K = 2^53 (M = 1 in slice 0) exactly 0
        const unsigned long long ln2_q64 = static_cast<unsigned long long>(ldexpl(logl(2.0L), 64) + 0.5L);
        std::vector<unsigned long long> nln2(kLogExponents);
        for (unsigned s = 0; s < 64; ++s) {
            const unsigned __int128 prod = static_cast<unsigned __int128>(s + 1) * ln2_q64 + 32u;
            nln2[s] = static_cast<unsigned long long>(prod >> 6);
        }
        nln2[64] = 0ull - log_core(0x80000000u, 0u, t[0]);
        // before the first slice stand zeros, for the look-ups of rare words (neg_log_impl)
        t.insert(t.begin(), kLogSlices, LogSlice{0, 0, 0});
        const size_t slice_bytes = t.size() * sizeof(LogSlice);
        LogSlice* p = nullptr;
        cudaError_t e = cudaMalloc(&p, slice_bytes + nln2.size() * sizeof(unsigned long long));
        if (e == cudaSuccess) e = cudaMemcpy(p, t.data(), slice_bytes, cudaMemcpyHostToDevice);
        if (e == cudaSuccess)
            e = cudaMemcpy(reinterpret_cast<char*>(p) + slice_bytes, nln2.data(),
                           nln2.size() * sizeof(unsigned long long), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) {
            if (p) cudaFree(p);
            return cuda_status(e, "log table upload");
        }
        d.log_slices = p;
    }
    out->slice = reinterpret_cast<const ulonglong2*>(d.log_slices);
    out->nln2_shared = 0;
    out->nln2 = reinterpret_cast<const unsigned long long*>(d.log_slices + 2 * kLogSlices);
    return MRIP_OK;
}

int sm_count() {
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    DeviceScratch& d = dev_scratch();
    if (d.sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev);
        if (d.sms <= 0) d.sms = 1;
    }
    return d.sms;
}

// ---------------------------------------------------------------------------
// Random-stream stages
// ---------------------------------------------------------------------------
__global__ void philox_kernel(const uint4* __restrict__ ctr, const uint2* __restrict__ key,
                              long long n, uint4* __restrict__ out) {
    long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    if (i >= n) return;
    uint4 c = ctr[i];
    uint2 k = key[i];
    uint32_t a = k.x, b = k.y;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        philox_round(c.x, c.y, c.z, c.w, a, b);
        a += 0x9E3779B9u;
        b += 0xBB67AE85u;
    }
    out[i] = c;
}

__global__ void expo_kernel(const uint32_t* __restrict__ lo, const uint32_t* __restrict__ hi,
                            const double* __restrict__ rate, long long n, double* __restrict__ u_out,
                            double* __restrict__ e_out, LogTable tab) {
    long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    if (i >= n) return;
    if (u_out) u_out[i] = u53(lo[i], hi[i]);
    if (e_out) e_out[i] = expo_fast<false>(lo[i], hi[i], tab, 0x1p-58 / rate[i]);
}

}  // namespace mrip

using namespace mrip;

extern "C" const char* mrip_last_error(void) { return g_last_error.c_str(); }

extern "C" mrip_status mrip_philox(const uint32_t* d_ctr, const uint32_t* d_key, int64_t n,
                                   uint32_t* d_out, void* stream) {
    if (n < 0) return fail(MRIP_EINVAL, "mrip_philox: n < 0");
    if (n == 0) return MRIP_OK;
    if (!d_ctr || !d_key || !d_out) return fail(MRIP_EINVAL, "mrip_philox: null pointer");
    if ((reinterpret_cast<uintptr_t>(d_ctr) | reinterpret_cast<uintptr_t>(d_out)) & 15u ||
        reinterpret_cast<uintptr_t>(d_key) & 7u)
        return fail(MRIP_EINVAL, "mrip_philox: misaligned buffer (ctr/out need 16 B, key 8 B)");
    philox_kernel<<<ceil_div_u(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        reinterpret_cast<const uint4*>(d_ctr), reinterpret_cast<const uint2*>(d_key), n,
        reinterpret_cast<uint4*>(d_out));
    return launch_status("mrip_philox");
}

extern "C" mrip_status mrip_expo(const uint32_t* d_lo, const uint32_t* d_hi, const double* d_rate,
                                 int64_t n, double* d_u, double* d_e, void* stream) {
    if (n < 0) return fail(MRIP_EINVAL, "mrip_expo: n < 0");
    if (n == 0) return MRIP_OK;
    if (!d_lo || !d_hi || (d_e && !d_rate)) return fail(MRIP_EINVAL, "mrip_expo: null pointer");
    LogTable tab;
    mrip_status s = log_table(&tab);
    if (s != MRIP_OK) return s;
    expo_kernel<<<ceil_div_u(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        d_lo, d_hi, d_rate, n, d_u, d_e, tab);
    return launch_status("mrip_expo");
}

#ifdef MRIP_DEBUG
namespace mrip {
namespace {
// One deliberately failed check (site 999, index 12345): no access is
// guarded by it, it only exercises the record.
__global__ void debug_selftest_kernel() { (void)MRIP_CHECK(threadIdx.x != 0, 999, 12345); }
}  // namespace
mrip_status debug_take_runtime(unsigned long long* rec);
mrip_status debug_take_forest_fire(unsigned long long* rec);
mrip_status debug_take_queues(unsigned long long* rec);
mrip_status debug_take_walk(unsigned long long* rec);
mrip_status debug_take_mlp(unsigned long long* rec);
mrip_status debug_take_cv(unsigned long long* rec);
mrip_status debug_take_area_walk(unsigned long long* rec);
mrip_status debug_take_stats(unsigned long long* rec);
}  // namespace mrip
#endif

extern "C" mrip_status mrip_debug_checks(int32_t* enabled, uint64_t* first) {
    if (!enabled || !first) return fail(MRIP_EINVAL, "mrip_debug_checks: null argument");
    *first = 0;
#ifdef MRIP_DEBUG
    *enabled = 1;
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return cuda_status(e, "mrip_debug_checks");
    using Take = mrip_status (*)(unsigned long long*);
    const Take units[] = {debug_take_runtime, debug_take_forest_fire, debug_take_queues,
                          debug_take_walk,    debug_take_mlp,         debug_take_cv,
                          debug_take_area_walk, debug_take_stats};
    for (Take take : units) {  // every unit is read (and cleared); the first record is kept
        unsigned long long rec = 0;
        const mrip_status s = take(&rec);
        if (s != MRIP_OK) return s;
        if (*first == 0) *first = rec;
    }
#else
    *enabled = 0;
#endif
    return MRIP_OK;
}

extern "C" mrip_status mrip_debug_selftest(void) {
#ifdef MRIP_DEBUG
    debug_selftest_kernel<<<1, 32>>>();
    return launch_status("mrip_debug_selftest");
#else
    return fail(MRIP_EINVAL, "mrip_debug_selftest: not a debug build");
#endif
}

extern "C" mrip_status mrip_check_device_flags(void) {
    int* flags = device_error_flags();
    if (!flags) return fail(MRIP_ENOMEM, "device error flags: allocation failed");
    int host[16];
    cudaError_t e = cudaMemcpy(host, flags, sizeof(host), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_status(e, "mrip_check_device_flags");
    if (host[0] != 0) {
        cudaMemset(flags, 0, sizeof(host));
        return fail(MRIP_ESTEPCAP, "a replication reached its step cap (its output is -1)");
    }
    return MRIP_OK;
}

MRIP_DEBUG_UNIT(runtime)

// Median spacing of a sorted grid of epochs, and the grid's ends, on the device.
//
// The default phase step is the median of t[i+1] - t[i].  Copying the epochs to
// the host and sorting the differences there took 112 us of a mixed fold's 281 at
// 16 000 epochs and 232 of 431 at 30 000.  Here one block selects the middle
// element (or the two middle ones) by radix, eight bits of an order-preserving key
// per pass, and 32 bytes come back: 35 and 79 us with the wait for them.
#include <algorithm>
#include <cstring>
#include <vector>

#include "nu_internal.cuh"

namespace nu {

__host__ __device__ inline unsigned long long bits_key(unsigned long long b) {
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ unsigned long long diff_key(double x) {
    return bits_key((unsigned long long)__double_as_longlong(x));
}
__device__ __forceinline__ double key_diff(unsigned long long k) {
    const unsigned long long b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double((long long)b);
}

// The differences' keys once: an FP64 subtraction holds its pipe for 64 cycles
// per warp, and the selection reads every difference up to nine times.
__global__ void k_diff_keys(const double* __restrict__ t, int64_t m,
                            unsigned long long* __restrict__ key) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < m) key[i] = diff_key(t[i + 1] - t[i]);
}

// out = {element (m - 1) / 2, element m / 2 of the sorted differences, t[0], t[m]}.
// key: those of k_diff_keys.
__global__ void __launch_bounds__(1024)
k_median(const double* __restrict__ t, int64_t m, const unsigned long long* __restrict__ key,
         double* __restrict__ out) {
    __shared__ unsigned hist[256];
    __shared__ unsigned long long sh_prefix, sh_next;
    __shared__ unsigned sh_rank, sh_left;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        sh_prefix = 0ull;
        sh_rank = (unsigned)((m - 1) / 2);      // (m < 2^31)
        sh_next = ~0ull;
    }
    for (int shift = 56; shift >= 0; shift -= 8) {
        if (threadIdx.x < 256) hist[threadIdx.x] = 0u;
        __syncthreads();
        const unsigned long long prefix = sh_prefix;
        for (int64_t base = 0; base < m; base += blockDim.x) {
            const int64_t i = base + threadIdx.x;
            const unsigned long long k = i < m ? key[i] : 0ull;
            // (shift + 8 = 64: every key has the empty prefix)
            const bool in = i < m && (shift == 56 || (k >> (shift + 8)) == prefix);
            const unsigned bin = in ? (unsigned)(k >> shift) & 255u : 256u;
            // most spacings are the cadence: one atomic per distinct bin and warp
            const unsigned same = __match_any_sync(FULL, bin);
            if (in && lane == __ffs(same) - 1) atomicAdd(&hist[bin], (unsigned)__popc(same));
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            // the bin of the rank: eight bins a lane, prefix sums over the lanes
            unsigned h[8], sum = 0u;
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                h[b] = hist[8 * lane + b];
                sum += h[b];
            }
            unsigned before = sum;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned v = __shfl_up_sync(FULL, before, o);
                if (lane >= o) before += v;
            }
            before -= sum;
            const unsigned r = sh_rank;
            __syncwarp();
            if (r >= before && r < before + sum) {          // (one lane)
                int b = 0;
                while (r >= before + h[b]) before += h[b++];
                sh_rank = r - before;
                sh_prefix = (prefix << 8) | (unsigned)(8 * lane + b);
                sh_left = h[b];
            }
        }
        __syncthreads();
    }
    const unsigned long long lo = sh_prefix;
    // the next element: the same value when more of it are left, else the
    // smallest larger one
    const bool again = sh_rank + 1u < sh_left || (m & 1);
    if (!again) {
        unsigned long long best = ~0ull;
        for (int64_t i = threadIdx.x; i < m; i += blockDim.x) {
            const unsigned long long k = key[i];
            if (k > lo && k < best) best = k;
        }
        if (best != ~0ull) atomicMin(&sh_next, best);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        out[0] = key_diff(lo);
        out[1] = again ? out[0] : key_diff(sh_next);
        out[2] = t[0];
        out[3] = t[m];
    }
}

// Grids this short: the same selection on the host.  The copy and the selection
// take less than the kernel's eight dependent passes (14 us) and its launch
// (whole fold of 1 100 epochs x 4 durations x 300 periods, mixed: 128 -> 108 us).
constexpr int64_t MEDIAN_HOST = 4096;

static cudaError_t median_on_host(const double* t_dev, int64_t n, cudaStream_t st, double* step,
                                  double* t_first, double* t_last) {
    std::vector<double> t(n);
    cudaError_t e = cudaMemcpyAsync(t.data(), t_dev, n * sizeof(double), cudaMemcpyDeviceToHost,
                                    st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    const int64_t m = n - 1;
    std::vector<unsigned long long> key(m);
    for (int64_t i = 0; i < m; ++i) {
        const double d = t[i + 1] - t[i];
        unsigned long long b;
        std::memcpy(&b, &d, 8);
        key[i] = bits_key(b);
    }
    auto value = [](unsigned long long k) {
        const unsigned long long b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
        double d;
        std::memcpy(&d, &b, 8);
        return d;
    };
    const auto mid = key.begin() + m / 2;
    std::nth_element(key.begin(), mid, key.end());
    const double hi = value(*mid);
    *step = (m % 2) ? hi : 0.5 * (value(*std::max_element(key.begin(), mid)) + hi);
    *t_first = t[0];
    *t_last = t[m];
    return cudaSuccess;
}

cudaError_t median_spacing(const double* t_dev, int64_t n, cudaStream_t st, double* step,
                           double* t_first, double* t_last) {
    const int64_t m = n - 1;
    if (m > 0 && n <= MEDIAN_HOST) return median_on_host(t_dev, n, st, step, t_first, t_last);
    char* mem = nullptr;
    pool_keep_memory();
    cudaError_t e = cudaMallocAsync((void**)&mem, (size_t)m * 8 + 256, st);
    if (e != cudaSuccess) return e;
    unsigned long long* key = (unsigned long long*)(mem + 256);
    if (m > 0) k_diff_keys<<<div_up(m, 256), 256, 0, st>>>(t_dev, m, key);
    k_median<<<1, 1024, 0, st>>>(t_dev, m, key, (double*)mem);
    count_launches(m > 0 ? 2 : 1);
    double h[4];
    e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(h, mem, sizeof(h), cudaMemcpyDeviceToHost, st);
    const cudaError_t f = cudaFreeAsync(mem, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    *step = (m % 2) ? h[1] : 0.5 * (h[0] + h[1]);
    *t_first = h[2];
    *t_last = h[3];
    return f;
}

}  // namespace nu

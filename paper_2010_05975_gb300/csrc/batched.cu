// Batched LU: many independent small matrices (n <= 1024), one persistent
// launch.  Each CTA takes matrices from a queue ordered largest first and
// runs the whole blocked tournament-pivoting factorization of one matrix on
// its own (batched_lu.cuh).
#include "batched_lu.cuh"
#include "batched_solve.cuh"
#include "common.cuh"
#include "ddiv.cuh"
#include "node_gepp.cuh"
#include "prof.cuh"
#include <climits>
#include <mutex>

namespace lu {
namespace bat {

// Panel width by size class: class c holds 2^(c+4) < n <= 2^(c+5) (class 0
// also n <= 32), c = 0..5 up to n = 1024.  The defaults are the fastest of
// 8 / 16 / 32 per class measured on GB300 (2048 matrices per class, both
// precisions): 32 everywhere, 10-17 % ahead of 16 for 129 <= n <= 512 and
// level with it (within timing noise) for n <= 64.
// lu_batched_set_panel_widths replaces them for a tuning sweep.
constexpr int kWidthClasses = 6;
struct Widths {
    int w[kWidthClasses];
};
__host__ __device__ inline int width_class(int n) {
    int c = 0;
    while (c < kWidthClasses - 1 && n > (32 << c)) ++c;
    return c;
}
__host__ __device__ inline int panel_width(const Widths& t, int n) { return t.w[width_class(n)]; }

// The queue of matrices, largest first, zeroed before the size kernels.
// Binary32 CTAs take from its front.  In binary64 the FP64 pipes of an SM are
// shared by its CTAs, so two large matrices on one SM both run at half its
// rate: with 2 048 matrices of n log-uniform in [16, 1024] the SM that got the
// two largest finished after 202 ms, the work of all SMs being 105 ms each.
// There an SM's first CTA takes from the front; its second one takes from the
// front as long as the SM's share of the whole batch's work (plus a
// sixteenth and kSlackWork, below which nothing is bound by the FP64 pipes)
// allows it, then from the back, the smallest, and ends when not even those
// fit: 132 ms.  What a CTA takes is what one atomic addition gives it: a look at
// the queue first decides the end, and what arrives from the front meanwhile is
// no larger.  (With a compare-and-swap on what was looked at, the CTAs took one matrix
// in 0.4 us between them all: 349 us for 600 of n = 16, now 94.)
constexpr int kSmIds = 256;
constexpr unsigned kQueueBias = 1u << 20; // both ends start here: takes past the end (one a CTA) do not wrap
constexpr unsigned long long kSlackWork = 512;           // a matrix of order 128
struct Queue {
    unsigned long long ends;              // next at the front (low word), end of the queue (high word)
    unsigned long long total;             // the batch's work
    unsigned long long load[kSmIds];      // work taken by each SM
    int slot[kSmIds];                     // CTAs seen on each SM
};
__host__ __device__ inline unsigned long long matrix_work(int n) {
    if (n <= 0 || n > kMaxN) return 1;
    const unsigned long long m = (n + 15) / 16;
    return m * m * m;
}

// The position in `order` of the CTA's next matrix, or -1 (thread 0).
__device__ __forceinline__ int queue_take(Queue* q, bool back) {
    const unsigned long long e = atomicAdd(&q->ends, back ? 0xffffffff00000000ull : 1ull);
    const unsigned f = static_cast<unsigned>(e), b = static_cast<unsigned>(e >> 32);
    return f < b ? static_cast<int>((back ? b - 1 : f) - kQueueBias) : -1;
}
__device__ __forceinline__ int take_shared(Queue* q, const int* order, const int* ns, unsigned sm, bool first,
                                           unsigned long long limit) {
    bool back = false;
    if (!first) {
        const unsigned long long load = *reinterpret_cast<volatile unsigned long long*>(&q->load[sm]);
        const unsigned long long e = *reinterpret_cast<volatile unsigned long long*>(&q->ends);
        const unsigned f = static_cast<unsigned>(e), b = static_cast<unsigned>(e >> 32);
        if (f >= b) return -1;
        if (load + matrix_work(ns[order[f - kQueueBias]]) > limit) {
            if (load + matrix_work(ns[order[b - 1 - kQueueBias]]) > limit) return -1;
            back = true;
        }
    }
    const int t = queue_take(q, back);
    if (t >= 0) atomicAdd(&q->load[sm], matrix_work(ns[order[t]]));
    return t;
}

template <typename T>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 ? 3 : 2)
    batched_lu_kernel(int batch, const int* __restrict__ ns, T* const* __restrict__ As, const int* __restrict__ ldas,
                      int* const* __restrict__ pivs, int* __restrict__ info, const int* __restrict__ order, Queue* q,
                      int sms, Widths widths) {
    Smem<T>& sm = shared_mem<T>();
    unsigned smid = 0;
    bool first = true;
    unsigned long long limit = 0;
    if (sizeof(T) == 8 && threadIdx.x == 0) {
        asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
        smid %= kSmIds;
        first = atomicAdd(&q->slot[smid], 1) == 0;
        limit = q->total / sms + q->total / sms / 16 + kSlackWork;
        // a later CTA of the SM waits (a fraction of a millisecond at most)
        // until the first one has taken its matrix
        for (int i = 0; !first && i < 4096; ++i) {
            const unsigned long long e = *reinterpret_cast<volatile unsigned long long*>(&q->ends);
            if (*reinterpret_cast<volatile unsigned long long*>(&q->load[smid]) != 0 ||
                static_cast<unsigned>(e) >= static_cast<unsigned>(e >> 32))
                break;
            __nanosleep(64);
        }
    }
    for (;;) {
        if (threadIdx.x == 0)
            sm.next = sizeof(T) == 4 ? queue_take(q, false) : take_shared(q, order, ns, smid, first, limit);
        __syncthreads();
        const int t = sm.next;
        __syncthreads();
        if (t < 0) break;
        const int mi = order[t];
        const int n = ns[mi];
        T* A = As[mi];
        const int lda = ldas[mi];
        int* piv = pivs[mi];
        if (n < 0 || n > kMaxN || (n > 0 && (A == nullptr || piv == nullptr || lda < n))) {
            if (threadIdx.x == 0) info[mi] = -1;
            continue;
        }
        if (threadIdx.x == 0) sm.zero_first = -1;
        int first_zero = -1;
        const int b = panel_width(widths, n);
        for (int k = 0; k < n; k += b) {
            const int w = min(b, n - k);
            tournament(sm, A, lda, n, k, w);
            if (threadIdx.x == 0 && first_zero < 0 && sm.zero_first >= 0) first_zero = k + sm.zero_first;
            if (threadIdx.x == 0) sm.zero_first = -1;
            if (threadIdx.x < 32) resolve_swaps(sm, k, w, piv);
            __syncthreads();
            swap_and_u12<T>(A, lda, n, k, w);
            __syncthreads();
            if (k + w >= n) break;
            solve_l21<T>(A, lda, n, k, w);
            // (a remainder of up to 64 or, in binary64, any: 64 x 64 tiles)
            if (sizeof(T) == 8 || n - k - w <= 64)
                schur<T, 4>(A, lda, n, k, w);
            else
                schur<T, tile_rows<T>()>(A, lda, n, k, w);
        }
        if (threadIdx.x == 0) info[mi] = first_zero >= 0 ? first_zero + 1 : 0;
        __syncthreads();
    }
}

// Largest-first order by a counting sort on n (sizes outside [0, kMaxN] go last).
__global__ void size_hist_kernel(int batch, const int* __restrict__ ns, int* __restrict__ hist) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < batch; i += gridDim.x * blockDim.x) {
        const int n = ns[i];
        const int key = (n >= 0 && n <= kMaxN) ? kMaxN - n : kMaxN + 1;
        atomicAdd(&hist[key], 1);
    }
}
// (one CTA: warp sums of the kMaxN + 2 counts, then their prefix)
__global__ void __launch_bounds__(1024) size_scan_kernel(int batch, int* __restrict__ hist, Queue* __restrict__ q) {
    __shared__ int part[33];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int N = kMaxN + 2;
    const int i0 = 2 * tid, a = i0 < N ? hist[i0] : 0, b = i0 + 1 < N ? hist[i0 + 1] : 0;
    int v = a + b;
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) part[warp] = v;
    __syncthreads();
    if (warp == 0) {
        int s = part[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += u;
        }
        part[lane] = s;
    }
    __syncthreads();
    const int before = v - a - b + (warp > 0 ? part[warp - 1] : 0);
    if (i0 < N) hist[i0] = before;
    if (i0 + 1 < N) hist[i0 + 1] = before + a;
    // (the count at key i is that of order kMaxN - i)
    unsigned long long work = static_cast<unsigned long long>(a) * matrix_work(kMaxN - i0) +
                              static_cast<unsigned long long>(b) * matrix_work(kMaxN - i0 - 1);
    for (int o = 16; o > 0; o >>= 1) work += __shfl_xor_sync(0xffffffffu, work, o);
    if (lane == 0 && work != 0) atomicAdd(&q->total, work);
    if (tid == 0) q->ends = (static_cast<unsigned long long>(kQueueBias + static_cast<unsigned>(batch)) << 32) | kQueueBias;
}
__global__ void size_scatter_kernel(int batch, const int* __restrict__ ns, int* __restrict__ hist,
                                    int* __restrict__ order) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < batch; i += gridDim.x * blockDim.x) {
        const int n = ns[i];
        const int key = (n >= 0 && n <= kMaxN) ? kMaxN - n : kMaxN + 1;
        order[atomicAdd(&hist[key], 1)] = i;
    }
}

template <typename T>
__global__ void __launch_bounds__(kThreads) batched_solve_kernel(int batch, const int* __restrict__ ns,
                                                                 const int* __restrict__ nrhss,
                                                                 T* const* __restrict__ LUs, const int* __restrict__ ldas,
                                                                 int* const* __restrict__ pivs, T* const* __restrict__ Bs,
                                                                 const int* __restrict__ ldbs) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SolveSmem<T>& sm = *reinterpret_cast<SolveSmem<T>*>(smem_raw);
    for (int mi = blockIdx.x; mi < batch; mi += gridDim.x) {
        const int n = ns[mi], nr = nrhss[mi];
        if (n <= 0 || n > kMaxN || nr <= 0 || nr > kSolveNr) continue;
        batched_solve_one(sm, n, nr, LUs[mi], ldas[mi], pivs[mi], Bs[mi], ldbs[mi]);
    }
}

// measured defaults per dtype (index 0 binary64, 1 binary32) and the
// table in use
constexpr Widths kDefaultWidths[2] = {{{32, 32, 32, 32, 32, 32}}, {{32, 32, 32, 32, 32, 32}}};
static std::mutex g_width_mu;
static Widths g_widths[2] = {kDefaultWidths[0], kDefaultWidths[1]};

static Widths widths_for(int dtype) {
    std::lock_guard<std::mutex> lk(g_width_mu);
    return g_widths[dtype == LU_PREC_F32 ? 1 : 0];
}

}  // namespace bat

static int sms() {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 148;
}

template <typename T>
static int factor_batched(int batch, const int* n, T* const* A, const int* lda, int* const* piv, int* info,
                          const bat::Widths& widths, cudaStream_t s) {
    void* ws = nullptr;
    const size_t zeroed = sizeof(bat::Queue) + (bat::kMaxN + 2) * sizeof(int);
    if (lu_malloc_async(&ws, zeroed + static_cast<size_t>(batch) * sizeof(int), s) != cudaSuccess) {
        cudaGetLastError();
        return LU_ENOMEM;
    }
    bat::Queue* q = static_cast<bat::Queue*>(ws);
    int* hist = reinterpret_cast<int*>(q + 1);
    int* order = hist + bat::kMaxN + 2;
    int rc = 0;
    if (cudaMemsetAsync(ws, 0, zeroed, s) != cudaSuccess) rc = LU_ELAUNCH;
    if (!rc) {
        ProfScope ps(LU_PROF_OTHER, s);
        bat::size_hist_kernel<<<cdiv(batch, 256), 256, 0, s>>>(batch, n, hist);
        bat::size_scan_kernel<<<1, 1024, 0, s>>>(batch, hist, q);
        bat::size_scatter_kernel<<<cdiv(batch, 256), 256, 0, s>>>(batch, n, hist, order);
        count_launches(3);
        if (cudaPeekAtLastError() != cudaSuccess) rc = LU_ELAUNCH;
    }
    if (!rc) {
        const size_t smem = sizeof(bat::Smem<T>);
        rc = smem_attr(bat::batched_lu_kernel<T>, smem);
        int per_sm = 0;
        if (!rc && cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bat::batched_lu_kernel<T>, bat::kThreads,
                                                                 smem) != cudaSuccess)
            rc = LU_ELAUNCH;
        if (!rc) {
            const int nsm = sms(), grid = nsm * (per_sm > 0 ? per_sm : 1);
            ProfScope ps(LU_PROF_SCHUR, s);
            bat::batched_lu_kernel<T><<<grid < batch ? grid : batch, bat::kThreads, smem, s>>>(
                batch, n, A, lda, piv, info, order, q, nsm, widths);
            count_launches(1);
            if (cudaPeekAtLastError() != cudaSuccess) rc = LU_ELAUNCH;
        }
    }
    cudaGetLastError();
    cudaFreeAsync(ws, s);
    return rc;
}

}  // namespace lu

using namespace lu;

extern "C" int lu_batched_panel_width(int n) { return bat::panel_width(bat::widths_for(LU_PREC_F64), n); }

extern "C" int lu_batched_panel_width_dt(int n, int dtype) {
    if (dtype != LU_PREC_F64 && dtype != LU_PREC_F32) return -2;
    return bat::panel_width(bat::widths_for(dtype), n);
}

extern "C" int lu_batched_set_panel_widths(int dtype, const int* widths, int count) {
    if (dtype != LU_PREC_F64 && dtype != LU_PREC_F32) return -1;
    const int d = dtype == LU_PREC_F32 ? 1 : 0;
    if (widths == nullptr) {
        std::lock_guard<std::mutex> lk(bat::g_width_mu);
        bat::g_widths[d] = bat::kDefaultWidths[d];
        return 0;
    }
    if (count != bat::kWidthClasses) return -3;
    bat::Widths t{};
    for (int c = 0; c < count; ++c) {
        if (widths[c] < 1 || widths[c] > bat::kMaxB) return -2;
        t.w[c] = widths[c];
    }
    std::lock_guard<std::mutex> lk(bat::g_width_mu);
    bat::g_widths[d] = t;
    return 0;
}

extern "C" int lu_factor_batched(int batch, const int* n, void* const* A, const int* lda, int* const* piv, int* info,
                                 int dtype, cudaStream_t stream) {
    if (batch < 0) return -1;
    if (batch == 0) return 0;
    if (n == nullptr) return -2;
    if (A == nullptr) return -3;
    if (lda == nullptr) return -4;
    if (piv == nullptr) return -5;
    if (info == nullptr) return -6;
    if (dtype == LU_PREC_F64)
        return factor_batched<double>(batch, n, reinterpret_cast<double* const*>(A), lda, piv, info,
                                      bat::widths_for(dtype), stream);
    if (dtype == LU_PREC_F32)
        return factor_batched<float>(batch, n, reinterpret_cast<float* const*>(A), lda, piv, info,
                                     bat::widths_for(dtype), stream);
    return -7;
}

extern "C" int lu_solve_batched(int batch, const int* n, const int* nrhs, void* const* LU, const int* lda,
                                int* const* piv, void* const* B, const int* ldb, int dtype, cudaStream_t stream) {
    if (batch < 0) return -1;
    if (batch == 0) return 0;
    if (!n || !nrhs || !LU || !lda || !piv || !B || !ldb) return -2;
    // one CTA per matrix: the device hands the next one out when a CTA ends
    const int grid = batch < (1 << 20) ? batch : (1 << 20);
    ProfScope ps(LU_PROF_SOLVE, stream);
    if (dtype == LU_PREC_F64) {
        const size_t smem = sizeof(bat::SolveSmem<double>);
        if (int rc_ = smem_attr(bat::batched_solve_kernel<double>, smem)) return rc_;
        bat::batched_solve_kernel<double><<<grid, bat::kThreads, smem, stream>>>(
            batch, n, nrhs, reinterpret_cast<double* const*>(LU), lda, piv, reinterpret_cast<double* const*>(B), ldb);
    } else if (dtype == LU_PREC_F32) {
        const size_t smem = sizeof(bat::SolveSmem<float>);
        if (int rc_ = smem_attr(bat::batched_solve_kernel<float>, smem)) return rc_;
        bat::batched_solve_kernel<float><<<grid, bat::kThreads, smem, stream>>>(
            batch, n, nrhs, reinterpret_cast<float* const*>(LU), lda, piv, reinterpret_cast<float* const*>(B), ldb);
    } else {
        return -9;
    }
    count_launches(1);
    LU_LAUNCHED();
    return 0;
}

// Solve A X = B with the factors P A = L U (getrs): X = U^{-1} L^{-1} P B.
// The linear solve is what the paper's factorization serves ("linear
// solvers", Section 1); the paper does not spell it out.  A Cholesky factor
// L goes through the same machinery with U = L^T and no permutation.
//
// A solve plan holds what depends on the factors only: the row permutation
// composed from the swap sequence piv, and the inverses of the NB x NB
// diagonal blocks of L (unit lower) and U (upper), stored row-major.  The
// refinement keeps one plan per factorization; the one-shot entry points
// build and drop one per call.
//
// Applying a plan: B is gathered through the permutation into Y (row stride
// nc, padded to a width of 8, 16, 32 or 64), then one kernel runs the
// blocked forward and backward substitutions: in binary64 as a list of work
// items taken in order from an atomic counter, in binary32 as a chain of steps
// in one cluster that the other CTAs feed.  Every wait is bounded and on work
// that a running CTA holds or that the waiting one can take, so the kernels
// progress whatever number of their CTAs is resident.  Every product has a
// fixed order, so results do not depend on timing.  Right-hand sides go
// through in passes of up to 64 (binary32: 32).
#include "common.cuh"
#include "ddiv.cuh"
#include "prof.cuh"
#include <climits>
#include <mutex>

namespace lu {

// perm[i] = the row that the swap sequence piv brings to position i, by one
// CTA, 256 swaps at a time (a replay by one thread takes 35 ns a swap: 20 us at
// n = 512, 1.1 ms at 32768).  Before swap j of a batch, position i0 + j holds
// C(j): the row that the last earlier swap j' aiming there displaced, C(j'),
// or its own.  The swap brings there what its target holds: C(j') of the last
// earlier swap j' with the same target, or the target's own row.  A target
// past the batch ends with C(j) of the last swap aiming at it.  "The last
// earlier swap aiming at v" is a scan of the batch in shared memory, done for
// all swaps at once.
constexpr int kPermBatch = 256;
__global__ void __launch_bounds__(kPermBatch) perm_from_piv(int n, const int* __restrict__ piv,
                                                            int* __restrict__ perm) {
    __shared__ int s_p[kPermBatch], s_prev[kPermBatch];
    const int t = threadIdx.x;
    for (int i = t; i < n; i += kPermBatch) perm[i] = i;
    for (int i0 = 0; i0 < n; i0 += kPermBatch) {
        const int m = min(kPermBatch, n - i0), i = i0 + t;
        const int p = t < m ? piv[i] : -1;
        // (the previous batch's perm is written after this barrier)
        if (__syncthreads_or(t < m && p < i)) {          // not a sequence that LAPACK makes: replay it
            if (t == 0)
                for (int j = i0; j < i0 + m; ++j) {
                    const int q = piv[j], a = perm[j];
                    perm[j] = perm[q];
                    perm[q] = a;
                }
            continue;
        }
        s_p[t] = p;
        __syncthreads();
        // the last earlier swap aiming at this position, and at this target;
        // whether a later one aims at this target
        int here = -1, same = -1;
        bool last = true;
        for (int j = 0; j < m; ++j) {
            const int pj = s_p[j];
            if (j < t && pj == i) here = j;
            if (j < t && pj == p) same = j;
            if (j > t && pj == p) last = false;
        }
        s_prev[t] = here;
        __syncthreads();
        auto content = [&](int j) {                      // C(j), a position before the batch
            while (s_prev[j] >= 0) j = s_prev[j];
            return i0 + j;
        };
        int to = -1, from_target = -1, own = -1;
        if (t < m) {
            own = content(t);
            to = perm[p == i ? own : same >= 0 ? content(same) : p];
            if (last && p >= i0 + m) from_target = perm[own];
        }
        __syncthreads();
        if (t < m) {
            perm[i] = to;
            if (last && p >= i0 + m) perm[p] = from_target;
        }
    }
}

// Block size of the substitution: NB = 128 for binary32, 64 for binary64
// (the inversion kernel holds two NB x NB tiles in shared memory).
template <typename T>
struct SolveNB {
    static constexpr int value = sizeof(T) == 4 ? 128 : 64;
};

// Dinv[blk][kind] = inv(diag block), row-major, one CTA per block, factor and
// quarter of its columns, which are independent; right-looking in shared
// memory: at step p every row after p (before it, for U) takes its update from
// the finished row p of the inverse, sixteen threads per column, the rows
// between them.  (A thread that summed its column's rows one after another
// waited for a shared-memory read per term: 126 us for 64-wide binary64 blocks
// and 215 us for 128-wide binary32 ones; right-looking on one CTA 60 and 197, the
// FP64 pipes' share of one SM and two barriers a step; now 38 and 104.)  With chol
// set the factors are L (non-unit lower, from a Cholesky factorization) and
// L^T: both kinds compute inv(L_bb), kind 1 stores inv(L_bb^T) = inv(L_bb)^T.
__device__ __forceinline__ unsigned inv_rec(float) { return 0u; }
__device__ __forceinline__ unsigned inv_rec(double x) { return div_rec(x); }
__device__ __forceinline__ float inv_div(float a, float b, unsigned) { return a / b; }
__device__ __forceinline__ double inv_div(double a, double b, unsigned rec) { return div_by(a, b, rec); }

constexpr int kInvParts = 4;

template <typename T>
__global__ void __launch_bounds__(4 * SolveNB<T>::value) invert_diag_kernel(int n, const T* __restrict__ LU, int lda,
                                                                            T* __restrict__ Dinv, int chol) {
    constexpr int NB = SolveNB<T>::value, SP = NB + 1;
    constexpr int QC = NB / kInvParts;                   // columns of this CTA
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* S = reinterpret_cast<T*>(smem_raw);              // NB x SP
    T* Xs = S + NB * SP;                                 // NB x (QC + 1), column c0 + c at Xs[p][c]
    const int blk = blockIdx.x, kind = blockIdx.y, c0 = blockIdx.z * QC;   // kind 0: L (unit lower), 1: U (upper)
    const int r0 = blk * NB, nb = min(NB, n - r0);
    const int tid = threadIdx.x, c = tid % QC, g = tid / QC;
    constexpr int G = 4 * NB / QC;                       // threads per column
    __shared__ unsigned s_rec[NB];
#pragma unroll 4
    for (int e = tid; e < NB * NB; e += 4 * NB) {
        const int i = e / NB, j = e % NB;
        S[i * SP + j] = (i < nb && j < nb) ? LU[idx(r0 + i, r0 + j, lda)] : T(0);
    }
    for (int e = tid; e < NB * QC; e += 4 * NB) {
        const int i = e / QC, j = e % QC;
        Xs[i * (QC + 1) + j] = (i == c0 + j && i < nb) ? T(1) : T(0);
    }
    __syncthreads();
    if (tid < NB) s_rec[tid] = inv_rec(S[tid * SP + tid]);
    __syncthreads();
    const bool lower = chol || kind == 0, divide = chol || kind == 1;
    // the steps before the first of these columns (after the last, for U) have nothing to do
    for (int s = lower ? c0 : max(0, nb - c0 - QC); s < nb; ++s) {
        const int p = lower ? s : nb - 1 - s;
        const bool col = lower ? c0 + c <= p : (c0 + c >= p && c0 + c < nb);   // columns with a value in row p
        T x = T(0);
        if (col) {
            x = Xs[p * (QC + 1) + c];
            if (divide) x = inv_div(x, S[p * SP + p], s_rec[p]);
        }
        __syncthreads();                                 // row p has been read by all
        if (col) {
            if (g == 0) Xs[p * (QC + 1) + c] = x;
            if (lower) {
                for (int i = p + 1 + g; i < nb; i += G)
                    Xs[i * (QC + 1) + c] = fma(-S[i * SP + p], x, Xs[i * (QC + 1) + c]);
            } else {
                for (int i = p - 1 - g; i >= 0; i -= G)
                    Xs[i * (QC + 1) + c] = fma(-S[i * SP + p], x, Xs[i * (QC + 1) + c]);
            }
        }
        __syncthreads();
    }
    // row-major: out[i][p] = inv[i][p] (rows arrive in the solve by 16-byte copies)
    T* out = Dinv + (static_cast<size_t>(blk) * 2 + kind) * NB * NB;
    if (chol && kind == 1) {
        // out[i][p] = inv(L^T)[i][p] = inv(L)[p][i]
        for (int e = tid; e < NB * QC; e += 4 * NB) out[(c0 + e / NB) * NB + e % NB] = Xs[(e % NB) * (QC + 1) + e / NB];
    } else {
        for (int e = tid; e < NB * QC; e += 4 * NB) out[e / QC * NB + c0 + e % QC] = Xs[e / QC * (QC + 1) + e % QC];
    }
}

// Right-hand sides per pass (binary32: as many as the chain's shared memory holds).
template <typename T>
constexpr int kSolveRhs = sizeof(T) == 8 ? 64 : 32;

// Item list bookkeeping (device memory, zeroed before each pass but for timeout,
// which a call's passes share and the host reads once, after the last).
struct SolveSync {
    int timeout;       // 1: a wait ran out; 2: an exchange of the chain's cluster did
    int next;          // next item to take
    int pad[2];
};

// Wait by thread 0 until *flag >= want, at most limit_ns of wall-clock time
// (%globaltimer, read every 64 polls); a wait that runs out records the
// timeout.  After any timeout every such wait returns at once, so a broken run
// ends quickly (its results are then invalid and the host reports
// LU_ETIMEOUT).  The waits of a CTA's warps for one another, and of the
// chain's CTAs for their exchanges, do not return then: they keep the CTA's
// barriers in step, and end as soon as the waits that they depend on have.
__device__ __forceinline__ void solve_wait(const int* flag, int want, SolveSync* sy, unsigned long long limit_ns) {
    const volatile int* f = flag;
    const volatile int* to = &sy->timeout;
    unsigned long long t0 = 0;
    for (unsigned it = 1; *f < want; ++it) {
        if ((it & 63) == 0) {
            if (*to) return;
            const unsigned long long now = global_ns();
            if (t0 == 0) {
                t0 = now;
            } else if (now - t0 > limit_ns) {
                atomicMax(&sy->timeout, 1);
                return;
            }
        }
        __nanosleep(32);
    }
}

// ---------------------------------------------------------------------------
// The binary32 substitution.  With V the right-hand side, step s of a phase
// (forward: block s; backward: block nblk - 1 - s) is
//   Z_s = inv(C_ss) (V_s - C_{s,s-4} Z_{s-4} - .. - C_{s,s-1} Z_{s-1}),
// V_s having taken the updates of the steps up to s - 5.  The steps run in one
// cluster of eight CTAs, 16 rows of the block each, that keeps the last
// solutions in its shared memory (results go to all eight by asynchronous
// stores that count on the receivers' barriers, twice a step).  Eight warps do
// the products, eight fetch the next step's coefficients, one waits for the
// next step's V_s and fetches it, one publishes the last step's solution: only
// two products and two exchanges are on the chain.  The other CTAs bring V_t,
// t >= 5, up to date, taking the blocks (or 64 or 32 of their rows, so that the
// blocks of a smaller system occupy them all) in order: such a task holds its
// sums in registers and follows the chain, step by step, its coefficients
// fetched ahead.  A solution's way to the task of the block after next and
// back to the chain takes about 8 us, which the four blocks that the chain treats
// itself (kChainNear) cover.  Steps by way of work items took 7.5 to 10 us each (17
// with 64 right-hand sides): two products of a whole block on one CTA, and a
// block's updates one after another through counters.  Measured against
// those, 16 right-hand sides: n = 12001 1.57 -> 0.75 ms, 32768 5.08 -> 1.95 (four: 8192 0.97 -> 0.32).
//
// Progress needs the cluster only: while it waits for updates that nobody has
// taken its waiting warps take them over, each CTA's its own 16 rows.  With no
// other CTA resident n = 4000 takes 22 ms and 8192 109 (16 right-hand sides; 281 and
// 2 734 when one warp did a whole task, an element at a time).  Beside a stream
// of matrix products that fills the chip n = 4000 takes 2.5 ms, 32768 5 (by way of
// work items 3.5 and 9.5).
// ---------------------------------------------------------------------------
constexpr int kChainCtas = 8;
constexpr int kChainThreads = 256;                           // of the products; as many fetch coefficients
constexpr int kChainBlock = 2 * kChainThreads + 64;          // and two warps
constexpr int kChainNear = 4;                                // blocks before its own that a step treats itself
constexpr int kChainNb = SolveNB<float>::value;              // 128
constexpr int kChainRows = kChainNb / kChainCtas;            // 16: a chain CTA's rows, an urgent item's rows
constexpr int kChainPitch = kChainNb + 4;                    // floats: 16-byte rows in distinct bank groups
constexpr unsigned long long kChainPatience = 20000;         // ns until a waiting chain CTA takes a task
constexpr int kChainTaken = 256;                             // done[]: units below, taken tasks from here on

// Shared memory (floats).  Chain: two sums of 16-row products, two sets of
// coefficients, the ring of solutions, U, two V.  Task of RT rows: the sums' last
// step, and stages of coefficients and a solution.
__host__ __device__ constexpr int chain_stages(int rt) { return rt == 128 ? 2 : 4; }
template <int NCW>
constexpr size_t chain_words() {
    return 16 * static_cast<size_t>(kChainRows) * NCW + 2 * static_cast<size_t>(kChainNear + 1) * kChainRows * kChainPitch +
           (kChainNear + 2) * static_cast<size_t>(kChainNb) * NCW + 2 * static_cast<size_t>(kChainRows) * NCW;
}
template <int NCW, int RT>
constexpr size_t chain_smem() {
    const size_t work = 16 * static_cast<size_t>(kChainThreads) +
                        chain_stages(RT) * (static_cast<size_t>(RT) * kChainPitch + static_cast<size_t>(kChainNb) * NCW);
    return (chain_words<NCW>() > work ? chain_words<NCW>() : work) * sizeof(float);
}
static_assert(chain_smem<32, 128>() <= 227 * 1024 && chain_smem<32, 64>() <= 227 * 1024, "one CTA per SM");

// 4-byte asynchronous copy, zero when bytes is 0.
__device__ __forceinline__ void chain_cp4(float* dst, const float* src, int bytes) {
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}

// Coefficient block of target rows [r0, r0 + rows) and source columns
// [c0, c0 + 128) to shared memory, zero outside the matrix; trans: the
// transposed element (a Cholesky factor's U = L^T).
__device__ __forceinline__ void chain_stage(float* dst, const float* LU, int lda, int n, int r0, int rows, int c0,
                                            bool trans, bool vec, int tid) {
    if (trans) {
        for (int e = tid; e < rows * kChainNb; e += kChainThreads) {
            const int i = e % rows, p = e / rows;
            const bool ok = r0 + i < n && c0 + p < n;
            chain_cp4(dst + i * kChainPitch + p, ok ? LU + idx(c0 + p, r0 + i, lda) : LU, ok ? 4 : 0);
        }
    } else if (vec) {
        for (int e = tid; e < rows * (kChainNb / 4); e += kChainThreads) {
            const int i = e / (kChainNb / 4), p = 4 * (e % (kChainNb / 4));
            const int bytes = r0 + i < n ? 4 * max(0, min(4, n - c0 - p)) : 0;
            cp_async16(dst + i * kChainPitch + p, bytes ? LU + idx(r0 + i, c0 + p, lda) : LU, bytes);
        }
    } else {
        for (int e = tid; e < rows * kChainNb; e += kChainThreads) {
            const int i = e / kChainNb, p = e % kChainNb;
            const bool ok = r0 + i < n && c0 + p < n;
            chain_cp4(dst + i * kChainPitch + p, ok ? LU + idx(r0 + i, c0 + p, lda) : LU, ok ? 4 : 0);
        }
    }
}

// acc += C (16 x 128) B (128 x NCW), this warp's sixteen terms: a lane's rows
// rg + 32 / CG i and four columns.
template <int NCW>
__device__ __forceinline__ void chain_product(const float* C, const float* B, float (&acc)[NCW / 8][4]) {
    constexpr int CG = NCW / 4, RL = NCW / 8;
    const int lane = threadIdx.x & 31, k0 = 16 * (threadIdx.x >> 5), cg = lane % CG, rg = lane / CG;
#pragma unroll
    for (int p = 0; p < 16; p += 4) {
        float4 b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) b[q] = *reinterpret_cast<const float4*>(B + (k0 + p + q) * NCW + 4 * cg);
#pragma unroll
        for (int i = 0; i < RL; ++i) {
            const float4 c = *reinterpret_cast<const float4*>(C + (rg + 32 / CG * i) * kChainPitch + k0 + p);
            const float cv[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                acc[i][0] = fmaf(cv[q], b[q].x, acc[i][0]);
                acc[i][1] = fmaf(cv[q], b[q].y, acc[i][1]);
                acc[i][2] = fmaf(cv[q], b[q].z, acc[i][2]);
                acc[i][3] = fmaf(cv[q], b[q].w, acc[i][3]);
            }
        }
    }
}

// The eight warps' sums of a 16-row product to shared memory; after a barrier
// chain_sum adds them for one row and four columns, in warp order.
template <int NCW>
__device__ __forceinline__ void chain_put(float* red, const float (&acc)[NCW / 8][4]) {
    constexpr int CG = NCW / 4, RL = NCW / 8;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, cg = lane % CG, rg = lane / CG;
#pragma unroll
    for (int i = 0; i < RL; ++i)
        *reinterpret_cast<float4*>(red + (warp * kChainRows + rg + 32 / CG * i) * NCW + 4 * cg) =
            make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
}
template <int NCW>
__device__ __forceinline__ float4 chain_sum(const float* red, int row, int c) {
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        const float4 x = *reinterpret_cast<const float4*>(red + (w * kChainRows + row) * NCW + c);
        s.x += x.x;
        s.y += x.y;
        s.z += x.z;
        s.w += x.w;
    }
    return s;
}
__device__ __forceinline__ float4 chain_sub(float4 a, float4 b) {
    return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}

// Tasks in order: phase, step t >= kChainNear + 1, rows RT part ..
struct ChainTask {
    int ph, t, part;         // t: -1 past the last one
};
__host__ __device__ inline int chain_tasks(int nblk, int rt) {            // of both phases
    return nblk > kChainNear + 1 ? 2 * (nblk - kChainNear - 1) * (kChainNb / rt) : 0;
}
__device__ __forceinline__ ChainTask chain_task(int nblk, int rt, int i) {
    const int parts = kChainNb / rt, per = chain_tasks(nblk, rt) / 2;
    ChainTask k;
    k.ph = i < per ? 0 : 1;
    const int e = i - k.ph * per;
    k.t = e / parts + kChainNear + 1;
    k.part = e % parts;
    return k;
}

// What the kernel works on.  Y: V forward and the result backward; X: the other.
struct ChainArgs {
    int n, nblk, lda, chol, vec, inject;
    const float* LU;
    const float* DT;
    float* Y;
    float* X;
    int* done[2];            // per step: 16-row units of its block that are up to date
    int* solved[2];          // per step: chain CTAs that have published it
    SolveSync* sy;
    unsigned long long wait_ns;
};
__device__ __forceinline__ int chain_block(const ChainArgs& a, int ph, int s) { return ph == 0 ? s : a.nblk - 1 - s; }

__device__ __forceinline__ void chain_bar_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void chain_bar_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
constexpr int kChainPair = kChainThreads + 32;       // the product warps and one other
constexpr int kChainFed = 2 * kChainThreads + 32;    // and the fetching warps

// A helper warp's wait for a counter in shared memory, which the other warps of the
// CTA advance after bounded waits of their own.  It does not look at the
// timeout: a helper that ran ahead of the others would arrive at their barriers
// out of turn.  The limit lies beyond any that it can depend on.
__device__ __forceinline__ void chain_follow(const volatile int* at, int want, const ChainArgs& a) {
    unsigned long long t0 = 0;
    while (*at < want) {
        __nanosleep(20);
        const unsigned long long now = global_ns();
        if (t0 == 0) t0 = now;
        else if (now - t0 > 64 * (a.wait_ns + 1000000000ull)) {
            atomicMax(&a.sy->timeout, 1);
            break;
        }
    }
    __syncwarp();
}

// How a task's 256 product threads divide RT x NCW sums over 128 terms a step:
// 4 rows and 4 columns each, KS shares of the terms.
template <int NCW, int RT>
struct ChainTile {
    static constexpr int CG = NCW / 4, RG = RT / 4, KS = kChainThreads / (CG * RG), KN = kChainNb / KS;
    static_assert(KS >= 1 && KN % 4 == 0, "a share is a multiple of four terms");
};

// 16 rows of a task that the chain took over, whose steps are all solved: by one
// warp, from global memory, in the order of the other form.  A lane has one
// column and NCW / 2 rows, eight at a time.
template <int NCW, int RT>
__device__ __noinline__ void chain_unit_direct(const ChainArgs& a, int ph, int t, int rank) {
    constexpr int KS = ChainTile<NCW, RT>::KS, KN = ChainTile<NCW, RT>::KN;
    constexpr int J = NCW / 2 < 8 ? NCW / 2 : 8, RS = 32 / NCW;
    const int lane = threadIdx.x & 31, c = lane % NCW, r0 = chain_block(a, ph, t) * kChainNb + rank * kChainRows;
    const bool trans = a.chol && ph == 1;
    const size_t rs = trans ? 1 : a.lda, ps = trans ? a.lda : 1;    // element (row, p) at rs row + ps p
    float* V = (ph == 0 ? a.Y : a.X) + c;
    const float* Z = (ph == 0 ? a.X : a.Y) + c;
#pragma unroll 1
    for (int r = r0 + lane / NCW; r < r0 + kChainRows && r0 < a.n; r += RS * J) {
        const float* L[J];
        float acc[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            L[j] = a.LU + rs * min(r + RS * j, a.n - 1);
            acc[j] = 0.0f;
        }
#pragma unroll 1
        for (int ks = 0; ks < KS; ++ks) {
            float sum[J];
#pragma unroll
            for (int j = 0; j < J; ++j) sum[j] = 0.0f;
#pragma unroll 1
            for (int s = 0; s < t - kChainNear; ++s) {
                const int p0 = chain_block(a, ph, s) * kChainNb + ks * KN, p1 = min(p0 + KN, a.n);
                float run[J];
#pragma unroll
                for (int j = 0; j < J; ++j) run[j] = 0.0f;
#pragma unroll 4
                for (int p = p0; p < p1; ++p) {
                    const float z = __ldcg(Z + static_cast<size_t>(p) * NCW);
#pragma unroll
                    for (int j = 0; j < J; ++j) run[j] = fmaf(L[j][ps * p], z, run[j]);
                }
#pragma unroll
                for (int j = 0; j < J; ++j) sum[j] += run[j];
            }
#pragma unroll
            for (int j = 0; j < J; ++j) acc[j] += sum[j];
        }
#pragma unroll
        for (int j = 0; j < J; ++j)
            if (r + RS * j < a.n) {
                float* v = V + static_cast<size_t>(r + RS * j) * NCW;
                *v = __ldcg(v) - acc[j];
            }
    }
    __syncwarp();
    if (lane == 0) {
        __threadfence();
        atomicAdd(a.done[ph] + t, 1);
    }
    __syncwarp();
}

// The bounded wait for the rest of a block's units.
__device__ __forceinline__ void chain_wait_units(const int* done, const ChainArgs& a) {
    const volatile int* f = done;
    const unsigned long long t0 = global_ns();
    while ((*f & (kChainTaken - 1)) < kChainNb / kChainRows && *static_cast<volatile int*>(&a.sy->timeout) == 0) {
        __nanosleep(32);
        if (global_ns() - t0 > a.wait_ns) atomicMax(&a.sy->timeout, 1);
    }
}

// One warp of chain CTA `rank`: the wait for its block (phase ph, step s).
// done[ph][s] holds the units that are up to date and, above them, a bit per task
// of the block that the chain took over: after kChainPatience one of the eight
// CTAs takes the next task if it is the block's, and each CTA does its own 16
// rows of it.
template <int NCW, int RT>
__device__ __forceinline__ void chain_wait(const ChainArgs& a, int ph, int s, int rank) {
    if (s <= kChainNear) return;
    const int total = chain_tasks(a.nblk, RT), bit = kChainTaken << (rank * kChainRows / RT);
    int* f = a.done[ph] + s;
    bool own = false;                                        // its rows are still to be done here
    if ((threadIdx.x & 31) == 0) {
        const unsigned long long t0 = global_ns();
        for (;;) {
            const int v = *static_cast<volatile int*>(f);
            if ((v & (kChainTaken - 1)) >= kChainNb / kChainRows || *static_cast<volatile int*>(&a.sy->timeout)) break;
            if (v & bit) {
                own = true;
                break;
            }
            const unsigned long long t = global_ns() - t0;
            if (t < kChainPatience) continue;
            const int next = *static_cast<volatile int*>(&a.sy->next);
            const ChainTask k = chain_task(a.nblk, RT, next);
            if (next < total && k.ph == ph && k.t == s) {
                if (atomicCAS(&a.sy->next, next, next + 1) == next) atomicAdd(f, kChainTaken << k.part);
            } else if (t > a.wait_ns) {                      // taken by others
                atomicMax(&a.sy->timeout, 1);
                break;
            } else {
                __nanosleep(32);
            }
        }
        __threadfence();
    }
    if (__shfl_sync(0xffffffffu, own ? 1 : 0, 0) == 0) return;
    chain_unit_direct<NCW, RT>(a, ph, s, rank);
    if ((threadIdx.x & 31) == 0) {
        chain_wait_units(f, a);
        __threadfence();
    }
    __syncwarp();
}

__device__ __forceinline__ void chain_mbar_init(unsigned long long* b, int count) {
    asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(static_cast<unsigned>(__cvta_generic_to_shared(b))), "r"(count)
                 : "memory");
}
__device__ __forceinline__ void chain_mbar_expect(unsigned long long* b, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared.b64 _, [%0], %1;" ::"r"(
                     static_cast<unsigned>(__cvta_generic_to_shared(b))), "r"(bytes)
                 : "memory");
}
// The stores of all eight CTAs for one exchange (the copies of a stage) are in.
// They come within the time limit of the waits that their senders may be in; past
// that (and once another such wait has found so) they are given up: false, and
// the chain goes through its remaining steps without exchanges.
__device__ __forceinline__ bool chain_mbar_wait(unsigned long long* b, unsigned parity, const ChainArgs& a) {
    const unsigned at = static_cast<unsigned>(__cvta_generic_to_shared(b));
    unsigned long long t0 = 0;
    for (unsigned it = 1;; ++it) {
        unsigned ok;
        asm volatile(
            "{\n.reg .pred p;\n"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(at), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((it & 63) == 0) {
            if (*static_cast<volatile int*>(&a.sy->timeout) == 2) return false;
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > 2 * a.wait_ns + 1000000000ull) {
                atomicExch(&a.sy->timeout, 2);
                return false;
            }
        }
    }
}
// 16 bytes to another CTA's shared memory, counted by its barrier.
__device__ __forceinline__ void chain_st4(unsigned addr, unsigned bar, float4 v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%2, %3, %4, %5}, [%1];" ::"r"(addr),
                 "r"(bar), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}
__device__ __forceinline__ void chain_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Buffers in use: U is written for step k + 1 only after every CTA has sent Z_k,
// so after it has read U; slot s % 5 of Z only after every CTA has sent its U of
// the step, so after the last read of Z_{s-5}.  When the copies of a result
// are shared out among threads, U's arrival does not show that every thread of
// this CTA has summed up its own: the second product has sums of its own.
template <int NCW, int RT>
__device__ __forceinline__ void chain_run(const ChainArgs& a, float* smem, int rank) {
    constexpr int ROWS = kChainRows, CP = kChainPitch, NB = kChainNb, Q = NCW / 4;
    constexpr int DUP = kChainThreads / (ROWS * Q);          // threads per four results: they share the eight copies
    constexpr int RING = kChainNear + 1, SET = (kChainNear + 1) * ROWS * CP;
    constexpr unsigned kBytes = NB * NCW * sizeof(float);
    float* red = smem;
    float* red2 = red + 8 * ROWS * NCW;                      // (see the note on buffers)
    float* Cf = red2 + 8 * ROWS * NCW;                       // 2 x (inv(C_ss), C_{s,s-1}, .., C_{s,s-4}) x 16 rows
    float* Zr = Cf + 2 * SET;                                // RING x NB x NCW: Z of the last steps
    float* Us = Zr + RING * NB * NCW;                        // NB x NCW
    float* Vs = Us + NB * NCW;                               // 2 x ROWS x NCW: V of this and the next step
    __shared__ __align__(8) unsigned long long bars[2];      // U, Z
    __shared__ volatile int s_prog;                          // steps whose products are done
    const int tid = threadIdx.x & (kChainThreads - 1), warp = threadIdx.x >> 5, lane = tid & 31, nblk = a.nblk, steps = 2 * nblk;
    if (threadIdx.x == 0) {
        chain_mbar_init(bars, 1);
        chain_mbar_init(bars + 1, 1);
        s_prog = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    chain_cluster_sync();
    auto grow = [&](int k) {                                 // k: step counted over both phases
        const int ph = k < nblk ? 0 : 1;
        return chain_block(a, ph, k - ph * nblk) * NB + rank * ROWS;
    };
    if (warp == 16) {
        for (int k = 0; k < steps; ++k) {
            const int ph = k < nblk ? 0 : 1, s = k - ph * nblk, r0 = grow(k);
            if (a.inject && k == 0 && lane == 0) solve_wait(&a.sy->pad[0], 1, a.sy, a.wait_ns);   // test hook
            // (a buffer of two steps ago; the first V of the second phase is the last solution of the first)
            chain_follow(&s_prog, ph == 1 && s == 0 ? k : k - 1, a);
            chain_wait<NCW, RT>(a, ph, s, rank);
            __syncwarp();
            const float* V = ph == 0 ? a.Y : a.X;
            for (int e = lane; e < ROWS * Q; e += 32)
                *reinterpret_cast<float4*>(Vs + (k & 1) * ROWS * NCW + 4 * e) =
                    r0 + e / Q < a.n
                        ? __ldcg(reinterpret_cast<const float4*>(V + static_cast<size_t>(r0) * NCW + 4 * e))
                        : make_float4(0.f, 0.f, 0.f, 0.f);
            chain_bar_arrive(2 + (k & 1), kChainFed);
        }
    } else if (warp == 17) {
        for (int k = 0; k < steps; ++k) {
            chain_bar_sync(4 + (k & 1), kChainPair);
            if (lane == 0) {
                __threadfence();
                s_prog = k + 1;
                const int ph = k < nblk ? 0 : 1;
                atomicAdd(a.solved[ph] + (k - ph * nblk), 1);
            }
            __syncwarp();
        }
    } else if (warp >= 8) {
        for (int k = 0; k < steps; ++k) {
            const int ph = k < nblk ? 0 : 1, s = k - ph * nblk, r0 = grow(k);
            chain_follow(&s_prog, k - 1, a);
            float* d = Cf + (k & 1) * SET;
            const float* D = a.DT + ((static_cast<size_t>(chain_block(a, ph, s)) * 2 + ph) * NB + rank * ROWS) * NB;
            for (int e = tid; e < ROWS * (NB / 4); e += kChainThreads)
                cp_async16(d + e / (NB / 4) * CP + 4 * (e % (NB / 4)), D + 4 * e, 16);
            for (int j = 1; j <= kChainNear && j <= s; ++j)
                chain_stage(d + j * ROWS * CP, a.LU, a.lda, a.n, r0, ROWS, chain_block(a, ph, s - j) * NB, a.chol && ph,
                            a.vec, tid);
            cp_async_wait_all();
            chain_bar_arrive(2 + (k & 1), kChainFed);
        }
    } else {
        const int o = tid % (ROWS * Q), row = o / Q, c = 4 * (o % Q), dup = tid / (ROWS * Q);
        // results of four columns to the same place in all eight CTAs
        auto spread = [&](float* at, unsigned long long* bar, float4 v) {
            const unsigned l = static_cast<unsigned>(__cvta_generic_to_shared(at));
            const unsigned lb = static_cast<unsigned>(__cvta_generic_to_shared(bar));
#pragma unroll
            for (int r = 0; r < kChainCtas / DUP; ++r) {
                unsigned d, db;
                const int to = dup * (kChainCtas / DUP) + r;
                asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(l), "r"(to));
                asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(db) : "r"(lb), "r"(to));
                chain_st4(d, db, v);
            }
        };
        bool on = true;                                      // every exchange so far has come
        for (int k = 0; k < steps; ++k) {
            const int ph = k < nblk ? 0 : 1, s = k - ph * nblk, gr = grow(k) + row;
            const float* d = Cf + (k & 1) * SET;
            if (tid == 0 && on) chain_mbar_expect(bars, kBytes);
            chain_bar_sync(2 + (k & 1), kChainFed);          // V and the coefficients are in
            float4 u = *reinterpret_cast<const float4*>(Vs + (k & 1) * ROWS * NCW + row * NCW + c);
            float acc[NCW / 8][4] = {};
#pragma unroll 1
            for (int j = min(kChainNear, s); j >= 2; --j)
                chain_product<NCW>(d + j * ROWS * CP, Zr + (s - j) % RING * NB * NCW, acc);
            if (k >= 1) on = on && chain_mbar_wait(bars + 1, (k - 1) & 1, a);
            if (tid == 0 && on) chain_mbar_expect(bars + 1, kBytes);
            if (s >= 1) {
                chain_product<NCW>(d + ROWS * CP, Zr + (s - 1) % RING * NB * NCW, acc);
                chain_put<NCW>(red, acc);
                chain_bar_sync(1, kChainThreads);
                if (gr < a.n) u = chain_sub(u, chain_sum<NCW>(red, row, c));
            }
            if (on) spread(Us + (rank * ROWS + row) * NCW + c, bars, u);
            on = on && chain_mbar_wait(bars, k & 1, a);
            float acd[NCW / 8][4] = {};
            chain_product<NCW>(d, Us, acd);
            chain_put<NCW>(red2, acd);
            chain_bar_sync(1, kChainThreads);
            float4 z = chain_sum<NCW>(red2, row, c);
            if (gr >= a.n) z = make_float4(0.f, 0.f, 0.f, 0.f);
            if (on) spread(Zr + (s % RING * NB + rank * ROWS + row) * NCW + c, bars + 1, z);
            if (dup == 0 && gr < a.n)
                *reinterpret_cast<float4*>((ph == 0 ? a.X : a.Y) + static_cast<size_t>(gr) * NCW + c) = z;
            chain_bar_arrive(4 + (k & 1), kChainPair);
        }
        if (on) chain_mbar_wait(bars + 1, (steps - 1) & 1, a);   // (nothing is on its way here any more)
    }
    __syncwarp();
    chain_cluster_sync();
}

__device__ __forceinline__ void chain_mbar_arrive(unsigned long long* b) {
    asm volatile("mbarrier.arrive.shared.b64 _, [%0];" ::"r"(static_cast<unsigned>(__cvta_generic_to_shared(b))) : "memory");
}
// arrives when the thread's copies so far are in
__device__ __forceinline__ void chain_mbar_arrive_copies(unsigned long long* b) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared.b64 [%0];" ::"r"(static_cast<unsigned>(__cvta_generic_to_shared(b)))
                 : "memory");
}

template <int NCW, int RT>
__device__ __forceinline__ void chain_work(const ChainArgs& a, float* smem) {
    constexpr int CP = kChainPitch, NB = kChainNb, ST = chain_stages(RT), WORDS = RT * CP + NB * NCW;
    constexpr int CG = ChainTile<NCW, RT>::CG, RG = ChainTile<NCW, RT>::RG;
    constexpr int KS = ChainTile<NCW, RT>::KS, KN = ChainTile<NCW, RT>::KN;
    float* red = smem;                                       // KS x RT x NCW
    float* Sg = red + 16 * kChainThreads;                    // ST x (RT x CP coefficients, NB x NCW solution)
    __shared__ ChainTask s_task[4];
    __shared__ __align__(8) unsigned long long s_full[ST], s_empty[ST];
    __shared__ volatile int s_known, s_prog, s_ready;        // tasks taken, tasks done, steps (over the tasks) solved
    const int tid = threadIdx.x & (kChainThreads - 1), warp = threadIdx.x >> 5, lane = tid & 31, nblk = a.nblk;
    if (threadIdx.x == 0) {
        s_known = s_prog = s_ready = 0;
        for (int i = 0; i < ST; ++i) {
            chain_mbar_init(s_full + i, kChainThreads);
            chain_mbar_init(s_empty + i, kChainThreads / 32);
        }
    }
    __syncthreads();
    if (warp == 16) {
        // takes tasks, at most three ahead of the products, and follows the chain for them
        const int total = chain_tasks(nblk, RT);
        int lead[2] = {0, 0}, unit = 0;                      // steps known to be solved
        for (int i = 0;; ++i) {
            chain_follow(&s_prog, i - 3, a);
            ChainTask k{0, -1, 0};
            if (lane == 0) {
                const int e = atomicAdd(&a.sy->next, 1);
                if (e < total) k = chain_task(nblk, RT, e);
                s_task[i & 3] = k;
                __threadfence_block();
                s_known = i + 1;
            }
            k.ph = __shfl_sync(0xffffffffu, k.ph, 0);
            k.t = __shfl_sync(0xffffffffu, k.t, 0);
            if (k.t < 0) return;
            for (int s = 0; s < k.t - kChainNear; ++s) {
                if (s >= lead[k.ph]) {
                    if (lane == 0) {
                        solve_wait(a.solved[k.ph] + s, kChainCtas, a.sy, a.wait_ns);
                        __threadfence();
                    }
                    lead[k.ph] = s + 1;
                }
                ++unit;
                if (lane == 0 && (s + 1 >= lead[k.ph] || s + 1 == k.t - kChainNear || (unit & 3) == 0)) s_ready = unit;
            }
            __syncwarp();
        }
    }
    if (warp == 17) {
        for (int i = 0;; ++i) {
            chain_bar_sync(4 + (i & 1), kChainPair);
            const ChainTask k = s_task[i & 3];
            __syncwarp();
            if (k.t < 0) return;
            if (lane == 0) {
                __threadfence();
                atomicAdd(a.done[k.ph] + k.t, RT / kChainRows);
                s_prog = i + 1;
            }
            __syncwarp();
        }
    }
    int unit = 0;                                            // steps over the tasks
    if (warp >= 8) {
        for (int i = 0;; ++i) {
            chain_follow(&s_known, i + 1, a);
            __threadfence_block();
            const ChainTask k = s_task[i & 3];
            if (k.t < 0) return;
            const int r0 = chain_block(a, k.ph, k.t) * NB + RT * k.part;
            const float* Z = k.ph == 0 ? a.X : a.Y;
            for (int s = 0; s < k.t - kChainNear; ++s, ++unit) {
                const int st = unit % ST, c0 = chain_block(a, k.ph, s) * NB;
                if (unit >= ST) chain_mbar_wait(s_empty + st, (unit / ST - 1) & 1, a);
                float* C = Sg + st * WORDS;
                chain_stage(C, a.LU, a.lda, a.n, r0, RT, c0, a.chol && k.ph, a.vec, tid);
                chain_follow(&s_ready, unit + 1, a);
                __threadfence_block();
#pragma unroll
                for (int e = tid; e < NB * CG; e += kChainThreads) {
                    const int bytes = c0 + e / CG < a.n ? 16 : 0;
                    cp_async16(C + RT * CP + 4 * e, bytes ? Z + static_cast<size_t>(c0) * NCW + 4 * e : Z, bytes);
                }
                chain_mbar_arrive_copies(s_full + st);
            }
        }
    }
    const int cg = tid % CG, rg = tid / CG % RG, ks = tid / (CG * RG);
    for (int i = 0;; ++i) {
        chain_follow(&s_known, i + 1, a);
        __threadfence_block();
        const ChainTask k = s_task[i & 3];
        if (k.t < 0) {
            chain_follow(&s_prog, i - 1, a);
            chain_bar_arrive(4 + (i & 1), kChainPair);
            return;
        }
        float4 acc[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s = 0; s < k.t - kChainNear; ++s, ++unit) {
            const int st = unit % ST;
            chain_mbar_wait(s_full + st, (unit / ST) & 1, a);
            const float* C = Sg + st * WORDS + rg * CP + ks * KN;
            const float* Zs = Sg + st * WORDS + RT * CP + ks * KN * NCW + 4 * cg;
            float4 run[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) run[r] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
            for (int p = 0; p < KN; p += 4) {
                float4 b[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) b[q] = *reinterpret_cast<const float4*>(Zs + (p + q) * NCW);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float4 l = *reinterpret_cast<const float4*>(C + r * RG * CP + p);
                    const float lv[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        run[r].x = fmaf(lv[q], b[q].x, run[r].x);
                        run[r].y = fmaf(lv[q], b[q].y, run[r].y);
                        run[r].z = fmaf(lv[q], b[q].z, run[r].z);
                        run[r].w = fmaf(lv[q], b[q].w, run[r].w);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) chain_mbar_arrive(s_empty + st);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                acc[r].x += run[r].x;
                acc[r].y += run[r].y;
                acc[r].z += run[r].z;
                acc[r].w += run[r].w;
            }
        }
        // the shares together, in order
        chain_bar_sync(1, kChainThreads);                    // (the last task's sums have been read)
#pragma unroll
        for (int r = 0; r < 4; ++r)
            *reinterpret_cast<float4*>(red + (ks * RT + rg + RG * r) * NCW + 4 * cg) = acc[r];
        chain_bar_sync(1, kChainThreads);
        const int r0 = chain_block(a, k.ph, k.t) * NB + RT * k.part;
        float* V = (k.ph == 0 ? a.Y : a.X) + static_cast<size_t>(r0) * NCW;
        for (int e = tid; e < RT * CG; e += kChainThreads) {
            if (r0 + e / CG >= a.n) break;
            float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int q = 0; q < KS; ++q) {
                const float4 x = *reinterpret_cast<const float4*>(red + static_cast<size_t>(q) * RT * NCW + 4 * e);
                sum.x += x.x;
                sum.y += x.y;
                sum.z += x.z;
                sum.w += x.w;
            }
            float4* v = reinterpret_cast<float4*>(V + 4 * e);
            *v = chain_sub(__ldcg(v), sum);
        }
        chain_follow(&s_prog, i - 1, a);
        chain_bar_arrive(4 + (i & 1), kChainPair);
    }
}

template <int NCW, int RT>
__global__ void __launch_bounds__(kChainBlock, 1) solve_chain_kernel(const ChainArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* smem = reinterpret_cast<float*>(smem_raw);
    if (blockIdx.x < kChainCtas)
        chain_run<NCW, RT>(a, smem, static_cast<int>(blockIdx.x));
    else
        chain_work<NCW, RT>(a, smem);
}

// ---------------------------------------------------------------------------
// The binary64 substitution.  An SM's FP64 pipes do two multiply-adds a cycle,
// so a 64 x 64 x 16 block product takes one CTA 16 us; the products on the
// critical path (a block's diagonal solve and its update of the next block)
// are therefore split into items of kSub = 128 / min(NCW, 16) rows, one output
// column group per 16 (8) lanes, which eight (four) CTAs take side by side;
// the updates of the blocks after that go in tiles of 32 rows.  Step b of the
// forward list (the backward list mirrors it from the last block):
//   parts  of block b             X_b = inv(L_bb) Y_b
//   near   rows of block b + 1    Y -= L X_b
//   far    32-row tiles of the blocks from b + 2 on.
// Counters hold, per 32-row tile, the 8-row units that have taken a step's
// update, and per block the parts solved.  Measured, 16 right-hand sides (8 for
// n = 512), against 32-row items throughout on eight CTAs per SM: n = 512 263 ->
// 170 us, 1999 1.82 -> 0.80 ms, 4096 3.88 -> 1.66, 8192 8.48 -> 4.03; 64 right-hand
// sides at 4096 14.0 -> 5.1.
// ---------------------------------------------------------------------------
constexpr int kPartsTile = 32;           // rows of a far tile
constexpr int kPartsUnit = 8;            // rows per unit of a tile's counter
constexpr int kPartsThreads = 128;
constexpr int kPartsNb = SolveNB<double>::value;

template <int NCW>
__host__ __device__ constexpr int parts_cols() { return NCW < 16 ? NCW : 16; }      // lanes along a row
template <int NCW>
__host__ __device__ constexpr int parts_sub() { return kPartsThreads / parts_cols<NCW>(); }   // kSub

// Items of step b: parts, near items, far tiles (forward; backward with the
// blocks counted from the end, block nblk - 1 - st at step st).
struct PartsStep {
    int b, parts, near, far;             // counts
    int near0, far0;                     // first row of block b +- 1; first far tile (backward: the last one)
};
__host__ __device__ inline PartsStep parts_step(int n, int nblk, int st, int sub) {
    PartsStep s{};
    const bool fwd = st < nblk;
    s.b = fwd ? st : 2 * nblk - 1 - st;
    const int NB = kPartsNb, ntile = cdiv(n, kPartsTile), tpb = NB / kPartsTile;
    s.parts = cdiv(n - s.b * NB < NB ? n - s.b * NB : NB, sub);
    if (fwd) {
        s.near0 = (s.b + 1) * NB;
        if (s.near0 < n) s.near = cdiv(n - s.near0 < NB ? n - s.near0 : NB, sub);
        s.far0 = (s.b + 2) * tpb;
        s.far = ntile > s.far0 ? ntile - s.far0 : 0;
    } else {
        s.near0 = (s.b - 1) * NB;
        s.near = s.b > 0 ? NB / sub : 0;
        s.far0 = (s.b - 1) * tpb - 1;
        s.far = s.b > 1 ? (s.b - 1) * tpb : 0;
    }
    return s;
}

// off[st] = items before step st, off[2 nblk] = their number, for a pass of one
// width (the splits differ); one CTA of 256 threads, launched for every pass.
__global__ void solve_parts_offsets_kernel(int n, int sub, int* __restrict__ off) {
    __shared__ int part[257];
    const int nblk = cdiv(n, kPartsNb), t = threadIdx.x;
    const int per = cdiv(2 * nblk, 256), s0 = t * per, s1 = min(s0 + per, 2 * nblk);
    int sum = 0;
    for (int st = s0; st < s1; ++st) {
        const PartsStep s = parts_step(n, nblk, st, sub);
        sum += s.parts + s.near + s.far;
    }
    part[t + 1] = sum;
    __syncthreads();
    if (t == 0) {
        part[0] = 0;
        for (int i = 1; i <= 256; ++i) part[i] += part[i - 1];
    }
    __syncthreads();
    int acc = part[t];
    for (int st = s0; st < s1; ++st) {
        const PartsStep s = parts_step(n, nblk, st, sub);
        off[st] = acc;
        acc += s.parts + s.near + s.far;
    }
    if (t == 0) off[2 * nblk] = part[256];
}

// Forward (L: Y -> X) then backward (U: X -> Y); right-hand sides row-major
// with stride NCW (columns >= nc are zero and stay zero).  With chol set, U is
// L^T: the backward tiles read L transposed.
template <int NCW>
__global__ void __launch_bounds__(kPartsThreads) solve_parts_kernel(int n, const double* __restrict__ LU, int lda,
                                                                    const double* __restrict__ DT,
                                                                    const int* __restrict__ off, double* Y, double* X,
                                                                    int* fdone, int* bdone, int* xpf, int* xpb,
                                                                    SolveSync* sy, int chol,
                                                                    unsigned long long wait_ns, int inject) {
    constexpr int NB = kPartsNb, TR = kPartsTile, SP = NB + 1;
    constexpr int CT = parts_cols<NCW>(), SUB = parts_sub<NCW>();
    constexpr int MR = TR / SUB;                     // rows per thread of a tile
    constexpr int MC = NCW / CT;                     // columns per thread
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* Ls = reinterpret_cast<double*>(smem_raw);   // TR x SP: the item's coefficient rows
    double* Bs = Ls + TR * SP;                       // NB x NCW: the right operand
    int* s_off = reinterpret_cast<int*>(Bs + NB * NCW);
    __shared__ int s_item, s_st;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int nwarp = kPartsThreads / 32;
    const int nblk = cdiv(n, NB);
    for (int i = tid; i <= 2 * nblk; i += kPartsThreads) s_off[i] = off[i];
    __syncthreads();
    const int total = s_off[2 * nblk];
    auto units = [&](int t) { return cdiv(min(TR, n - t * TR), kPartsUnit); };
    int bs_key = -1;                                 // which block Bs holds: (ph * 2 + kind) * nblk + b
    int lo = 0;                                      // thread 0: the last item's step
    for (;;) {
        if (tid == 0) {
            const int item = atomicAdd(&sy->next, 1);
            if (item < total) {
                int hi = 2 * nblk - 1;               // (a CTA's items come in list order)
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (s_off[mid] <= item) lo = mid; else hi = mid - 1;
                }
            }
            s_item = item;
            s_st = lo;
        }
        __syncthreads();
        const int item = s_item;
        if (item >= total) break;
        const PartsStep ps = parts_step(n, nblk, s_st, SUB);
        const int ph = s_st < nblk ? 0 : 1, b = ps.b, k = item - s_off[s_st];
        const int r0 = b * NB, nb = min(NB, n - r0);
        const bool part = k < ps.parts, near = !part && k < ps.parts + ps.near;
        // 1. the coefficient rows (independent of everything in flight)
        int ra, nr;                                  // first output row, rows
        if (part) {
            ra = r0 + k * SUB;
            nr = min(SUB, r0 + nb - ra);
        } else if (near) {
            ra = ps.near0 + (k - ps.parts) * SUB;
            nr = min(SUB, min(ps.near0 + NB, n) - ra);
        } else {
            const int t = ps.far0 + (ph == 0 ? 1 : -1) * (k - ps.parts - ps.near);
            ra = t * TR;
            nr = min(TR, n - ra);
        }
        const int t = ra / TR;                       // the rows' tile
        if (part) {
            const double* D = DT + (static_cast<size_t>(b) * 2 + ph) * NB * NB + static_cast<size_t>(ra - r0) * NB;
            for (int i = warp; i < nr; i += nwarp)
#pragma unroll
                for (int p = lane; p < NB; p += 32) Ls[i * SP + p] = D[static_cast<size_t>(i) * NB + p];
        } else if (chol && ph == 1) {
            // U[ra + i][r0 + p] = L[r0 + p][ra + i]: lanes along the L row
#pragma unroll 4
            for (int p = warp; p < nb; p += nwarp)
                if (lane < nr) Ls[lane * SP + p] = LU[idx(r0 + p, ra + lane, lda)];
        } else {
#pragma unroll 4
            for (int i = warp; i < nr; i += nwarp)
                for (int p = lane; p < nb; p += 32) Ls[i * SP + p] = LU[idx(ra + i, r0 + p, lda)];
        }
        // 2. dependencies, all on earlier items
        if (tid < 4) {                               // a counter per thread
            const int* done = ph == 0 ? fdone : bdone;
            const int steps = ph == 0 ? b : nblk - 1 - b;
            const int* flag = nullptr;
            int want = 0;
            if (tid == 0) {                          // the rows' (or the block's first) tile
                const int u = part ? r0 / TR : t;
                flag = done + u;
                want = steps * units(u);
            } else if (tid == 1) {
                if (!part) {
                    flag = ph == 0 ? xpf + b : xpb + b;
                    want = ps.parts;
                } else if (r0 + TR < r0 + nb) {
                    flag = done + r0 / TR + 1;
                    want = steps * units(r0 / TR + 1);
                }
            } else if (tid == 2) {
                if (ph == 1) {                       // the forward solution of the rows' block
                    const int tb = ra / NB;
                    flag = xpf + tb;
                    want = cdiv(min(NB, n - tb * NB), SUB);
                }
            } else if (inject && item == 0) {        // test hook: a counter nothing increments
                flag = &sy->pad[0];
                want = 1;
            }
            if (flag != nullptr) solve_wait(flag, want, sy, wait_ns);
            __threadfence();
        }
        __syncthreads();
        // 3. the right operand: the block's right-hand side (part) or its solution;
        //    written by other CTAs, so read past L1
        const int key = (ph * 2 + (part ? 0 : 1)) * nblk + b;
        if (bs_key != key) {
            const double* src = (part ? (ph == 0 ? Y : X) : (ph == 0 ? X : Y)) + static_cast<size_t>(r0) * NCW;
#pragma unroll 4
            for (int e = tid; e < nb * NCW; e += kPartsThreads) Bs[e] = __ldcg(src + e);
            bs_key = key;
        }
        __syncthreads();
        // 4. rows tid / CT + SUB m, columns tid % CT + CT k: out = Ls Bs
        const int rr = tid / CT, cc = tid % CT;
        double* out = (part == (ph == 0) ? X : Y) + static_cast<size_t>(ra) * NCW;
        auto rows = [&](auto count) {
            constexpr int M = decltype(count)::value;
            double old[M][MC], acc[M][MC];
#pragma unroll
            for (int m = 0; m < M; ++m)
#pragma unroll
                for (int k2 = 0; k2 < MC; ++k2) {
                    acc[m][k2] = 0.0;
                    const int i = rr + SUB * m;
                    old[m][k2] = (!part && i < nr) ? __ldcg(out + static_cast<size_t>(i) * NCW + cc + CT * k2) : 0.0;
                }
#pragma unroll 4
            for (int p = 0; p < nb; ++p) {
                double bv[MC];
#pragma unroll
                for (int k2 = 0; k2 < MC; ++k2) bv[k2] = Bs[p * NCW + cc + CT * k2];
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    const double l = Ls[(rr + SUB * m) * SP + p];
#pragma unroll
                    for (int k2 = 0; k2 < MC; ++k2) acc[m][k2] = fma(l, bv[k2], acc[m][k2]);
                }
            }
#pragma unroll
            for (int m = 0; m < M; ++m)
#pragma unroll
                for (int k2 = 0; k2 < MC; ++k2) {
                    const int i = rr + SUB * m;
                    if (i < nr)
                        out[static_cast<size_t>(i) * NCW + cc + CT * k2] =
                            part ? acc[m][k2] : old[m][k2] - acc[m][k2];
                }
        };
        if (part || near)
            rows(std::integral_constant<int, 1>{});
        else
            rows(std::integral_constant<int, MR>{});
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            if (part) atomicAdd(ph == 0 ? xpf + b : xpb + b, 1);
            else atomicAdd((ph == 0 ? fdone : bdone) + t, cdiv(nr, kPartsUnit));
        }
    }
}

template <int NCW>
static size_t parts_smem(int n) {
    constexpr int NB = kPartsNb;
    return (static_cast<size_t>(kPartsTile) * (NB + 1) + static_cast<size_t>(NB) * NCW) * sizeof(double) +
           (2 * static_cast<size_t>(cdiv(n, NB)) + 1) * sizeof(int);
}

static int solve_sms() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

// CTAs of the binary64 kernel (none need to be resident together): one per SM
// while a step's far tiles do not outnumber the SMs, else two.  Far tiles on an
// SM delay a part there by the FP64 pipes they take, and a second CTA only
// pays once its staging hides behind another's products (16 right-hand
// sides, one CTA per SM against two and eight: n = 4096 1.66, 1.88, 3.31 ms;
// n = 8192 4.63, 4.03, 7.16).
template <int NCW>
static int parts_grid(int n) {
    const int sms = solve_sms();
    const size_t smem = parts_smem<NCW>(n);
    int per = 0;
    if (smem_attr(solve_parts_kernel<NCW>, smem) != 0) return -1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, solve_parts_kernel<NCW>, kPartsThreads, smem);
    cudaGetLastError();
    if (per < 1 || sms < 1) return -1;
    const int most = cdiv(n, kPartsTile) <= sms ? 1 : 2;
    return sms * (per < most ? per : most);
}

// The chain's cluster and up to `work` CTAs for the tasks: no more than a phase
// has, so that a small system leaves the other SMs to other streams.
template <int NCW, int RT>
static int chain_launch(const ChainArgs& a, int work, cudaStream_t s) {
    const size_t smem = chain_smem<NCW, RT>();
    if (smem_attr(solve_chain_kernel<NCW, RT>, smem) != 0) return LU_EUNSUPPORTED;
    const int tasks = chain_tasks(a.nblk, RT) / 2;
    const int ctas = tasks < work ? tasks : work > kChainCtas ? work : kChainCtas;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((cdiv(ctas, kChainCtas) + 1) * kChainCtas);
    cfg.blockDim = dim3(kChainBlock);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kChainCtas;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, solve_chain_kernel<NCW, RT>, a) != cudaSuccess) {
        cudaGetLastError();
        return LU_ELAUNCH;
    }
    return 0;
}

template <typename T, int NCW>
static int solve_launch(int n, const SolvePlan<T>& p, T* Y, T* X, int* fdone, int* bdone, int* xpf, int* xpb,
                        SolveSync* sy, cudaStream_t s) {
    const WaitCfg wc = wait_cfg(LU_WAIT_SITE_SOLVE);
    if constexpr (sizeof(T) == 8) {
        const int G = parts_grid<NCW>(n);
        if (G <= 0) return LU_EUNSUPPORTED;
        solve_parts_offsets_kernel<<<1, 256, 0, s>>>(n, parts_sub<NCW>(), p.off);
        solve_parts_kernel<NCW><<<G, kPartsThreads, parts_smem<NCW>(n), s>>>(
            n, p.LU, p.lda, p.DT, p.off, Y, X, fdone, bdone, xpf, xpb, sy, p.chol, wc.wait_ns, wc.inject);
        count_launches(2);
    } else {
        ChainArgs a{};
        a.n = n;
        a.nblk = cdiv(n, kChainNb);
        a.lda = p.lda;
        a.chol = p.chol;
        a.vec = (reinterpret_cast<uintptr_t>(p.LU) & 15) == 0 && (p.lda & 3) == 0 ? 1 : 0;
        a.inject = wc.inject;
        a.LU = p.LU;
        a.DT = p.DT;
        a.Y = Y;
        a.X = X;
        a.done[0] = fdone;
        a.done[1] = bdone;
        a.solved[0] = xpf;
        a.solved[1] = xpb;
        a.sy = sy;
        a.wait_ns = wc.wait_ns;
        // tasks of 32 or 64 rows as long as every block's fit on the device at once
        const int work = solve_sms() - kChainCtas;
        const int rc = 4 * a.nblk <= work   ? chain_launch<NCW, 32>(a, work, s)
                       : 2 * a.nblk <= work ? chain_launch<NCW, 64>(a, work, s)
                                            : chain_launch<NCW, 128>(a, work, s);
        if (rc) return rc;
        count_launches(1);
    }
    return 0;
}

// gather with zero padding: Y[i][c] = B[perm[i]][c0 + c] for c < nc, 0 for nc <= c < w
template <typename T>
__global__ void gather_rows_pad(int n, int nc, int w, const int* __restrict__ perm, const T* __restrict__ B, int ldb,
                                T* __restrict__ Y) {
    const long long tot = static_cast<long long>(n) * w;
    for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < tot;
         e += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int i = static_cast<int>(e / w), c = static_cast<int>(e % w);
        Y[e] = c < nc ? B[idx(perm[i], c, ldb)] : T(0);
    }
}

template <typename T>
__global__ void copy_out_pad(int n, int nc, int w, const T* __restrict__ Y, T* __restrict__ B, int ldb) {
    const long long tot = static_cast<long long>(n) * nc;
    for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < tot;
         e += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int i = static_cast<int>(e / nc), c = static_cast<int>(e % nc);
        B[idx(i, c, ldb)] = Y[static_cast<size_t>(i) * w + c];
    }
}

__global__ void perm_identity(int n, int* __restrict__ perm) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) perm[i] = i;
}

// piv == nullptr: LU holds a Cholesky factor L (lower triangle), solved as
// L (L^T X) = B with no permutation.
template <typename T>
int solve_plan_make(int n, const T* LU, int lda, const int* piv, SolvePlan<T>* p, cudaStream_t s) {
    constexpr int NB = SolveNB<T>::value;
    *p = SolvePlan<T>{};
    p->n = n;
    p->LU = LU;
    p->lda = lda;
    p->chol = piv == nullptr ? 1 : 0;
    if (n == 0) return 0;
    const int nblk = cdiv(n, NB);
    if (lu_malloc_async(reinterpret_cast<void**>(&p->perm), sizeof(int) * static_cast<size_t>(n), s) != cudaSuccess ||
        lu_malloc_async(reinterpret_cast<void**>(&p->DT), sizeof(T) * static_cast<size_t>(nblk) * 2 * NB * NB, s) !=
            cudaSuccess ||
        (sizeof(T) == 8 &&
         lu_malloc_async(reinterpret_cast<void**>(&p->off), sizeof(int) * (2 * static_cast<size_t>(nblk) + 1), s) !=
             cudaSuccess)) {
        cudaGetLastError();
        solve_plan_free(p, s);
        return LU_ENOMEM;
    }
    if (p->chol) {
        ProfScope ps(LU_PROF_SOLVE, s);
        perm_identity<<<cdiv(n, 256) < 1024 ? cdiv(n, 256) : 1024, 256, 0, s>>>(n, p->perm);
        count_launches(1);
    } else {
        ProfScope ps(LU_PROF_SOLVE, s);
        perm_from_piv<<<1, kPermBatch, 0, s>>>(n, piv, p->perm);
        count_launches(1);
    }
    LU_LAUNCHED();
    {
        const size_t ismem = static_cast<size_t>(NB) * (NB + 1 + NB / kInvParts + 1) * sizeof(T);
        if (int rc_ = smem_attr(invert_diag_kernel<T>, ismem)) return rc_;
        ProfScope ps(LU_PROF_SOLVE, s);
        invert_diag_kernel<T><<<dim3(nblk, 2, kInvParts), 4 * NB, ismem, s>>>(n, LU, lda, p->DT, p->chol);
        count_launches(1);
    }
    LU_LAUNCHED();
    return 0;
}

template <typename T>
void solve_plan_free(SolvePlan<T>* p, cudaStream_t s) {
    if (p->perm) cudaFreeAsync(p->perm, s);
    if (p->DT) cudaFreeAsync(p->DT, s);
    if (p->off) cudaFreeAsync(p->off, s);
    p->perm = nullptr;
    p->DT = nullptr;
    p->off = nullptr;
}

template <typename T>
int solve_plan_apply(const SolvePlan<T>& p, int nrhs, T* B, int ldb, cudaStream_t s) {
    constexpr int NB = SolveNB<T>::value;
    const int n = p.n;
    if (n == 0 || nrhs == 0) return 0;
    const int nblk = cdiv(n, NB), ntile = cdiv(n, kPartsTile);
    const int nflag = sizeof(T) == 8 ? ntile : nblk;           // per-tile (binary64) or per-block counters
    const size_t vs = static_cast<size_t>(n) * kSolveRhs<T>;
    const size_t flags = sizeof(SolveSync) + sizeof(int) * (2 * static_cast<size_t>(nflag) + 2 * nblk);
    const size_t fbytes = (flags + 255) / 256 * 256;
    void* ws = nullptr;
    if (lu_malloc_async(&ws, fbytes + sizeof(T) * 2 * vs, s) != cudaSuccess) {
        cudaGetLastError();
        return LU_ENOMEM;
    }
    SolveSync* sy = static_cast<SolveSync*>(ws);
    int* fdone = reinterpret_cast<int*>(sy + 1);
    int* bdone = fdone + nflag;
    int* xpf = bdone + nflag;
    int* xpb = xpf + nblk;
    T* Y = reinterpret_cast<T*>(static_cast<unsigned char*>(ws) + fbytes);
    T* X = Y + vs;
    int rc = 0;
    int timeout = 0;
    for (int c0 = 0; c0 < nrhs && !rc; c0 += kSolveRhs<T>) {
        const int nc = (nrhs - c0) < kSolveRhs<T> ? (nrhs - c0) : kSolveRhs<T>;
        const int w = nc <= 8 ? 8 : nc <= 16 ? 16 : nc <= 32 ? 32 : 64;
        const long long tot = static_cast<long long>(n) * w;
        const int gblocks = static_cast<int>(tot / 256 + 1 < 4096 ? tot / 256 + 1 : 4096);
        const size_t kept = c0 > 0 ? offsetof(SolveSync, next) : 0;
        if (cudaMemsetAsync(static_cast<unsigned char*>(ws) + kept, 0, flags - kept, s) != cudaSuccess) {
            rc = LU_ELAUNCH;
            break;
        }
        {
            ProfScope ps(LU_PROF_SOLVE, s);
            gather_rows_pad<T><<<gblocks, 256, 0, s>>>(n, nc, w, p.perm, B + c0, ldb, Y);
            count_launches(1);
        }
        {
            ProfScope ps(LU_PROF_SOLVE, s, 2.0 * static_cast<double>(n) * n * nc);
            if constexpr (sizeof(T) == 8)
                rc = w == 8    ? solve_launch<T, 8>(n, p, Y, X, fdone, bdone, xpf, xpb, sy, s)
                     : w == 16 ? solve_launch<T, 16>(n, p, Y, X, fdone, bdone, xpf, xpb, sy, s)
                     : w == 32 ? solve_launch<T, 32>(n, p, Y, X, fdone, bdone, xpf, xpb, sy, s)
                               : solve_launch<T, 64>(n, p, Y, X, fdone, bdone, xpf, xpb, sy, s);
            else
                rc = w == 8    ? solve_launch<T, 8>(n, p, Y, X, fdone, bdone, xpf, xpb, sy, s)
                     : w == 16 ? solve_launch<T, 16>(n, p, Y, X, fdone, bdone, xpf, xpb, sy, s)
                               : solve_launch<T, 32>(n, p, Y, X, fdone, bdone, xpf, xpb, sy, s);
        }
        if (rc) break;
        {
            ProfScope ps(LU_PROF_SOLVE, s);
            copy_out_pad<T><<<gblocks, 256, 0, s>>>(n, nc, w, Y, B + c0, ldb);
            count_launches(1);
        }
        if (cudaPeekAtLastError() != cudaSuccess) {
            cudaGetLastError();
            rc = LU_ELAUNCH;
            break;
        }
    }
    if (!rc && (cudaMemcpyAsync(&timeout, &sy->timeout, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                cudaStreamSynchronize(s) != cudaSuccess))
        rc = LU_ELAUNCH;
    if (!rc && timeout) rc = LU_ETIMEOUT;
    cudaFreeAsync(ws, s);
    return rc;
}

template <typename T>
int getrs_alloc(int n, int nrhs, const T* LU, int lda, const int* piv, T* B, int ldb, cudaStream_t s) {
    if (n == 0 || nrhs == 0) return 0;
    SolvePlan<T> p;
    int rc = solve_plan_make<T>(n, LU, lda, piv, &p, s);
    if (!rc) rc = solve_plan_apply<T>(p, nrhs, B, ldb, s);
    solve_plan_free<T>(&p, s);
    return rc;
}

template int solve_plan_make<float>(int, const float*, int, const int*, SolvePlan<float>*, cudaStream_t);
template int solve_plan_apply<float>(const SolvePlan<float>&, int, float*, int, cudaStream_t);
template void solve_plan_free<float>(SolvePlan<float>*, cudaStream_t);

int getrs_f64(int n, int nrhs, const double* LU, int lda, const int* piv, double* B, int ldb, cudaStream_t s) {
    return getrs_alloc<double>(n, nrhs, LU, lda, piv, B, ldb, s);
}

int getrs_f32(int n, int nrhs, const float* LU, int lda, const int* piv, float* B, int ldb, cudaStream_t s) {
    return getrs_alloc<float>(n, nrhs, LU, lda, piv, B, ldb, s);
}

}  // namespace lu

using namespace lu;

// Cholesky solve: the same substitution with L and L^T.
template <typename T>
static int chol_solve_t(int n, int nrhs, const T* L, int lda, T* B, int ldb, cudaStream_t s) {
    if (n < 0) return -1;
    if (nrhs < 0 || nrhs > 384) return -2;
    if (n > 0 && L == nullptr) return -3;
    if (lda < (n > 1 ? n : 1)) return -4;
    if (n > 0 && nrhs > 0 && B == nullptr) return -5;
    if (ldb < (nrhs > 1 ? nrhs : 1)) return -6;
    return getrs_alloc<T>(n, nrhs, L, lda, nullptr, B, ldb, s);
}

extern "C" int chol_solve(int n, int nrhs, const double* L, int lda, double* B, int ldb, cudaStream_t stream) {
    return chol_solve_t<double>(n, nrhs, L, lda, B, ldb, stream);
}

extern "C" int chol_solve_f32(int n, int nrhs, const float* L, int lda, float* B, int ldb, cudaStream_t stream) {
    return chol_solve_t<float>(n, nrhs, L, lda, B, ldb, stream);
}


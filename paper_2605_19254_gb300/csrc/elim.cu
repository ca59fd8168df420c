// Elimination over Z/(m) with unit pivots, on the device.  Two uses in the
// Smith-form driver (Section 2):
//  - the last iteration of Phase 2 works modulo a word-size s: the Smith form
//    of A over Z/(s) is the product over the prime powers q^e || s of the
//    local Smith forms over Z/(q^e), and each of those is found by
//    elimination with pivots that are units modulo q;
//  - Phase 3 checks prod s_i = +-det A modulo primes q: det A mod q by
//    Gaussian elimination over GF(q).
//
// Every column takes as pivot a row not yet used whose entry in it is a unit (not
// divisible by q), and every other unused row i subtracts f_i = M[i][k] / M[p][k]
// times the pivot row (no row is moved, so the determinant is the sign of the
// permutation k -> pivot row times the product of the pivots).  A column without
// a unit is left for later ("deferred"): in the local form, once every column has
// been seen, the unused rows and the deferred columns hold a square block whose
// entries are all divisible by q; it is divided by q and reduced again modulo
// q^(e-1).  Its size at each level counts the invariant factors divisible by the
// next power of q.
//
// Moduli below 2^31 go by panels of columns at every size (from the threshold of
// smf_set_elim_panels on), each panel reduced by one thread-block cluster: see
// "Elimination by panels" below, and panel.h.
//
// Wider moduli, and matrices below the threshold, go column by column, with the
// first unused unit row as the pivot.  Products modulo m use Shoup's method there:
// for a multiplier f fixed across a row, f' = floor(f 2^w / m) makes f y mod m =
// f y - floor(y f' / 2^w) m, at most one m too large (w = 32 for m < 2^31, 64 for
// m < 2^62).  Determinants and lockstep local forms (two or more lanes) take one
// launch per column: the launch for column k eliminates it and, in the threads that
// update column k+1, copies that column's new values into a compact buffer and finds
// its first unused unit row (atomicMin).  The last of those blocks to finish (a
// counter, no waiting) takes that row as column k+1's pivot, marks it used and stores
// its inverse, so the next launch finds everything it needs; each block then forms
// the multipliers of its own rows from the compact column.  A local form in one lane
// keeps two launches per column (a one-block pivot step that writes every row's
// multiplier, then the update): there every column stays live and the per-block
// multipliers cost more than the pivot step saves (measured at n = 5003: 0.185 s
// against 0.227 s for one local form; four lockstep determinants 0.527 s against
// 0.418 s fused; four lockstep local forms 0.645 s against 0.604 s fused).
#include <algorithm>
#include <vector>

#include "modarith.h"
#include "panel.h"
#include "smf_internal.h"

namespace smf {
namespace {

constexpr int kPivThreads = 256;
constexpr int kUpdThreads = 256;
// rows per update thread (the pivot row's entry is loaded once for them): eight
// for entries of up to 16 bytes, fewer for wider ones to stay in registers
template <typename T, int L>
__host__ __device__ constexpr int upd_rows() {
    return sizeof(T) * L <= 16 ? 8 : sizeof(T) * L <= 32 ? 4 : 2;
}

template <typename T>
struct ModOps;

template <>
struct ModOps<uint32_t> {
    __host__ __device__ static uint32_t shoup(uint32_t f, uint32_t m) {
        return (uint32_t)(((uint64_t)f << 32) / m);
    }
    __device__ static uint32_t mul(uint32_t y, uint32_t f, uint32_t fs, uint32_t m) {
        uint32_t r = f * y - __umulhi(y, fs) * m;
        return r >= m ? r - m : r;
    }
    __device__ static uint32_t mulmod(uint32_t a, uint32_t b, uint32_t m) {
        return (uint32_t)(((uint64_t)a * b) % m);
    }
    // shoup(f, m) from rcp = floor((2^64 - 1) / m): x = f 2^32 < 2^63, and
    // floor(x rcp / 2^64) is floor(x / m) or one less (x (2^64 / m - rcp) / 2^64 < 1/2)
    __device__ static uint32_t shoup_rcp(uint32_t f, uint32_t m, uint64_t rcp) {
        const uint64_t x = (uint64_t)f << 32;
        uint64_t q = __umul64hi(x, rcp);
        if (x - q * m >= m) q++;
        return (uint32_t)q;
    }
};

template <>
struct ModOps<uint64_t> {
    __host__ __device__ static uint64_t shoup(uint64_t f, uint64_t m) {
        return (uint64_t)(((unsigned __int128)f << 64) / m);
    }
    __device__ static uint64_t mul(uint64_t y, uint64_t f, uint64_t fs, uint64_t m) {
        uint64_t r = f * y - __umul64hi(y, fs) * m;
        return r >= m ? r - m : r;
    }
    __device__ static uint64_t mulmod(uint64_t a, uint64_t b, uint64_t m) {
        return (uint64_t)(((unsigned __int128)a * b) % m);
    }
};

// a^-1 mod m for a unit a (extended Euclid on signed 64-bit values, m < 2^62)
__device__ int64_t inv_mod(int64_t a, int64_t m) {
    int64_t r0 = m, r1 = a, t0 = 0, t1 = 1;
    while (r1) {
        const int64_t qq = r0 / r1;
        int64_t x = r0 - qq * r1;
        r0 = r1;
        r1 = x;
        x = t0 - qq * t1;
        t0 = t1;
        t1 = x;
    }
    return t0 < 0 ? t0 + m : t0;
}

// Up to L moduli m_l (units tested modulo the primes q_l | m_l) run in
// lockstep on one matrix whose entries hold L residues side by side: the
// pivot of a column is the first unused row that is a unit modulo every q_l,
// so one column loop serves all of them (Phase 3's primes; Phase 2's prime
// powers of s').
template <typename T, int L>
struct Lanes {
    int n;      // lanes in use (<= L)
    T m[L];
    T q[L];
    uint64_t rcp[L];  // floor((2^64 - 1) / m_l)
};

// A pivot's inverse and a multiplier's Shoup companion in lane l: 32-bit
// lanes (m < 2^31) by 32-bit Euclid and the lane's reciprocal of m, which keep
// 64-bit divisions (emulated on the device) off the column loop's critical
// path; 64-bit lanes as before.
template <typename T, int L>
__device__ __forceinline__ T inv_lane(T a, const Lanes<T, L>& md, int l) {
    if constexpr (sizeof(T) == 4) return inv_mod32(a, md.m[l]);
    else return (T)inv_mod((int64_t)a, (int64_t)md.m[l]);
}
template <typename T, int L>
__device__ __forceinline__ T shoup_lane(T f, const Lanes<T, L>& md, int l) {
    if constexpr (sizeof(T) == 4) return ModOps<uint32_t>::shoup_rcp(f, md.m[l], md.rcp[l]);
    else return ModOps<T>::shoup(f, md.m[l]);
}

// A (int64, row-major, lda) -> M[i][j][l] = A[i][j] mod m_l, canonical.
template <typename T, int L>
__global__ void elim_init_kernel(const int64_t* __restrict__ A, int64_t lda, int64_t n, T* __restrict__ M,
                                 Lanes<T, L> md) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * n) return;
    const int64_t i = e / n, j = e - i * n;
    const int64_t a = A[i * lda + j];
#pragma unroll
    for (int l = 0; l < L; l++) {
        const int64_t m = (int64_t)md.m[l < md.n ? l : 0];  // (lanes not in use repeat lane 0)
        const int64_t r = a % m;
        M[e * L + l] = (T)(r < 0 ? r + m : r);
    }
}

template <typename T, int L>
__device__ __forceinline__ bool joint_unit(const T* __restrict__ x, const Lanes<T, L>& md) {
    bool u = true;
#pragma unroll
    for (int l = 0; l < L; l++)
        if (l < md.n) u &= x[l] % md.q[l] != 0;
    return u;
}

// One column's pivot: the first unused row that is a unit in every lane, then
// the multipliers of every other unused row (0 for used rows).
template <typename T, int L>
__global__ void __launch_bounds__(kPivThreads)
elim_pivot_kernel(T* __restrict__ M, int64_t n, int64_t k, Lanes<T, L> md, int field, int* __restrict__ used,
                  int64_t* __restrict__ pivrow, T* __restrict__ pivval, T* __restrict__ f, T* __restrict__ fs,
                  int* __restrict__ dead) {
    pdl_wait();
    __shared__ int64_t best;
    __shared__ T sinv[L], sinvs[L];
    if (threadIdx.x == 0) best = n;
    __syncthreads();
    const bool stop = *dead != 0;
    if (!stop) {
        // every row of the thread's stride is tested (independent loads), the first kept
        int64_t mine = n;
#pragma unroll 4
        for (int64_t i = threadIdx.x; i < n; i += kPivThreads)
            if (!used[i] && joint_unit<T, L>(M + (i * n + k) * L, md) && i < mine) mine = i;
        if (mine < n) atomicMin((unsigned long long*)&best, (unsigned long long)mine);
    }
    __syncthreads();
    const int64_t p = best;
    if (stop || p >= n) {
        if (threadIdx.x == 0) {
            pivrow[k] = -1;
            if (field) *dead = 1;  // the determinant: a column without a pivot means det = 0 (in some lane)
        }
        for (int64_t i = threadIdx.x; i < n * L; i += kPivThreads) f[i] = 0;
        pdl_trigger();
        return;
    }
    if (threadIdx.x < md.n) {
        const int l = threadIdx.x;
        const T pv = M[(p * n + k) * L + l];
        pivval[k * L + l] = pv;
        sinv[l] = inv_lane<T, L>(pv, md, l);
        sinvs[l] = shoup_lane<T, L>(sinv[l], md, l);
    }
    if (threadIdx.x == 0) {
        used[p] = 1;
        pivrow[k] = p;
    }
    __syncthreads();
    for (int64_t i = threadIdx.x; i < n; i += kPivThreads) {
        const bool live = !used[i];
#pragma unroll
        for (int l = 0; l < L; l++) {
            if (l >= md.n) break;
            T fi = 0;
            if (live) fi = ModOps<T>::mul(M[(i * n + k) * L + l], sinv[l], sinvs[l], md.m[l]);
            f[i * L + l] = fi;
            fs[i * L + l] = fi ? shoup_lane<T, L>(fi, md, l) : 0;
        }
    }
    pdl_trigger();
}

// The L residues of one entry, loaded and stored as one vector when they fill
// 8 or 16 bytes.
template <typename T, int L>
struct Entry {
    T v[L];
    __device__ __forceinline__ void load(const T* p) {
        if constexpr (sizeof(T) * L == 16) {
            const uint4 u = *reinterpret_cast<const uint4*>(p);
            memcpy(v, &u, 16);
        } else if constexpr (sizeof(T) * L == 8) {
            const uint2 u = *reinterpret_cast<const uint2*>(p);
            memcpy(v, &u, 8);
        } else {
#pragma unroll
            for (int l = 0; l < L; l++) v[l] = p[l];
        }
    }
    __device__ __forceinline__ void store(T* p) const {
        if constexpr (sizeof(T) * L == 16) {
            uint4 u;
            memcpy(&u, v, 16);
            *reinterpret_cast<uint4*>(p) = u;
        } else if constexpr (sizeof(T) * L == 8) {
            uint2 u;
            memcpy(&u, v, 8);
            *reinterpret_cast<uint2*>(p) = u;
        } else {
#pragma unroll
            for (int l = 0; l < L; l++) p[l] = v[l];
        }
    }
};

// Row i -= f_i * row p over the live columns (after k, or every column not yet
// a pivot column), every lane.  A thread takes one column and kUpdRows rows:
// it loads every row's multipliers and entries first, then updates them, so
// the loads of the rows overlap.
template <typename T, int L>
__global__ void __launch_bounds__(kUpdThreads)
elim_update_kernel(T* __restrict__ M, int64_t n, int64_t k, int64_t c0, Lanes<T, L> md,
                   const int64_t* __restrict__ pivrow, const T* __restrict__ f, const T* __restrict__ fs,
                   const int64_t* __restrict__ colpiv) {
    pdl_wait();
    const int64_t p = pivrow[k];
    const int64_t j = c0 + (int64_t)blockIdx.x * kUpdThreads + threadIdx.x;
    // colpiv (local form): columns that already have a pivot are never read again
    if (p >= 0 && j < n && j != k && !(colpiv && j < k && colpiv[j] >= 0)) {
        Entry<T, L> y;
        y.load(M + (p * n + j) * L);
        constexpr int kUpdRows = upd_rows<T, L>();
        const int64_t r0 = (int64_t)blockIdx.y * kUpdRows;
        T fi[kUpdRows][L];
        bool live[kUpdRows];
#pragma unroll
        for (int rr = 0; rr < kUpdRows; rr++) {
            const int64_t i = r0 + rr;
            live[rr] = false;
#pragma unroll
            for (int l = 0; l < L; l++) {
                fi[rr][l] = (i < n && l < md.n) ? f[i * L + l] : 0;
                live[rr] |= fi[rr][l] != 0;
            }
        }
        Entry<T, L> x[kUpdRows];
#pragma unroll
        for (int rr = 0; rr < kUpdRows; rr++)
            if (live[rr]) x[rr].load(M + ((r0 + rr) * n + j) * L);
#pragma unroll
        for (int rr = 0; rr < kUpdRows; rr++) {
            if (!live[rr]) continue;
            const int64_t i = r0 + rr;
#pragma unroll
            for (int l = 0; l < L; l++) {
                if (l >= md.n) break;
                const T t = ModOps<T>::mul(y.v[l], fi[rr][l], fs[i * L + l], md.m[l]);
                const T v = x[rr].v[l];
                x[rr].v[l] = v >= t ? v - t : v + (md.m[l] - t);
            }
            x[rr].store(M + (i * n + j) * L);
        }
    }
    pdl_trigger();
}

constexpr int kCountGroup = 32;  // blocks per first-level counter of the last-block count
constexpr int kStepRows = 8;  // rows per block of the column step (many blocks: the update is latency-bound)

// Column k: row i -= f_i * row p over the live columns (after k for a
// determinant; every column without a pivot yet for the local form), every
// lane, with f_i = M[i][k] / M[p][k] formed per block from the compact copy of
// column k; and column k+1's pivot search (see the top of this file).  A thread
// takes one column and kStepRows rows in groups of upd_rows, loading a group's
// entries before updating them.  k = -1 only searches column 0.
template <typename T, int L>
__global__ void __launch_bounds__(kUpdThreads)
elim_step_kernel(T* __restrict__ M, int64_t n, int64_t k, int64_t c0, Lanes<T, L> md, int field,
                 int* __restrict__ used, int64_t* __restrict__ pivrow, T* __restrict__ pivval, T* __restrict__ pinv,
                 T* __restrict__ pinvs, T* __restrict__ colbuf, unsigned* __restrict__ cand,
                 unsigned* __restrict__ counter, int* __restrict__ dead) {
    pdl_wait();
    constexpr int R = upd_rows<T, L>();
    static_assert(kStepRows % R == 0, "whole row groups");
    __shared__ T sf[kStepRows][L], sfs[kStepRows][L];
    __shared__ int s_last;
    const int64_t r0 = (int64_t)blockIdx.y * kStepRows;
    const bool stop = *dead != 0;  // a determinant that is already 0 in some lane
    const int64_t p = k >= 0 && !stop ? pivrow[k] : -1;
    const T* cur = colbuf + (size_t)(k & 1) * n * L;     // column k, copied by the launch before
    T* nxt = colbuf + (size_t)((k + 1) & 1) * n * L;     // column k+1, copied here
    if (p >= 0) {
        for (int t = threadIdx.x; t < kStepRows * L; t += kUpdThreads) {
            const int rr = t / L, l = t % L;
            const int64_t i = r0 + rr;
            T fi = 0;
            if (l < md.n && i < n && i != p && !used[i])
                fi = ModOps<T>::mul(cur[i * L + l], pinv[k * L + l], pinvs[k * L + l], md.m[l]);
            sf[rr][l] = fi;
            if constexpr (sizeof(T) == 4) sfs[rr][l] = fi ? ModOps<T>::shoup_rcp(fi, md.m[l], md.rcp[l]) : 0;
            else sfs[rr][l] = fi ? ModOps<T>::shoup(fi, md.m[l]) : 0;
        }
    }
    __syncthreads();
    const int64_t j = c0 + (int64_t)blockIdx.x * kUpdThreads + threadIdx.x;
    // local form: columns that already have a pivot are never read again
    const bool col_live = p >= 0 && j < n && j != k && !(!field && j < k && pivrow[j] >= 0);
    const bool search = !stop && k + 1 < n && j == k + 1;  // this thread copies column k+1 and searches it
    if (col_live || search) {
        Entry<T, L> y;
        if (col_live) y.load(M + (p * n + j) * L);
        unsigned best = 0xFFFFFFFFu;
        for (int g = 0; g < kStepRows; g += R) {
            bool live[R];
            Entry<T, L> x[R];
#pragma unroll
            for (int rr = 0; rr < R; rr++) {
                const int64_t i = r0 + g + rr;
                live[rr] = false;
                if (col_live && i < n) {
#pragma unroll
                    for (int l = 0; l < L; l++)
                        if (l < md.n) live[rr] |= sf[g + rr][l] != 0;
                }
            }
#pragma unroll
            for (int rr = 0; rr < R; rr++)
                if (live[rr] || (search && r0 + g + rr < n)) x[rr].load(M + ((r0 + g + rr) * n + j) * L);
#pragma unroll
            for (int rr = 0; rr < R; rr++) {
                const int64_t i = r0 + g + rr;
                if (live[rr]) {
#pragma unroll
                    for (int l = 0; l < L; l++) {
                        if (l >= md.n) break;
                        const T t = ModOps<T>::mul(y.v[l], sf[g + rr][l], sfs[g + rr][l], md.m[l]);
                        const T v = x[rr].v[l];
                        x[rr].v[l] = v >= t ? v - t : v + (md.m[l] - t);
                    }
                    x[rr].store(M + (i * n + j) * L);
                }
                if (search && i < n) {
                    x[rr].store(nxt + i * L);
                    if (i != p && !used[i] && joint_unit<T, L>(x[rr].v, md) && (unsigned)i < best) best = (unsigned)i;
                }
            }
        }
        // (the first unit row usually comes from an early block: skip the atomic when beaten)
        if (best != 0xFFFFFFFFu && best < *(volatile unsigned*)(cand + (k + 1))) atomicMin(cand + (k + 1), best);
    }
    // the last block over column k+1 settles its pivot; blocks are counted in groups
    // of kCountGroup (counter[1 + g]) and the groups in counter[0], so that no
    // address takes more than a few tens of atomics
    if (!stop && k + 1 < n && (k + 1 - c0) / kUpdThreads == (int64_t)blockIdx.x) {
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned g = blockIdx.y / kCountGroup, ng = (gridDim.y + kCountGroup - 1) / kCountGroup;
            const unsigned in_g = min((unsigned)kCountGroup, gridDim.y - g * kCountGroup);
            s_last = 0;
            if (atomicAdd(counter + 1 + g, 1u) == in_g - 1) {
                counter[1 + g] = 0u;  // for the next launch
                __threadfence();
                s_last = atomicAdd(counter, 1u) == ng - 1;
            }
        }
        __syncthreads();
        if (s_last) {
            __threadfence();
            const unsigned q = atomicAdd(cand + (k + 1), 0u);
            if (q < (unsigned)n) {
                if (threadIdx.x < md.n) {
                    const int l = threadIdx.x;
                    const T pv = __ldcg(nxt + (size_t)q * L + l);
                    pivval[(k + 1) * L + l] = pv;
                    const T iv = inv_lane<T, L>(pv, md, l);
                    pinv[(k + 1) * L + l] = iv;
                    pinvs[(k + 1) * L + l] = shoup_lane<T, L>(iv, md, l);
                }
                if (threadIdx.x == 0) {
                    used[q] = 1;
                    pivrow[k + 1] = q;
                }
            } else if (threadIdx.x == 0) {
                pivrow[k + 1] = -1;
                if (field) *dead = 1;  // the determinant: a column without a pivot means det = 0 (in some lane)
            }
            if (threadIdx.x == 0) *counter = 0u;  // for the next launch
        }
    }
    pdl_trigger();
}

// out[a][b] = M[rows[a]][cols[b]][lane] / div (exact), a square block of size nb, one lane.
template <typename T, int L>
__global__ void elim_gather_kernel(const T* __restrict__ M, int64_t n, const int64_t* __restrict__ rows,
                                   const int64_t* __restrict__ cols, int64_t nb, int lane, T div,
                                   T* __restrict__ out) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nb * nb) return;
    const int64_t a = e / nb, b = e - a * nb;
    out[e] = M[(rows[a] * n + cols[b]) * L + lane] / div;
}

// Scratch of an elimination of an n x n matrix with L lanes of type T.
// (stream-ordered: freeing them does not synchronise the device)
template <typename T, int L>
struct ElimBufs {
    StreamBuf M, used, pivrow, pivval, pinv, pinvs, colbuf, cand, counter, dead, f, fs;
    // the last-block count: one total and one per group of kCountGroup row blocks
    static size_t counters(int64_t n) {
        return 1 + (size_t)(((n + kStepRows - 1) / kStepRows + kCountGroup - 1) / kCountGroup);
    }
    cudaError_t alloc(smf_ctx* ctx, int64_t n, cudaStream_t s) { return M.alloc(ctx, sizeof(T) * L * (size_t)n * (size_t)n, s); }
    // what the column loop needs beside the matrix
    cudaError_t alloc_columns(smf_ctx* ctx, int64_t n, cudaStream_t s) {
        cudaError_t e;
        if (used.p) return cudaSuccess;
        const size_t nl = sizeof(T) * L * (size_t)n;
        if ((e = used.alloc(ctx, sizeof(int) * (size_t)n, s)) ||
            (e = pivrow.alloc(ctx, sizeof(int64_t) * (size_t)n, s)) || (e = pivval.alloc(ctx, nl, s)) ||
            (e = pinv.alloc(ctx, nl, s)) || (e = pinvs.alloc(ctx, nl, s)) || (e = colbuf.alloc(ctx, 2 * nl, s)) ||
            (e = cand.alloc(ctx, sizeof(unsigned) * (size_t)(n + 1), s)) ||
            (e = counter.alloc(ctx, sizeof(unsigned) * counters(n), s)) || (e = f.alloc(ctx, nl, s)) || (e = fs.alloc(ctx, nl, s)) ||
            (e = dead.alloc(ctx, sizeof(int), s)))
            return e;
        return cudaSuccess;
    }
};

// The column loop on the n x n matrix in `M`: each column's pivot row (-1 for a
// deferred column) and its values in every lane.  field: a determinant (only
// the columns after k are updated, a column without a pivot ends it); else the
// local form (every column but k stays current: deferred columns are kept).
template <typename T, int L>
cudaError_t elim_columns(smf_ctx* ctx, ElimBufs<T, L>& b, T* M, int64_t n, const Lanes<T, L>& md, bool field,
                         std::vector<int64_t>* pivrow, std::vector<T>* pivval, cudaStream_t s) {
    cudaError_t e;
    if ((e = b.alloc_columns(ctx, n, s)) || (e = cudaMemsetAsync(b.used.p, 0, sizeof(int) * (size_t)n, s)) ||
        (e = cudaMemsetAsync(b.dead.p, 0, sizeof(int), s)) ||
        (e = cudaMemsetAsync(b.counter.p, 0, sizeof(unsigned) * ElimBufs<T, L>::counters(n), s)) ||
        (e = cudaMemsetAsync(b.cand.p, 0xFF, sizeof(unsigned) * (size_t)(n + 1), s)) ||
        (e = cudaMemsetAsync(b.pivrow.p, 0xFF, sizeof(int64_t) * (size_t)n, s)))
        return e;
    const bool fused = field || L > 1;
    for (int64_t k = 0; !fused && k < n; k++) {  // a one-lane local form: pivot step, then update
        e = launch_pdl(elim_pivot_kernel<T, L>, dim3(1), dim3(kPivThreads), 0, s, M, n, k, md, 0, (int*)b.used.p,
                       (int64_t*)b.pivrow.p, (T*)b.pivval.p, (T*)b.f.p, (T*)b.fs.p, (int*)b.dead.p);
        if (e) return e;
        constexpr int R = upd_rows<T, L>();
        const dim3 grid((unsigned)((n + kUpdThreads - 1) / kUpdThreads), (unsigned)((n + R - 1) / R));
        e = launch_pdl(elim_update_kernel<T, L>, grid, dim3(kUpdThreads), 0, s, M, n, k, (int64_t)0, md,
                       (const int64_t*)b.pivrow.p, (const T*)b.f.p, (const T*)b.fs.p, (const int64_t*)b.pivrow.p);
        if (e) return e;
    }
    // one launch per column (k = -1 only searches column 0)
    for (int64_t k = -1; fused && k < n; k++) {
        const int64_t c0 = field ? k + 1 : 0;
        if (c0 >= n) continue;
        const dim3 grid((unsigned)((n - c0 + kUpdThreads - 1) / kUpdThreads), (unsigned)((n + kStepRows - 1) / kStepRows));
        e = launch_pdl(elim_step_kernel<T, L>, grid, dim3(kUpdThreads), 0, s, M, n, k, c0, md, field ? 1 : 0,
                       (int*)b.used.p, (int64_t*)b.pivrow.p, (T*)b.pivval.p, (T*)b.pinv.p, (T*)b.pinvs.p,
                       (T*)b.colbuf.p, (unsigned*)b.cand.p, (unsigned*)b.counter.p, (int*)b.dead.p);
        if (e) return e;
    }
    pivrow->resize(n);
    pivval->resize((size_t)n * L);
    if ((e = cudaMemcpyAsync(pivrow->data(), b.pivrow.p, sizeof(int64_t) * n, cudaMemcpyDeviceToHost, s)) ||
        (e = cudaMemcpyAsync(pivval->data(), b.pivval.p, sizeof(T) * L * n, cudaMemcpyDeviceToHost, s)))
        return e;
    return cudaStreamSynchronize(s);
}

// ---------------------------------------------------------------------------
// Elimination by panels (32-bit lanes).  The column loop above reads and writes
// the whole trailing block once per column, one launch each.  Here one cluster
// reduces a panel of kPanel columns (panel.h) to its transform S, and one pass
// applies it to the trailing columns, M[i][j] += sum_t S[i][t] M[p_t][j], for the
// rows i without a pivot, whose list each panel hands to the next: the matrix is
// read and written once per panel, and the pivot rows stay as they are.
//
//  - a determinant: a column without a unit ends the call (*fallback);
//  - a local Smith form: such a column is deferred and stays live; the deferred
//    columns are listed in increasing order (dcols[0 .. *ndef)), and the trailing
//    columns are all of them, the panel's own too, followed by [c1, n).
//
// GB300, four 31-bit primes: n = 2003 6.6 ms (44 ms with a launch per column; 8.1 ms
// without the look-ahead of elim_blocked).  With it 63 panels of 36 to 97 us, 4.1 ms
// in all, run beside passes of 11 to 157 us, 4.6 ms in all.  n = 5003 59 ms, 10007 0.46 s.
constexpr int kPanel = 32;
constexpr int64_t kLookAhead = 2 << 20;  // words of a pass (about 20 us)

// 32-bit entries go by panels from the context's threshold up to the largest
// matrix of which one column fits the cluster.
bool by_panels(const smf_ctx* ctx, int64_t n, int L) {
    return n >= ctx->elim_panel_min_n && panel_width(n, L, kPanel) > 0;
}

// trailing column x of a panel: a deferred column, then [c1, n)
__device__ __forceinline__ int64_t trail_col(int64_t x, int64_t nd, const int* __restrict__ dcols, int64_t c1) {
    return x < nd ? dcols[x] : c1 + (x - nd);
}

__global__ void bd_init_kernel(int64_t n, int* __restrict__ live, int* __restrict__ count, int* __restrict__ flag,
                               int* __restrict__ ndef, uint32_t* __restrict__ det, int dets) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) live[i] = (int)i;
    if (i < dets) det[i] = 1;
    if (i == 0) {
        *count = (int)n;
        *flag = 0;
        *ndef = 0;
    }
}

// The pass over the trailing block: 64 live rows by 128 words per block.  A
// thread keeps its word of the panel's KT pivot rows in registers and takes 32
// rows, four at a time, whose multipliers it reads from shared memory.  Bound by
// the integer pipe: KT 64-bit multiply-adds per word (28 a clock and SM), against
// 8 bytes of memory traffic.
constexpr int kTrailRows = 64, kTrailWords = 128;
template <int L, PanelRed RED, int KT, bool LOC>
__global__ void __launch_bounds__(256)
bd_trail_kernel(uint32_t* __restrict__ M, int64_t n, int64_t c0, int w, int64_t c1, int64_t ce,
                const __grid_constant__ PanelMod<L> md, const int* __restrict__ live, const int* __restrict__ count,
                const int* __restrict__ piv, const uint32_t* __restrict__ G, const int* __restrict__ flag,
                const int* __restrict__ dcols, const int* __restrict__ ndef) {
    constexpr int SW = KT + 4;  // padded row of multipliers of one lane
    __shared__ __align__(16) uint32_t ss[kTrailRows * L * SW];
    __shared__ int sid[kTrailRows], sp[KT];
    pdl_wait();
    pdl_trigger();
    if (*flag) return;
    const int64_t nd = LOC && ndef ? (int64_t)*ndef : 0;
    const int64_t ncols = nd + (ce - c1);
    const int nl = *count;
    const int64_t x0 = (int64_t)blockIdx.x * (kTrailWords / L);
    const int r0 = (int)blockIdx.y * kTrailRows;
    if (x0 >= ncols || r0 >= nl) return;  // (the grid bounds both)
    const int nr = min(kTrailRows, nl - r0);
    const int tid = threadIdx.x;
    if (tid < nr) sid[tid] = live[r0 + tid];
    if (tid < KT) sp[tid] = tid < w ? piv[c0 + tid] : -1;
    for (int e = tid; e < nr * L * (KT / 4); e += 256) {
        const uint4 v = *reinterpret_cast<const uint4*>(G + (size_t)r0 * L * KT + 4 * (size_t)e);
        *reinterpret_cast<uint4*>(ss + e / (KT / 4) * SW + e % (KT / 4) * 4) = v;
    }
    __syncthreads();
    const int c = tid % kTrailWords, l = c % L;
    const int64_t xx = x0 + c / L;
    if (xx >= ncols) return;
    uint32_t* Mj = M + trail_col(xx, nd, dcols, c1) * L + l;
    const size_t ld = (size_t)n * L;
    uint32_t y[KT];
#pragma unroll
    for (int t = 0; t < KT; t++) y[t] = sp[t] >= 0 ? Mj[sp[t] * ld] : 0u;
    const uint32_t m = md.m[l], ninv = md.ninv[l];
    for (int r = tid / kTrailWords; r < nr; r += 8) {
        uint64_t acc[4];
        const uint32_t* f[4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int ri = r + 2 * i < nr ? r + 2 * i : r;
            f[i] = ss + (ri * L + l) * SW;
            acc[i] = mac_start<RED>(Mj[sid[ri] * ld], m);
        }
#pragma unroll
        for (int t = 0; t < KT; t += 4)
#pragma unroll
            for (int i = 0; i < 4; i++) acc[i] = mac4<RED>(acc[i], *reinterpret_cast<const uint4*>(f[i] + t), y + t, m);
#pragma unroll
        for (int i = 0; i < 4; i++)
            if (r + 2 * i < nr) Mj[sid[r + 2 * i] * ld] = mac_end<RED>(acc[i], m, ninv);
    }
}

// The trailing columns [c1, ce) of a panel, and the deferred ones when ndef is given.
// dependent: launched while the kernel before it on the stream still runs (not
// where an event comes between).
template <int L, bool LOC>
cudaError_t launch_trail(const PanelArgs<L>& a, int64_t c1, int64_t ce, const int* ndef, int64_t rows, bool dependent,
                         cudaStream_t s) {
    const int64_t cols = ce - c1 + (ndef ? c1 : 0);  // (deferred columns lie before c1)
    const dim3 grid((unsigned)((cols + kTrailWords / L - 1) / (kTrailWords / L)),
                    (unsigned)((rows + kTrailRows - 1) / kTrailRows));
    auto go = [&](auto kernel) {
        if (dependent)
            return launch_pdl(kernel, grid, dim3(256), 0, s, a.M, a.n, a.c0, a.w, c1, ce, a.md, (const int*)a.live_out,
                              (const int*)a.count_out, (const int*)a.piv, (const uint32_t*)a.G, (const int*)a.flag,
                              (const int*)a.dcols, ndef);
        kernel<<<grid, 256, 0, s>>>(a.M, a.n, a.c0, a.w, c1, ce, a.md, a.live_out, a.count_out, a.piv, a.G, a.flag,
                                    a.dcols, ndef);
        return cudaGetLastError();
    };
    if (panel_red(a.md) == PanelRed::kNarrow)
        return a.gw > 16 ? go(bd_trail_kernel<L, PanelRed::kNarrow, 32, LOC>) : go(bd_trail_kernel<L, PanelRed::kNarrow, 16, LOC>);
    return a.gw > 16 ? go(bd_trail_kernel<L, PanelRed::kWide, 32, LOC>) : go(bd_trail_kernel<L, PanelRed::kWide, 16, LOC>);
}

// An elimination by panels on the stream: what it leaves on the device.
struct Blocked {
    StreamBuf buf;
    int* piv;       // [n] each column's pivot row (-1 for a local form's deferred column)
    int* flag;      // a determinant: a column without a pivot that is a unit in every lane
    uint32_t* det;  // [2 L] its pivots' product in every lane, numerators and denominators
    int* live;      // the rows without a pivot, and their count
    int* count;
    int* dcols;     // the deferred columns
};

// The n x n matrix in M (32-bit lanes) by panels.  Only enqueues.
template <int L, bool LOC>
cudaError_t elim_blocked(smf_ctx* ctx, uint32_t* M, int64_t n, const Lanes<uint32_t, L>& md, Blocked* out,
                         cudaStream_t s) {
    cudaError_t e;
    PanelArgs<L> a{};
    for (int l = 0; l < L; l++) panel_mod(a.md, l, md.m[l < md.n ? l : 0], md.q[l < md.n ? l : 0]);
    const int pw = panel_width(n, L, kPanel), gw = pw > 16 ? 32 : 16;
    const int64_t panels = (n + pw - 1) / pw;
    // scratch: G (two, see below), ybuf, then [piv n | flag | det 2L] read back in one copy, live lists, counts,
    // deferred columns and their number before each panel
    const size_t gwords = (size_t)n * L * gw;
    const size_t words = 2 * gwords + panel_scratch(pw * L) + (size_t)n + 1 + 2 * L + 2 * (size_t)n + 2 + (size_t)n +
                         (size_t)panels + 1;
    if ((e = out->buf.alloc(ctx, sizeof(uint32_t) * words, s))) return e;
    uint32_t* G = (uint32_t*)out->buf.p;
    uint32_t* ybuf = G + 2 * gwords;
    int* piv = (int*)(ybuf + panel_scratch(pw * L));
    int* flag = piv + n;
    uint32_t* det = (uint32_t*)flag + 1;
    int* live[2] = {(int*)det + 2 * L, (int*)det + 2 * L + n};
    int* count = live[1] + n;
    int* dcols = count + 2;
    int* ndef = dcols + n;
    bd_init_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, live[0], count, flag, ndef, det, 2 * L);
    if ((e = cudaGetLastError())) return e;
    a.M = M;
    a.n = a.ld = n;
    a.ybuf = ybuf;
    a.piv = piv;
    a.flag = flag;
    a.gw = gw;
    a.det = det;
    a.dcols = dcols;
    int k = 0;
    // Look-ahead: the columns of the next panel first, then the next panel (16
    // SMs, a serial chain) beside the pass over the rest, on the context's side
    // stream.  What the two share is apart: M's columns; G and the live lists, two
    // of each; the deferred columns, whose number is kept for each panel.  The rest
    // is done before anything touches its columns or the buffers it reads: the next
    // panel's own columns wait for it.  Where the rest is short the events cost more
    // than they hide: below kLookAhead words everything stays on one stream.
    struct Events {  // the call's own: calls on other streams may share the context
        cudaEvent_t fork = nullptr, join = nullptr;
        cudaError_t make() {
            cudaError_t e = cudaSuccess;
            if (!fork) e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
            if (!e && !join) e = cudaEventCreateWithFlags(&join, cudaEventDisableTiming);
            return e;
        }
        ~Events() {
            if (fork) cudaEventDestroy(fork);
            if (join) cudaEventDestroy(join);
        }
    } ev;
    bool side = false;  // a pass on the side stream that s has not waited for
    auto join = [&] {
        if (!side) return cudaSuccess;
        side = false;
        return cudaStreamWaitEvent(s, ev.join, 0);
    };
    auto enqueue = [&]() -> cudaError_t {
        for (int64_t c0 = 0, i = 0; c0 < n; c0 += pw, k ^= 1, i++) {
            const int64_t c1 = std::min<int64_t>(n, c0 + pw), c2 = std::min<int64_t>(n, c1 + pw);
            a.c0 = c0;
            a.w = (int)(c1 - c0);
            a.live = live[k];
            a.count = count + k;
            a.live_out = live[k ^ 1];
            a.count_out = count + (k ^ 1);
            a.G = G + (i & 1) * gwords;
            a.ndef = ndef + i;
            a.ndef_out = ndef + i + 1;
            if ((e = launch_panel<L, LOC ? PanelKind::kLocal : PanelKind::kDet>(a, n, s))) return e;
            const bool dependent = !side;
            if ((e = join())) return e;
            if (!LOC && c1 >= n) continue;
            // a determinant leaves n - c1 rows; a local form's rows and deferred columns are known on the device
            const int64_t rows = LOC ? n : n - c1;
            const int* nd = LOC ? a.ndef_out : nullptr;
            if ((n - c1) * (n - c2) * L < kLookAhead) {
                if ((e = launch_trail<L, LOC>(a, c1, n, nd, rows, dependent, s))) return e;
                continue;
            }
            if ((e = ev.make()) || (e = launch_trail<L, LOC>(a, c1, c2, nullptr, rows, dependent, s)) ||
                (e = cudaEventRecord(ev.fork, s)) || (e = cudaStreamWaitEvent(ctx->aux, ev.fork, 0)))
                return e;
            side = true;
            e = launch_trail<L, LOC>(a, c2, n, nd, rows, false, ctx->aux);
            const cudaError_t e2 = cudaEventRecord(ev.join, ctx->aux);
            if (e || e2) return e ? e : e2;
        }
        return cudaSuccess;
    };
    e = enqueue();
    const cudaError_t ej = join();  // (the scratch goes back on s)
    if (e || ej) return e ? e : ej;
    out->piv = piv;
    out->flag = flag;
    out->det = det;
    out->live = live[k];
    out->count = count + k;
    out->dcols = dcols;
    return cudaSuccess;
}

// Waits for it: the pivot rows, and for a determinant (dets not null) the
// fractions dets[l] / dets[L + l] and whether a column had no pivot.
template <int L>
cudaError_t read_blocked(const Blocked& b, int64_t n, std::vector<int64_t>* pivrow, uint32_t* dets, bool* no_pivot,
                         cudaStream_t s) {
    cudaError_t e;
    std::vector<int> h((size_t)n + 1 + 2 * L);
    if ((e = cudaMemcpyAsync(h.data(), b.piv, sizeof(int) * h.size(), cudaMemcpyDeviceToHost, s)) ||
        (e = cudaStreamSynchronize(s)))
        return e;
    pivrow->assign(h.begin(), h.begin() + n);
    if (!dets) return cudaSuccess;
    *no_pivot = h[n] != 0;
    for (int l = 0; l < 2 * L; l++) dets[l] = (uint32_t)h[n + 1 + l];
    return cudaSuccess;
}

// The levels of a small block that a joint elimination leaves (rows live[],
// columns dcols[], nb of each): block l of the grid takes modulus l = q^e.
// While an entry is a unit it is a pivot and its row and column go; then every
// entry left is divided by q, and the rest goes on over Z/(q^(e-1)).
// out[l][t]: the size left after level t, the number of invariant factors
// divisible by q^(t+1); out[L][0] = nb, and nothing else when nb > kSmallBlock.
// One launch and one read, where each level took an elimination, a read and a
// gather (about 0.3 ms a level).
constexpr int kSmallBlock = 192, kSmallThreads = 256, kSmallLevels = 32;
struct SmallLevels {
    uint32_t m[4], q[4];
    int e[4];
};
template <int L>
__global__ void __launch_bounds__(kSmallThreads)
local_small_kernel(const uint32_t* __restrict__ M, int64_t n, const int* __restrict__ live,
                   const int* __restrict__ count, const int* __restrict__ dcols, SmallLevels lv, int* __restrict__ out) {
    extern __shared__ uint32_t B[];  // [nb][nb]
    __shared__ int ri[kSmallBlock], ci[kSmallBlock];
    __shared__ unsigned s_at;
    __shared__ uint32_t s_inv;
    const int nb = *count, l = blockIdx.x, tid = threadIdx.x;
    if (l == 0 && tid == 0) out[L * kSmallLevels] = nb;
    if (nb > kSmallBlock) return;
    const uint32_t q = lv.q[l];
    uint32_t m = lv.m[l];
    for (int x = tid; x < nb * nb; x += kSmallThreads) {
        const int a = x / nb, b = x % nb;
        B[x] = M[((size_t)live[a] * n + dcols[b]) * L + l];
    }
    for (int x = tid; x < nb; x += kSmallThreads) ri[x] = ci[x] = x;  // the rows and columns left: [0, k)
    int k = nb;
    for (int t = 0; t < lv.e[l] && k > 0; t++, m /= q) {
        const uint64_t rcp = UINT64_MAX / m;
        for (;;) {
            __syncthreads();
            if (tid == 0) s_at = 0xFFFFFFFFu;
            __syncthreads();
            for (int x = tid; x < k * k; x += kSmallThreads)
                if (B[ri[x / k] * nb + ci[x % k]] % q != 0) {
                    atomicMin(&s_at, (unsigned)x);
                    break;
                }
            __syncthreads();
            const unsigned at = s_at;
            if (at == 0xFFFFFFFFu) break;
            const int pr = ri[at / k], pc = ci[at % k], lr = ri[k - 1], lc = ci[k - 1];
            if (tid == 0) s_inv = inv_mod32(B[pr * nb + pc], m);
            __syncthreads();
            if (tid == 0) {  // the last row and column take the places of the pivot's
                ri[at / k] = lr;
                ci[at % k] = lc;
            }
            k--;
            __syncthreads();
            for (int x = tid; x < k * k; x += kSmallThreads) {
                const int r = ri[x / k], c = ci[x % k];
                const uint32_t f = mulmod32_rcp(B[r * nb + pc], s_inv, m, rcp);
                const uint32_t y = mulmod32_rcp(f, B[pr * nb + c], m, rcp), v = B[r * nb + c];
                B[r * nb + c] = v >= y ? v - y : v + m - y;
            }
        }
        if (tid == 0) out[l * kSmallLevels + t] = k;
        for (int x = tid; x < k * k; x += kSmallThreads) B[ri[x / k] * nb + ci[x % k]] /= q;
    }
}

// The column loop of a local form (every column but k stays current), by
// panels when the entries are 32-bit (by_panels).
template <typename T, int L>
cudaError_t elim_local(smf_ctx* ctx, ElimBufs<T, L>& b, T* M, int64_t n, const Lanes<T, L>& md,
                       std::vector<int64_t>* pivrow, std::vector<T>* pivval, cudaStream_t s) {
    if constexpr (sizeof(T) == 4) {
        if (by_panels(ctx, n, L)) {
            Blocked r;
            const cudaError_t e = elim_blocked<L, true>(ctx, M, n, md, &r, s);
            return e ? e : read_blocked<L>(r, n, pivrow, nullptr, nullptr, s);
        }
    }
    return elim_columns<T, L>(ctx, b, M, n, md, false, pivrow, pivval, s);
}

uint64_t mulmod_host(uint64_t a, uint64_t b, uint64_t m) { return (uint64_t)((unsigned __int128)a * b % m); }

int elim_fail(smf_ctx* ctx, const char* what, cudaError_t e) {
    cudaGetLastError();
    ctx->err = std::string(what) + ": " + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? SMF_E_NOMEM : SMF_E_CUDA;
}

// det A mod q_l for nq <= L primes in one column loop.  A column without a
// pivot that is nonzero modulo every prime sends the call back to one prime
// at a time (then such a column means det = 0 for that prime).
template <typename T, int L>
int det_lanes(smf_ctx* ctx, const int64_t* A, int64_t lda, int64_t n, const uint64_t* q, int nq, uint64_t* det,
              cudaStream_t s) {
    if (n == 0) {
        for (int l = 0; l < nq; l++) det[l] = 1 % q[l];
        return SMF_OK;
    }
    Lanes<T, L> md{};
    md.n = nq;
    for (int l = 0; l < nq; l++) {
        md.m[l] = md.q[l] = (T)q[l];
        md.rcp[l] = UINT64_MAX / (uint64_t)q[l];
    }
    ElimBufs<T, L> b;
    cudaError_t e = b.alloc(ctx, n, s);
    if (e) return elim_fail(ctx, "det_mod: device allocation", e);
    T* M = (T*)b.M.p;
    elim_init_kernel<T, L><<<(unsigned)((n * n + 255) / 256), 256, 0, s>>>(A, lda, n, M, md);
    std::vector<int64_t> pr;
    std::vector<T> pv;
    if ((e = cudaGetLastError())) return elim_fail(ctx, "det_mod", e);
    bool blocked = false;
    if constexpr (sizeof(T) == 4) {
        // 31-bit primes: by panels.  A column without a joint unit pivot sends
        // several primes back to one at a time (below); with one prime det = 0
        if (by_panels(ctx, n, L)) {
            bool no_pivot = false;
            uint32_t dets[2 * L];
            Blocked r;
            if ((e = elim_blocked<L, false>(ctx, M, n, md, &r, s)) ||
                (e = read_blocked<L>(r, n, &pr, dets, &no_pivot, s)))
                return elim_fail(ctx, "det_mod", e);
            blocked = true;
            if (no_pivot) pr.assign(n, -1);
            else pv.assign(dets, dets + 2 * L);
        }
    }
    if (!blocked && (e = elim_columns<T, L>(ctx, b, M, n, md, true, &pr, &pv, s))) return elim_fail(ctx, "det_mod", e);
    if (std::any_of(pr.begin(), pr.end(), [](int64_t r) { return r < 0; })) {
        if (nq == 1) {
            det[0] = 0;
            return SMF_OK;
        }
        for (int l = 0; l < nq; l++) {
            const int st = det_lanes<T, 1>(ctx, A, lda, n, q + l, 1, det + l, s);
            if (st) return st;
        }
        return SMF_OK;
    }
    // sign of the permutation k -> pr[k]: (-1)^(n - cycles)
    std::vector<char> seen(n, 0);
    int64_t cycles = 0;
    for (int64_t k = 0; k < n; k++) {
        if (seen[k]) continue;
        cycles++;
        for (int64_t j = k; !seen[j]; j = pr[j]) seen[j] = 1;
    }
    for (int l = 0; l < nq; l++) {
        uint64_t d = 1 % q[l];
        if (blocked) d = mulmod_host(pv[l], inv_mod32((uint32_t)pv[L + l], (uint32_t)q[l]), q[l]);
        else
            for (int64_t k = 0; k < n; k++) d = mulmod_host(d, (uint64_t)pv[k * L + l], q[l]);
        if (((n - cycles) & 1) && d) d = q[l] - d;
        det[l] = d;
    }
    return SMF_OK;
}

// The local Smith form at q over Z/(q^e) of the nb x nb matrix already in M
// (one lane, canonical modulo q^e): counts[t] += #(invariant factors divisible
// by q^t) for t = 1 .. e.
template <typename T>
int local_levels(smf_ctx* ctx, ElimBufs<T, 1>& b, StreamBuf& M2, int64_t nb, uint64_t q, int e, int64_t* counts,
                 cudaStream_t s) {
    uint64_t m = 1;
    for (int t = 0; t < e; t++) m *= q;
    T* M = (T*)b.M.p;
    T* Mn = (T*)M2.p;
    StreamBuf idx;
    cudaError_t ce = idx.alloc(ctx, sizeof(int64_t) * 2 * (size_t)std::max<int64_t>(nb, 1), s);
    if (ce) return elim_fail(ctx, "smith_local: device allocation", ce);
    int64_t size = nb;
    std::vector<int64_t> pr;
    std::vector<T> pv;
    // level t: the block left holds the invariant factors divisible by q^t, over Z/(q^(e-t))
    for (int t = 0; t < e && size > 0; t++) {
        Lanes<T, 1> md{};
        md.n = 1;
        md.m[0] = (T)m;
        md.q[0] = (T)q;
        md.rcp[0] = UINT64_MAX / m;
        if ((ce = elim_local<T, 1>(ctx, b, M, size, md, &pr, &pv, s))) return elim_fail(ctx, "smith_local", ce);
        std::vector<char> row_used(size, 0);
        std::vector<int64_t> id;  // unused rows, then deferred columns
        for (int64_t k = 0; k < size; k++)
            if (pr[k] >= 0) row_used[pr[k]] = 1;
        for (int64_t i = 0; i < size; i++)
            if (!row_used[i]) id.push_back(i);
        const int64_t k2 = (int64_t)id.size();
        for (int64_t k = 0; k < size; k++)
            if (pr[k] < 0) id.push_back(k);
        if ((int64_t)id.size() != 2 * k2) {
            ctx->err = "smith_local: unused rows and deferred columns differ in number";
            return SMF_E_INVALID;
        }
        counts[t + 1] += k2;  // invariant factors with q-valuation above t
        if (k2 == 0) break;
        m /= q;
        if (t + 1 == e) break;
        if ((ce = cudaMemcpyAsync(idx.p, id.data(), sizeof(int64_t) * 2 * k2, cudaMemcpyHostToDevice, s)))
            return elim_fail(ctx, "smith_local", ce);
        elim_gather_kernel<T, 1><<<(unsigned)((k2 * k2 + 255) / 256), 256, 0, s>>>(
            M, size, (const int64_t*)idx.p, (const int64_t*)idx.p + k2, k2, 0, (T)q, Mn);
        if ((ce = cudaGetLastError())) return elim_fail(ctx, "smith_local", ce);
        std::swap(M, Mn);
        size = k2;
    }
    return SMF_OK;
}

// The local Smith forms of A at the prime powers q_l^e_l (l < nq <= L) with one
// joint column loop over Z/(prod q_l^e_l) - pivots that are units modulo every
// q_l - and then, per prime, the levels of local_levels on the block of unused
// rows and deferred columns that is left.  counts[l][t], t = 0 .. e_l.
template <typename T, int L>
int local_lanes(smf_ctx* ctx, const int64_t* A, int64_t lda, int64_t n, const uint64_t* q, const int* e, int nq,
                std::vector<std::vector<int64_t>>* counts, cudaStream_t s) {
    counts->assign(nq, {});
    for (int l = 0; l < nq; l++) {
        (*counts)[l].assign(e[l] + 1, 0);
        (*counts)[l][0] = n;
    }
    if (n == 0) return SMF_OK;
    Lanes<T, L> md{};
    md.n = nq;
    for (int l = 0; l < nq; l++) {
        uint64_t m = 1;
        for (int t = 0; t < e[l]; t++) m *= q[l];
        md.m[l] = (T)m;
        md.q[l] = (T)q[l];
        md.rcp[l] = UINT64_MAX / m;
    }
    int64_t nb;
    std::vector<int64_t> id;
    StreamBuf joint, idx;
    {
        ElimBufs<T, L> b;
        cudaError_t ce = b.alloc(ctx, n, s);
        if (ce) return elim_fail(ctx, "smith_local: device allocation", ce);
        T* M = (T*)b.M.p;
        elim_init_kernel<T, L><<<(unsigned)((n * n + 255) / 256), 256, 0, s>>>(A, lda, n, M, md);
        std::vector<int64_t> pr;
        std::vector<T> pv;
        if ((ce = cudaGetLastError())) return elim_fail(ctx, "smith_local", ce);
        bool done = false;
        if constexpr (sizeof(T) == 4) {
            if (by_panels(ctx, n, L)) {  // by panels, and the block left at once when it is small
                Blocked r;
                StreamBuf ob;
                constexpr int words = L * kSmallLevels + 1;
                int h[words];
                const size_t sm = sizeof(uint32_t) * kSmallBlock * kSmallBlock;
                SmallLevels lv{};
                for (int l = 0; l < nq; l++) {
                    lv.m[l] = md.m[l];
                    lv.q[l] = md.q[l];
                    lv.e[l] = e[l];
                }
                if ((ce = elim_blocked<L, true>(ctx, M, n, md, &r, s)) || (ce = ob.alloc(ctx, sizeof(h), s)) ||
                    (ce = cudaMemsetAsync(ob.p, 0, sizeof(h), s)) ||
                    (ce = cudaFuncSetAttribute(local_small_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)))
                    return elim_fail(ctx, "smith_local", ce);
                local_small_kernel<L><<<(unsigned)nq, kSmallThreads, sm, s>>>(M, n, r.live, r.count, r.dcols, lv, (int*)ob.p);
                if ((ce = cudaGetLastError()) || (ce = cudaMemcpyAsync(h, ob.p, sizeof(h), cudaMemcpyDeviceToHost, s)) ||
                    (ce = cudaStreamSynchronize(s)))
                    return elim_fail(ctx, "smith_local", ce);
                if (h[words - 1] <= kSmallBlock) {
                    for (int l = 0; l < nq; l++)
                        for (int t = 0; t < e[l]; t++) (*counts)[l][t + 1] += h[l * kSmallLevels + t];
                    return SMF_OK;
                }
                if ((ce = read_blocked<L>(r, n, &pr, nullptr, nullptr, s))) return elim_fail(ctx, "smith_local", ce);
                done = true;
            }
        }
        if (!done && (ce = elim_local<T, L>(ctx, b, M, n, md, &pr, &pv, s))) return elim_fail(ctx, "smith_local", ce);
        std::vector<char> row_used(n, 0);
        for (int64_t k = 0; k < n; k++)
            if (pr[k] >= 0) row_used[pr[k]] = 1;
        for (int64_t i = 0; i < n; i++)
            if (!row_used[i]) id.push_back(i);
        nb = (int64_t)id.size();
        for (int64_t k = 0; k < n; k++)
            if (pr[k] < 0) id.push_back(k);
        if ((int64_t)id.size() != 2 * nb) {
            ctx->err = "smith_local: unused rows and deferred columns differ in number";
            return SMF_E_INVALID;
        }
        if (nb == 0) return SMF_OK;  // every invariant factor is prime to every q_l
        // keep the joint matrix, free the rest of the scratch
        std::swap(joint.p, b.M.p);
        joint.s = s;
        if ((ce = idx.alloc(ctx, sizeof(int64_t) * 2 * nb, s)) ||
            (ce = cudaMemcpyAsync(idx.p, id.data(), sizeof(int64_t) * 2 * nb, cudaMemcpyHostToDevice, s)))
            return elim_fail(ctx, "smith_local", ce);
    }
    // each prime on the block that is left (the joint pivots are units for all of them)
    ElimBufs<T, 1> b1;
    StreamBuf M2;
    cudaError_t ce = b1.alloc(ctx, nb, s);
    if (!ce) ce = M2.alloc(ctx, sizeof(T) * (size_t)nb * nb, s);
    if (ce) return elim_fail(ctx, "smith_local: device allocation", ce);
    for (int l = 0; l < nq; l++) {
        elim_gather_kernel<T, L><<<(unsigned)((nb * nb + 255) / 256), 256, 0, s>>>(
            (const T*)joint.p, n, (const int64_t*)idx.p, (const int64_t*)idx.p + nb, nb, l, (T)1, (T*)b1.M.p);
        if ((ce = cudaGetLastError())) return elim_fail(ctx, "smith_local", ce);
        const int st = local_levels<T>(ctx, b1, M2, nb, q[l], e[l], (*counts)[l].data(), s);
        if (st) return st;
    }
    return SMF_OK;
}

// How many 32-bit moduli one elimination of an n x n matrix takes at most.  By
// panels the moduli share the cluster's shared memory: with more of them a large
// matrix's panels get narrower, and a pass over the rest (which multiplies by 16
// or 32 columns) comes more often.  Four 31-bit determinants, four at a time /
// one at a time (start of the panels' 16 and 8 columns with four moduli: n = 5345
// and 10705):
//   n = 8009 0.243 / 0.248 s, 10007 0.461 / 0.458, 12007 1.54 / 0.76, 20501 14.9 / 3.6
// (two at a time, panels of 16 columns: 0.80 and 3.8 s at the last two).
int elim_group(const smf_ctx* ctx, int64_t n) {
    if (!by_panels(ctx, n, 1)) return 4;  // by columns
    return panel_width(n, 4, kPanel) >= 16 ? 4 : panel_width(n, 2, kPanel) >= kPanel ? 2 : 1;
}

template <typename T>
int det_dispatch(smf_ctx* ctx, const int64_t* A, int64_t lda, int64_t n, const uint64_t* q, int nq, uint64_t* det,
                 cudaStream_t s) {
    const int most = sizeof(T) == 4 ? elim_group(ctx, n) : 4;
    for (int i = 0; i < nq; i += most) {
        const int k = std::min(most, nq - i);
        const int st = k == 1   ? det_lanes<T, 1>(ctx, A, lda, n, q + i, k, det + i, s)
                       : k == 2 ? det_lanes<T, 2>(ctx, A, lda, n, q + i, k, det + i, s)
                                : det_lanes<T, 4>(ctx, A, lda, n, q + i, k, det + i, s);
        if (st) return st;
    }
    return SMF_OK;
}

// Prime powers below 2^31 in lockstep groups of up to four 32-bit lanes
// (elim_group), wider ones one at a time in 64-bit words.
// A joint loop of all eleven prime powers of the n = 5003 test in 64-bit lanes
// was slower than one at a time (4.35 s against 1.94 s): every update moved 88
// bytes per entry.
int local_dispatch(smf_ctx* ctx, const int64_t* A, int64_t lda, int64_t n, const uint64_t* q, const int* e, int nq,
                   const std::vector<char>& wide, std::vector<std::vector<int64_t>>* counts, cudaStream_t s) {
    counts->assign(nq, {});
    std::vector<int> narrow;
    for (int l = 0; l < nq; l++) {
        if (!wide[l]) {
            narrow.push_back(l);
            continue;
        }
        std::vector<std::vector<int64_t>> one;
        const int st = local_lanes<uint64_t, 1>(ctx, A, lda, n, q + l, e + l, 1, &one, s);
        if (st) return st;
        (*counts)[l] = std::move(one[0]);
    }
    const size_t most = (size_t)elim_group(ctx, n);
    for (size_t g = 0; g < narrow.size(); g += most) {
        const int k = (int)std::min(most, narrow.size() - g);
        std::vector<uint64_t> qg;
        std::vector<int> eg;
        for (int t = 0; t < k; t++) {
            qg.push_back(q[narrow[g + t]]);
            eg.push_back(e[narrow[g + t]]);
        }
        std::vector<std::vector<int64_t>> grp;
        const int st = k == 1   ? local_lanes<uint32_t, 1>(ctx, A, lda, n, qg.data(), eg.data(), 1, &grp, s)
                       : k == 2 ? local_lanes<uint32_t, 2>(ctx, A, lda, n, qg.data(), eg.data(), 2, &grp, s)
                                : local_lanes<uint32_t, 4>(ctx, A, lda, n, qg.data(), eg.data(), k, &grp, s);
        if (st) return st;
        for (int t = 0; t < k; t++) (*counts)[narrow[g + t]] = std::move(grp[t]);
    }
    return SMF_OK;
}

}  // namespace

int det_mod_device(smf_ctx* ctx, const int64_t* A, int64_t lda, int64_t n, const uint64_t* q, int nq, uint64_t* det,
                   cudaStream_t s) {
    bool wide = false;
    for (int l = 0; l < nq; l++) {
        if (q[l] < 2 || q[l] >= (1ull << 62)) {
            ctx->err = "det_mod: q must be a prime below 2^62";
            return SMF_E_INVALID;
        }
        wide |= q[l] >= (1ull << 31);
    }
    return wide ? det_dispatch<uint64_t>(ctx, A, lda, n, q, nq, det, s)
                : det_dispatch<uint32_t>(ctx, A, lda, n, q, nq, det, s);
}

int local_smith_device(smf_ctx* ctx, const int64_t* A, int64_t lda, int64_t n, const uint64_t* q, const int* e,
                       int nq, std::vector<std::vector<int64_t>>* counts, cudaStream_t s) {
    if (nq < 1 || nq > 16) {
        ctx->err = "smith_local: 1 to 16 prime powers";
        return SMF_E_INVALID;
    }
    std::vector<char> wide(nq, 0);
    for (int l = 0; l < nq; l++) {
        unsigned __int128 m = 1;
        for (int t = 0; t < e[l]; t++) m *= q[l];
        if (q[l] < 2 || e[l] < 1 || e[l] > 62 || m >= ((unsigned __int128)1 << 62)) {
            ctx->err = "smith_local: need primes q and q^e below 2^62";
            return SMF_E_INVALID;
        }
        wide[l] = m >= (1u << 31);
    }
    return local_dispatch(ctx, A, lda, n, q, e, nq, wide, counts, s);
}

}  // namespace smf

// One panel of w columns of an elimination over Z/(m), reduced in place
// (Gauss-Jordan without row moves) by one thread-block cluster: A^-1 mod p
// (inverse.cu), determinants and local Smith forms (elim.cu).
//
// With pivot rows p_t (t < w) the panel T (the columns of the rows given) ends
// as its own transform S: every row i of the matrix becomes, on every other
// column,
//   M[i] + sum_t S[i][t] M[p_t]   (i no pivot row),   sum_t S[i][t] M[p_t]   (i a pivot row),
// with M[p_t] as it was before the panel; column t of S is zero where the
// column had no pivot.  The caller applies that as one product with K = w.
//
// The columns are a serial chain.  One launch per column costs 10 to 20 us and
// one cluster barrier per column 1.1 us (measured, n = 64, 24-bit p).  Here a
// column costs no barrier at all: any unit is as good a pivot as another in
// Z/(m), so one block takes the pivots of up to 16 columns from 32 rows, in four
// warps per modulus, and publishes the 16 pivot rows already multiplied by the
// inverse of the pivot block, Y = B^-1 T[Q]; then every block updates its rows by
// T[i] - T[i][J] Y, 16 multiply-adds and one reduction per word.
//
// The 32 rows: where the first 32 open rows of some block hold several units in
// every column at hand (dense matrices), that block takes them, with two
// barriers a round.  Else (sparse matrices, small primes, the last rows) the
// blocks first hand it a row or two for each column, from wherever there are
// units: one barrier and one way through L2 more.  (With own rows only, a
// planted n = 1009 matrix, mostly zeros, took a round for every column or two:
// 9.2 ms against 2.9 ms for a dense one.)  Columns in which these rows came to
// hold no unit stay pending for the next round; when no block has a unit in them,
// they have no pivot.
//
// The 32 x 16 tile is reduced without a division: the update is left unscaled,
// x[j] <- (v x[j] - f y[j]) / R (one Montgomery reduction, R = 2^32; for m = 2^e
// the low e bits, R = 1), which multiplies every row but the pivot's by v / R.
// With sigma_0 = 1, sigma_(t+1) = sigma_t v_t / R, the pivot row stays as it is
// with sigma_t in its pivot column, and at the end carries the factor
// R sigma / sigma_t: one inverse per 16 columns.
//
// The sums are 64-bit multiply-adds written in C (28 a clock and SM; the same as
// mad.wide.u32 in inline assembly 25 with four warps per scheduler, 10 against 17
// with one).
#pragma once

#include "cluster.h"
#include "modarith.h"
#include "smf_internal.h"

namespace smf {

constexpr int kSub = 16;            // columns per round of pivots
constexpr int kPanelThreads = 512;
constexpr int kPanelBatch = 32;     // rows updated between two block barriers
constexpr int kFbStride = kSub + 4; // words of one row's multipliers in one lane (padded: no bank conflicts)
constexpr int kParts = 4;            // warps that share the columns of a tile
constexpr size_t kPanelSmem = 216 * 1024;  // of a block's 227 KB: the rows of the panel and the kernel's static arrays

// Words of a panel row in shared memory: an odd multiple of four, so that one
// column of consecutive rows takes eight banks.
constexpr int panel_stride(int W) { return ((W + 3) & ~3) | 4; }

// Up to L moduli side by side in each entry; lanes beyond those in use repeat
// lane 0.  A modulus is a prime or a prime power, R = 2^32.
template <int L>
struct PanelMod {
    uint32_t m[L];
    uint32_t ninv[L];  // m odd: -m^-1 mod R
    uint32_t r1[L];    //        R mod m
    uint32_t r2[L];    //        R^2 mod m
    uint32_t ord[L];   //        phi(m) - 1
    uint32_t qinv[L];  // x is divisible by the prime q of m iff x qinv <= qlim (mod 2^32)
    uint32_t qlim[L];
    uint64_t rcp[L];   // floor((2^64 - 1) / m)
};

inline uint32_t inv_mod_2_32(uint32_t a) {  // a odd, Newton's steps
    uint32_t x = a;
    for (int k = 0; k < 5; k++) x *= 2 - a * x;
    return x;
}

template <int L>
void panel_mod(PanelMod<L>& d, int l, uint32_t m, uint32_t q) {
    d.m[l] = m;
    d.rcp[l] = UINT64_MAX / m;
    d.ninv[l] = m & 1 ? 0u - inv_mod_2_32(m) : 0u;
    d.r1[l] = (uint32_t)((1ull << 32) % m);
    d.r2[l] = (uint32_t)((uint64_t)d.r1[l] * d.r1[l] % m);
    d.ord[l] = m / q * (q - 1) - 1;
    if (q == 2) {  // x 2^31 mod 2^32 is 0 iff x is even
        d.qinv[l] = 1u << 31;
        d.qlim[l] = 0;
    } else {
        d.qinv[l] = inv_mod_2_32(q);
        d.qlim[l] = UINT32_MAX / q;
    }
}

// How a launch's moduli are reduced: below 2^28 and odd, below 2^28, below 2^31.
enum class PanelRed { kOddNarrow, kNarrow, kWide };

template <int L>
PanelRed panel_red(const PanelMod<L>& d) {
    bool narrow = true;
    for (int l = 0; l < L; l++) narrow &= d.m[l] < (1u << 28);
    return narrow ? PanelRed::kNarrow : PanelRed::kWide;
}

template <int L>
struct PanelArgs {
    uint32_t* M;          // [n][ld] entries of L words
    int64_t ld;           // entries
    int64_t c0;
    int w, wpad;          // panel columns; threads per row group (half the panel's words, rounded up to a power of two)
    PanelMod<L> md;
    int rows_max;         // rows per block at most
    uint32_t* ybuf;       // panel_scratch(w L) words: [kSub][w L] Y, [32][w L] candidate rows, [32] where they are
    int* piv;             // pivot row of each column (-1: none), written at [c0, c0 + w)
    int* flag;            // set when a column has no pivot (not for LOC); every later panel returns
    // whole inverse: all n rows, rows with a pivot are reduced on
    int64_t n;
    int* rowcol;          // [n] column whose pivot the row is, or -1
    int32_t* S;           // [n][w], or null
    int* status;
    // elimination: the live rows only
    const int* live;      // row ids before the panel, and their count
    const int* count;
    int* live_out;        // after it
    int* count_out;
    uint32_t* G;          // [live after the panel][L][gw] rows of S (times R for odd moduli), zero beyond w
    int gw;
    uint32_t* det;        // [2 L] the pivots' product as a fraction, numerators and denominators (kDet)
    int* dcols;           // columns without a pivot, ascending, and their count (LOC)
    const int* ndef;      // the latter before the panel and after it
    int* ndef_out;
};

// Blocks of a panel's cluster: 16 (the largest), fewer for matrices of few rows
// (a block wants 32 candidate rows).
inline int panel_cluster(int64_t n) {
    int C = 16;
    while (C > 1 && n < 32 * C) C /= 2;
    return C;
}

inline size_t panel_smem(int64_t rows_max, int64_t W, int64_t w) {
    return sizeof(uint32_t) * (size_t)(rows_max * (panel_stride((int)W) + 2) + w + 32 * W);
}

// words of a panel's scratch in global memory
constexpr size_t panel_scratch(size_t W) { return (kSub + 32) * W + 32; }

// dynamic shared memory a panel kernel of L lanes may take
constexpr size_t panel_smem_limit(int L) {
    return kPanelSmem - sizeof(uint32_t) * (size_t)(kSub + 2 * kPanelBatch) * L * kFbStride;
}

// The widest panel of at most `most` columns (a power of two) whose rows fit the
// blocks; 0 where no panel fits (one lane: n above 142,000).
inline int panel_width(int64_t n, int L, int most) {
    const int64_t rows = (n + 15) / 16;
    int w = most;
    while (w > 0 && panel_smem(rows, (int64_t)w * L, w) > panel_smem_limit(L)) w /= 2;
    return w;
}

#ifdef __CUDACC__
namespace {

enum class PanelKind { kInverse, kDet, kLocal };

__device__ __forceinline__ uint64_t mad_wide(uint32_t a, uint32_t b, uint64_t c) {
    return (uint64_t)a * b + c;
}

// x / R mod m for odd m and x < 2 m^2 < 2^63 (Montgomery)
__device__ __forceinline__ uint32_t mred(uint64_t x, uint32_t m, uint32_t ninv) {
    const uint32_t q = (uint32_t)x * ninv;
    const uint32_t r = (uint32_t)(mad_wide(q, m, x) >> 32);  // < 2m
    return min(r, r - m);
}

// acc_i,c + sum of 16 products f_i[t] y_c[t] of values below m, for N rows of
// multipliers (read from shared memory once) and two columns.  Below 2^28, up
// to 32 products stay below 2^61 beside an acc below 2^60.  Else (m < 2^31) the high
// word of a product is below m / 2: with the high word of acc below m, it stays
// below 2 m < 2^32 over two products, and then m 2^32 is taken off where it fits.
template <PanelRed RED>
__device__ __forceinline__ uint64_t mac4(uint64_t s, const uint4& q, const uint32_t* y, uint32_t m) {
    s = mad_wide(q.x, y[0], s);
    s = mad_wide(q.y, y[1], s);
    if constexpr (RED == PanelRed::kWide) {
        const uint32_t hi = (uint32_t)(s >> 32);
        s = ((uint64_t)min(hi, hi - m) << 32) | (uint32_t)s;
    }
    s = mad_wide(q.z, y[2], s);
    s = mad_wide(q.w, y[3], s);
    if constexpr (RED == PanelRed::kWide) {
        const uint32_t hi = (uint32_t)(s >> 32);
        s = ((uint64_t)min(hi, hi - m) << 32) | (uint32_t)s;
    }
    return s;
}
template <PanelRed RED, int N>
__device__ __forceinline__ void mac16(uint64_t (&acc)[N][2], const uint32_t* const (&f)[N],
                                      const uint32_t (&y)[2][kSub], uint32_t m) {
#pragma unroll
    for (int t4 = 0; t4 < kSub; t4 += 4) {
#pragma unroll
        for (int i = 0; i < N; i++) {
            const uint4 q = *reinterpret_cast<const uint4*>(f[i] + t4);
            acc[i][0] = mac4<RED>(acc[i][0], q, y[0] + t4, m);
            acc[i][1] = mac4<RED>(acc[i][1], q, y[1] + t4, m);
        }
    }
}

// The start and the end of x + sum f y.  m odd: y holds y R, x goes into the
// high word (x R), and one Montgomery reduction ends it.  m = 2^e: x and y as
// they are, and the low e bits.  (Barrett's reduction for both takes a 64-bit
// high product, 7 a clock and SM: it made the local forms that have the prime 2
// as slow as the multiply-adds themselves.)
template <PanelRed RED>
__device__ __forceinline__ uint64_t mac_start(uint32_t x, uint32_t m) {
    if constexpr (RED == PanelRed::kOddNarrow) return (uint64_t)x << 32;
    return m & 1 ? (uint64_t)x << 32 : x;
}
template <PanelRed RED>
__device__ __forceinline__ uint32_t mac_end(uint64_t acc, uint32_t m, uint32_t ninv) {
    const uint32_t q = (uint32_t)acc * ninv;
    uint32_t r = (uint32_t)(mad_wide(q, m, acc) >> 32);  // < 2m; below 2^28 < 4m
    if constexpr (RED != PanelRed::kWide) r = min(r, r - 2 * m);
    r = min(r, r - m);
    if constexpr (RED == PanelRed::kOddNarrow) return r;
    return m & 1 ? r : (uint32_t)acc & (m - 1);
}
// y to y R (m odd) and back
__device__ __forceinline__ uint32_t scale_r(uint32_t y, uint32_t m, uint32_t ninv, uint32_t r2) {
    return m & 1 ? mred((uint64_t)y * r2, m, ninv) : y;
}

// The tile's own unscaled step: x / R mod m as above, or x mod 2^e
template <bool EVEN>
__device__ __forceinline__ uint32_t tred(uint64_t x, uint32_t m, uint32_t ninv) {
    if constexpr (EVEN) return (uint32_t)x & (m - 1);
    return mred(x, m, ninv);
}

// a^-1 R^2 mod m (odd m: a^(phi(m) - 1) by squarings, which do not wait for the
// products; Euclid's divisions take four times as long), a^-1 mod 2^e
template <bool EVEN>
__device__ __forceinline__ uint32_t tinv(uint32_t a, uint32_t m, uint32_t ninv, uint32_t r1, uint32_t ord) {
    if constexpr (EVEN) {
        uint32_t x = a;
#pragma unroll
        for (int k = 0; k < 5; k++) x *= 2 - a * x;
        return x & (m - 1);
    }
    uint32_t p = r1;
    for (uint32_t e = ord; e; e >>= 1) {
        if (e & 1) p = mred((uint64_t)p * a, m, ninv);
        a = mred((uint64_t)a * a, m, ninv);
    }
    return p;
}

// The tile of one modulus (lane l of the entries) in four warps, a candidate
// row (list[.] of T, or -1) per thread and four columns per warp (part g): pivots for the pending
// columns, and the pivot rows reduced by them to yv[t][l][j] (t: the row of
// column t's pivot; times R^2 for odd m).  In step t the part that
// holds column t hands the column and its units to all; the warps of the L lanes
// agree on the pivot row.
template <int L, bool EVEN>
__device__ __forceinline__ void panel_tile(const uint32_t* T, int stride, int sub0, unsigned pend, int l, int g,
                                           const PanelMod<L>& md, const int* list, uint32_t* yv, int* s_piv,
                                           uint32_t (*sf)[L][32], unsigned (*sb)[L], uint32_t* det) {
    constexpr int P = kSub / kParts;
    const int lane = threadIdx.x & 31;
    const uint32_t m = md.m[l], ninv = md.ninv[l], qinv = md.qinv[l], qlim = md.qlim[l];
    const int slot = list[lane];
    uint32_t x[P];
#pragma unroll
    for (int j = 0; j < P; j++)
        x[j] = slot >= 0 && (pend >> (g * P + j) & 1) ? T[slot * stride + (sub0 + g * P + j) * L + l] : 0u;
    bool open = slot >= 0;
    int mine = -1, par = 0;
    uint32_t sig = 1, mysig = 1, num = 1, den = 1;
    // the column at hand is always x[0] of its part, whose results go one place
    // down: one small loop body (unrolled it does not fit the instruction cache)
#pragma unroll 1
    for (int t = 0; t < kSub; t++) {
        const bool own = t / P == g;
        unsigned b = 0;
        if (pend >> t & 1) {
            if (own) {
                const unsigned u = __ballot_sync(0xffffffffu, open && x[0] * qinv > qlim);
                sf[par][l][lane] = x[0];
                if (lane == 0) sb[par][l] = u;
            }
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kParts * L) : "memory");
            b = sb[par][0];
#pragma unroll
            for (int k = 1; k < L; k++) b &= sb[par][k];
        }
        if (b == 0) {  // no joint unit among these rows: the column stays pending
            if (own) {
                const uint32_t f = x[0];
#pragma unroll
                for (int j = 1; j < P; j++) x[j - 1] = x[j];
                x[P - 1] = f;
            }
            if (pend >> t & 1) par ^= 1;
            continue;
        }
        const int r = 31 - __clz(b);
        const bool me = lane == r;
        const uint32_t f = sf[par][l][lane], v = sf[par][l][r];
        par ^= 1;
        uint32_t y[P];
#pragma unroll
        for (int j = 0; j < P; j++) {
            const uint32_t pj = __shfl_sync(0xffffffffu, x[j], r);
            const uint32_t z = tred<EVEN>(mad_wide(f, m - pj, (uint64_t)v * x[j]), m, ninv);
            y[j] = me ? x[j] : z;
        }
        if (own) {
            const uint32_t z = me ? sig : tred<EVEN>((uint64_t)f * (m - sig), m, ninv);
#pragma unroll
            for (int j = 1; j < P; j++) x[j - 1] = y[j];
            x[P - 1] = z;
        } else {
#pragma unroll
            for (int j = 0; j < P; j++) x[j] = y[j];
        }
        if (me) {
            open = false;
            mine = t;
            mysig = sig;
        }
        if (det) {  // the true pivot is v / sigma
            num = tred<EVEN>((uint64_t)num * v, m, ninv);
            den = tred<EVEN>((uint64_t)den * sig, m, ninv);
        }
        sig = tred<EVEN>((uint64_t)sig * v, m, ninv);
        if (l == 0 && g == 0 && lane == 0) s_piv[t] = list[r];
    }
    uint32_t kn = tinv<EVEN>(sig, m, ninv, md.r1[l], md.ord[l]);
    if constexpr (!EVEN) kn = mred((uint64_t)kn * md.r2[l], m, ninv);
    if (det && lane == 0) {  // (another block's turn may come next: past the L1 caches)
        __stcg(det, mulmod32_rcp(__ldcg(det), num, m, md.rcp[l]));
        __stcg(det + L, mulmod32_rcp(__ldcg(det + L), den, m, md.rcp[l]));
    }
    if (mine >= 0) {
        const uint32_t k = tred<EVEN>((uint64_t)mysig * kn, m, ninv);
#pragma unroll
        for (int j = 0; j < P; j++)
            yv[(mine * L + l) * kFbStride + g * P + j] = tred<EVEN>((uint64_t)x[j] * k, m, ninv);
    }
}

template <int L, PanelRed RED, PanelKind KIND>
__global__ void __launch_bounds__(kPanelThreads, 1) panel_kernel(const __grid_constant__ PanelArgs<L> a) {
    extern __shared__ __align__(16) uint32_t sm[];
    __shared__ __align__(16) uint32_t yv[kSub * L * kFbStride];
    __shared__ __align__(16) uint32_t fb[2][kPanelBatch * L * kFbStride];
    __shared__ uint32_t sf[2][L][32];
    __shared__ unsigned sb[2][L];
    __shared__ uint32_t flags[2][16];
    __shared__ int s_list[32], s_first[kSub], s_last[kSub], s_id[32], s_piv[kSub], s_slots[kSub], s_n, s_base[17];
    __shared__ unsigned s_has, s_thin;
    constexpr bool INV = KIND == PanelKind::kInverse;
    pdl_wait();
    pdl_trigger();
    if (a.flag && *a.flag) return;  // a column had no pivot (the same for every block)
    const int C = (int)gridDim.x, rank = (int)blockIdx.x;  // one cluster
    const int w = a.w, W = w * L, stride = panel_stride(W);
    const int nrows = INV ? (int)a.n : *a.count;
    const int rows = (nrows - rank + C - 1) / C;  // <= rows_max
    uint32_t* T = sm;                             // [rows_max][stride]
    int* rid = (int*)(T + (size_t)a.rows_max * stride);  // [rows_max] row ids
    int* state = rid + a.rows_max;                // [rows_max] panel column whose pivot the row is; -1 none yet, -2 no candidate
    int* got = state + a.rows_max;                // [w] pivot found
    uint32_t* cr = (uint32_t*)(got + w);          // [32][W] candidate rows of all blocks
    uint32_t* cbuf = a.ybuf + kSub * W;
    int* cid = (int*)(cbuf + 32 * W);
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tid = threadIdx.x, c = tid % a.wpad, rg = tid / a.wpad, G = kPanelThreads / a.wpad;
    // a thread's two words of a row: c and c + W2, of the same lane
    const int W2 = (w + 1) / 2 * L;
    const bool col = c < W2, col2 = col && c + W2 < W;
    const int l = c % L;
    const uint32_t m = a.md.m[l];
    const uint32_t ninv = a.md.ninv[l];
    for (int s = tid; s < rows; s += kPanelThreads) {
        const int r = INV ? s * C + rank : a.live[s * C + rank];
        rid[s] = r;
        state[s] = INV && a.rowcol[r] >= 0 ? -2 : -1;
    }
    for (int j = tid; j < w; j += kPanelThreads) got[j] = 0;
    __syncthreads();
    for (int s = rg; s < rows; s += G)
        for (int k = c; k < W; k += a.wpad) T[s * stride + k] = a.M[((size_t)rid[s] * a.ld + a.c0) * L + k];
    cluster_sync();
    int fx = 0;
    bool missing = false;
    for (int sub0 = 0; sub0 < w && !missing; sub0 += kSub) {
        const int ks = min(kSub, w - sub0);
        unsigned pend = (1u << ks) - 1;
        while (pend) {
            // this block's first 32 open rows, and for each pending column (a warp each) whether they
            // hold units, else the first and the last open row that does
            if (wid == 0) {
                int k = 0;
                for (int s0 = 0; s0 < rows && k < 32; s0 += 32) {
                    const bool open = s0 + lane < rows && state[s0 + lane] == -1;
                    const unsigned b = __ballot_sync(0xffffffffu, open);
                    const int at = k + __popc(b & ((1u << lane) - 1));
                    if (open && at < 32) s_list[at] = s0 + lane;
                    k += __popc(b);
                }
                if (lane >= k) s_list[lane] = -1;
                if (lane == 0) s_has = s_thin = 0;
            }
            __syncthreads();
            if (pend >> wid & 1) {
                auto unit = [&](int s) {
                    bool u = true;
#pragma unroll
                    for (int k = 0; k < L; k++) u &= T[s * stride + (sub0 + wid) * L + k] * a.md.qinv[k] > a.md.qlim[k];
                    return u;
                };
                const int s = s_list[lane];
                const unsigned b = __ballot_sync(0xffffffffu, s >= 0 && unit(s));
                if (__popc(b) < 4) {
                    int first = -1, last = -1;
                    for (int s0 = 0; s0 < rows; s0 += 32) {
                        const int r = s0 + lane;
                        const unsigned v = __ballot_sync(0xffffffffu, r < rows && state[r] == -1 && unit(r));
                        if (v == 0) continue;
                        if (first < 0) first = s0 + __ffs(v) - 1;
                        last = s0 + 31 - __clz(v);
                    }
                    if (lane == 0) {
                        s_first[wid] = first;
                        s_last[wid] = last;
                        atomicOr(&s_thin, 1u << wid);
                        if (first >= 0) atomicOr(&s_has, 1u << wid);
                    }
                } else if (lane == 0) {
                    s_first[wid] = s_list[__ffs(b) - 1];
                    s_last[wid] = s_list[31 - __clz(b)];
                    atomicOr(&s_has, 1u << wid);
                }
            }
            __syncthreads();
            if (tid < C) cluster_store(&flags[fx & 1][rank], tid, s_has | (s_thin ? 0u : 1u << kSub));
            cluster_sync();
            const unsigned info = lane < C ? flags[fx & 1][lane] : 0u;
            const unsigned any = __ballot_sync(0xffffffffu, info & pend);
            const unsigned dense = __ballot_sync(0xffffffffu, info >> kSub);
            fx++;
            if (any == 0) break;  // no unit left in these columns
            // (the same block again and again: its instruction cache holds the tile's code)
            const int src = dense ? __ffs(dense) - 1 : 0;
            if (!dense) {
                for (int k = wid; k < 32; k += kPanelThreads / 32) {  // candidate k: for column j, from the k / 16-th block with a unit
                    const int j = k % kSub, rot = (j + fx) % C;
                    const unsigned b = __ballot_sync(0xffffffffu, info >> j & 1);
                    int owner = -1, row = -1;
                    if ((pend >> j & 1) && b) {
                        const unsigned hi = b >> rot << rot;
                        owner = __ffs(hi ? hi : b) - 1;
                        if (k >= kSub) {  // the next one, or this block's last row
                            const unsigned up = b & (0xFFFFFFFEu << owner);
                            const int o2 = __ffs(up ? up : b) - 1;
                            row = o2 == owner ? s_last[j] : s_first[j];
                            owner = o2;
                        } else {
                            row = s_first[j];
                        }
                    }
                    if (owner == rank) {
                        for (int e = lane; e < W; e += 32) __stcg(cbuf + k * W + e, T[row * stride + e]);
                        if (lane == 0) __stcg(cid + k, rank << 16 | row);
                    } else if (owner < 0 && rank == 0 && lane == 0) {
                        __stcg(cid + k, -1);
                    }
                }
                cluster_sync();
            }
            if (rank == src) {
                if (!dense) {
                    for (int e = tid; e < 32 * W; e += kPanelThreads) cr[e] = __ldcg(cbuf + e);
                    if (tid < 32) {
                        s_id[tid] = __ldcg(cid + tid);
                        s_list[tid] = s_id[tid] >= 0 ? tid : -1;
                    }
                }
                const uint32_t* base = dense ? T : cr;
                const int bst = dense ? stride : W;
                for (int k = tid; k < kSub * L * kFbStride; k += kPanelThreads) yv[k] = 0;
                if (tid < kSub) s_piv[tid] = -1;
                __syncthreads();
                if (tid < 32 * kParts * L) {
                    const int tl = tid / (32 * kParts), tg = tid / 32 % kParts;
                    uint32_t* det = KIND == PanelKind::kDet && tg == 0 ? a.det + tl : nullptr;
                    if (RED == PanelRed::kOddNarrow || (a.md.m[tl] & 1))
                        panel_tile<L, false>(base, bst, sub0, pend, tl, tg, a.md, s_list, yv, s_piv, sf, sb, det);
                    else
                        panel_tile<L, true>(base, bst, sub0, pend, tl, tg, a.md, s_list, yv, s_piv, sf, sb, det);
                }
                __syncthreads();
                if (tid < kSub * C) {  // where the pivot rows are: block and slot
                    const int p = s_piv[tid % kSub];
                    const int id = p < 0 ? -1 : dense ? rank << 16 | p : s_id[p];
                    cluster_store((uint32_t*)s_slots + tid % kSub, tid / kSub, (uint32_t)id);
                }
                // -Y = -B^-1 T[Q] on every column (in the pending ones the tile holds Y)
                if (col) {
                    bool tile[2];
                    uint32_t tq[2][kSub];
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const int ch = c + h * W2, j = ch / L - sub0;
                        tile[h] = j >= 0 && j < ks && (pend >> j & 1);
#pragma unroll
                        for (int t = 0; t < kSub; t++)
                            tq[h][t] = !tile[h] && (h == 0 || col2) && s_piv[t] >= 0 ? base[s_piv[t] * bst + ch] : 0u;
                    }
                    const uint32_t* b0 = yv + l * kFbStride;
                    for (int t = rg; t < kSub; t += 2 * G) {
                        const uint32_t* bt[2];
                        uint64_t acc[2][2] = {};
#pragma unroll
                        for (int i = 0; i < 2; i++) bt[i] = b0 + (t + i * G < kSub ? t + i * G : t) * (L * kFbStride);
                        mac16<RED, 2>(acc, bt, tq, m);
#pragma unroll
                        for (int i = 0; i < 2; i++) {
                            if (t + i * G >= kSub) break;
#pragma unroll
                            for (int h = 0; h < 2; h++) {
                                const int ch = c + h * W2;
                                if (h == 1 && !col2) break;
                                if (tile[h]) acc[i][h] = bt[i][ch / L - sub0];
                                const uint32_t y = mac_end<RED>(acc[i][h], m, ninv);
                                __stcg(a.ybuf + (t + i * G) * W + ch, y ? m - y : 0u);
                            }
                        }
                    }
                }
            }
            cluster_sync();
            uint32_t y[2][kSub];
#pragma unroll
            for (int t = 0; t < kSub; t++) {
                y[0][t] = col ? __ldcg(a.ybuf + t * W + c) : 0u;
                y[1][t] = col2 ? __ldcg(a.ybuf + t * W + c + W2) : 0u;
            }
            unsigned now = 0;
#pragma unroll
            for (int t = 0; t < kSub; t++) now |= (unsigned)(s_slots[t] >= 0) << t;
            if (tid < kSub && s_slots[tid] >= 0) {
                got[sub0 + tid] = 1;
                if (s_slots[tid] >> 16 == rank) {
                    state[s_slots[tid] & 0xFFFF] = sub0 + tid;
                    a.piv[a.c0 + sub0 + tid] = rid[s_slots[tid] & 0xFFFF];
                }
            }
            const int j0 = c / L - sub0, j1 = j0 + W2 / L;
            const bool p0 = j0 >= 0 && j0 < kSub && (now >> j0 & 1);  // a pivot column: its old values go
            const bool p1 = j1 >= 0 && j1 < kSub && (now >> j1 & 1);
            for (int s0 = 0, bi = 0; s0 < rows; s0 += kPanelBatch, bi ^= 1) {
                for (int e = tid; e < kPanelBatch * kSub * L; e += kPanelThreads) {
                    const int r = e / (kSub * L), k = e % (kSub * L), t = k / L;
                    fb[bi][(r * L + k % L) * kFbStride + t] =
                        s0 + r < rows && (now >> t & 1) ? T[(s0 + r) * stride + sub0 * L + k] : 0u;
                }
                __syncthreads();
                if (!col) continue;
                const uint32_t* fl = fb[bi] + l * kFbStride;
                for (int r = rg; r < kPanelBatch && s0 + r < rows; r += 4 * G) {  // four rows at a time
                    uint64_t acc[4][2];
                    const uint32_t* f[4];
                    bool on[4];
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        const int ri = r + i * G, s = s0 + ri;
                        on[i] = ri < kPanelBatch && s < rows;
                        f[i] = fl + (on[i] ? ri : r) * (L * kFbStride);
                        acc[i][0] = mac_start<RED>(on[i] && !p0 ? T[s * stride + c] : 0u, m);
                        acc[i][1] = mac_start<RED>(on[i] && !p1 && col2 ? T[s * stride + c + W2] : 0u, m);
                        if (on[i]) {
                            // the new pivot rows become Y; an elimination is done with its pivot rows
                            const int st = state[s];
                            if (INV ? st >= sub0 && (now >> (st - sub0) & 1) : st >= 0) on[i] = false;
                        }
                    }
                    mac16<RED, 4>(acc, f, y, m);
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        if (!on[i]) continue;
                        uint32_t* to = T + (s0 + r + i * G) * stride + c;
                        to[0] = mac_end<RED>(acc[i][0], m, ninv);
                        if (col2) to[W2] = mac_end<RED>(acc[i][1], m, ninv);
                    }
                }
            }
            if (INV && col && rg == 0) {
#pragma unroll
                for (int t = 0; t < kSub; t++) {
                    if (s_slots[t] < 0 || s_slots[t] >> 16 != rank) continue;
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        if (h == 1 && !col2) break;
                        const uint32_t v = mred(y[h][t], m, ninv);  // (an inverse: m odd)
                        T[(s_slots[t] & 0xFFFF) * stride + c + h * W2] = v ? m - v : 0u;
                    }
                }
            }
            pend &= ~now;
            __syncthreads();
        }
        if (pend && KIND != PanelKind::kLocal) missing = true;
    }
    __syncthreads();
    if (missing) {  // every block, at the same columns
        if (rank == 0 && tid == 0) {
            *a.flag = 1;
            if (INV) atomicOr(a.status, kStatusSingular);
        }
        return;
    }
    if constexpr (INV) {
        for (int s = rg; s < rows; s += G) {
            for (int k = c; k < W; k += a.wpad) {
                const uint32_t v = T[s * stride + k];
                if (a.S) a.S[(size_t)rid[s] * W + k] = (int32_t)v;
                a.M[(size_t)rid[s] * a.ld + a.c0 + k] = v;
            }
        }
        for (int s = tid; s < rows; s += kPanelThreads)
            if (state[s] >= 0) a.rowcol[rid[s]] = (int)(a.c0 + state[s]);
    } else {
        // the rows still live, in block order, and their rows of S
        if (tid == 0) s_n = 0;
        __syncthreads();
        for (int s = tid; s < rows; s += kPanelThreads) {
            const bool keep = state[s] == -1;
            if (keep) state[s] = -3 - atomicAdd(&s_n, 1);  // its place in the block
        }
        __syncthreads();
        if (tid < C) cluster_store(&flags[fx & 1][rank], tid, (uint32_t)s_n);
        cluster_sync();
        if (tid == 0) {
            int b = 0;
            for (int k = 0; k < C; k++) {
                s_base[k] = b;
                b += (int)flags[fx & 1][k];
            }
            if (rank == 0) *a.count_out = b;
        }
        if (rank == 0 && tid < w && got[tid] == 0) a.piv[a.c0 + tid] = -1;
        if (KIND == PanelKind::kLocal && rank == 0 && tid == 0) {
            int d = *a.ndef;
            for (int j = 0; j < w; j++)
                if (!got[j]) a.dcols[d++] = (int)(a.c0 + j);
            *a.ndef_out = d;
        }
        __syncthreads();
        const int base = s_base[rank];
        for (int s = tid; s < rows; s += kPanelThreads)
            if (state[s] <= -3) a.live_out[base - 3 - state[s]] = rid[s];
        const int gw = a.gw;
        for (int s = tid / (gw * L); s < rows; s += kPanelThreads / (gw * L)) {
            if (state[s] > -3) continue;
            const int e = tid % (gw * L), k = e / gw, t = e % gw;  // lane k, column t
            uint32_t v = t < w && got[t] ? T[s * stride + t * L + k] : 0u;
            v = scale_r(v, a.md.m[k], a.md.ninv[k], a.md.r2[k]);
            a.G[(size_t)(base - 3 - state[s]) * gw * L + e] = v;
        }
    }
}

}  // namespace

template <int L, PanelRed RED, PanelKind KIND>
cudaError_t launch_panel_red(PanelArgs<L>& a, int64_t n, cudaStream_t s) {
    const int C = panel_cluster(n);
    a.wpad = 32;
    while (a.wpad < (a.w + 1) / 2 * L) a.wpad *= 2;
    a.rows_max = (int)((n + C - 1) / C);
    return launch_cluster(panel_kernel<L, RED, KIND>, C, kPanelThreads, panel_smem(a.rows_max, (int64_t)a.w * L, a.w),
                          panel_smem_limit(L), s, a);
}
template <int L, PanelKind KIND>
cudaError_t launch_panel(PanelArgs<L>& a, int64_t n, cudaStream_t s) {
    switch (panel_red(a.md)) {
    case PanelRed::kNarrow: return launch_panel_red<L, PanelRed::kNarrow, KIND>(a, n, s);
    default: return launch_panel_red<L, PanelRed::kWide, KIND>(a, n, s);
    }
}
#endif  // __CUDACC__

}  // namespace smf

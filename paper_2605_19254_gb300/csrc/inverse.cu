// A^-1 mod p by Gauss-Jordan elimination over GF(p): the initialization of
// the p-adic lifting (Section 3 notes that it costs about as much as the
// lifting itself).
//
// The augmented n x 2n matrix [A mod p | I] is reduced column by column.
// Column k takes two launches:
//   gj_pivot: one block finds the first row r >= k whose entry in column k is
//             non-zero, swaps rows r and k, scales row k by that entry's
//             inverse (Fermat: a^(p-2)), and copies column k aside (f_i, with
//             f_k = 0);
//   gj_elim:  every row i != k subtracts f_i times row k, over the columns
//             j >= k (row k is zero left of column k).
// Afterwards the right half is A^-1 mod p.  That is the general form; matrices
// of 2 to kInvSingle columns, and larger ones in the limb form, go by panels
// instead (below).  A column without a pivot means p | det A: the pivot launch
// sets kStatusSingular and a device flag, and every later launch returns at once.
#include <algorithm>

#include "panel.h"
#include "smf_internal.h"

namespace smf {
namespace {

constexpr int kPivotThreads = 1024;
constexpr int kElimThreads = 256;
constexpr int kMaxGridY = 65535;
constexpr int64_t kElimBlocksPerSM = 16;

// Barrett reduction of a product of two residues (p < 2^31): with
// mu = floor((2^64 - 1) / p) the estimate q falls short of the quotient by at
// most 2.
__device__ __forceinline__ uint32_t mulmod(uint32_t a, uint32_t b, uint32_t p, uint64_t mu) {
    const uint64_t x = (uint64_t)a * b;
    uint64_t r = x - __umul64hi(x, mu) * p;
    while (r >= p) r -= p;
    return (uint32_t)r;
}

__device__ uint32_t powmod(uint32_t a, uint32_t e, uint32_t p, uint64_t mu) {
    uint32_t r = 1 % p;
    while (e) {
        if (e & 1) r = mulmod(r, a, p, mu);
        a = mulmod(a, a, p, mu);
        e >>= 1;
    }
    return r;
}

__global__ void __launch_bounds__(kElimThreads) gj_init_kernel(const int32_t* __restrict__ res, int64_t n,
                                                               uint32_t* __restrict__ M) {
    const int64_t e = (int64_t)blockIdx.x * kElimThreads + threadIdx.x;
    if (e >= 2 * n * n) return;
    const int64_t i = e / (2 * n), j = e - i * 2 * n;
    M[e] = j < n ? (uint32_t)res[i * n + j] : (uint32_t)(j - n == i);
}

__global__ void __launch_bounds__(kPivotThreads) gj_pivot_kernel(uint32_t* __restrict__ M, int64_t n, int64_t k,
                                                                 uint32_t p, uint64_t mu, uint32_t* __restrict__ col,
                                                                 int* flag, int* status) {
    __shared__ unsigned long long s_piv;
    __shared__ uint32_t s_inv;
    pdl_wait();
    pdl_trigger();
    if (*flag) return;  // an earlier column had no pivot
    const int64_t ld = 2 * n;
    if (threadIdx.x == 0) s_piv = (unsigned long long)n;
    __syncthreads();
    for (int64_t r = k + threadIdx.x; r < n; r += kPivotThreads) {
        if (M[r * ld + k] != 0) {
            atomicMin(&s_piv, (unsigned long long)r);
            break;
        }
    }
    __syncthreads();
    const int64_t r = (int64_t)s_piv;
    if (r == n) {
        if (threadIdx.x == 0) {
            *flag = 1;
            atomicOr(status, kStatusSingular);
        }
        return;
    }
    if (r != k) {
        for (int64_t j = threadIdx.x; j < ld; j += kPivotThreads) {
            const uint32_t t = M[r * ld + j];
            M[r * ld + j] = M[k * ld + j];
            M[k * ld + j] = t;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) s_inv = powmod(M[k * ld + k], p - 2, p, mu);
    __syncthreads();
    const uint32_t inv = s_inv;
    for (int64_t j = k + threadIdx.x; j < ld; j += kPivotThreads) M[k * ld + j] = mulmod(M[k * ld + j], inv, p, mu);
    for (int64_t i = threadIdx.x; i < n; i += kPivotThreads) col[i] = i == k ? 0u : M[i * ld + k];
}

__global__ void __launch_bounds__(kElimThreads) gj_elim_kernel(uint32_t* __restrict__ M, int64_t n, int64_t k,
                                                               uint32_t p, uint64_t mu,
                                                               const uint32_t* __restrict__ col, const int* flag) {
    pdl_wait();
    pdl_trigger();
    if (*flag) return;
    const int64_t ld = 2 * n;
    const int64_t j = k + (int64_t)blockIdx.x * kElimThreads + threadIdx.x;
    if (j >= ld) return;
    const uint32_t rk = M[k * ld + j];
    const int64_t gy = gridDim.y;
    int64_t i = blockIdx.y;
    // four rows at a time: their loads are issued before any store
    for (; i + 3 * gy < n; i += 4 * gy) {
        uint32_t f[4], v[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            f[u] = col[i + u * gy];  // 0 for row k
            v[u] = M[(i + u * gy) * ld + j];
        }
#pragma unroll
        for (int u = 0; u < 4; u++) {
            if (f[u] == 0) continue;
            const uint32_t t = mulmod(f[u], rk, p, mu);
            M[(i + u * gy) * ld + j] = v[u] >= t ? v[u] - t : v[u] + p - t;
        }
    }
    for (; i < n; i += gy) {
        const uint32_t f = col[i];
        if (f == 0) continue;
        const uint32_t t = mulmod(f, rk, p, mu);
        uint32_t* e = M + i * ld + j;
        const uint32_t v = *e;
        *e = v >= t ? v - t : v + p - t;
    }
}

// ---- by panels (panel.h)
//
// M (n x n) is inverted in place: the panel's columns become its transform S,
// the other columns M + S Mp (the panel's pivot rows S Mp), one residue product
// with K = w and one pass.  When every column has had its pivot,
// A^-1[k][c] = M[piv[k]][rowcol[c]].  Up to kInvSingle columns the matrix is one
// panel, in the shared memory of one cluster (n = 512: 0.70 ms, n = 513 in five
// panels 0.63 ms, n = 384 0.61 ms).  Above 5900 the rows of 128 columns do not fit
// the cluster: those panels are reduced by narrower ones (64 columns up to 11,700,
// 32 up to 22,000, ...) whose products stay within the 128 columns, so that the
// whole matrix is still read and written once per 128: n = 10007 138 ms (217 ms
// with a product over the matrix per narrow panel, 325 ms by two launches a
// column), n = 20501 0.95 s (3.09 s, 1.72 s).
//
// GB300, 24-bit p: n = 1500 2.5 ms (15.3 ms with two launches per column of a
// panel), n = 1024 1.3 ms, n = 128 0.12 ms.  Of a round of 16 columns at n = 1500
// (31,000 cycles): the multiply-adds of the update 14,000 (28 of them a clock and
// SM is what the integer pipe gives: 94 rows x 128 words x 16), the tile of the
// pivots 10,000, the barriers and the way of Y through L2 7,000; the products
// between panels add 60 us each.

// The other columns of a block of M's columns from b0, w of them from c0 being
// the panel: column x of the R others is b0 + x, or b0 + x + w from the panel on.
__global__ void __launch_bounds__(kElimThreads)
    inv_gather_kernel(const uint32_t* __restrict__ M, int64_t ld, int64_t b0, int64_t c0, int w, int64_t R,
                      const int* __restrict__ piv, int32_t* __restrict__ Mp, const int* flag) {
    const int64_t x = (int64_t)blockIdx.x * kElimThreads + threadIdx.x;
    if (x >= R || *flag) return;  // (without a pivot there is no row to read)
    const int t = blockIdx.y;
    Mp[(int64_t)t * R + x] = (int32_t)M[(int64_t)piv[c0 + t] * ld + b0 + (b0 + x < c0 ? x : x + w)];
}

// M[i] = C[i] on the panel's pivot rows, M[i] + C[i] mod p on the others
__global__ void __launch_bounds__(kElimThreads)
    inv_update_kernel(uint32_t* __restrict__ M, int64_t ld, int64_t n, int64_t b0, int64_t c0, int w, int64_t R,
                      const int* __restrict__ rowcol, const int32_t* __restrict__ C, uint32_t p) {
    const int64_t x = (int64_t)blockIdx.x * kElimThreads + threadIdx.x;
    if (x >= R) return;
    const int64_t c = b0 + (b0 + x < c0 ? x : x + w);
    for (int64_t i = blockIdx.y; i < n; i += gridDim.y) {
        const int q = rowcol[i];
        const uint32_t v = (uint32_t)C[i * R + x];
        uint32_t* m = M + i * ld + c;
        const uint32_t u = (q >= c0 && q < c0 + w) ? v : *m + v;  // both below p < 2^31
        *m = u >= p ? u - p : u;
    }
}

// A^-1[k][c] = M[piv[k]][rowcol[c]]
__global__ void __launch_bounds__(kElimThreads)
    inv_place_kernel(const uint32_t* __restrict__ M, int64_t n, const int* __restrict__ piv,
                     const int* __restrict__ rowcol, int32_t* __restrict__ out, const int* flag) {
    const int64_t c = (int64_t)blockIdx.x * kElimThreads + threadIdx.x;
    if (c >= n || *flag) return;
    const int64_t at = rowcol[c];
    for (int64_t k = blockIdx.y; k < n; k += gridDim.y) out[k * n + c] = (int32_t)M[(int64_t)piv[k] * n + at];
}

}  // namespace

int64_t inv_panel_width(int64_t n) { return n <= kInvSingle ? n : 128; }

int64_t inv_sub_width(int64_t n) { return n <= kInvSingle ? n : panel_width(n, 1, 128); }

size_t inv_scratch_bytes() { return sizeof(uint32_t) * panel_scratch(kInvSingle); }

cudaError_t launch_inv_panel(uint32_t* M, int64_t n, int64_t c0, int w, uint32_t p, int* rowcol, int* piv, int32_t* S,
                             void* scratch, int* flag, int* status, cudaStream_t s) {
    if (p >= kInvMaxP || !(p & 1)) return cudaErrorInvalidValue;
    PanelArgs<1> a{};
    a.M = M;
    a.n = a.ld = n;
    a.c0 = c0;
    a.w = w;
    panel_mod(a.md, 0, p, p);
    a.ybuf = (uint32_t*)scratch;
    a.piv = piv;
    a.flag = flag;
    a.rowcol = rowcol;
    a.S = S;
    a.status = status;
    return launch_panel_red<1, PanelRed::kOddNarrow, PanelKind::kInverse>(a, n, s);
}

cudaError_t launch_inv_gather(const uint32_t* M, int64_t n, int64_t b0, int64_t bw, int64_t c0, int w, const int* piv,
                              int32_t* Mp, const int* flag, cudaStream_t s) {
    const int64_t R = bw - w;
    inv_gather_kernel<<<dim3((unsigned)((R + kElimThreads - 1) / kElimThreads), (unsigned)w), kElimThreads, 0, s>>>(
        M, n, b0, c0, w, R, piv, Mp, flag);
    return cudaGetLastError();
}

cudaError_t launch_inv_update(uint32_t* M, int64_t n, int64_t b0, int64_t bw, int64_t c0, int w, const int* rowcol,
                              const int32_t* C, uint32_t p, cudaStream_t s) {
    const int64_t R = bw - w;
    inv_update_kernel<<<dim3((unsigned)((R + kElimThreads - 1) / kElimThreads), (unsigned)std::min<int64_t>(n, kMaxGridY)),
                        kElimThreads, 0, s>>>(M, n, n, b0, c0, w, R, rowcol, C, p);
    return cudaGetLastError();
}

cudaError_t launch_inv_place(const uint32_t* M, int64_t n, const int* piv, const int* rowcol, int32_t* out,
                             const int* flag, cudaStream_t s) {
    inv_place_kernel<<<dim3((unsigned)((n + kElimThreads - 1) / kElimThreads), (unsigned)std::min<int64_t>(n, kMaxGridY)),
                       kElimThreads, 0, s>>>(M, n, piv, rowcol, out, flag);
    return cudaGetLastError();
}

cudaError_t launch_inverse_mod_p(const int32_t* res, int64_t n, uint32_t p, uint32_t* M, uint32_t* col, int* flag,
                                 int32_t* C, int* status, int num_sms, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const uint64_t mu = UINT64_MAX / p;
    const int64_t blocks = kElimBlocksPerSM * (num_sms > 0 ? num_sms : 148);
    cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    gj_init_kernel<<<(unsigned)((2 * n * n + kElimThreads - 1) / kElimThreads), kElimThreads, 0, s>>>(res, n, M);
    for (int64_t k = 0; k < n; k++) {
        if ((e = launch_pdl(gj_pivot_kernel, dim3(1), dim3(kPivotThreads), 0, s, M, n, k, p, mu, col, flag, status)) !=
            cudaSuccess)
            return e;
        // about 16 blocks per SM in all, each over a strided set of rows
        const int64_t gx = (2 * n - k + kElimThreads - 1) / kElimThreads;
        const int64_t gy = std::min<int64_t>(std::min<int64_t>(n, kMaxGridY), std::max<int64_t>(1, blocks / gx));
        const dim3 grid((unsigned)gx, (unsigned)gy);
        if ((e = launch_pdl(gj_elim_kernel, grid, dim3(kElimThreads), 0, s, M, n, k, p, mu, (const uint32_t*)col,
                            (const int*)flag)) != cudaSuccess)
            return e;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return cudaMemcpy2DAsync(C, sizeof(int32_t) * n, M + n, sizeof(uint32_t) * 2 * n, sizeof(int32_t) * n, n,
                             cudaMemcpyDeviceToDevice, s);
}

}  // namespace smf

// p-adic (Dixon) lifting: the elementwise steps between the products.
// With C = A^-1 mod p, each step computes X_i = C R_i mod p (a residue product)
// and A X_i (an exact product); these kernels widen X_i to the product's word
// layout and form R_(i+1) = (R_i - A X_i) / p, an exact division whose
// remainder is checked (a non-zero remainder means C is not A^-1 mod p).
//
// The limb form runs each step as two residue products and two kernels that
// stand between them and take the products' K-split partials as they are:
//   lift_x:    X_i = sum of the partials of C R_i mod p, stored, and X_i's
//              centred residues modulo the product basis q_0 .. q_(L-1), split
//              into the digit planes of A X_i's B operand;
//   lift_step: A X_i mod q_j summed over its partials, A X_i itself by Garner's
//              mixed radix (|A X_i| < Q/2, Q = q_0 ... q_(L-1)),
//              R_(i+1) = (R_i - A X_i) / p in place, and the digit planes of
//              R_(i+1) mod p for the next step's C R_(i+1).
// The C and A digit planes are made once per call.
#include <cuda_bf16.h>

#include "smf_internal.h"

namespace smf {
namespace {

constexpr int kThreads = 256;

__global__ void __launch_bounds__(kThreads) widen_kernel(const int32_t* __restrict__ x, int64_t count,
                                                         int64_t* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i < count) out[i] = (int64_t)x[i];
}

__global__ void __launch_bounds__(kThreads) lift_update_kernel(int64_t* __restrict__ R, int64_t ldR,
                                                               const int64_t* __restrict__ AX, int64_t rows,
                                                               int64_t cols, int64_t p, int* status) {
    const int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (e >= rows * cols) return;
    const int64_t r = e / cols, c = e - r * cols;
    int64_t* rp = R + r * ldR + c;
    const int64_t t = *rp - AX[e];
    const int64_t q = t / p;
    if (q * p != t) atomicOr(status, kStatusInexact);
    *rp = q;
}

// Balanced base-2^8 digits of a centred value: t-1 digits in [-128, 127], then
// the remaining quotient (|v| <= 2^23 keeps it within +-128 for t = 3).  Digit u
// goes to d[u * plane].
__device__ __forceinline__ void put_digits(__nv_bfloat16* d, int64_t plane, int32_t v, int t) {
    for (int u = 0; u < t - 1; u++) {
        const int32_t lo = ((v + 128) & 255) - 128;
        d[u * plane] = __int2bfloat16_rn(lo);
        v = (v - lo) >> 8;  // exact: v - lo is a multiple of 256
    }
    d[(t - 1) * plane] = __int2bfloat16_rn(v);
}

// The step kernels work on tiles of 32 rows by 8 columns of the n x m matrices:
// entries are read and written along c (the matrices are row-major in k), and the
// digit planes [t][L][m][ldd], contiguous in k, are written along k after a
// transpose through shared memory.  One entry per thread.  The step is a chain of
// short launches, so what counts is one thread's way through it: tiles of 32 x 32 in
// 64 blocks, with 64-bit divisions emulated one after the other, took 12.1 us for
// lift_step and 5.6 us for lift_x at n = 1024, m = 64.  Every division is by a number
// fixed for the call, so all of them are products with constants (LiftBasis).  The
// whole Smith form of a planted n = 1009 matrix went from 37.9 to 35.5 ms; the loop at
// n = 1024, m = 64 from 34.6 to 33.9 us a step (32.7 with the tiles of columns along
// the grid's first dimension): the two products bound it.
constexpr int kTileK = 32, kTileC = 8;

// x mod q, rcp = floor(2^32 / q): the quotient is at most one low
__device__ __forceinline__ uint32_t mod32(uint32_t x, uint32_t q, uint32_t rcp) {
    const uint32_t r = x - __umulhi(x, rcp) * q;
    return min(r, r - q);
}
// v w mod q in [0, 2q) for any v, ws = floor(w 2^32 / q) (Shoup)
__device__ __forceinline__ uint32_t mul_shoup(uint32_t v, uint32_t w, uint32_t ws, uint32_t q) {
    return v * w - __umulhi(v, ws) * q;
}

// Sum of `split` canonical partials (at most 16 below 2^26: the sum stays
// below 2^32) at stride `stride`, reduced mod q once.  The loads are
// independent of one another and unrolled, so they are all in flight at once.
__device__ __forceinline__ uint32_t sum_parts(const int32_t* __restrict__ part, int split, int64_t stride,
                                              uint32_t q, uint32_t rcp) {
    uint32_t a0 = 0, a1 = 0, a2 = 0, a3 = 0;
    int sp = 0;
    for (; sp + 4 <= split; sp += 4) {
        a0 += (uint32_t)part[(sp + 0) * stride];
        a1 += (uint32_t)part[(sp + 1) * stride];
        a2 += (uint32_t)part[(sp + 2) * stride];
        a3 += (uint32_t)part[(sp + 3) * stride];
    }
    for (; sp < split; sp++) a0 += (uint32_t)part[sp * stride];
    return mod32(a0 + a1 + a2 + a3, q, rcp);
}

template <int LQ>
__global__ void __launch_bounds__(kThreads)
    lift_x_kernel(const int32_t* __restrict__ part, int split, int64_t n, int64_t m, int32_t* __restrict__ X,
                  const __grid_constant__ LiftBasis q, __nv_bfloat16* __restrict__ xdig, int64_t ldd, int t) {
    __shared__ uint32_t tile[kTileK][kTileC + 1];
    pdl_wait();
    pdl_trigger();
    const int64_t nm = n * m;
    const int64_t k0 = (int64_t)blockIdx.y * kTileK, c0 = (int64_t)blockIdx.x * kTileC;
    {  // X_i = the K-split partials summed mod p, along c
        const int tx = threadIdx.x % kTileC, ty = threadIdx.x / kTileC;
        const int64_t k = k0 + ty, c = c0 + tx;
        if (k < n && c < m) {
            const int64_t at = k * m + c;
            const uint32_t x = sum_parts(part + at, split, nm, q.p, q.prcp);
            X[at] = (int32_t)x;
            tile[ty][tx] = x;
        }
    }
    __syncthreads();
    // its centred residues modulo q_j, as digit planes, along k
    const int tx = threadIdx.x % kTileK, ty = threadIdx.x / kTileK;
    const int64_t k = k0 + tx, c = c0 + ty;
    if (k >= n || c >= m) return;
    const int64_t plane = (int64_t)LQ * m * ldd;
    const uint32_t x = tile[tx][ty];
#pragma unroll
    for (int j = 0; j < LQ; j++) {
        int32_t v = (int32_t)mod32(x, q.q[j], q.rcp[j]);
        if (v > (int32_t)(q.q[j] >> 1)) v -= (int32_t)q.q[j];
        put_digits(xdig + (j * m + c) * ldd + k, plane, v, t);
    }
}

template <int LQ>
__global__ void __launch_bounds__(kThreads)
    lift_step_kernel(const int32_t* __restrict__ part, int split, int64_t n, int64_t m,
                     const __grid_constant__ LiftBasis q, int64_t* __restrict__ R, int64_t ldR,
                     __nv_bfloat16* __restrict__ rdig, int64_t ldd, int t, int* status) {
    __shared__ int32_t tile[kTileK][kTileC + 1];
    pdl_wait();
    pdl_trigger();
    const int64_t nm = n * m;
    const int64_t k0 = (int64_t)blockIdx.y * kTileK, c0 = (int64_t)blockIdx.x * kTileC;
    {
        const int tx = threadIdx.x % kTileC, ty = threadIdx.x / kTileC;
        const int64_t k = k0 + ty, c = c0 + tx;
        if (k < n && c < m) {
            const int64_t at = k * m + c;
            int64_t* rp = R + k * ldR + c;
            const int64_t rv = *rp;
            // mixed-radix digits v_j of A X_i mod Q: with s_j = (v_0 + v_1 q_0 + ...
            // + v_(j-1) q_0...q_(j-2)) mod q_j, v_j = (r_j - s_j) (q_0...q_(j-1))^-1 mod q_j
            uint32_t rj[LQ], v[LQ];
#pragma unroll
            for (int j = 0; j < LQ; j++) rj[j] = sum_parts(part + j * nm + at, split, LQ * nm, q.q[j], q.rcp[j]);
            uint64_t x = 0;  // modulo 2^64: |A X_i| < 2^62
            int cmp = 0;     // against (Q - 1) / 2, whose digits are the (q_j - 1) / 2
#pragma unroll
            for (int j = 0; j < LQ; j++) {
                const uint32_t qj = q.q[j];
                uint32_t s = rj[j];
#pragma unroll
                for (int i = 0; i < j; i++) s += 2 * qj - mul_shoup(v[i], q.w[j][i], q.ws[j][i], qj);  // < 7 q_j
                if (j > 0) {
                    s = mul_shoup(s, q.inv[j], q.invs[j], qj);
                    s = min(s, s - qj);
                }
                v[j] = s;
                x += (uint64_t)s * q.W[j];
                if (s != (qj >> 1)) cmp = s > (qj >> 1) ? 1 : -1;
            }
            if (cmp > 0) x -= q.Q;
            const int64_t d = rv - (int64_t)x;
            // the quotient by p as a product with p^-1 mod 2^64: exact iff it is in range
            int64_t quo = (int64_t)((uint64_t)d * q.pinv);
            if (quo > q.qmax || quo < -q.qmax) {
                atomicOr(status, kStatusInexact);
                quo = d / (int64_t)q.p;
            }
            *rp = quo;
            const uint64_t u = quo < 0 ? 0 - (uint64_t)quo : (uint64_t)quo;
            const uint32_t lo = (uint32_t)u;
            uint32_t r = mul_shoup((uint32_t)(u >> 32), q.p32, q.p32s, q.p) + mod32(lo, q.p, q.prcp);  // < 3p
            r = min(r, r - 2 * q.p);
            r = min(r, r - q.p);
            int32_t res = quo < 0 && r ? (int32_t)(q.p - r) : (int32_t)r;
            if (res > (int32_t)(q.p >> 1)) res -= (int32_t)q.p;
            tile[ty][tx] = res;
        }
    }
    if (!rdig) return;  // uniform over the block
    __syncthreads();
    const int tx = threadIdx.x % kTileK, ty = threadIdx.x / kTileK;
    const int64_t k = k0 + tx, c = c0 + ty;
    if (k < n && c < m) put_digits(rdig + c * ldd + k, m * ldd, tile[tx][ty], t);
}

}  // namespace

void lift_basis(const smf_basis& Q, uint32_t p, LiftBasis* q) {
    q->L = (int)Q.primes.size();
    q->Q = 1;
    for (int j = 0; j < q->L; j++) {
        q->q[j] = Q.primes[j];
        q->rcp[j] = (uint32_t)((1ull << 32) / Q.primes[j]);
        q->inv[j] = Q.ginv[j];
        q->invs[j] = Q.ginvs[j];
        for (int i = 0; i < j; i++) {
            q->w[j][i] = Q.gw[(size_t)j * q->L + i];
            q->ws[j][i] = Q.gws[(size_t)j * q->L + i];
        }
        q->W[j] = q->Q;
        q->Q *= Q.primes[j];
    }
    q->p = p;
    q->prcp = (uint32_t)((1ull << 32) / p);
    q->p32 = (uint32_t)((1ull << 32) % p);
    q->p32s = (uint32_t)(((uint64_t)q->p32 << 32) / p);
    q->pinv = p;  // p odd: p p = 1 mod 8, and each Newton step doubles the bits
    for (int k = 0; k < 5; k++) q->pinv *= 2 - p * q->pinv;
    q->qmax = INT64_MAX / (int64_t)p;
}

// Tiles of columns along x, which takes 2^31 blocks (y: 65535; A is n x n, so n is
// never that large, but m can be).
static dim3 tile_grid(int64_t n, int64_t m) {
    return dim3((unsigned)((m + kTileC - 1) / kTileC), (unsigned)((n + kTileK - 1) / kTileK));
}

cudaError_t launch_lift_x(const int32_t* part, int split, int64_t n, int64_t m, int32_t* X, const LiftBasis& q,
                          void* xdig, int64_t ldd, int t, cudaStream_t s) {
    if (n * m == 0) return cudaSuccess;
    const dim3 grid = tile_grid(n, m);
    __nv_bfloat16* xd = (__nv_bfloat16*)xdig;
    switch (q.L) {
    case 1: return launch_pdl(lift_x_kernel<1>, grid, dim3(kThreads), 0, s, part, split, n, m, X, q, xd, ldd, t);
    case 2: return launch_pdl(lift_x_kernel<2>, grid, dim3(kThreads), 0, s, part, split, n, m, X, q, xd, ldd, t);
    case 3: return launch_pdl(lift_x_kernel<3>, grid, dim3(kThreads), 0, s, part, split, n, m, X, q, xd, ldd, t);
    case 4: return launch_pdl(lift_x_kernel<4>, grid, dim3(kThreads), 0, s, part, split, n, m, X, q, xd, ldd, t);
    default: return cudaErrorNotSupported;
    }
}

cudaError_t launch_lift_step(const int32_t* part, int split, int64_t n, int64_t m, const LiftBasis& q, int64_t* R,
                             int64_t ldR, void* rdig, int64_t ldd, int t, int* status, cudaStream_t s) {
    if (n * m == 0) return cudaSuccess;
    const dim3 grid = tile_grid(n, m);
    __nv_bfloat16* rd = (__nv_bfloat16*)rdig;
    switch (q.L) {
    case 1: return launch_pdl(lift_step_kernel<1>, grid, dim3(kThreads), 0, s, part, split, n, m, q, R, ldR, rd, ldd, t, status);
    case 2: return launch_pdl(lift_step_kernel<2>, grid, dim3(kThreads), 0, s, part, split, n, m, q, R, ldR, rd, ldd, t, status);
    case 3: return launch_pdl(lift_step_kernel<3>, grid, dim3(kThreads), 0, s, part, split, n, m, q, R, ldR, rd, ldd, t, status);
    case 4: return launch_pdl(lift_step_kernel<4>, grid, dim3(kThreads), 0, s, part, split, n, m, q, R, ldR, rd, ldd, t, status);
    default: return cudaErrorNotSupported;
    }
}

cudaError_t launch_widen(const int32_t* x, int64_t count, int64_t* out, cudaStream_t s) {
    if (count == 0) return cudaSuccess;
    widen_kernel<<<(unsigned)((count + kThreads - 1) / kThreads), kThreads, 0, s>>>(x, count, out);
    return cudaGetLastError();
}

cudaError_t launch_lift_update(int64_t* R, int64_t ldR, const int64_t* AX, int64_t rows, int64_t cols, uint32_t p,
                               int* status, cudaStream_t s) {
    const int64_t count = rows * cols;
    if (count == 0) return cudaSuccess;
    lift_update_kernel<<<(unsigned)((count + kThreads - 1) / kThreads), kThreads, 0, s>>>(R, ldR, AX, rows, cols,
                                                                                          (int64_t)p, status);
    return cudaGetLastError();
}

}  // namespace smf

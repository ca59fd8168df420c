// crt_reconstruct: residues -> the signed integer (Section 3.1: the exact
// product is recovered from its per-prime residues by CRT), one entry per
// thread, result in (-M/2, M/2] written as W two's complement words; and the
// conversion between RNS bases.  The per-entry reconstruction (Lagrange form
// with an fp32 quotient, exact mixed-radix fallback) is in crt_dev.h.
#include <vector>

#include "rns_mma.h"

namespace smf {
namespace {

template <int LMAX, bool FAST, int PB>
__global__ void __launch_bounds__(128)
crt_kernel(const __grid_constant__ CrtConst<LMAX, FAST, PB> q, const int32_t* __restrict__ R, int64_t rows,
           int64_t cols, uint64_t* __restrict__ X, int64_t ld, int W) {
    const int64_t count = rows * cols;
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= count) return;
    crt_entry<LMAX, FAST, PB>(q, R, count, cols, e, X, ld, W);
}

// Several outputs of one basis in one launch: block u takes unit u, the 128
// consecutive entries u - base_i of item i (found by bisection).  One unit per
// block keeps the register count of crt_kernel; the search is a few loads from
// L1 against a block's tens of thousands of modular products.
template <int LMAX, bool FAST, int PB>
__global__ void __launch_bounds__(128)
crt_grouped_kernel(const __grid_constant__ CrtConst<LMAX, FAST, PB> q, const CrtItem* __restrict__ items, int n) {
    const CrtItem* it = find_item(items, n, (int64_t)blockIdx.x);
    const int64_t count = it->rows * it->cols;
    const int64_t e = ((int64_t)blockIdx.x - it->base) * 128 + threadIdx.x;
    if (e < count) crt_entry<LMAX, FAST, PB>(q, it->R, count, it->cols, e, it->X, it->ld, it->W);
}

// ---------------------------------------------------------------------------
// Conversion between RNS bases (Section 3.1: the Lagrange shortcut with a
// floating-point correction, no reconstruction).  With xi_i and alpha as in
// the fast path above, x + H = sum_i xi_i M_i - alpha M, so for a target prime q
//   x mod q = (sum_i xi_i (M_i mod q) - alpha (M mod q) - (H mod q)) mod q.
// Each term xi_i (M_i mod q) < 2^52 and at most 48 of them are summed in a
// 64-bit register, then one Barrett reduction.  When the fp32 estimate of
// alpha is too close to an integer to call, alpha is settled exactly: the
// true value is within one of floor(f), and it is the one that puts
// sum_i xi_i M_i - alpha M in [0, M), checked limb by limb.
template <int LMAX>
struct ConvConst {
    static constexpr int MLMAX = (LMAX * 26 + 31) / 32 + 1;
    uint32_t p[LMAX], hmod[LMAX], c[LMAX], cs[LMAX];
    float invp[LMAX];
    uint32_t mi[LMAX * MLMAX];     // limbs of M_i (exact alpha)
    uint32_t m[MLMAX];             // limbs of M
    uint32_t wt[LMAX * LMAX];      // M_i mod q_j at j * LMAX + i (zero for i >= L)
    // per target prime: {q, 2^32 mod q, its Shoup companion, floor(2^32 / q),
    // M mod q, H mod q, 0, 0}
    uint32_t qr[LMAX * 8];
    int L, LQ, m_limbs;
};
static_assert(sizeof(ConvConst<48>) <= 32000, "kernel parameter space");

template <int LMAX>
__device__ __noinline__ uint32_t exact_alpha(const ConvConst<LMAX>& v, const int32_t* __restrict__ R, int64_t count,
                                             int64_t e, uint32_t fl) {
    constexpr int MLMAX = ConvConst<LMAX>::MLMAX;
    const int L = v.L, ml = v.m_limbs;
    uint32_t xi[LMAX];  // recomputed here, so that the common path keeps its xi in registers
#pragma unroll 1
    for (int i = 0; i < L; i++) {
        const uint32_t pi = v.p[i];
        uint32_t a = (uint32_t)__ldg(R + (size_t)i * count + e) + v.hmod[i];
        if (a >= pi) a -= pi;
        uint32_t z = shoup_mul(a, v.c[i], v.cs[i], pi);
        if (z >= pi) z -= pi;
        xi[i] = z;
    }
    uint32_t d[MLMAX + 1];  // sum_i xi_i M_i - fl M, two's complement over ml + 1 limbs
    uint64_t carry = 0;
    uint32_t borrow = 0;
#pragma unroll 1
    for (int j = 0; j <= ml; j++) {
        uint64_t col = carry;
        if (j < ml) {
#pragma unroll 1
            for (int i = 0; i < L; i++) col += (uint64_t)xi[i] * v.mi[i * MLMAX + j];  // < 48 * 2^58 + 2^32
        }
        const uint32_t y = (uint32_t)col;
        carry = col >> 32;
        const uint64_t am = (uint64_t)fl * (j < ml ? v.m[j] : 0u) + borrow;
        const uint64_t diff = (uint64_t)y - (uint32_t)am;
        borrow = (uint32_t)(am >> 32) + (uint32_t)(diff >> 63);
        d[j] = (uint32_t)diff;
    }
    if (d[ml] >> 31) return fl - 1;  // below 0
    bool ge = d[ml] != 0;            // compare with M
    if (!ge) {
        ge = true;  // equal counts as >= M
#pragma unroll 1
        for (int j = ml - 1; j >= 0; j--) {
            if (d[j] != v.m[j]) {
                ge = d[j] > v.m[j];
                break;
            }
        }
    }
    return ge ? fl + 1 : fl;
}

template <int LMAX>
__global__ void __launch_bounds__(128)
convert_kernel(const __grid_constant__ ConvConst<LMAX> v, const int32_t* __restrict__ R, int32_t* __restrict__ out,
               int64_t count) {
    // The [j][i] table of M_i mod q_j and the per-target-prime records are
    // staged once per block in shared memory; the block then walks chunks of
    // 128 entries.  The loop over source primes is unrolled against 16-byte
    // shared loads, so xi stays in registers.
    __shared__ __align__(16) uint32_t ws[LMAX * LMAX];
    __shared__ __align__(16) uint32_t qs[LMAX * 8];
    const int L = v.L, LQ = v.LQ;
    for (int k = threadIdx.x; k < LQ * LMAX; k += blockDim.x) ws[k] = v.wt[k];
    for (int k = threadIdx.x; k < LQ * 8; k += blockDim.x) qs[k] = v.qr[k];
    __syncthreads();
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x) {
        uint32_t rv[LMAX], xi[LMAX];
#pragma unroll
        for (int i = 0; i < LMAX; i++) rv[i] = i < L ? (uint32_t)__ldg(R + (size_t)i * count + e) : 0u;
        float f = 0.f;
#pragma unroll
        for (int i = 0; i < LMAX; i++) {
            xi[i] = 0;
            if (i < L) {
                const uint32_t pi = v.p[i];
                uint32_t a = rv[i] + v.hmod[i];
                if (a >= pi) a -= pi;
                uint32_t z = shoup_mul(a, v.c[i], v.cs[i], pi);
                if (z >= pi) z -= pi;
                xi[i] = z;
                f = fmaf((float)z, v.invp[i], f);
            }
        }
        const float fl = floorf(f);
        const float frac = f - fl;
        uint32_t alpha = (uint32_t)fl;
        if (frac < 0x1p-12f || frac > 1.f - 0x1p-12f) alpha = exact_alpha<LMAX>(v, R, count, e, alpha);
        int32_t* o = out + e;
#pragma unroll 1
        for (int j = 0; j < LQ; j++, o += count) {
            const uint4* wj = reinterpret_cast<const uint4*>(ws + j * LMAX);
            uint32_t l0 = 0, h0 = 0, l1 = 0, h1 = 0;  // two chains; xi_i = 0 and w = 0 beyond L
#pragma unroll
            for (int i4 = 0; i4 < LMAX / 4; i4++) {
                const uint4 w4 = wj[i4];
                mac64(l0, h0, xi[4 * i4], w4.x);
                mac64(l1, h1, xi[4 * i4 + 1], w4.y);
                mac64(l0, h0, xi[4 * i4 + 2], w4.z);
                mac64(l1, h1, xi[4 * i4 + 3], w4.w);
            }
            const uint4 c0 = *reinterpret_cast<const uint4*>(qs + 8 * j);
            const uint2 c1 = *reinterpret_cast<const uint2*>(qs + 8 * j + 4);
            const uint32_t qj = c0.x;
            // y - H = sum - alpha M - H; adding q 2^32 keeps it non-negative
            // (alpha (M mod q) + (H mod q) < 49 * 2^26 < 2^32) and below 2^59
            const uint64_t t = (((uint64_t)h0 << 32) | l0) + (((uint64_t)h1 << 32) | l1) + ((uint64_t)qj << 32) -
                               ((uint64_t)alpha * c1.x + c1.y);
            const uint32_t hi = (uint32_t)(t >> 32), lo = (uint32_t)t;
            const uint32_t t1 = hi * c0.y - __umulhi(hi, c0.z) * qj;  // [0, 2q)
            const uint32_t t2 = lo - __umulhi(lo, c0.w) * qj;         // [0, 2q)
            uint32_t r = t1 + t2;                                     // [0, 4q)
            if (r >= 2 * qj) r -= 2 * qj;
            if (r >= qj) r -= qj;
            *o = (int32_t)r;
        }
    }
}


// ---------------------------------------------------------------------------
// CRT of bases of 13 to 48 primes below 2^24, on the tensor cores (rns_mma.h).
// x = sum_i xi_i M_i - alpha M - H modulo 2^(8 N), where N bytes hold the signed
// result; the columns of the product are the balanced base-256 digits of the
// 2^(8u) M_i, lane 4g + t owns 2 NT consecutive ones (NT / 2 limbs), and the carry
// into the next lane's limbs is passed by a shuffle.  The limbs go through shared
// memory, so that the words are stored in order.
// 1300 thread instructions an entry with 23 primes (1815 as limb sums, one thread per
// entry) at half the issue slots: 18.6M entries 1.51 -> 1.47 ms.  The product of 1009 x 1009 by
// 1009 x 100 with 34 primes (reduction and CRT both so) went from 303 to 208 us, one
// of 64 x 64 by 64 x 16 from 38 to 25 us.
template <int LMAX>
struct CrtMma {
    static constexpr int NT = (3 * LMAX / 4 + 3) / 4 * 2;  // n8 tiles
    static constexpr int LPT = NT / 2, NL = 4 * LPT;       // limbs per lane, limbs
    static constexpr int SE = NL + 1;                      // staged entry (odd: no bank conflicts)
    static constexpr int KS = XiShape<LMAX>::KS;
    // the tables, made with the basis and copied to shared memory by each block:
    // fragments, pc, cn (per limb {128 (1 + 2^8 + 2^16) sum_i M_i - H, -M}: the digits
    // of xi are less 128), 1 / p_i
    static constexpr size_t kPc = sizeof(uint2) * NT * KS * 32, kCn = kPc + sizeof(uint4) * LMAX,
                            kIp = kCn + sizeof(uint2) * NL, kImage = kIp + sizeof(float) * LMAX;
    static constexpr size_t kSmem = kImage + sizeof(uint32_t) * (kMmaThreads * SE);
    static_assert(kCn % 16 == 0 && kIp % 16 == 0 && kImage % 16 == 0, "copied 16 bytes at a time");
};

template <int LMAX>
struct CrtSmem {
    const uint2* wf;
    const uint2* cn;
    const uint4* pc;
    const float* ip;
    uint32_t* st;
    __device__ CrtSmem(uint8_t* p, const uint8_t* image) {
        using Q = CrtMma<LMAX>;
        stage(p, image, Q::kImage);
        wf = (const uint2*)p;
        pc = (const uint4*)(p + Q::kPc);
        cn = (const uint2*)(p + Q::kCn);
        ip = (const float*)(p + Q::kIp);
        st = (uint32_t*)(p + Q::kImage) + (threadIdx.x >> 5) * 32 * Q::SE;
        __syncthreads();
    }
};

// The words of the staged entries 0 .. left - 1 (W each, the sign beyond the NL
// limbs), in order by the warp's lanes: word 32 k + lane to to[32 k], or where the
// rows lie apart (GAPS) gap words later for each end of a row passed; col: the
// column of this lane's first entry.  (Carried along: two 64-bit divisions a word
// took 194 us for 2M entries of 9 words, against 154 without gaps.)
template <int NL, int SE, bool GAPS>
__device__ __forceinline__ void put_words(const uint32_t* st, int left, int W, uint64_t* to, int64_t col, int64_t cols,
                                          int64_t gap) {
    const int lane = threadIdx.x & 31, de = 32 / W, dw = 32 % W;
    int e = lane / W, w = lane % W;
    while (e < left) {
        const uint32_t* s = st + e * SE;
        uint32_t lo, hi;
        if (2 * w + 1 < NL) {
            lo = s[2 * w];
            hi = s[2 * w + 1];
        } else {  // the sign
            hi = (uint32_t)((int32_t)s[NL - 1] >> 31);
            lo = 2 * w < NL ? s[2 * w] : hi;
        }
        *to = (uint64_t)hi << 32 | lo;
        to += 32;
        const int before = e;
        e += de;
        w += dw;
        if (w >= W) {
            w -= W;
            e++;
        }
        if constexpr (GAPS)
            for (col += e - before; col >= cols; col -= cols) to += gap;
    }
}

template <int NL, int SE>
__device__ __noinline__ void put_rows(const uint32_t* st, int left, int W, uint64_t* X, int64_t e0, int64_t count,
                                      int64_t cols, int64_t ld) {
    const int lane = threadIdx.x & 31;
    const int64_t q = e0 + lane / W;  // (below 2^32 for an entry that is there, if count is)
    const int64_t row = count <= 0xFFFFFFFFll ? (int64_t)((uint32_t)q / (uint32_t)cols) : q / cols;
    const int64_t gap = (ld - cols) * W;
    put_words<NL, SE, true>(st, left, W, X + e0 * W + lane + row * gap, q - row * cols, cols, gap);
}

// Entries e0 .. e0 + 31 (those below count) of one output, by one warp.
template <int LMAX>
__device__ __forceinline__ void crt_chunk(const XiExact& q, const CrtSmem<LMAX>& sm,
                                          const int32_t* __restrict__ R, int64_t count, int64_t cols, int64_t e0,
                                          uint64_t* __restrict__ X, int64_t ld, int W) {
    using Q = CrtMma<LMAX>;
    const int lane = threadIdx.x & 31, t = lane & 3;
    const bool vec = (count & 3) == 0 && ((uintptr_t)R & 15) == 0;
    uint32_t a[2][Q::KS][4], alpha[4];
    xi_frags<LMAX>(q, sm.pc, sm.ip, R, count, e0, vec, a, alpha);
    uint32_t x[Q::LPT][4];
    int32_t carry[4] = {0, 0, 0, 0};
#pragma unroll
    for (int l = 0; l < Q::LPT; l++) {
        float acc[2][2][4];
        mma_tiles<2, Q::KS>(acc, a, sm.wf + 2 * l * Q::KS * 32 + lane);
        const uint2 k = sm.cn[t * Q::LPT + l];
#pragma unroll
        for (int e = 0; e < 4; e++) {
            uint32_t s[4];  // the four column sums, each 0x4B400000 too large
#pragma unroll
            for (int b = 0; b < 4; b++) s[b] = __float_as_uint(acc[e >> 1][b >> 1][2 * (e & 1) + (b & 1)]);
            const int32_t lo = (int32_t)(s[0] + (s[1] << 8) - kMagicBits * 257u);  // below 2^30 in absolute value
            const int32_t hi = (int32_t)(s[2] + (s[3] << 8) - kMagicBits * 257u);
            const int64_t v = (int64_t)((uint64_t)alpha[e] * k.y + k.x) + (int64_t)hi * 65536 + ((int64_t)lo + carry[e]);
            x[l][e] = (uint32_t)v;
            carry[e] = (int32_t)(v >> 32);
        }
    }
    // the carries into the next lane's limbs; rarely more than one round (a carry
    // that passes all of a lane's limbs)
    for (;;) {
        bool more = false;
#pragma unroll
        for (int e = 0; e < 4; e++) {
            int32_t c = __shfl_up_sync(0xffffffffu, carry[e], 1);
            if (t == 0) c = 0;
#pragma unroll
            for (int l = 0; l < Q::LPT; l++) {
                const int64_t v = (int64_t)x[l][e] + c;
                x[l][e] = (uint32_t)v;
                c = (int32_t)(v >> 32);
            }
            carry[e] = t == 3 ? 0 : c;
            more |= carry[e] != 0;
        }
        if (!__any_sync(0xffffffffu, more)) break;
    }
#pragma unroll
    for (int e = 0; e < 4; e++)
#pragma unroll
        for (int l = 0; l < Q::LPT; l++) sm.st[((lane >> 2) * 4 + e) * Q::SE + t * Q::LPT + l] = x[l][e];
    __syncwarp();
    const int left = (int)min((int64_t)32, count - e0);
    if (ld == cols) {
        put_words<Q::NL, Q::SE, false>(sm.st, left, W, X + e0 * W + lane, 0, 0, 0);
    } else {  // (called: in line it cost the other path registers)
        put_rows<Q::NL, Q::SE>(sm.st, left, W, X, e0, count, cols, ld);
    }
    __syncwarp();
}

template <int LMAX>
__global__ void __launch_bounds__(kMmaThreads, LMAX <= 16 ? 5 : LMAX <= 32 ? 4 : 3)
crt_mma_kernel(const uint8_t* __restrict__ image, XiExact q, const int32_t* __restrict__ R, int64_t rows,
               int64_t cols, uint64_t* __restrict__ X, int64_t ld, int W) {
    extern __shared__ __align__(16) uint8_t dyn[];
    const CrtSmem<LMAX> sm(dyn, image);
    const int64_t count = rows * cols;
    for (int64_t e0 = (int64_t)blockIdx.x * kMmaThreads + (threadIdx.x & ~31); e0 < count;
         e0 += (int64_t)gridDim.x * kMmaThreads)
        crt_chunk<LMAX>(q, sm, R, count, cols, e0, X, ld, W);
}

// Several outputs of one basis in one launch: unit u is the 128 consecutive
// entries u - base_i of item i (found by bisection).
template <int LMAX>
__global__ void __launch_bounds__(kMmaThreads, LMAX <= 16 ? 5 : LMAX <= 32 ? 4 : 3)
crt_mma_grouped_kernel(const uint8_t* __restrict__ image, XiExact q, const CrtItem* __restrict__ items, int n,
                       int64_t units) {
    extern __shared__ __align__(16) uint8_t dyn[];
    const CrtSmem<LMAX> sm(dyn, image);
    for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
        const CrtItem* it = find_item(items, n, u);
        const int64_t count = it->rows * it->cols, e0 = (u - it->base) * kMmaThreads + (threadIdx.x & ~31);
        if (e0 < count) crt_chunk<LMAX>(q, sm, it->R, count, it->cols, e0, it->X, it->ld, it->W);
    }
}

// The fragments of a basis, a block for each tile, on the device from the limbs of
// the M_i.  Lane 4n + t of tile nt owns result bytes (n / 2) 2 NT + 2 nt and + 1, whose
// digit of 2^(8u) M_i is digit (byte - u) of M_i.
template <int LMAX>
__global__ void __launch_bounds__(kMmaThreads)
crt_image_kernel(const uint32_t* __restrict__ mi, int L, int m_limbs, __half* __restrict__ wf) {
    using Q = CrtMma<LMAX>;
    constexpr int NL = Q::NL;
    __shared__ uint32_t bal[LMAX * NL];  // M_i + 0x80..80: its bytes less 128 are the balanced digits of M_i
    const int nt = blockIdx.x;
    if (threadIdx.x < L) {
        uint64_t c = 0;
        for (int k = 0; k < NL; k++) {
            c += (uint64_t)(k < m_limbs ? mi[threadIdx.x * m_limbs + k] : 0u) + 0x80808080u;
            bal[threadIdx.x * NL + k] = (uint32_t)c;
            c >>= 32;
        }
    }
    __syncthreads();
    for (int x = threadIdx.x; x < Q::KS * 128; x += kMmaThreads) {
        const int ks = x / 128, lane = x / 4 % 32, n = lane >> 2, byte = (n >> 1) * 2 * Q::NT + 2 * nt + (n & 1);
        int i, u, d = 0;
        if (xi_slot<LMAX>(ks, x & 3, lane & 3, &i, &u) && i < L && byte >= u)
            d = (int)(bal[i * NL + ((byte - u) >> 2)] >> (8 * ((byte - u) & 3)) & 255u) - 128;
        wf[nt * Q::KS * 128 + x] = __int2half_rn(d);
    }
}

// The image's other tables.
template <int LMAX>
void crt_image(const CrtHost& h, uint8_t* image) {
    using Q = CrtMma<LMAX>;
    constexpr int NL = Q::NL;
    uint64_t sum[NL] = {};
    for (int i = 0; i < h.L; i++)
        for (int k = 0; k < NL && k < h.m_limbs; k++) sum[k] += h.mi[(size_t)i * h.m_limbs + k];
    uint4* pc = (uint4*)(image + Q::kPc);
    float* ip = (float*)(image + Q::kIp);
    for (int i = 0; i < LMAX; i++) {  // beyond L: xi = 0
        pc[i] = i < h.L ? make_uint4(h.p[i], h.hmod[i], h.c[i], h.cs[i]) : make_uint4(1, 0, 0, 0);
        ip[i] = i < h.L ? 1.0f / (float)h.p[i] : 0.f;
    }
    uint2* cn = (uint2*)(image + Q::kCn);
    uint64_t c = 0, b = 0, g = 0;
    for (int k = 0; k < NL; k++) {
        c += sum[k] * (128u * 65793u);
        b = (uint64_t)(uint32_t)c - (k < h.m_limbs ? h.h[k] : 0u) - b;
        g = 0ull - (k < h.m_limbs ? h.m[k] : 0u) - g;
        cn[k] = make_uint2((uint32_t)b, (uint32_t)g);
        b >>= 63;
        g >>= 63;
        c >>= 32;
    }
}

XiExact xi_exact(const CrtHost& h) { return {h.d_mi, h.d_m, h.d_rcp, h.L, h.m_limbs}; }

// As many blocks as are resident at once (each makes the tables once).
template <auto kernel>
cudaError_t mma_grid(size_t smem, int num_sms, int64_t units, unsigned* grid) {
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e) return e;
    }
    // a property of the kernel's code, asked once (1 us a call)
    static const int per = [smem] {
        int n = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kMmaThreads, smem);
        return n > 0 ? n : 1;
    }();
    const int64_t most = (int64_t)num_sms * per;
    *grid = (unsigned)(units < most ? units : most);
    return cudaSuccess;
}

template <int LMAX>
cudaError_t launch_crt_mma(const CrtHost& h, const int32_t* R, int64_t rows, int64_t cols, uint64_t* X, int64_t ld,
                           int W, int num_sms, cudaStream_t s) {
    using Q = CrtMma<LMAX>;
    unsigned grid;
    const cudaError_t e = mma_grid<crt_mma_kernel<LMAX>>(Q::kSmem, num_sms, (rows * cols + kMmaThreads - 1) / kMmaThreads, &grid);
    if (e) return e;
    crt_mma_kernel<LMAX><<<grid, kMmaThreads, Q::kSmem, s>>>(h.d_image, xi_exact(h), R, rows, cols, X, ld, W);
    return cudaGetLastError();
}

template <int LMAX>
cudaError_t launch_crt_mma_grouped(const CrtHost& h, const CrtItem* items, int n, int64_t units, int num_sms,
                                   cudaStream_t s) {
    using Q = CrtMma<LMAX>;
    unsigned grid;
    const cudaError_t e = mma_grid<crt_mma_grouped_kernel<LMAX>>(Q::kSmem, num_sms, units, &grid);
    if (e) return e;
    crt_mma_grouped_kernel<LMAX><<<grid, kMmaThreads, Q::kSmem, s>>>(h.d_image, xi_exact(h), items, n, units);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Conversion to primes below 2^24, on the tensor cores (rns_mma.h): the columns of
// the product are the balanced digits of w_ij 2^(8u) mod q_j, w_ij = M_i mod q_j.
// Lane 4g + t owns target primes j = 4b + t, three columns each; three n8 tiles
// hold two targets of a lane.  A residue is then
//   v = S_0 + 2^8 S_1 + 2^16 S_2 + C_j - alpha (M mod q_j)  mod q_j:
// sums_quot and sums_rem have the arithmetic.
// 23 -> 23 primes, 1M entries: 159 -> 68 us (28 us of HBM traffic); half the issue
// slots are busy, the chunks' latencies bound it.
template <int LMAX>
struct ConvMma {
    const uint4* pc;          // the source's constants (device)
    XiExact xi;
    alignas(16) uint32_t w[LMAX * LMAX];  // w_ij at j LMAX + i (0 for i >= L)
    uint4 ti[LMAX];           // q_j, M mod q_j, rem_const of C_j
    float4 tf[LMAX];          // 1 / q_j, (M mod q_j) / q_j, quot_const of C_j
    int LQ;
};
static_assert(sizeof(ConvMma<48>) <= 32000, "kernel parameter space");

template <int LMAX>
__global__ void __launch_bounds__(kMmaThreads, LMAX <= 24 ? 5 : LMAX <= 32 ? 4 : 3)
convert_mma_kernel(const __grid_constant__ ConvMma<LMAX> v, const int32_t* __restrict__ R, int32_t* __restrict__ out,
                   int64_t count) {
    constexpr int KS = XiShape<LMAX>::KS, NB = LMAX / 8;  // groups of eight targets
    __shared__ uint2 wf[NB * 3 * KS * 32];
    __shared__ uint4 pc[LMAX], ti[LMAX];
    __shared__ float4 tf[LMAX];
    __shared__ float ip[LMAX];
    const int LQ = v.LQ, L = v.xi.L, lane = threadIdx.x & 31, t = lane & 3;
    for (int i = threadIdx.x; i < LMAX; i += kMmaThreads) {
        const uint4 c = i < L ? __ldg(v.pc + i) : make_uint4(1, 0, 0, 0);
        pc[i] = c;
        ip[i] = i < L ? 1.0f / (float)c.x : 0.f;
    }
    for (int j = threadIdx.x; j < LQ; j += kMmaThreads) {
        ti[j] = v.ti[j];
        tf[j] = v.tf[j];
    }
    for (int x = threadIdx.x; x < (LQ + 7) / 8 * 3 * KS * 32; x += kMmaThreads) wf[x] = make_uint2(0, 0);
    __syncthreads();
    // the three digits of w_ij 2^(8u) mod q_j to where the fragments have them (xi_slot)
    // (four w at a time: loads of the parameter bank at an address per lane take turns)
    for (int x = threadIdx.x; x < LQ * (LMAX / 4) * 3; x += kMmaThreads) {
        const int a = x % (LMAX / 4), u = x / (LMAX / 4) % 3, j = x / (LMAX / 4 * 3);
        const int pr = u < 2 ? a : LMAX / 4 + a / 2, kap = 2 * (pr & 1) + (u < 2 ? u : a & 1);
        const uint4 w4 = *(const uint4*)(v.w + j * LMAX + 4 * a);
        const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w}, q = ti[j].x;
        const float s = (float)(1 << 8 * u) * tf[j].x;
#pragma unroll
        for (int z = 0; z < 4; z++) {  // prime 4a + z; w = 0 beyond L
            // to within half of q_j and a little (the quotient is below 2^16)
            int32_t r = (int32_t)((w[z] << 8 * u) - (uint32_t)__float2int_rn((float)w[z] * s) * q);
#pragma unroll
            for (int dig = 0; dig < 3; dig++) {
                const int c6 = (j >> 2 & 1) * 3 + dig, nt = (j >> 3) * 3 + c6 / 2, ln = (2 * (j & 3) + (c6 & 1)) * 4 + z;
                ((__half*)wf)[((nt * KS + pr / 2) * 32 + ln) * 4 + kap] = __int2half_rn(dig < 2 ? ((r + 128) & 255) - 128 : r);
                r = (r + 128) >> 8;
            }
        }
    }
    __syncthreads();
    const bool vec = (count & 3) == 0 && ((uintptr_t)R & 15) == 0, vout = (count & 3) == 0 && ((uintptr_t)out & 15) == 0;
    for (int64_t e0 = (int64_t)blockIdx.x * kMmaThreads + (threadIdx.x & ~31); e0 < count;
         e0 += (int64_t)gridDim.x * kMmaThreads) {
        uint32_t a[2][KS][4], alpha[4];
        float al[4];
        xi_frags<LMAX>(v.xi, pc, ip, R, count, e0, vec, a, alpha);
#pragma unroll
        for (int x = 0; x < 4; x++) al[x] = (float)alpha[x];
        const int64_t e = e0 + (lane >> 2) * 4;
#pragma unroll 1
        for (int nb = 0; 8 * nb < LQ; nb++) {
            float acc[2][3][4];
            mma_tiles<3, KS>(acc, a, wf + 3 * nb * KS * 32 + lane);
#pragma unroll
            for (int b = 0; b < 2; b++) {
                const int j = 8 * nb + 4 * b + t;
                if (j >= LQ) continue;
                const uint4 ci = ti[j];
                const float4 cf = tf[j];
                uint32_t r[4];
#pragma unroll
                for (int x = 0; x < 4; x++) {
                    float s[3];
#pragma unroll
                    for (int k = 0; k < 3; k++) s[k] = acc[x >> 1][(3 * b + k) >> 1][2 * (x & 1) + ((3 * b + k) & 1)];
                    const float f = fmaf(-al[x], cf.y, sums_quot(s[0], s[1], s[2], cf.x, cf.z));
                    const uint32_t y = sums_rem(s[0], s[1], s[2], ci.x, ci.z, f) - alpha[x] * ci.y;
                    r[x] = min(y, y - ci.x);
                }
                int32_t* o = out + (size_t)j * count + e;
                if (vout) {
                    if (e < count) *(int4*)o = make_int4((int)r[0], (int)r[1], (int)r[2], (int)r[3]);
                } else {
#pragma unroll
                    for (int x = 0; x < 4; x++)
                        if (e + x < count) o[x] = (int32_t)r[x];
                }
            }
        }
    }
}

// a mod q of the integer with 32-bit limbs x[0 .. n) (q < 2^32)
uint32_t limbs_mod(const uint32_t* x, int n, uint32_t q) {
    uint64_t r = 0;
    for (int k = n - 1; k >= 0; k--) r = ((r << 32) | x[k]) % q;
    return (uint32_t)r;
}

template <int LMAX>
cudaError_t launch_convert_mma(const CrtHost& h, const uint32_t* q, int LQ, const int32_t* R, int32_t* out,
                               int64_t count, int num_sms, cudaStream_t s) {
    ConvMma<LMAX> v{};
    v.pc = (const uint4*)h.d_pc;
    v.xi = xi_exact(h);
    const int L = h.L;
    for (int j = 0; j < LQ; j++) {
        const uint32_t qj = q[j];
        // M_i mod q_j by products of the primes before and after p_i
        uint32_t* w = v.w + j * LMAX;
        uint64_t before = 1 % qj, after = 1 % qj, sum = 0;
        for (int i = 0; i < L; i++) {
            w[i] = (uint32_t)before;
            before = before * h.p[i] % qj;
        }
        for (int i = L - 1; i >= 0; i--) {
            w[i] = (uint32_t)(w[i] * after % qj);
            after = after * h.p[i] % qj;
            sum += w[i];
        }
        const uint32_t m = (uint32_t)before, hm = limbs_mod(h.h, h.m_limbs, qj);
        const uint32_t c = (uint32_t)((sum * (128u * 65793u) + qj - hm) % qj);  // (every digit of xi is less 128)
        const float iq = 1.0f / (float)qj;
        v.ti[j] = make_uint4(qj, m, rem_const(c, qj), 0);
        v.tf[j] = make_float4(iq, (float)m / (float)qj, quot_const(c, iq, qj), 0.f);
    }
    v.LQ = LQ;
    unsigned grid;
    const cudaError_t e = mma_grid<convert_mma_kernel<LMAX>>(0, num_sms, (count + kMmaThreads - 1) / kMmaThreads, &grid);
    if (e) return e;
    convert_mma_kernel<LMAX><<<grid, kMmaThreads, 0, s>>>(v, R, out, count);
    return cudaGetLastError();
}

template <int LMAX, bool FAST, int PB>
cudaError_t launch_crt_t(const CrtHost& h, const int32_t* R, int64_t rows, int64_t cols, uint64_t* X, int64_t ld,
                         int W, cudaStream_t s) {
    CrtConst<LMAX, FAST, PB> q;
    crt_const(h, q);
    const int64_t count = rows * cols;
    const int threads = 128;
    crt_kernel<LMAX, FAST, PB><<<(unsigned)((count + threads - 1) / threads), threads, 0, s>>>(q, R, rows, cols, X, ld,
                                                                                          W);
    return cudaGetLastError();
}

template <int LMAX, bool FAST, int PB>
cudaError_t launch_crt_grouped_t(const CrtHost& h, const CrtItem* items, int n, int64_t units, cudaStream_t s) {
    CrtConst<LMAX, FAST, PB> q;
    crt_const(h, q);
    crt_grouped_kernel<LMAX, FAST, PB><<<(unsigned)units, 128, 0, s>>>(q, items, n);
    return cudaGetLastError();
}

template <int LMAX>
cudaError_t launch_convert_t(const CrtHost& h, const uint32_t* q, int LQ, const int32_t* R, int32_t* out,
                             int64_t count, int num_sms, cudaStream_t s) {
    using V = ConvConst<LMAX>;
    V v{};  // the parameter block, copied into the launch
    const int L = h.L;
    if (h.m_limbs > V::MLMAX) return cudaErrorInvalidValue;
    for (int i = 0; i < L; i++) {
        v.p[i] = h.p[i];
        v.hmod[i] = h.hmod[i];
        v.c[i] = h.c[i];
        v.cs[i] = h.cs[i];
        v.invp[i] = 1.0f / (float)h.p[i];
        for (int k = 0; k < h.m_limbs; k++) v.mi[i * V::MLMAX + k] = h.mi[(size_t)i * h.m_limbs + k];
    }
    for (int k = 0; k < h.m_limbs; k++) v.m[k] = h.m[k];
    for (int j = 0; j < LQ; j++) {
        const uint32_t qj = q[j];
        const uint32_t r32 = (uint32_t)((1ull << 32) % qj);
        uint32_t* rec = v.qr + 8 * j;
        rec[0] = qj;
        rec[1] = r32;
        rec[2] = (uint32_t)(((uint64_t)r32 << 32) / qj);
        rec[3] = (uint32_t)((1ull << 32) / qj);
        rec[4] = limbs_mod(h.m, h.m_limbs, qj);
        rec[5] = limbs_mod(h.h, h.m_limbs, qj);
        for (int i = 0; i < L; i++) v.wt[j * LMAX + i] = limbs_mod(h.mi + (size_t)i * h.m_limbs, h.m_limbs, qj);
    }
    v.L = L;
    v.LQ = LQ;
    v.m_limbs = h.m_limbs;
    // one block per 128 entries (measured faster than a persistent grid of
    // resident blocks walking the chunks: 0.164 against 0.183 ms for 1M entries)
    (void)num_sms;
    const int64_t chunks = (count + 127) / 128;
    if (chunks > 0x7FFFFFFF) return cudaErrorInvalidValue;
    convert_kernel<LMAX><<<(unsigned)chunks, 128, 0, s>>>(v, R, out, count);
    return cudaGetLastError();
}

// The tensor-core kernels take primes below 2^24 (the limb form's bases), whose
// three digits keep the fp32 sums exact; wider primes, and targets below 2^22
// (kMinPrime), keep the multiply-adds.
bool narrow_basis(const CrtHost& h) { return h.L > 0 && h.L <= 48 && h.p[0] < (1u << 24); }

// The CRT of up to twelve primes is few multiply-adds an entry, and no tables to
// copy: 1M entries as limb sums / digit products (of 8 or 16 primes, zeros or not)
// take 13.7 / 29.4 us with one prime, 18.2 / 28.9 with five, 22.2 / 28.0 with eight,
// 29.6 / 37.8 with nine, 34.8 / 40.2 with twelve (16 as limb sums 72, as digit products
// 43); 1024 entries about the same.
bool mma_crt(const CrtHost& h) { return narrow_basis(h) && h.L > 12; }

}  // namespace

size_t crt_image_bytes(const CrtHost& h, size_t* pc) {
    if (!narrow_basis(h)) return 0;
#define SMF_IMAGE(N) (*pc = CrtMma<N>::kPc, CrtMma<N>::kImage)
    return h.L <= 16 ? SMF_IMAGE(16) : h.L <= 24 ? SMF_IMAGE(24) : h.L <= 32 ? SMF_IMAGE(32) : SMF_IMAGE(48);
#undef SMF_IMAGE
}

void crt_image_make(const CrtHost& h, uint8_t* image) {
    if (h.L <= 16) crt_image<16>(h, image);
    else if (h.L <= 24) crt_image<24>(h, image);
    else if (h.L <= 32) crt_image<32>(h, image);
    else crt_image<48>(h, image);
}

cudaError_t launch_crt_image(const CrtHost& h, uint8_t* image, cudaStream_t s) {
    if (!mma_crt(h)) return cudaSuccess;
    __half* wf = (__half*)image;
    if (h.L <= 16) crt_image_kernel<16><<<CrtMma<16>::NT, kMmaThreads, 0, s>>>(h.d_mi, h.L, h.m_limbs, wf);
    else if (h.L <= 24) crt_image_kernel<24><<<CrtMma<24>::NT, kMmaThreads, 0, s>>>(h.d_mi, h.L, h.m_limbs, wf);
    else if (h.L <= 32) crt_image_kernel<32><<<CrtMma<32>::NT, kMmaThreads, 0, s>>>(h.d_mi, h.L, h.m_limbs, wf);
    else crt_image_kernel<48><<<CrtMma<48>::NT, kMmaThreads, 0, s>>>(h.d_mi, h.L, h.m_limbs, wf);
    return cudaGetLastError();
}

cudaError_t launch_crt(const CrtHost& h, const int32_t* R, int64_t rows, int64_t cols, uint64_t* X, int64_t ld,
                       int W, int num_sms, cudaStream_t s) {
    if (rows == 0 || cols == 0) return cudaSuccess;
    if (mma_crt(h)) {
        if (h.L <= 16) return launch_crt_mma<16>(h, R, rows, cols, X, ld, W, num_sms, s);
        if (h.L <= 24) return launch_crt_mma<24>(h, R, rows, cols, X, ld, W, num_sms, s);
        if (h.L <= 32) return launch_crt_mma<32>(h, R, rows, cols, X, ld, W, num_sms, s);
        return launch_crt_mma<48>(h, R, rows, cols, X, ld, W, num_sms, s);
    }
    if (h.L <= 8)  // primes below 2^24: fewer limbs of M
        return narrow_basis(h) ? launch_crt_t<8, true, 24>(h, R, rows, cols, X, ld, W, s)
                               : launch_crt_t<8, true, 26>(h, R, rows, cols, X, ld, W, s);
    if (h.L <= 12 && narrow_basis(h)) return launch_crt_t<12, true, 24>(h, R, rows, cols, X, ld, W, s);
    if (h.L <= 16) return launch_crt_t<16, true, 26>(h, R, rows, cols, X, ld, W, s);
    if (h.L <= 24) return launch_crt_t<24, true, 26>(h, R, rows, cols, X, ld, W, s);
    if (h.L <= 32) return launch_crt_t<32, true, 26>(h, R, rows, cols, X, ld, W, s);
    if (h.L <= 48) return launch_crt_t<48, true, 26>(h, R, rows, cols, X, ld, W, s);
    if (h.L <= 64) return launch_crt_t<64, false, 26>(h, R, rows, cols, X, ld, W, s);
    return cudaErrorNotSupported;
}

int64_t crt_units(int64_t rows, int64_t cols) { return (rows * cols + 127) / 128; }

cudaError_t launch_crt_grouped(const CrtHost& h, const CrtItem* items, int n, int64_t units, int num_sms,
                               cudaStream_t s) {
    if (n == 0 || units == 0) return cudaSuccess;
    if (units > 0x7FFFFFFF) return cudaErrorInvalidValue;
    if (mma_crt(h)) {
        if (h.L <= 16) return launch_crt_mma_grouped<16>(h, items, n, units, num_sms, s);
        if (h.L <= 24) return launch_crt_mma_grouped<24>(h, items, n, units, num_sms, s);
        if (h.L <= 32) return launch_crt_mma_grouped<32>(h, items, n, units, num_sms, s);
        return launch_crt_mma_grouped<48>(h, items, n, units, num_sms, s);
    }
    if (h.L <= 8)
        return narrow_basis(h) ? launch_crt_grouped_t<8, true, 24>(h, items, n, units, s)
                               : launch_crt_grouped_t<8, true, 26>(h, items, n, units, s);
    if (h.L <= 12 && narrow_basis(h)) return launch_crt_grouped_t<12, true, 24>(h, items, n, units, s);
    if (h.L <= 16) return launch_crt_grouped_t<16, true, 26>(h, items, n, units, s);
    if (h.L <= 24) return launch_crt_grouped_t<24, true, 26>(h, items, n, units, s);
    if (h.L <= 32) return launch_crt_grouped_t<32, true, 26>(h, items, n, units, s);
    if (h.L <= 48) return launch_crt_grouped_t<48, true, 26>(h, items, n, units, s);
    if (h.L <= 64) return launch_crt_grouped_t<64, false, 26>(h, items, n, units, s);
    return cudaErrorNotSupported;
}

cudaError_t launch_convert(const CrtHost& from, const uint32_t* q, int LQ, const int32_t* R, int32_t* out,
                           int64_t count, int num_sms, cudaStream_t s) {
    if (count == 0 || LQ == 0) return cudaSuccess;
    const int n = from.L > LQ ? from.L : LQ;
    // Between few primes the multiply-adds (about L + 2 LQ of them count) are fewer than
    // the digit products of eight primes: 1M entries 1 -> 1 prime 12.0 / 16.7 us, 2 -> 2
    // 15.0 / 16.6, 4 -> 1 14.9 / 16.8; 6 -> 1 17.3 / 17.5, 1 -> 4 17.9 / 16.7, 3 -> 3 18.7 / 17.2
    bool narrow = narrow_basis(from) && from.L + 2 * LQ > 7;
    for (int j = 0; j < LQ; j++) narrow &= q[j] < (1u << 24) && q[j] >= kMinPrime;
    if (narrow) {
        if (n <= 8) return launch_convert_mma<8>(from, q, LQ, R, out, count, num_sms, s);
        if (n <= 16) return launch_convert_mma<16>(from, q, LQ, R, out, count, num_sms, s);
        if (n <= 24) return launch_convert_mma<24>(from, q, LQ, R, out, count, num_sms, s);
        if (n <= 32) return launch_convert_mma<32>(from, q, LQ, R, out, count, num_sms, s);
        if (n <= 48) return launch_convert_mma<48>(from, q, LQ, R, out, count, num_sms, s);
        return cudaErrorNotSupported;
    }
    if (n <= 8) return launch_convert_t<8>(from, q, LQ, R, out, count, num_sms, s);
    if (n <= 16) return launch_convert_t<16>(from, q, LQ, R, out, count, num_sms, s);
    if (n <= 24) return launch_convert_t<24>(from, q, LQ, R, out, count, num_sms, s);
    if (n <= 32) return launch_convert_t<32>(from, q, LQ, R, out, count, num_sms, s);
    if (n <= 48) return launch_convert_t<48>(from, q, LQ, R, out, count, num_sms, s);
    return cudaErrorNotSupported;
}

}  // namespace smf

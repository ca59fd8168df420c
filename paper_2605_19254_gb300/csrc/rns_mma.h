// Constant-matrix products of residues on the tensor cores, in registers: the
// sums sum_i xi_i M_i of the Lagrange form (CRT and base conversion, crt.cu).
//
// Per entry that is a product of a row of L 24-bit values with a constant table
// of L x L words (conversion) or L x 3L bytes (CRT): 23 x 23 wide multiply-adds
// and 23 x 19, on a pipe that takes 28 a clock and SM.  As 8-bit digits it is
// one m16n8k16 product of 16 entries at a time with fp32 sums, exact: K = 3L
// digits of at most 2^7 in absolute value on both sides sum below 2^22.
// mma.sync and not tcgen05: the digits are made in the registers in which the
// instruction takes them and the sums come back in registers, so there is no
// shared-memory tile to fill, no TMEM to read back and nothing to wait for (a
// tcgen05 version of the CRT was no faster than the multiply-adds); the tensor
// pipe is far from full either way, the integer pipes are what bounds both.
//
// A warp takes 32 consecutive entries as two m16 tiles.  Lane 4g + t holds
// entries 4g .. 4g+3 (so that it loads 16 bytes per prime, and stores 16 per
// target) and primes i = 4a + t: K is a sum, its order is free, so every lane's
// digits are its own fragment and nothing is shuffled.
#pragma once

#include "crt_dev.h"

#ifdef __CUDACC__
#include <cuda_fp16.h>

namespace smf {
namespace {

constexpr int kMmaThreads = 128;
constexpr float kMagic = 12582912.0f;           // 1.5 2^23: x + kMagic holds the integer x, |x| < 2^22,
constexpr uint32_t kMagicBits = 0x4B400000u;    // in its low bits

// LMAX primes: primes per lane, pairs of digits per lane, K steps of two pairs
template <int LMAX>
struct XiShape {
    static constexpr int NQ = LMAX / 4, NP = 3 * NQ / 2, KS = (NP + 1) / 2;
    static constexpr int ML = LMAX * 24 / 32 + 1;  // limbs of M
};

// The Lagrange form's constants of a basis on the device, for the entries whose
// alpha is settled exactly; pc[i] = {p_i, H mod p_i, c_i, its Shoup companion}.
struct XiExact {
    const uint32_t* mi;  // [L][m_limbs] limbs of M_i
    const uint32_t* m;   // [m_limbs] limbs of M
    const uint64_t* rcp; // [L] floor(2^64 / p_i)
    int L, m_limbs;
};

// The prime and digit of the fragment's element kap (0 .. 3) of lane 4g + t in K
// step ks: pair 2 ks + kap / 2 is (digit 0, digit 1) of prime a, or digit 2 of
// primes 2b and 2b + 1.  False where the fragment is padding.
template <int LMAX>
__host__ __device__ inline bool xi_slot(int ks, int kap, int t, int* i, int* u) {
    constexpr int NQ = XiShape<LMAX>::NQ;
    const int pr = 2 * ks + (kap >> 1), e = kap & 1;
    const int a = pr < NQ ? pr : 2 * (pr - NQ) + e;
    *i = 4 * a + t;
    *u = pr < NQ ? e : 2;
    return a < NQ;
}

// d = kMagic + a b: the sums start at kMagic, so that they are integers in their
// low bits as they stand (integers in [2^23, 2^24) all along, exact)
__device__ __forceinline__ void mma_f16_first(float (&d)[4], const uint32_t (&a)[4], const uint2& b) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%10, %10, %10, %10};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y), "f"(kMagic));
}
__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], const uint2& b) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// The sums of N n8 tiles over KS steps for both m16 tiles; wf: the tiles' fragments of this lane
template <int N, int KS>
__device__ __forceinline__ void mma_tiles(float (&acc)[2][N][4], const uint32_t (&a)[2][KS][4], const uint2* wf) {
#pragma unroll
    for (int ks = 0; ks < KS; ks++) {
#pragma unroll
        for (int h = 0; h < N; h++) {
            const uint2 b = wf[(h * KS + ks) * 32];
            if (ks == 0) {
                mma_f16_first(acc[0][h], a[0][ks], b);
                mma_f16_first(acc[1][h], a[1][ks], b);
            } else {
                mma_f16(acc[0][h], a[0][ks], b);
                mma_f16(acc[1][h], a[1][ks], b);
            }
        }
    }
}

// v mod q, or that plus q, for v = S_0 + 2^8 S_1 + 2^16 S_2 + constants, from the sums as
// they stand (kMagic too large each): the quotient in fp32, f_c (quot_const) holding
// the constants' part of it and the biases', less 1/2 + 2^-5, and the remainder in
// wrapping 32 bits, i_c (rem_const) holding the constants, the sums' biases and the
// quotient's.  For q >= 2^22 the fp32 error is below 2^-5 (2^15 / q of the sum, whose
// biases are 2^39.6, half a unit of f_c, at most 2^-7, and little of a quotient below
// 2^14), so the result lies in [0, 1.07 q): min(y, y - q) ends it.
constexpr uint32_t kMinPrime = 1u << 22;
__host__ __device__ inline float quot_const(double c, float iq, uint32_t q) {
    return (float)(c / q - 0.5 - 0x1p-5 - 12582912.0 * 65793.0 * (double)iq);
}
__host__ __device__ inline uint32_t rem_const(uint32_t c, uint32_t q) { return c - kMagicBits * 65793u + q * kMagicBits; }
__device__ __forceinline__ float sums_quot(float s0, float s1, float s2, float iq, float f_c) {
    return fmaf(fmaf(s2, 65536.f, fmaf(s1, 256.f, s0)), iq, f_c);
}
__device__ __forceinline__ uint32_t sums_rem(float s0, float s1, float s2, uint32_t q, uint32_t i_c, float f) {
    const uint32_t y = __float_as_uint(s0) + (__float_as_uint(s1) << 8) + (__float_as_uint(s2) << 16) + i_c;
    return y - __float_as_uint(f + kMagic) * q;
}

// two bytes, each in the low bits of 0x6400 (the fp16 value 1024 + byte), as byte - 128
__device__ __forceinline__ uint32_t centre2(uint32_t x) {
    const __half2 c = __half2half2(__ushort_as_half(0x6480));  // 1152
    const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&x), c);
    return *reinterpret_cast<const uint32_t*>(&r);
}

// n bytes (a multiple of 16) from device to shared memory, by the block: eight
// loads a thread in flight (a small call is little else than this copy; one load at
// a time made the CRT of 256 entries of 32 primes 10.2 us after other work, 7.0 so)
__device__ __forceinline__ void stage(void* to, const void* from, size_t n) {
    const int m = (int)(n / 16);
    for (int x0 = threadIdx.x; x0 < m; x0 += 8 * kMmaThreads) {
        uint4 v[8];
#pragma unroll
        for (int k = 0; k < 8; k++)
            if (x0 + k * kMmaThreads < m) v[k] = __ldg((const uint4*)from + x0 + k * kMmaThreads);
#pragma unroll
        for (int k = 0; k < 8; k++)
            if (x0 + k * kMmaThreads < m) ((uint4*)to)[x0 + k * kMmaThreads] = v[k];
    }
}

// alpha where the estimate's fraction is too near an integer: within one of its
// floor, and the one that puts sum_i xi_i M_i - alpha M into [0, M), limb by limb.
template <int LMAX>
__device__ __noinline__ uint32_t settle_alpha(const XiExact& v, const uint4* pc, const int32_t* __restrict__ R,
                                              int64_t count, int64_t e, uint32_t fl) {
    constexpr int ML = XiShape<LMAX>::ML;
    const int L = v.L, ml = v.m_limbs;
    uint32_t xi[LMAX];
#pragma unroll 1
    for (int i = 0; i < L; i++) {
        const uint4 c = pc[i];
        uint32_t a = (uint32_t)__ldg(R + (size_t)i * count + e) + c.y;
        a = min(a, a - c.x);
        const uint32_t z = shoup_mul(a, c.z, c.w, c.x);
        xi[i] = min(z, z - c.x);
    }
    uint32_t d[ML + 1];  // sum_i xi_i M_i - fl M, two's complement over ml + 1 limbs
    uint64_t carry = 0;
    uint32_t borrow = 0;
#pragma unroll 1
    for (int j = 0; j <= ml; j++) {
        uint64_t col = carry;
        if (j < ml) {
#pragma unroll 1
            for (int i = 0; i < L; i++) col += (uint64_t)xi[i] * v.mi[i * ml + j];  // < 48 * 2^56 + 2^32
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

// The warp's entries e0 .. e0 + 31 (those below count): xi_i = ((r_i + H) c_i) mod
// p_i as centred digits in the fragments of the two m16 tiles (every digit less
// 128: the tables' constants put that back), and alpha of this lane's four entries.
template <int LMAX>
__device__ __forceinline__ void xi_frags(const XiExact& v, const uint4* pc, const float* ip,
                                         const int32_t* __restrict__ R, int64_t count, int64_t e0, bool vec,
                                         uint32_t (&a)[2][XiShape<LMAX>::KS][4], uint32_t (&alpha)[4]) {
    constexpr int NQ = XiShape<LMAX>::NQ, NP = XiShape<LMAX>::NP, KS = XiShape<LMAX>::KS;
    const int lane = threadIdx.x & 31, t = lane & 3, L = v.L;
    const int64_t e = e0 + (lane >> 2) * 4;
    uint32_t r[NQ][4];
#pragma unroll
    for (int k = 0; k < NQ; k++) {
        const int i = 4 * k + t;
        const int32_t* src = R + (size_t)i * count + e;
        r[k][0] = r[k][1] = r[k][2] = r[k][3] = 0;
        if (i < L) {
            if (vec) {  // count is a multiple of four
                if (e < count) {
                    const int4 q = __ldg((const int4*)src);
                    r[k][0] = (uint32_t)q.x;
                    r[k][1] = (uint32_t)q.y;
                    r[k][2] = (uint32_t)q.z;
                    r[k][3] = (uint32_t)q.w;
                }
            } else {
#pragma unroll
                for (int x = 0; x < 4; x++)
                    if (e + x < count) r[k][x] = (uint32_t)__ldg(src + x);
            }
        }
    }
    float f[4] = {0.f, 0.f, 0.f, 0.f};
    if constexpr (NP % 2) {  // the last step's second pair: zeros
#pragma unroll
        for (int x = 0; x < 4; x++) a[x >> 1][KS - 1][(x & 1) + 2] = 0u;
    }
#pragma unroll
    for (int k = 0; k < NQ; k++) {
        const uint4 c = pc[4 * k + t];
        const float iv = ip[4 * k + t];
#pragma unroll
        for (int x = 0; x < 4; x++) {
            uint32_t s = r[k][x] + c.y;
            s = min(s, s - c.x);
            uint32_t z = shoup_mul(s, c.z, c.w, c.x);
            z = min(z, z - c.x);
            f[x] = fmaf((float)z, iv, f[x]);
            r[k][x] = z;
            a[x >> 1][k / 2][(x & 1) + 2 * (k & 1)] = centre2(__byte_perm(z, 0x64u, 0x4140));
        }
        if (k & 1) {
            const int pr = NQ + k / 2;
#pragma unroll
            for (int x = 0; x < 4; x++)
                a[x >> 1][pr / 2][(x & 1) + 2 * (pr & 1)] =
                    centre2(__byte_perm(r[k - 1][x], r[k][x], 0x7632) | 0x64006400u);
        }
    }
    bool unsure = false;
#pragma unroll
    for (int x = 0; x < 4; x++) {
        f[x] += __shfl_xor_sync(0xffffffffu, f[x], 1);
        f[x] += __shfl_xor_sync(0xffffffffu, f[x], 2);  // the same value in the quad's lanes
        const float fl = floorf(f[x]);
        const float frac = f[x] - fl;
        alpha[x] = (uint32_t)fl;
        unsure |= frac < 0x1p-12f || frac > 1.f - 0x1p-12f;
    }
    // One entry in 2000 (of a range taken in full: a warp in 64 has one; results well
    // inside the range have none).  2^64 times the fraction in wrapping integers, too
    // small by less than the sum of the xi_i (below 2^30), tells on which side of the
    // integer the sum lies; what that leaves open (the ends of the range) goes limb
    // by limb.  (All of them so left a tail of warps that had several, half of the
    // conversion's 148 us at 1M entries; the sum in double precision, with a division
    // per prime, 3 us in a call of a few.)
    if (__any_sync(0xffffffffu, unsure)) {
        uint64_t d[4] = {0, 0, 0, 0};
#pragma unroll
        for (int k = 0; k < NQ; k++) {
            const uint64_t rc = 4 * k + t < L ? __ldg(v.rcp + 4 * k + t) : 0;
#pragma unroll
            for (int x = 0; x < 4; x++) d[x] += r[k][x] * rc;
        }
#pragma unroll
        for (int x = 0; x < 4; x++) {
            d[x] += __shfl_xor_sync(0xffffffffu, d[x], 1);
            d[x] += __shfl_xor_sync(0xffffffffu, d[x], 2);
            const float frac = f[x] - floorf(f[x]);
            if (frac >= 0x1p-12f && frac <= 1.f - 0x1p-12f) continue;
            if (d[x] < 0ull - (1ull << 30)) alpha[x] = (uint32_t)rintf(f[x]) - (uint32_t)(d[x] >> 63);
            else if (e + x < count) alpha[x] = settle_alpha<LMAX>(v, pc, R, count, e + x, alpha[x]);
        }
    }
    __syncwarp();
}

}  // namespace
}  // namespace smf
#endif

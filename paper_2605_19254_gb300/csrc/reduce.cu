// rns_reduce: big-integer matrices -> residues modulo each prime of a basis
// (Section 3.1: the product starts by mapping each operand to one residue
// matrix per word-size prime), plus the balanced 8-bit digit split of the
// residues that feeds the tensor-core residue product.
//
// A two's complement entry of W words is x = sum_j v_j 2^(32 j) - s 2^(64 W)
// over its 2W unsigned 32-bit limbs v_j and sign bit s.  Hence
//   x mod p = (sum_j v_j c_j - s c_(2W)) mod p,   c_j = 2^(32 j) mod p,
// where every product v_j c_j < 2^58, so sixteen of them sum below 2^62 in a
// 64-bit register before one Barrett reduction.  The c_j of the primes in a
// launch's group are built once per block in shared memory.
#include <cuda_bf16.h>

#include "rns_mma.h"

namespace smf {
namespace {

constexpr int kThreads = 256;
constexpr int kTableWords = 4096;  // shared-memory table capacity (uint32)

__device__ __forceinline__ uint32_t barrett64(uint64_t x, uint32_t p, uint64_t mu) {
    // mu = floor((2^64-1)/p): the estimate q is at most 2 below floor(x/p)
    uint64_t q = __umul64hi(x, mu);
    uint64_t r = x - q * (uint64_t)p;
    if (r >= p) r -= p;
    if (r >= p) r -= p;
    return (uint32_t)r;
}

// bf16 bit pattern of an integer |d| <= 2^15: the fp32 value is formed exactly by
// the 1.5 * 2^23 offset trick (integer add, then one float subtract), and any
// integer with at most 8 significant bits converts to bf16 by truncation of
// the fp32 bits, exactly.  Callers pass |d| <= 256.
__device__ __forceinline__ uint16_t bf16_bits_small(int32_t d) {
    const float f = __int_as_float(0x4B400000 + d) - 12582912.0f;
    return (uint16_t)(__float_as_uint(f) >> 16);
}

// Balanced digits: lower digits in [-128, 127], top digit = remaining quotient.
// With a = r + 128: d0 = (a & 255) - 128 and the rest is a >> 8 (floor), so for
// two or three digits (|r| < 2^23) the split is in closed form.
__device__ __forceinline__ void store_digits(int64_t r, int t, __nv_bfloat16* dst, int64_t plane) {
    uint16_t* o = reinterpret_cast<uint16_t*>(dst);
    if (t == 3 || t == 2) {
        const int32_t a = (int32_t)r + 128;
        o[0] = bf16_bits_small((a & 255) - 128);
        if (t == 2) {
            o[plane] = bf16_bits_small(a >> 8);
        } else {
            const int32_t b = (a >> 8) + 128;
            o[plane] = bf16_bits_small((b & 255) - 128);
            o[2 * plane] = bf16_bits_small(b >> 8);
        }
        return;
    }
    for (int u = 0; u < t - 1; u++) {
        const int32_t d = (int32_t)(((r + 128) & 255) - 128);
        o[u * plane] = bf16_bits_small(d);
        r = (r - d) >> 8;
    }
    o[(t - 1) * plane] = bf16_bits_small((int32_t)r);  // |top| <= 128
}

// Declared-bound check: does the two's complement value of the 2W limbs v[]
// lie outside [-2^bits, 2^bits]?  Negative values fit when every bit from
// `bits` up is one; non-negative ones when every bit above `bits` is zero and,
// if bit `bits` is set, every bit below it is zero (x = 2^bits).
template <int WC>
__device__ __forceinline__ bool over_bits(const uint32_t (&v)[2 * WC], int W, int bits) {
    if (bits >= 64 * W - 1) return false;
    const int L = bits >> 5, sh = bits & 31;
    const bool neg = (v[2 * W - 1] >> 31) != 0;
    bool over = false, low_zero = true;
#pragma unroll
    for (int j = 0; j < 2 * WC; j++) {
        if (j >= 2 * W) break;
        if (j < L) {
            low_zero &= v[j] == 0;
        } else if (j == L) {
            const uint32_t hi = v[j] >> sh;
            if (neg) over |= hi != (0xFFFFFFFFu >> sh);
            else over |= hi > 1 || (hi == 1 && (!low_zero || (sh && (v[j] << (32 - sh)) != 0)));
        } else {
            over |= v[j] != (neg ? 0xFFFFFFFFu : 0u);
        }
    }
    return over;
}

// The same check for an entry that is its own centred value (the shared-digit
// path reads only the low word): |v| <= 2^bits, and the words above the low
// one (W > 1) are its sign extension.
__device__ __forceinline__ bool over_bits_low(int64_t v, int bits) {
    return bits < 63 && (v > (1ll << bits) || v < -(1ll << bits));
}

__device__ __forceinline__ void flag_bound(int* status) {
    if (status) atomicOr(status, kStatusBound);
}

// Residue of one entry whose 2W 32-bit limbs are v[] (two's complement sign s)
// modulo prime e of the block's group.
template <int WC>
__device__ __forceinline__ uint32_t entry_mod(const uint32_t (&v)[2 * WC], int W, uint32_t s, const uint32_t* ct,
                                              uint32_t p, uint64_t mu) {
    uint64_t acc = 0;
    uint32_t rr = 0;
#pragma unroll
    for (int j4 = 0; j4 < 2 * WC; j4 += 4) {
        if (j4 < 2 * W) {
            const uint4 c4 = *(const uint4*)(ct + j4);  // ct rows are 16-byte aligned
            const uint32_t cj[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int j = j4 + q;
                if (j < 2 * W) {
                    acc += (uint64_t)v[j] * cj[q];
                    if ((j & 15) == 15) {  // 16 products: fold before 2^64
                        rr = barrett64(acc + rr, p, mu);
                        acc = 0;
                    }
                }
            }
        }
    }
    rr = barrett64(acc + rr, p, mu);
    if (s) {  // subtract 2^(64W) mod p
        const uint32_t cw = ct[2 * W];
        rr = rr >= cw ? rr - cw : rr + p - cw;
    }
    return rr;
}

// WC: compile-time word capacity (the entry's words are held in registers);
// W <= WC is the runtime word count.
template <ReduceOut KIND, int WC>
__global__ void __launch_bounds__(kThreads)
reduce_kernel(BasisDev b, ReduceArgs a, int group) {
    extern __shared__ uint32_t ctab[];  // [G][2W+1]
    const int i0 = blockIdx.z * group;
    const int G = min(group, b.L - i0);
    const int W = a.W;
    const int nw = (2 * W + 1 + 3) & ~3;  // row of one prime's constants, padded to 16 bytes
    if (!a.identity) {
        for (int e = threadIdx.x; e < G; e += blockDim.x) {
            const uint32_t p = b.p[i0 + e];
            const uint64_t mu = b.mu[i0 + e];
            const uint32_t r32 = b.pow32[i0 + e];
            uint32_t c = 1 % p;
            for (int j = 0; j < nw; j++) {
                ctab[e * nw + j] = j <= 2 * W ? c : 0u;
                c = barrett64((uint64_t)c * r32, p, mu);
            }
        }
        __syncthreads();
    }
    // Thread mapping: consecutive threads take consecutive output addresses.
    // Transposed digit planes are contiguous along rows, the others along cols.
    constexpr bool trans = KIND == ReduceOut::kDigitsT;
    const int64_t minor_n = trans ? a.rows : a.cols;
    const int64_t major_n = trans ? a.cols : a.rows;
    const int64_t minor = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (minor >= minor_n) return;
    for (int64_t major = blockIdx.y; major < major_n; major += gridDim.y) {
        const int64_t r = trans ? minor : major;
        const int64_t c = trans ? major : minor;
        const uint64_t* x = a.X + (size_t)(r * a.ld + c) * W;
        // the entry's words, loaded once (16-byte loads when aligned)
        uint32_t v[2 * WC];
#pragma unroll
        for (int j = 0; j < WC; j++) {
            if (j < W) {
                uint64_t w;
                if ((W & 1) == 0 && (j & 1) == 0) {
                    const ulonglong2 q = __ldg((const ulonglong2*)(x + j));
                    w = q.x;
                    v[2 * j + 2] = (uint32_t)q.y;
                    v[2 * j + 3] = (uint32_t)(q.y >> 32);
                } else if ((W & 1) == 0) {
                    w = ((uint64_t)v[2 * j + 1] << 32) | v[2 * j];  // already loaded
                } else {
                    w = __ldg(x + j);
                }
                v[2 * j] = (uint32_t)w;
                v[2 * j + 1] = (uint32_t)(w >> 32);
            }
        }
        const uint32_t s = v[2 * W - 1] >> 31;
        if (a.status && blockIdx.z == 0) {
            bool over;
            if (a.identity) {
                const int64_t lo = (int64_t)(((uint64_t)v[1] << 32) | v[0]);
                over = over_bits_low(lo, a.bits);
                for (int j = 2; j < 2 * W; j++) over |= v[j] != (lo < 0 ? 0xFFFFFFFFu : 0u);
            } else {
                over = over_bits<WC>(v, W, a.bits);
            }
            if (over) flag_bound(a.status);
        }
        for (int e = 0; e < (a.identity ? 1 : G); e++) {
            const int i = i0 + e;
            int64_t val;  // centred residue, or the value itself (identity)
            uint32_t canon = 0;
            if (a.identity) {
                val = (int64_t)(((uint64_t)v[1] << 32) | v[0]);
            } else {
                const uint32_t p = b.p[i];
                canon = entry_mod<WC>(v, W, s, ctab + e * nw, p, b.mu[i]);
                val = (int64_t)canon > (int64_t)(p >> 1) ? (int64_t)canon - p : (int64_t)canon;
            }
            if constexpr (KIND == ReduceOut::kCanonical) {
                ((int32_t*)a.out)[((size_t)i * a.rows + r) * a.cols + c] = (int32_t)canon;
            } else if constexpr (KIND == ReduceOut::kCentered) {
                ((int32_t*)a.out)[((size_t)i * a.rows + r) * a.cols + c] = (int32_t)val;
            } else if constexpr (KIND == ReduceOut::kDigits) {  // [L][t][rows][ld_out]
                const int64_t plane = a.rows * a.ld_out;
                __nv_bfloat16* base = (__nv_bfloat16*)a.out + (size_t)i * a.t * plane;
                store_digits(val, a.t, base + r * a.ld_out + c, plane);
            } else {  // [t][L][cols][ld_out]
                const int64_t plane = a.cols * a.ld_out;
                __nv_bfloat16* base = (__nv_bfloat16*)a.out + (size_t)i * plane;
                store_digits(val, a.t, base + c * a.ld_out + r, plane * b.L);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// The reductions modulo at most 64 primes in [2^22, 2^24) of entries of 1, 2, 4 or 8
// words, on the tensor cores (rns_mma.h has the layout).  x mod p_i is a product
// of the entry's 8 W bytes with the constants 2^(8b) mod p_i: bytes less 128 (the
// top one signed as it is) and balanced digits of the constants, fp32 sums below
// 2^20, exact.  Lane 4g + t takes a quarter of the bytes of entries 4g .. 4g+3,
// which follow one another along the output's contiguous dimension, so that its
// results are stored 8 or 16 bytes at a time (the limb sums stored two bytes at a
// time, 69 stores an entry with 23 primes).  512-bit entries and 23 primes take 700
// thread instructions an entry as canonical residues, 1200 as transposed digits
// (2016 as limb sums), at 49 and 61 % of the issue slots: the latency of the 32-entry
// chunks at 24 warps per SM bounds it.
struct RmArgs {
    const uint64_t* X;
    int64_t minor_n, major_n;  // entries along the output's contiguous dimension, and across it
    int64_t smin, smaj;        // their strides in X, in entries
    void* out;                 // element (i, u, major, minor) at i si + u su + major ldo + minor
    int64_t ldo, si, su;
    int t;                     // digits per residue
    int bits;
    int* status;
};

template <int W>
struct RmShape {
    static constexpr int KS = W == 1 ? 1 : W / 2;  // K steps of 16 bytes: a limb per lane and step
};

__host__ __device__ constexpr size_t rm_frag(int L, int KS) { return sizeof(uint2) * ((L + 7) / 8 * 3) * KS * 32; }

// The tables of a basis, made with it (on the device: on the host they took as long
// as a small product) and copied to shared memory by each block: the constants'
// fragments (three n8 tiles for the eight primes 8B .. 8B + 7, as in the
// conversion), and per prime {p, rem_const, 1 / p, quot_const} of the constant, for
// centred and then for canonical results: what the bytes' 128s take off, and
// (p - 1) / 2 for centred results.  A block makes prime i's part of the four (zeros
// beyond L), a thread that of 2^(8b) mod p.
struct ReduceImages {
    uint8_t* to[4];  // for entries of 1, 2, 4, 8 words
};
constexpr int kImageBytes = 64;  // bytes of the longest entry
__global__ void __launch_bounds__(kImageBytes)
reduce_images_kernel(const uint32_t* __restrict__ primes, int L, ReduceImages im) {
    __shared__ uint32_t ws[kImageBytes];
    const int i = blockIdx.x, b = threadIdx.x;
    const uint32_t p = i < L ? primes[i] : 1u;
    uint32_t w = 1 % p;
    for (int k = 0; k < b; k++) w = (w << 8) % p;  // (p below 2^24)
    ws[b] = w;
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 4; c++) {
        const int W = 1 << c, KS = W == 1 ? 1 : W / 2;
        if (b >= 16 * KS) continue;
        __half* wf = (__half*)im.to[c];
        int32_t r = i < L && b < 8 * W ? (int32_t)w : 0;
        if (r > (int32_t)(p >> 1)) r -= (int32_t)p;
        const int limb = b >> 2, t = limb / KS, ks = limb % KS;
        for (int dig = 0; dig < 3; dig++) {
            const int c6 = (i >> 2 & 1) * 3 + dig, nt = (i >> 3) * 3 + c6 / 2;
            const int ln = (2 * (i & 3) + (c6 & 1)) * 4 + t;
            wf[((nt * KS + ks) * 32 + ln) * 4 + (b & 3)] = __int2half_rn(dig < 2 ? ((r + 128) & 255) - 128 : r);
            r = (r + 128) >> 8;
        }
    }
    if (i >= L || b >= 8) return;
    const int c = b >> 1, ints = b & 1, n = (8 << c) - 1;
    uint64_t sum = 0;  // 128 times the 2^(8b) of the bytes below the top one
    for (int k = 0; k < n; k++) sum += 128ull * ws[k];
    const uint32_t k = (uint32_t)((sum + (ints ? 0u : p >> 1)) % p);
    const float ip = 1.0f / (float)p;
    uint4* ti = (uint4*)(im.to[c] + rm_frag(L, c == 0 ? 1 : 1 << (c - 1)));
    ti[ints * L + i] = make_uint4(p, rem_const(k, p), __float_as_uint(ip), __float_as_uint(quot_const(k, ip, p)));
}

template <int W, bool INT>
__device__ __forceinline__ void rm_tables(const uint8_t* __restrict__ image, int L, uint8_t* to) {
    const size_t nf = rm_frag(L, RmShape<W>::KS);
    stage(to, image, nf);
    stage(to + nf, image + nf + (INT ? sizeof(uint4) * L : 0), sizeof(uint4) * L);
    __syncthreads();
}

constexpr int word_class(int W) { return W == 1 ? 0 : W == 2 ? 1 : W == 4 ? 2 : 3; }

// Does one of the warp's 32 entries (four in a quad, their limbs spread over its
// lanes) lie outside [-2^bits, 2^bits] (as over_bits)?  Some lane knows from its own
// limbs, but for a value with bit `bits` set and none above it: whether a lower bit
// is set too.  (Three votes an entry instead took a quarter of the reduction's time.)
template <int W>
__device__ __forceinline__ bool rm_over(const uint32_t (&v)[4][RmShape<W>::KS], int bits) {
    constexpr int KS = RmShape<W>::KS;
    const int lane = threadIdx.x & 31, t = lane & 3, Lb = bits >> 5, sh = bits & 31;
    bool over = false;
    unsigned one = 0, nz = 0;  // a bit for each entry
#pragma unroll
    for (int x = 0; x < 4; x++) {
        const uint32_t sign = (uint32_t)((int32_t)__shfl_sync(0xffffffffu, v[x][KS - 1], lane | 3) >> 31);
#pragma unroll
        for (int k = 0; k < KS; k++) {
            const int j = t * KS + k;
            if (j < Lb) {
                nz |= (unsigned)(v[x][k] != 0) << x;
            } else if (j == Lb) {
                const uint32_t hi = (v[x][k] ^ sign) >> sh;
                over |= hi > (sign ? 0u : 1u);
                one |= (unsigned)(hi == 1 && !sign) << x;
                nz |= (unsigned)(sh && (v[x][k] << (32 - sh)) != 0) << x;
            } else {
                over |= v[x][k] != sign;
            }
        }
    }
    if (__any_sync(0xffffffffu, one)) {
#pragma unroll
        for (int d = 1; d < 4; d *= 2) {
            one |= __shfl_xor_sync(0xffffffffu, one, d);
            nz |= __shfl_xor_sync(0xffffffffu, nz, d);
        }
        over |= (one & nz) != 0;
    }
    return over;
}

// 32 entries from minor m0 of one major, by one warp.
template <int W, bool INT>
__device__ __forceinline__ void rm_chunk(const RmArgs& a, int L, const uint2* wf, const uint4* ti, int64_t m0,
                                         int64_t major) {
    constexpr int KS = RmShape<W>::KS;
    const int lane = threadIdx.x & 31, t = lane & 3;
    const int64_t m = m0 + (lane >> 2) * 4;
    uint32_t v[4][KS];
#pragma unroll
    for (int x = 0; x < 4; x++) {
#pragma unroll
        for (int k = 0; k < KS; k++) v[x][k] = 0;
        if (m + x < a.minor_n && (W > 1 || t < 2)) {
            const uint32_t* src = (const uint32_t*)(a.X + (size_t)((m + x) * a.smin + major * a.smaj) * W) + t * KS;
            if constexpr (KS == 4) {
                const uint4 q = __ldg((const uint4*)src);
                v[x][0] = q.x;
                v[x][1] = q.y;
                v[x][2] = q.z;
                v[x][3] = q.w;
            } else if constexpr (KS == 2) {
                const uint2 q = __ldg((const uint2*)src);
                v[x][0] = q.x;
                v[x][1] = q.y;
            } else {
                v[x][0] = __ldg(src);
            }
        }
    }
    if (!INT && a.status && a.bits < 64 * W - 1) {
        if constexpr (W == 1) {  // an entry per lane, from L1: 60 instructions fewer a warp than from the limbs at hand
            const int64_t e = m0 + lane;
            if (e < a.minor_n && over_bits_low((int64_t)__ldg(a.X + (size_t)(e * a.smin + major * a.smaj)), a.bits))
                flag_bound(a.status);
        } else if (rm_over<W>(v, a.bits)) {
            flag_bound(a.status);
        }
    }
    uint32_t f[2][KS][4];
    const uint32_t top = t == (W == 1 ? 1 : 3) ? 0x80000000u : 0u;  // the sign: the top byte as it is
#pragma unroll
    for (int x = 0; x < 4; x++) {
#pragma unroll
        for (int k = 0; k < KS; k++) {
            const uint32_t z = k == KS - 1 ? v[x][k] ^ top : v[x][k];
            f[x >> 1][k][x & 1] = centre2(__byte_perm(z, 0x64u, 0x4140));
            f[x >> 1][k][(x & 1) + 2] = centre2(__byte_perm(z, 0x64u, 0x4342));
        }
    }
    const int64_t at0 = major * a.ldo + m;
    const bool full = m + 3 < a.minor_n &&
                      (((uint64_t)a.si | (uint64_t)a.su | (uint64_t)a.ldo) & 3) == 0 && ((uintptr_t)a.out & (INT ? 15 : 7)) == 0;
    // a centred residue plus this has its balanced digits plus 128 as bytes
    const uint32_t bias = a.t == 3 ? 0x808080u : a.t == 2 ? 0x8080u : 0x80u;
#pragma unroll 1
    for (int nb = 0; 8 * nb < L; nb++) {
        float acc[2][3][4];
        mma_tiles<3, KS>(acc, f, wf + 3 * nb * KS * 32 + lane);
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const int i = 8 * nb + 4 * q + t;
            if (i >= L || m >= a.minor_n) continue;
            const uint4 c = ti[i];
            uint32_t r[4];
#pragma unroll
            for (int x = 0; x < 4; x++) {
                float s[3];
#pragma unroll
                for (int k = 0; k < 3; k++) s[k] = acc[x >> 1][(3 * q + k) >> 1][2 * (x & 1) + ((3 * q + k) & 1)];
                const uint32_t y =
                    sums_rem(s[0], s[1], s[2], c.x, c.y, sums_quot(s[0], s[1], s[2], __uint_as_float(c.z), __uint_as_float(c.w)));
                r[x] = min(y, y - c.x);  // [0, p)
            }
            const int64_t at = at0 + i * a.si;
            if constexpr (INT) {
                int32_t* o = (int32_t*)a.out + at;
                if (full) {
                    *(int4*)o = make_int4((int)r[0], (int)r[1], (int)r[2], (int)r[3]);
                } else {
#pragma unroll
                    for (int x = 0; x < 4; x++)
                        if (m + x < a.minor_n) o[x] = (int32_t)r[x];
                }
            } else {
                const uint32_t off = bias - (c.x >> 1);
                uint16_t* o = (uint16_t*)a.out + at;
#pragma unroll
                for (int u = 0; u < 3; u++) {
                    if (u >= a.t) break;
                    uint32_t d[4];
#pragma unroll
                    for (int x = 0; x < 4; x++) {
                        const uint32_t z = r[x] + off;
                        // byte u, or all that is left (up to 256) at the top, in the low bits of 0x4B400000
                        const uint32_t e = u == 2              ? __byte_perm(z, kMagicBits, 0x7632)
                                           : u == a.t - 1      ? (z >> 8 * u) + kMagicBits
                                                               : __byte_perm(z, kMagicBits, 0x7640 + u);
                        d[x] = __float_as_uint(__uint_as_float(e) - (kMagic + 128.f));
                    }
                    const uint32_t lo = __byte_perm(d[0], d[1], 0x7632), hi = __byte_perm(d[2], d[3], 0x7632);
                    if (full) {
                        *(uint2*)o = make_uint2(lo, hi);
                    } else {
                        if (m + 0 < a.minor_n) o[0] = (uint16_t)lo;
                        if (m + 1 < a.minor_n) o[1] = (uint16_t)(lo >> 16);
                        if (m + 2 < a.minor_n) o[2] = (uint16_t)hi;
                        if (m + 3 < a.minor_n) o[3] = (uint16_t)(hi >> 16);
                    }
                    o += a.su;
                }
            }
        }
    }
}

// Unit: 128 entries along the minor dimension of one major, 32 per warp, where X is
// contiguous along it (smin 1): rows of the output whose ends are not multiples of 32
// bytes then have the halves of a sector written together (2003 x 2003 entries of one
// word modulo 25 primes, as digits of rows of 2008: 45 us less than with a row per
// warp).  Else 32 entries of four majors, adjacent in X's sectors.
template <int W, bool INT>
__global__ void __launch_bounds__(kMmaThreads, 6)
reduce_mma_kernel(BasisDev b, const __grid_constant__ RmArgs a) {
    extern __shared__ __align__(16) uint8_t dyn[];
    uint2* wf = (uint2*)dyn;
    uint4* ti = (uint4*)(dyn + rm_frag(b.L, RmShape<W>::KS));
    rm_tables<W, INT>(b.red[word_class(W)], b.L, dyn);
    const bool along = a.smin == 1;
    const int64_t nm = along ? (a.minor_n + 127) / 128 : (a.minor_n + 31) / 32;
    const int64_t units = along ? nm * a.major_n : nm * ((a.major_n + 3) / 4);
    for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
        const int64_t q = u / nm, r = u - q * nm, wid = threadIdx.x >> 5;
        const int64_t major = along ? q : q * 4 + wid, m0 = along ? r * 128 + wid * 32 : r * 32;
        if (major < a.major_n && m0 < a.minor_n) rm_chunk<W, INT>(a, b.L, wf, ti, m0, major);
    }
}

// The transposed reduce of several B operands (all of W words) in one persistent
// launch.  Unit: 32 rows by kRmCols columns of one item, adjacent columns in
// adjacent warps (an item's rows are contiguous in memory).
constexpr int kRmCols = 16;
template <int W>
__global__ void __launch_bounds__(kMmaThreads)
reduce_mma_grouped_kernel(BasisDev b, const ReduceItem* __restrict__ items, int n, int64_t units, int* status) {
    extern __shared__ __align__(16) uint8_t dyn[];
    uint2* wf = (uint2*)dyn;
    uint4* ti = (uint4*)(dyn + rm_frag(b.L, RmShape<W>::KS));
    rm_tables<W, false>(b.red[word_class(W)], b.L, dyn);
    for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
        const ReduceItem* it = find_item(items, n, u);
        const int64_t plane = it->cols * it->ld_out;
        const RmArgs a{it->X, it->rows, it->cols, it->ld, 1, it->out, it->ld_out, plane, plane * b.L, it->t, it->bits, status};
        const int64_t nm = (it->rows + 31) / 32, lu = u - it->base;
        for (int k = threadIdx.x >> 5; k < kRmCols; k += kMmaThreads / 32) {
            const int64_t c = lu / nm * kRmCols + k;
            if (c < it->cols) rm_chunk<W, false>(a, b.L, wf, ti, lu % nm * 32, c);
        }
    }
}

// Blocks of `kernel` resident at once with the tables of 24 primes (asked once: a property of its code).
template <auto kernel, int W>
int64_t rm_resident() {
    static const int per = [] {
        int nb = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, kMmaThreads, rm_frag(24, RmShape<W>::KS) + 24 * sizeof(uint4));
        return nb > 0 ? nb : 1;
    }();
    return per;
}

// The transposed reduction of entries of one or two words modulo few primes
// (limb_sums_t): planes [t][L][cols][ld_out] as above, but limb sums, two or four
// multiply-adds a prime, where the digit products always work on eight primes.  A
// block takes 256 rows by four columns (32 bytes of a row of one-word entries); per
// prime the table has {p, 2^32 mod p, its Shoup companion, floor(2^32 / p)}, then
// c_j = 2^(32 j) mod p for j <= 2W.  Bound by instruction issue and two-byte stores.
constexpr int kTCols = 4, kTSumRow = 12;
template <int W>
__global__ void __launch_bounds__(kThreads)
reduce_sums_t_kernel(BasisDev b, const __grid_constant__ ReduceArgs a) {
    static_assert(4 + 2 * W + 1 <= kTSumRow, "a row of the table");
    extern __shared__ __align__(16) uint32_t ctab[];  // [L][kTSumRow]
    for (int e = threadIdx.x; e < b.L; e += kThreads) {
        const uint32_t p = b.p[e], r32 = b.pow32[e];
        uint32_t* row = ctab + e * kTSumRow;
        row[0] = p;
        row[1] = r32;
        row[2] = (uint32_t)(((uint64_t)r32 << 32) / p);
        row[3] = (uint32_t)((1ull << 32) / p);
        uint32_t c = 1 % p;
        for (int j = 0; j <= 2 * W; j++) {
            row[4 + j] = c;
            c = barrett64((uint64_t)c * r32, p, b.mu[e]);
        }
    }
    __syncthreads();
    const int64_t r = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (r >= a.rows) return;
    const int64_t plane = a.cols * a.ld_out, dstride = plane * b.L, cb = (int64_t)blockIdx.y * kTCols;
    for (int cc = 0; cc < kTCols; cc++) {
        const int64_t c = cb + cc;
        if (c >= a.cols) break;
        const uint64_t* x = a.X + (size_t)(r * a.ld + c) * W;
        uint32_t v[2 * W];
        if constexpr (W == 2) {
            const ulonglong2 q = __ldg((const ulonglong2*)x);
            v[0] = (uint32_t)q.x;
            v[1] = (uint32_t)(q.x >> 32);
            v[2] = (uint32_t)q.y;
            v[3] = (uint32_t)(q.y >> 32);
        } else {
            const uint64_t q = __ldg(x);
            v[0] = (uint32_t)q;
            v[1] = (uint32_t)(q >> 32);
        }
        const bool neg = v[2 * W - 1] >> 31;
        if (a.status && over_bits<W>(v, W, a.bits)) flag_bound(a.status);
        uint16_t* o = (uint16_t*)a.out + c * a.ld_out + r;
        for (int e = 0; e < b.L; e++, o += plane) {
            const uint32_t* ct = ctab + e * kTSumRow;
            const uint4 hd = *(const uint4*)ct, c4 = *(const uint4*)(ct + 4);
            const uint32_t p = hd.x, cj[4] = {c4.x, c4.y, c4.z, c4.w};
            uint32_t lo = 0, hi = 0;  // sum_j v_j c_j < 4 * 2^56
#pragma unroll
            for (int j = 0; j < 2 * W; j++) mac64(lo, hi, v[j], cj[j]);
            // hi (2^32 mod p) by Shoup, lo by its reciprocal quotient
            const uint32_t t1 = hi * hd.y - __umulhi(hi, hd.z) * p;  // [0, 2p)
            const uint32_t t2 = lo - __umulhi(lo, hd.w) * p;         // [0, 2p)
            uint32_t rr = t1 + t2;                                   // [0, 4p)
            if (rr >= 2 * p) rr -= 2 * p;
            if (rr >= p) rr -= p;
            if (neg) {  // subtract 2^(64W) mod p
                const uint32_t cw = W == 1 ? c4.z : ct[8];
                rr = rr >= cw ? rr - cw : rr + p - cw;
            }
            const int32_t val = rr > (p >> 1) ? (int32_t)rr - (int32_t)p : (int32_t)rr;
            if (a.t == 3) {
                const int32_t d = val + 128, f = (d >> 8) + 128;
                o[0] = bf16_bits_small((d & 255) - 128);
                o[dstride] = bf16_bits_small((f & 255) - 128);
                o[2 * dstride] = bf16_bits_small(f >> 8);
            } else {
                store_digits(val, a.t, (__nv_bfloat16*)o, dstride);
            }
        }
    }
}

// Digit split of a matrix whose int64 entries (low word of W) are their own
// centred residues (|x| <= (p_L - 1)/2): planes [t][rows][ld_out].  Eight
// consecutive entries per thread: 64 bytes in, 16 bytes out per plane.
__global__ void __launch_bounds__(kThreads)
split_digits8_kernel(const uint64_t* __restrict__ X, int64_t rows, int64_t cols, int64_t ld, int W,
                     __nv_bfloat16* __restrict__ out, int64_t ld_out, int t, int bits, int* status) {
    const int64_t groups = cols / 8;
    const int64_t g = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (g >= groups) return;
    const int64_t plane = rows * ld_out;
    for (int64_t r = blockIdx.y; r < rows; r += gridDim.y) {
        const uint64_t* x = X + (size_t)(r * ld + g * 8) * W;
        int64_t v[8];
        if (W == 1) {
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const ulonglong2 w = __ldg((const ulonglong2*)x + q);
                v[2 * q] = (int64_t)w.x;
                v[2 * q + 1] = (int64_t)w.y;
            }
        } else {
            bool ext = false;  // the upper words must be the low word's sign extension
#pragma unroll
            for (int q = 0; q < 8; q++) {
                v[q] = (int64_t)__ldg(x + (size_t)q * W);
                for (int j = 1; j < W; j++) ext |= __ldg(x + (size_t)q * W + j) != (v[q] < 0 ? ~0ull : 0ull);
            }
            if (ext) flag_bound(status);
        }
        {
            bool over = false;
#pragma unroll
            for (int q = 0; q < 8; q++) over |= over_bits_low(v[q], bits);
            if (over) flag_bound(status);
        }
        __nv_bfloat16* o = out + r * ld_out + g * 8;
        for (int u = 0; u < t; u++) {
            float f[8];
#pragma unroll
            for (int q = 0; q < 8; q++) {
                int32_t dq;
                if (u < t - 1) {
                    dq = (int32_t)(((v[q] + 128) & 255) - 128);
                    v[q] = (v[q] - dq) >> 8;
                } else {
                    dq = (int32_t)v[q];  // |top| <= 128
                }
                f[q] = __int_as_float(0x4B400000 + dq) - 12582912.0f;  // exact, |dq| <= 256
            }
            uint32_t w[4];
#pragma unroll
            for (int q = 0; q < 4; q++)
                w[q] = (__float_as_uint(f[2 * q]) >> 16) | (__float_as_uint(f[2 * q + 1]) & 0xFFFF0000u);
            *(uint4*)(o + u * plane) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// Digit split of several centred-value operands (shared-digit A: every entry
// is its own centred residue for all primes) in one persistent launch.  A thread
// takes eight consecutive entries of a row (the last of a row fewer), so that a
// digit plane gets 16 bytes at a time, a unit is 256 such groups of one item in
// row-major order.  One entry per thread took 86 instructions an entry and two-byte
// stores: 447 us for the 78.6 M entries of 512 products, issue-bound; the batch went
// from 7.03 to 6.81 ms.
constexpr int kSplitPer = 8;
__global__ void __launch_bounds__(kThreads, 5)
split_digits_grouped_kernel(const ReduceItem* __restrict__ items, int n, int64_t units, int* status) {
    for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
        const ReduceItem* it = find_item(items, n, u);
        const int64_t cols = it->cols, per_row = (cols + kSplitPer - 1) / kSplitPer, count = it->rows * per_row;
        const int64_t g = (u - it->base) * kThreads + threadIdx.x;
        if (g >= count) continue;
        int64_t r;
        if (count <= 0xFFFFFFFFll)  // quotient by the item's precomputed multiplier
            r = (uint32_t)(((uint64_t)__umulhi((uint32_t)g, it->div_m) + (uint32_t)g) >> it->div_s);
        else
            r = g / per_row;
        const int64_t c = (g - r * per_row) * kSplitPer;
        const int left = (int)min((int64_t)kSplitPer, cols - c), W = it->W, t = it->t;
        const uint64_t* x = it->X + (size_t)(r * it->ld + c) * W;
        int64_t v[kSplitPer];
        bool over = false;
        if (W == 1 && left == kSplitPer && ((uintptr_t)x & 15) == 0) {
#pragma unroll
            for (int q = 0; q < kSplitPer; q += 2) {
                const ulonglong2 w = __ldg((const ulonglong2*)(x + q));
                v[q] = (int64_t)w.x;
                v[q + 1] = (int64_t)w.y;
            }
        } else {
#pragma unroll
            for (int q = 0; q < kSplitPer; q++) {
                v[q] = 0;
                if (q < left) {
                    v[q] = (int64_t)__ldg(x + (size_t)q * W);
                    for (int j = 1; j < W; j++) over |= __ldg(x + (size_t)q * W + j) != (v[q] < 0 ? ~0ull : 0ull);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < kSplitPer; q++) over |= over_bits_low(v[q], it->bits);
        if (over) flag_bound(status);
        // at most three digits: an entry plus this has its balanced digits plus 128 as
        // bytes (the top one up to 256); each goes to the low bits of 0x4B400000
        const uint32_t bias = t == 3 ? 0x808080u : t == 2 ? 0x8080u : 0x80u;
        const int64_t plane = it->rows * it->ld_out;
        uint16_t* o = (uint16_t*)it->out + r * it->ld_out + c;
        const bool vec = left == kSplitPer && ((uintptr_t)o & 15) == 0 && (plane & 7) == 0;
        for (int k = 0; k < t; k++, o += plane) {
            uint32_t w[kSplitPer / 2];
#pragma unroll
            for (int q = 0; q < kSplitPer; q += 2) {
                uint32_t d[2];
#pragma unroll
                for (int z = 0; z < 2; z++) {
                    const uint32_t e = ((uint32_t)v[q + z] + bias) >> (8 * k);
                    d[z] = __float_as_uint(__uint_as_float((k == t - 1 ? e : e & 255u) + kMagicBits) - (kMagic + 128.f));
                }
                w[q / 2] = __byte_perm(d[0], d[1], 0x7632);
            }
            if (vec) {
                *(uint4*)o = make_uint4(w[0], w[1], w[2], w[3]);
            } else {
#pragma unroll
                for (int q = 0; q < kSplitPer; q++)
                    if (q < left) o[q] = (uint16_t)(w[q / 2] >> (16 * (q & 1)));
            }
        }
    }
}

// int32 residues (any representative in (-p, p)) -> digit planes.
// Non-transposed: elementwise.  Transposed: 32 x 32 tiles through shared memory.
__global__ void __launch_bounds__(kThreads)
digits_kernel(BasisDev b, const int32_t* R, int64_t prime_stride, int64_t rows, int64_t cols,
              __nv_bfloat16* out, int64_t ld_out, int t, int shared_a) {
    const int i = blockIdx.z;
    const int32_t* Ri = R + (size_t)i * prime_stride;
    const int64_t plane = rows * ld_out;
    __nv_bfloat16* base = out + (size_t)i * t * plane;
    const uint32_t p = b.p[shared_a ? b.L - 1 : i];
    const int32_t h = (int32_t)(p >> 1);
    const int64_t c = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (c >= cols) return;
    for (int64_t r = blockIdx.y; r < rows; r += gridDim.y) {
        int32_t v = Ri[r * cols + c];
        if (!shared_a) {
            if (v > h) v -= (int32_t)p;
            if (v < -h) v += (int32_t)p;
        }
        store_digits(v, t, base + r * ld_out + c, plane);
    }
}

__global__ void __launch_bounds__(256)
digits_t_kernel(BasisDev b, const int32_t* R, int64_t prime_stride, int64_t rows, int64_t cols,
                __nv_bfloat16* out, int64_t ld_out, int t) {
    // R_i is rows x cols; the planes are cols x ld_out (transposed), digit-major
    // across the primes: digit u of prime i at plane u * L + i.
    __shared__ int32_t tile[32][33];
    const int i = blockIdx.z;
    const int32_t* Ri = R + (size_t)i * prime_stride;
    const int64_t plane = cols * ld_out;
    __nv_bfloat16* base = out + (size_t)i * plane;
    const uint32_t p = b.p[i];
    const int32_t h = (int32_t)(p >> 1);
    const int64_t r0 = (int64_t)blockIdx.x * 32, c0 = (int64_t)blockIdx.y * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int k = ty; k < 32; k += 8) {
        const int64_t r = r0 + k, c = c0 + tx;
        int32_t v = 0;
        if (r < rows && c < cols) {
            v = Ri[r * cols + c];
            if (v > h) v -= (int32_t)p;
            if (v < -h) v += (int32_t)p;
        }
        tile[k][tx] = v;
    }
    __syncthreads();
    for (int k = ty; k < 32; k += 8) {
        const int64_t c = c0 + k, r = r0 + tx;
        if (c < cols && r < rows) store_digits(tile[tx][k], t, base + c * ld_out + r, plane * gridDim.z);
    }
}

}  // namespace

template <ReduceOut KIND>
cudaError_t launch_reduce_kind(const BasisDev& b, const ReduceArgs& a, dim3 grid, size_t smem, int group,
                               cudaStream_t s) {
    if (a.W <= 1) reduce_kernel<KIND, 1><<<grid, kThreads, smem, s>>>(b, a, group);
    else if (a.W <= 2) reduce_kernel<KIND, 2><<<grid, kThreads, smem, s>>>(b, a, group);
    else if (a.W <= 4) reduce_kernel<KIND, 4><<<grid, kThreads, smem, s>>>(b, a, group);
    else if (a.W <= 8) reduce_kernel<KIND, 8><<<grid, kThreads, smem, s>>>(b, a, group);
    else if (a.W <= 16) reduce_kernel<KIND, 16><<<grid, kThreads, smem, s>>>(b, a, group);
    else return cudaErrorNotSupported;
    return cudaGetLastError();
}

// The tensor-core reduction takes whole limbs per lane and three digits; other
// word counts, wider primes and larger bases keep reduce_kernel.
static bool mma_reducible(const BasisDev& b, const ReduceArgs& a) {
    return !a.identity && b.L <= 64 && b.p_top < (1u << 24) && b.p_low >= kMinPrime && (a.W == 1 || a.W == 2 || a.W == 4 || a.W == 8) &&
           ((uintptr_t)a.X & (a.W == 8 ? 15 : 7)) == 0;
}

// Large matrices of short entries modulo few primes, which limb sums reduce faster
// (us, limb sums / digit products; small ones the digit products, by a us or so).
// Canonical residues, 1M entries: one word, one prime 9.7 / 13.5, two primes 11.8 /
// 13.3, three 14.6 / 13.5; two words, one prime 11.7 / 13.3, two 14.1 / 13.5; four
// words, one prime 14.7 / 15.7.  Transposed digits, where the digit products take
// 20 with up to eight primes and 27 with nine to sixteen: one word, four primes 13.2,
// six 17.2, eleven 28.9; two words, seven 20.6, nine 24.7, twelve 31.7.
static bool limb_sums(const BasisDev& b, const ReduceArgs& a, ReduceOut kind) {
    if (a.rows * a.cols < (1 << 18) || (a.W % 2 == 0 && ((uintptr_t)a.X & 15))) return false;
    if (kind == ReduceOut::kCanonical) return b.L * a.W <= 2 || (b.L == 1 && a.W == 4);
    return kind == ReduceOut::kDigitsT && a.W <= 2 && 2 * b.L < (b.L + 7) / 8 * 7 + 9 - a.W && a.rows >= 128 &&
           a.cols <= 65535 * kTCols;
}

template <int W>
static cudaError_t launch_reduce_mma(const BasisDev& b, const ReduceArgs& a, ReduceOut kind, cudaStream_t s) {
    const bool trans = kind == ReduceOut::kDigitsT, ints = kind == ReduceOut::kCanonical;
    RmArgs r{a.X, trans ? a.rows : a.cols, trans ? a.cols : a.rows, trans ? a.ld : 1, trans ? 1 : a.ld,
             a.out, ints ? a.cols : a.ld_out, 0, 0, a.t, a.bits, a.status};
    if (ints) {  // [L][rows][cols]
        r.si = r.su = a.rows * a.cols;
    } else if (trans) {  // [t][L][cols][ld_out]
        r.si = a.cols * a.ld_out;
        r.su = r.si * b.L;
    } else {  // [L][t][rows][ld_out]
        r.su = a.rows * a.ld_out;
        r.si = r.su * a.t;
    }
    const size_t sm = rm_frag(b.L, RmShape<W>::KS) + (size_t)b.L * sizeof(uint4);
    const int64_t units = r.smin == 1 ? ((r.minor_n + 127) / 128) * r.major_n : ((r.minor_n + 31) / 32) * ((r.major_n + 3) / 4);
    if (ints) {
        const int64_t most = b.sms * rm_resident<reduce_mma_kernel<W, true>, W>();
        reduce_mma_kernel<W, true><<<(unsigned)(units < most ? units : most), kMmaThreads, sm, s>>>(b, r);
    } else {
        const int64_t most = b.sms * rm_resident<reduce_mma_kernel<W, false>, W>();
        reduce_mma_kernel<W, false><<<(unsigned)(units < most ? units : most), kMmaThreads, sm, s>>>(b, r);
    }
    return cudaGetLastError();
}

size_t reduce_image_bytes(const std::vector<uint32_t>& p, int W) {
    const int L = (int)p.size();
    if (L > 64 || p[0] >= (1u << 24) || p[L - 1] < kMinPrime) return 0;
    return rm_frag(L, W == 1 ? 1 : W / 2) + 2 * (size_t)L * sizeof(uint4);
}

cudaError_t launch_reduce_images(const uint32_t* d_p, int L, uint8_t* const (&to)[4], cudaStream_t s) {
    ReduceImages im;
    for (int k = 0; k < 4; k++) im.to[k] = to[k];
    reduce_images_kernel<<<(unsigned)((L + 7) / 8 * 8), kImageBytes, 0, s>>>(d_p, L, im);
    return cudaGetLastError();
}

cudaError_t launch_reduce(const BasisDev& b, const ReduceArgs& a_in, ReduceOut kind, int* d_status,
                          cudaStream_t s) {
    if (a_in.rows == 0 || a_in.cols == 0) return cudaSuccess;
    // entries outside the declared bound set kStatusBound (bits <= 0: not checked)
    ReduceArgs a = a_in;
    if (a.bits <= 0) a.bits = 64 * a.W;
    a.status = a.bits < 64 * a.W - 1 ? d_status : nullptr;
    if (kind == ReduceOut::kDigits && a.identity && a.cols % 8 == 0 && a.ld % 2 == 0 && a.ld_out % 8 == 0 &&
        ((uintptr_t)a.X & 15) == 0 && ((uintptr_t)a.out & 15) == 0) {
        const int64_t groups = a.cols / 8;
        dim3 grid((unsigned)((groups + kThreads - 1) / kThreads), (unsigned)(a.rows < 65535 ? a.rows : 65535));
        split_digits8_kernel<<<grid, kThreads, 0, s>>>(a.X, a.rows, a.cols, a.ld, a.W, (__nv_bfloat16*)a.out,
                                                       a.ld_out, a.t, a.bits, a.status);
        return cudaGetLastError();
    }
    const int nw = (2 * a.W + 1 + 3) & ~3;
    int group = a.identity ? 1 : max(1, min(b.L, kTableWords / (nw + 4)));
    // (canonical residues are asked for without a bound)
    if (mma_reducible(b, a) && (kind == ReduceOut::kCanonical ? !a.status : kind != ReduceOut::kCentered && a.t <= 3)) {
        if (!limb_sums(b, a, kind))
            return a.W == 1   ? launch_reduce_mma<1>(b, a, kind, s)
                   : a.W == 2 ? launch_reduce_mma<2>(b, a, kind, s)
                   : a.W == 4 ? launch_reduce_mma<4>(b, a, kind, s)
                              : launch_reduce_mma<8>(b, a, kind, s);
        if (kind == ReduceOut::kDigitsT) {
            const dim3 grid((unsigned)((a.rows + kThreads - 1) / kThreads), (unsigned)((a.cols + kTCols - 1) / kTCols));
            const size_t sm = sizeof(uint32_t) * (size_t)b.L * kTSumRow;
            if (a.W == 1) reduce_sums_t_kernel<1><<<grid, kThreads, sm, s>>>(b, a);
            else reduce_sums_t_kernel<2><<<grid, kThreads, sm, s>>>(b, a);
            return cudaGetLastError();
        }
    }
    const int groups = a.identity ? 1 : (b.L + group - 1) / group;
    const bool trans = kind == ReduceOut::kDigitsT;
    const int64_t minor_n = trans ? a.rows : a.cols;
    const int64_t major_n = trans ? a.cols : a.rows;
    dim3 grid((unsigned)((minor_n + kThreads - 1) / kThreads), (unsigned)(major_n < 65535 ? major_n : 65535),
              (unsigned)groups);
    size_t smem = a.identity ? 0 : sizeof(uint32_t) * (size_t)group * nw;
    switch (kind) {
        case ReduceOut::kCanonical: return launch_reduce_kind<ReduceOut::kCanonical>(b, a, grid, smem, group, s);
        case ReduceOut::kCentered: return launch_reduce_kind<ReduceOut::kCentered>(b, a, grid, smem, group, s);
        case ReduceOut::kDigits: return launch_reduce_kind<ReduceOut::kDigits>(b, a, grid, smem, group, s);
        case ReduceOut::kDigitsT: return launch_reduce_kind<ReduceOut::kDigitsT>(b, a, grid, smem, group, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_residue_digits(const BasisDev& b, const int32_t* R, int64_t prime_stride,
                                  int Lcount, int64_t rows, int64_t cols, void* out,
                                  int64_t ld_out, int t, bool transpose, cudaStream_t s) {
    if (rows == 0 || cols == 0 || Lcount == 0) return cudaSuccess;
    if (!transpose) {
        dim3 grid((unsigned)((cols + kThreads - 1) / kThreads), (unsigned)(rows < 65535 ? rows : 65535),
                  (unsigned)Lcount);
        digits_kernel<<<grid, kThreads, 0, s>>>(b, R, prime_stride, rows, cols, (__nv_bfloat16*)out,
                                                ld_out, t, prime_stride == 0 ? 1 : 0);
    } else {
        dim3 grid((unsigned)((rows + 31) / 32), (unsigned)((cols + 31) / 32), (unsigned)Lcount);
        digits_t_kernel<<<grid, 256, 0, s>>>(b, R, prime_stride, rows, cols, (__nv_bfloat16*)out,
                                             ld_out, t);
    }
    return cudaGetLastError();
}

namespace {
// blocks of `kernel` resident per SM (at least one), computed once per kernel
template <class Kern>
int resident(Kern kernel, int threads, size_t smem) {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        nb = 1;
    }
    return nb > 0 ? nb : 1;
}

int64_t persistent_grid(int64_t units, int num_sms, int per_sm) {
    const int64_t g = (int64_t)(num_sms > 0 ? num_sms : 148) * per_sm;
    return units < g ? units : g;
}

template <int W>
cudaError_t launch_rt_grouped_w(const BasisDev& b, const ReduceItem* items, int n, int64_t units, int num_sms,
                                int* status, cudaStream_t s) {
    const size_t sm = rm_frag(b.L, RmShape<W>::KS) + (size_t)b.L * sizeof(uint4);
    const int64_t grid = persistent_grid(units, num_sms, (int)rm_resident<reduce_mma_grouped_kernel<W>, W>());
    reduce_mma_grouped_kernel<W><<<(unsigned)grid, kMmaThreads, sm, s>>>(b, items, n, units, status);
    return cudaGetLastError();
}
}  // namespace

int64_t reduce_t_units(int64_t rows, int64_t cols) { return ((rows + 31) / 32) * ((cols + kRmCols - 1) / kRmCols); }

bool reduce_t_groupable(const BasisDev& b, const ReduceArgs& a) { return mma_reducible(b, a) && a.t <= 3; }

int64_t split_units(int64_t rows, int64_t cols, uint32_t* div_m, int* div_s) {
    // m = ceil(2^(32+s) / d) with 2^s >= d lies in (2^32, 2^33]; its low 32 bits
    // are kept and the 2^32 e term is added back in the kernel
    const int64_t per_row = (cols + kSplitPer - 1) / kSplitPer;  // a thread's groups in a row
    const uint64_t d = per_row > 0 ? (uint64_t)per_row : 1;
    int sh = 0;
    while (sh < 32 && (1ull << sh) < d) sh++;
    const unsigned __int128 num = (unsigned __int128)1 << (32 + sh);
    const unsigned __int128 m = (num + d - 1) / d;
    *div_m = (uint32_t)(m - ((unsigned __int128)1 << 32));
    *div_s = sh;
    return (rows * per_row + kThreads - 1) / kThreads;
}

cudaError_t launch_reduce_t_grouped(const BasisDev& b, int W, const ReduceItem* items, int n, int64_t units,
                                    int num_sms, int* status, cudaStream_t s) {
    if (n == 0 || units == 0) return cudaSuccess;
    switch (W) {
        case 1: return launch_rt_grouped_w<1>(b, items, n, units, num_sms, status, s);
        case 2: return launch_rt_grouped_w<2>(b, items, n, units, num_sms, status, s);
        case 4: return launch_rt_grouped_w<4>(b, items, n, units, num_sms, status, s);
        case 8: return launch_rt_grouped_w<8>(b, items, n, units, num_sms, status, s);
    }
    return cudaErrorNotSupported;
}

cudaError_t launch_split_grouped(const ReduceItem* items, int n, int64_t units, int num_sms, int* status,
                                 cudaStream_t s) {
    if (n == 0 || units == 0) return cudaSuccess;
    static int per_sm = 0;
    if (!per_sm) per_sm = resident(split_digits_grouped_kernel, kThreads, 0);
    const int64_t grid = persistent_grid(units, num_sms, per_sm);
    split_digits_grouped_kernel<<<(unsigned)grid, kThreads, 0, s>>>(items, n, units, status);
    return cudaGetLastError();
}

}  // namespace smf

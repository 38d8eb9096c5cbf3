// kernels.cu -- sampling, pointwise, exact RNS and linear kernels of the BFV evaluator.
//
// Randomness: Philox4x64-10 (Salmon et al., SC'11) with key (seed, purpose)
// and counter (block, poly, limb, kind): uniform residues use the word pair
// (w_hi, w_lo) of block n>>1 at offset 2(n&1) reduced as (w_hi 2^64 + w_lo)
// mod q; small samples use word n&3 of block n>>2 (kind 1): ternary {0, 1,
// -1}[w mod 3], centred binomial popcount(w & (2^21-1)) - popcount((w >> 21)
// & (2^21-1)).
//
// The exact base extensions (lift, scale-and-round, mod-down, decryption's
// last step) are in ext.cu.
#include <algorithm>

#include "rows.cuh"

namespace {

constexpr int TPB = 256;

inline int grid_for(size_t work) {
    size_t b = (work + TPB - 1) / TPB;
    if (b > (size_t)1 << 30) b = (size_t)1 << 30;
    return (int)(b ? b : 1);
}

// ---------------------------------------------------------------- Philox4x64-10
__device__ __forceinline__ void philox4x64(u64 c[4], u64 k0, u64 k1) {
    const u64 M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
    const u64 W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) {
            k0 += W0;
            k1 += W1;
        }
        const u64 lo0 = M0 * c[0], hi0 = __umul64hi(M0, c[0]);
        const u64 lo1 = M1 * c[2], hi1 = __umul64hi(M1, c[2]);
        const u64 n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = lo1;
        c[2] = n2;
        c[3] = lo0;
    }
}

__global__ void k_sample_uniform(u64* out, int n_polys, int n_limbs, LimbMap map, PrimeTab tab, const u64* R2,
                                 u64 seed, u64 purpose, u64 poly_base, int N) {
    pdl_begin();
    const size_t half = (size_t)N >> 1;
    const size_t total = (size_t)n_polys * n_limbs * half;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const size_t blk = idx % half;
        const int limb = (int)((idx / half) % n_limbs);
        const int poly = (int)(idx / (half * n_limbs));
        const int p = map(limb);
        const u64 q = tab.q[p], qinv = tab.qinv[p], mu = tab.mu[p], r2 = R2[p];
        u64 c[4] = {(u64)blk, poly_base + (u64)poly, (u64)limb, 0ull};
        philox4x64(c, seed, purpose);
        u64* o = out + ((size_t)poly * n_limbs + limb) * N + 2 * blk;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const u64 lo = c[2 * h], hi = reduce64(c[2 * h + 1], q, mu);
            const u64 t1 = redc(hi, lo, q, qinv);                 // (hi 2^64 + lo) 2^-64
            o[h] = redc(__umul64hi(t1, r2), t1 * r2, q, qinv);   // * 2^128 * 2^-64
        }
    }
}

__global__ void k_sample_small(i64* out, int n_polys, u64 seed, u64 purpose, u64 poly_base, int cbd, int N) {
    pdl_begin();
    const size_t quarter = (size_t)N >> 2;
    const size_t total = (size_t)n_polys * quarter;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const size_t blk = idx % quarter;
        const int poly = (int)(idx / quarter);
        u64 c[4] = {(u64)blk, poly_base + (u64)poly, 0ull, 1ull};
        philox4x64(c, seed, purpose);
        i64* o = out + (size_t)poly * N + 4 * blk;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const u64 w = c[h];
            if (cbd) {
                o[h] = (i64)__popcll(w & 0x1FFFFFull) - (i64)__popcll((w >> 21) & 0x1FFFFFull);
            } else {
                const u64 m = w % 3ull;
                o[h] = m == 0 ? 0 : (m == 1 ? 1 : -1);
            }
        }
    }
}

__global__ void k_spread(const i64* in, u64* out, int n_polys, int n_limbs, LimbMap map, PrimeTab tab, int N) {
    pdl_begin();
    const size_t total = (size_t)n_polys * n_limbs * N;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(idx % N);
        const int limb = (int)((idx / N) % n_limbs);
        const int poly = (int)(idx / ((size_t)N * n_limbs));
        const u64 q = tab.q[map(limb)];
        const i64 v = in[(size_t)poly * N + k];
        out[idx] = v >= 0 ? (u64)v : q - (u64)(-v);
    }
}

// ---------------------------------------------------------------- pointwise (NTT domain)
__global__ void k_pointwise(const u64* A, const u64* B, u64* out, int n, int polys, int n_limbs, LimbMap map,
                            PrimeTab tab, PwStrides s, int N) {
    pdl_begin();
    const size_t total = (size_t)n * polys * n_limbs * N;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(idx % N);
        const int limb = (int)((idx / N) % n_limbs);
        const size_t cp = idx / ((size_t)N * n_limbs);
        const int p = (int)(cp % polys);
        const size_t c = cp / polys;
        const int pi = map(limb);
        const u64 q = tab.q[pi], qinv = tab.qinv[pi];
        const size_t off = (size_t)limb * N + k;
        const u64 a = A[c * s.a_cs + p * s.a_ps + off];
        const u64 b = B[c * s.b_cs + p * s.b_ps + off];
        out[c * s.o_cs + p * s.o_ps + off] = redc(__umul64hi(a, b), a * b, q, qinv);
    }
}

// tensor in place: X[c][0..3] = (a0, a1, b0, b1) -> X[c][0..2] = (d0, d1, d2), Montgomery factor 2^-64
// Each thread takes two consecutive words (one 16-byte load per operand; N is even, so a pair never
// straddles limbs, and every limb starts 16-byte aligned).
__device__ __forceinline__ void tensor_word(u64 a0, u64 a1, u64 b0, u64 b1, u64 q, u64 qinv, u64& d0, u64& d1,
                                            u64& d2) {
    d0 = redc(__umul64hi(a0, b0), a0 * b0, q, qinv);
    u64 hi = 0, lo = 0;
    mac128(hi, lo, a0, b1);
    mac128(hi, lo, a1, b0);
    d1 = redc(hi, lo, q, qinv);
    d2 = redc(__umul64hi(a1, b1), a1 * b1, q, qinv);
}

// the same words with moduli 2^b - d: inputs below 2^(b+1), outputs plain residues (signed, within 2^(63-b) d of [0, 2^b)),
// each sum folded instead of reduced by Montgomery's ten further multiplies (28 wide multiplies per word against 46: 64
// pairs at N = 16384, L = 8 166 -> 149 us, 6.1 TB/s)
__device__ __forceinline__ void tensor_word_pm(u64 a0, u64 a1, u64 b0, u64 b1, int b, uint32_t d, u64& d0, u64& d1, u64& d2) {
    const int hs = (b + 2) >> 1;
    const uint32_t mask = (1u << hs) - 1u;
    const uint32_t a0l = (uint32_t)a0 & mask, a0h = (uint32_t)(a0 >> hs), a1l = (uint32_t)a1 & mask, a1h = (uint32_t)(a1 >> hs);
    const uint32_t b0l = (uint32_t)b0 & mask, b0h = (uint32_t)(b0 >> hs), b1l = (uint32_t)b1 & mask, b1h = (uint32_t)(b1 >> hs);
    d0 = pm_fold(pm_fold3((u64)a0l * b0l, mad_wide_u(a0h, b0l, (u64)a0l * b0h), (u64)a0h * b0h, b, d), b, d);
    d2 = pm_fold(pm_fold3((u64)a1l * b1l, mad_wide_u(a1h, b1l, (u64)a1l * b1h), (u64)a1h * b1h, b, d), b, d);
    u64 pm = (u64)a0l * b1h;
    pm = mad_wide_u(a0h, b1l, pm);
    pm = mad_wide_u(a1l, b0h, pm);
    pm = mad_wide_u(a1h, b0l, pm);
    d1 = pm_fold(pm_fold3(mad_wide_u(a1l, b0l, (u64)a0l * b1l), pm, mad_wide_u(a1h, b0h, (u64)a0h * b1h), b, d), b, d);
}

// tensor (SQ: squaring, b = a) in place as k_tensor; a block of 256 threads takes 512 words of one limb
template <bool SQ>
__global__ void __launch_bounds__(256) k_tensor_pm(u64* X, int LK, LimbMap map, PrimeTab tab, int logN, int b) {
    pdl_next();
    const int sh = logN - 9;
    const uint32_t row = blockIdx.x >> sh, c = row / (uint32_t)LK, limb = row - c * LK;
    const uint32_t d = (uint32_t)(((u64)1 << b) - tab.q[map((int)limb)]);
    const size_t p2 = ((size_t)LK << logN) / 2;   // one plane in 16-byte units
    ulonglong2* x = reinterpret_cast<ulonglong2*>(X + ((size_t)(c * 4 * LK + limb) << logN)) +
                    (blockIdx.x & ((1u << sh) - 1u)) * 256 + threadIdx.x;
    pdl_wait();
    const ulonglong2 a0 = x[0], a1 = x[p2], b0 = SQ ? a0 : x[2 * p2], b1 = SQ ? a1 : x[3 * p2];
    u64 e0, e1, e2, f0, f1, f2;
    tensor_word_pm(a0.x, a1.x, b0.x, b1.x, b, d, e0, e1, e2);
    tensor_word_pm(a0.y, a1.y, b0.y, b1.y, b, d, f0, f1, f2);
    x[0] = make_ulonglong2(e0, f0);
    x[p2] = make_ulonglong2(e1, f1);
    x[2 * p2] = make_ulonglong2(e2, f2);
}

__global__ void k_tensor(u64* X, int n, int LK, LimbMap map, PrimeTab tab, int N) {
    pdl_begin();
    const size_t plane = (size_t)LK * N, half = plane / 2;
    const size_t total = (size_t)n * half;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const size_t c = idx / half, off = (idx % half) * 2;
        const int pi = map((int)(off / N));
        const u64 q = tab.q[pi], qinv = tab.qinv[pi];
        ulonglong2* x = reinterpret_cast<ulonglong2*>(X + c * 4 * plane + off);
        const size_t p2 = half;   // one plane in 16-byte units
        const ulonglong2 a0 = x[0], a1 = x[p2], b0 = x[2 * p2], b1 = x[3 * p2];
        u64 e0, e1, e2, f0, f1, f2;
        tensor_word(a0.x, a1.x, b0.x, b1.x, q, qinv, e0, e1, e2);
        tensor_word(a0.y, a1.y, b0.y, b1.y, q, qinv, f0, f1, f2);
        x[0] = make_ulonglong2(e0, f0);
        x[p2] = make_ulonglong2(e1, f1);
        x[2 * p2] = make_ulonglong2(e2, f2);
    }
}

// squaring: X[c][0..1] = (a0, a1) -> X[c][0..2] = (a0^2, 2 a0 a1, a1^2), same sums as the general tensor
__global__ void k_tensor_sq(u64* X, int n, int LK, LimbMap map, PrimeTab tab, int N) {
    pdl_begin();
    const size_t plane = (size_t)LK * N, half = plane / 2;
    const size_t total = (size_t)n * half;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const size_t c = idx / half, off = (idx % half) * 2;
        const int pi = map((int)(off / N));
        const u64 q = tab.q[pi], qinv = tab.qinv[pi];
        ulonglong2* x = reinterpret_cast<ulonglong2*>(X + c * 4 * plane + off);
        const size_t p2 = half;
        const ulonglong2 a0 = x[0], a1 = x[p2];
        u64 e0, e1, e2, f0, f1, f2;
        tensor_word(a0.x, a1.x, a0.x, a1.x, q, qinv, e0, e1, e2);
        tensor_word(a0.y, a1.y, a0.y, a1.y, q, qinv, f0, f1, f2);
        x[0] = make_ulonglong2(e0, f0);
        x[p2] = make_ulonglong2(e1, f1);
        x[2 * p2] = make_ulonglong2(e2, f2);
    }
}

// z = sl + sm 2^28 + sh 2^56 as a 128-bit (hi, lo)
__device__ __forceinline__ void join28(u64 sl, u64 sm, u64 sh, u64& hi, u64& lo) {
    const u64 mlo = sm << 28, hlo = sh << 56;
    u64 r = sl + mlo;
    u64 c = r < mlo ? 1ull : 0ull;
    lo = r + hlo;
    c += lo < hlo ? 1ull : 0ull;
    hi = (sm >> 36) + (sh >> 8) + c;
}

// key-switch inner product: W[c][comp][k] = sum_j Dg[c][j][k] * rlk[j][comp][k]  (REDC).
// A thread owns one word (k, coefficient) of Q u P: it keeps the 2L key words of that word in
// registers and walks a group of ciphertexts, so the key is read once per group.  Up to 8 data primes
// the digits of the next two ciphertexts are in flight while the current one is accumulated; above 8
// there is no look-ahead, so that two CTAs of 256 threads still fit an SM (at 16 primes: 166 -> 128
// registers, +3% mul_relin at N = 32768).
// SPLIT (every prime below 2^50, so digits < 64q < 2^56 and key words < 2^50): each operand is cut at bit
// 28, a = ah 2^28 + al, b = bh 2^28 + bl (al, ah, bl < 2^28, bh < 2^22), and the three partial sums
// sum al bl, sum (al bh + ah bl), sum ah bh (weights 1, 2^28, 2^56) are 32 x 32 -> 64-bit multiply-adds into
// 64-bit accumulators: below 16 (2^56 + 2^56) = 2^61 for up to 16 terms, so none overflows; they are joined
// into the 128-bit sum once per output.  Otherwise each term is a full 64 x 64 -> 128-bit product.
template <int L, bool SPLIT>
__global__ void __launch_bounds__(256, 2) k_inner(const u64* Dg, const u64* rlk, u64* W, int n, int QP,
                                                              int cpg, PrimeTab tab, int N) {
    pdl_begin();
    static_assert(!SPLIT || L <= 16, "the split sums are bounded for at most 16 terms");
    constexpr int D = L <= 8 ? 2 : 0;
    constexpr uint32_t M28 = (1u << 28) - 1;
    const size_t plane = (size_t)QP * N;
    const int groups = (n + cpg - 1) / cpg;
    const size_t total = plane * groups;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const size_t off = idx % plane;
        const int grp = (int)(idx / plane);
        const int k = (int)(off / N);
        const u64 q = tab.q[k], qinv = tab.qinv[k];
        u64 k0[L], k1[L];   // SPLIT: (bh << 32) | bl
#pragma unroll
        for (int j = 0; j < L; ++j) {
            k0[j] = rlk[((size_t)j * 2 + 0) * plane + off];
            k1[j] = rlk[((size_t)j * 2 + 1) * plane + off];
            if constexpr (SPLIT) {
                k0[j] = ((k0[j] >> 28) << 32) | ((uint32_t)k0[j] & M28);
                k1[j] = ((k1[j] >> 28) << 32) | ((uint32_t)k1[j] & M28);
            }
        }
        const int c0 = grp * cpg, c_end = min(n, (grp + 1) * cpg);
        u64 buf[D + 1][L];
#pragma unroll
        for (int b = 0; b < D; ++b) {
            if (c0 + b < c_end) {
                const u64* d = Dg + (size_t)(c0 + b) * L * plane + off;
#pragma unroll
                for (int j = 0; j < L; ++j) buf[b][j] = d[(size_t)j * plane];
            }
        }
        for (int c = c0; c < c_end; ++c) {
            if (c + D < c_end) {
                const u64* d = Dg + (size_t)(c + D) * L * plane + off;
#pragma unroll
                for (int j = 0; j < L; ++j) buf[D][j] = d[(size_t)j * plane];
            }
            u64 h0 = 0, l0 = 0, h1 = 0, l1 = 0;
            if constexpr (SPLIT) {
                u64 s0l = 0, s0m = 0, s0h = 0, s1l = 0, s1m = 0, s1h = 0;
#pragma unroll
                for (int j = 0; j < L; ++j) {
                    const uint32_t al = (uint32_t)buf[0][j] & M28, ah = (uint32_t)(buf[0][j] >> 28);
                    const uint32_t b0l = (uint32_t)k0[j], b0h = (uint32_t)(k0[j] >> 32);
                    const uint32_t b1l = (uint32_t)k1[j], b1h = (uint32_t)(k1[j] >> 32);
                    s0l += (u64)al * b0l;
                    s0m += (u64)al * b0h;
                    s0m += (u64)ah * b0l;
                    s0h += (u64)ah * b0h;
                    s1l += (u64)al * b1l;
                    s1m += (u64)al * b1h;
                    s1m += (u64)ah * b1l;
                    s1h += (u64)ah * b1h;
                }
                join28(s0l, s0m, s0h, h0, l0);
                join28(s1l, s1m, s1h, h1, l1);
            } else {
#pragma unroll
                for (int j = 0; j < L; ++j) {
                    mac128(h0, l0, buf[0][j], k0[j]);
                    mac128(h1, l1, buf[0][j], k1[j]);
                }
            }
            W[((size_t)c * 2 + 0) * plane + off] = redc(h0, l0, q, qinv);
            W[((size_t)c * 2 + 1) * plane + off] = redc(h1, l1, q, qinv);
#pragma unroll
            for (int b = 0; b < D; ++b)
#pragma unroll
                for (int j = 0; j < L; ++j) buf[b][j] = buf[b + 1][j];
        }
    }
}

// the same inner product for moduli 2^b - d: digits below 2^(b+1) and key words cut at bit hs, the three limb sums in
// 64 bits, one fold per output, plain residues out (no Montgomery factor).  Up to 8 primes the middle sum comes from
// (x0 + x1)(y0 + y1), three products per term with the key words' sums kept in registers; above, four.  The kernel with
// Montgomery's reduction was bound by the multiplier pipe (97%): 28 instead of 42 multiplies per output at L = 8, where
// it now waits on its digit loads (64 ciphertexts at N = 16384: 172 -> 158 us, 5.4 TB/s).
template <int L>
__global__ void __launch_bounds__(256, 2) k_inner_pm(const u64* Dg, const u64* rlk, u64* W,
                                                     int n, int QP, int cpg, PrimeTab tab, int logN, int b) {
    pdl_begin();
    constexpr bool KARA = L <= 8;
    constexpr int D = L <= 8 ? 2 : 0;   // ciphertexts of look-ahead
    const int hs = (b + 2) >> 1;
    const uint32_t mask = (1u << hs) - 1u;
    const size_t plane = (size_t)QP << logN;
    const int groups = (n + cpg - 1) / cpg;
    const size_t total = plane * groups;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const uint32_t row = (uint32_t)(idx >> logN), grp = row / (uint32_t)QP, k = row - grp * QP;
        const size_t off = ((size_t)k << logN) + (idx & (((size_t)1 << logN) - 1));
        const u64 q = tab.q[k];
        const uint32_t d = (uint32_t)(((u64)1 << b) - q);
        uint32_t yl[2][L], yh[2][L], ys[2][KARA ? L : 1];
#pragma unroll
        for (int j = 0; j < L; ++j)
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const u64 y = rlk[((size_t)j * 2 + m) * plane + off];
                yl[m][j] = (uint32_t)y & mask;
                yh[m][j] = (uint32_t)(y >> hs);
                if constexpr (KARA) ys[m][j] = yl[m][j] + yh[m][j];
            }
        const int c0 = grp * cpg, c_end = min(n, (int)(grp + 1) * cpg);
        u64 buf[D + 1][L];
#pragma unroll
        for (int p = 0; p < D; ++p) {
            if (c0 + p < c_end) {
                const u64* s = Dg + (size_t)(c0 + p) * L * plane + off;
#pragma unroll
                for (int j = 0; j < L; ++j) buf[p][j] = s[(size_t)j * plane];
            }
        }
        for (int c = c0; c < c_end; ++c) {
            if (c + D < c_end) {
                const u64* s = Dg + (size_t)(c + D) * L * plane + off;
#pragma unroll
                for (int j = 0; j < L; ++j) buf[D][j] = s[(size_t)j * plane];
            }
            u64 p00[2] = {0, 0}, pm[2] = {0, 0}, p11[2] = {0, 0};
#pragma unroll
            for (int j = 0; j < L; ++j) {
                const uint32_t xl = (uint32_t)buf[0][j] & mask, xh = (uint32_t)(buf[0][j] >> hs);
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    p00[m] += (u64)xl * yl[m][j];
                    p11[m] += (u64)xh * yh[m][j];
                    if constexpr (KARA) {
                        pm[m] += (u64)(xl + xh) * ys[m][j];
                    } else {
                        pm[m] += (u64)xl * yh[m][j];
                        pm[m] += (u64)xh * yl[m][j];
                    }
                }
            }
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                if constexpr (KARA) pm[m] -= p00[m] + p11[m];
                W[((size_t)c * 2 + m) * plane + off] = pm_fold(pm_fold3(p00[m], pm[m], p11[m], b, d), b, d);
            }
#pragma unroll
            for (int p = 0; p < D; ++p)
#pragma unroll
                for (int j = 0; j < L; ++j) buf[p][j] = buf[p + 1][j];
        }
    }
}

// the same inner product for 17 or more data primes (insecure test-only parameter sets): sizes at run time,
// one thread per (ciphertext, word), the key re-read per ciphertext
__global__ void k_inner_n(const u64* Dg, const u64* rlk, u64* W, int n, int QP, int L, PrimeTab tab, int N) {
    pdl_begin();
    const size_t plane = (size_t)QP * N;
    const size_t total = plane * n;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const size_t off = idx % plane;
        const size_t c = idx / plane;
        const int k = (int)(off / N);
        const u64 q = tab.q[k], qinv = tab.qinv[k];
        const u64* d = Dg + c * L * plane + off;
        u64 h0 = 0, l0 = 0, h1 = 0, l1 = 0;
#pragma unroll 1
        for (int j = 0; j < L; ++j) {
            const u64 dj = d[(size_t)j * plane];
            mac128(h0, l0, dj, rlk[((size_t)j * 2 + 0) * plane + off]);
            mac128(h1, l1, dj, rlk[((size_t)j * 2 + 1) * plane + off]);
        }
        W[(c * 2 + 0) * plane + off] = redc(h0, l0, q, qinv);
        W[(c * 2 + 1) * plane + off] = redc(h1, l1, q, qinv);
    }
}

// ---------------------------------------------------------------- encode/decode, encrypt, keygen
__global__ void k_permute(const u64* in, u64* out, const uint32_t* brv, int n, int scatter, int N, u64 t,
                          uint32_t* flags) {
    pdl_begin();
    const size_t total = (size_t)n * N;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int j = (int)(idx % N);
        const size_t base = idx - j;
        if (scatter) {
            const u64 v = in[idx];   // a slot value being encoded: must be < t
            if (v >= t) atomicOr(flags, BFHE_FLAG_PLAINTEXT);
            out[base + brv[j]] = v;
        } else {
            out[idx] = in[base + brv[j]];
        }
    }
}

// out = -(as + e) [+ [P]_{q_j} s2 on limb j of poly j when gadget]
__global__ void k_neg_add_small(const u64* as, const i64* e, u64* out, int n_polys, int n_limbs, LimbMap map,
                                PrimeTab tab, const u64* s2, int gadget, const u64* Pq, int L, int N) {
    pdl_begin();
    const size_t total = (size_t)n_polys * n_limbs * N;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(idx % N);
        const int limb = (int)((idx / N) % n_limbs);
        const int poly = (int)(idx / ((size_t)N * n_limbs));
        const u64 q = tab.q[map(limb)];
        const i64 ev = e[(size_t)poly * N + k];
        u64 v = as[idx];
        v = ev >= 0 ? add_mod(v, (u64)ev, q) : sub_mod(v, (u64)(-ev), q);
        v = v == 0 ? 0 : q - v;
        if (gadget && limb == poly) {
            const u64 g = shoup(s2[(size_t)limb * N + k], Pq[limb], Pq[L + limb], q);
            v = add_mod(v, g, q);
        }
        out[idx] = v;
    }
}

template <int W>
__global__ void __launch_bounds__(256) k_lincomb(u64* out, const u64* x, const u64* y, const u64* z, const u64* p, LinCoef cf,
                                                 u64 cval, int L, const u64* qtab, const u64* delta, int logN) {
    pdl_begin();
    const Row<W> r(logN);
    const uint32_t h = r.row / (uint32_t)L;
    const int i = (int)(r.row - h * L);
    store_words<W>(out + r.off, lin_words<W>(cf.cc, cf.cx, cf.cy, cf.cz, cf.cp, cval, x, y, z, p, r.off,
                                             (h & 1) == 0 && r.k == 0, qtab[i], delta[i], delta[L + i]));
}

struct ScalarPairs {
    u64 w[BFHE_MAX_L], ws[BFHE_MAX_L];
};

template <int W>
__global__ void __launch_bounds__(256) k_mul_scalar(const u64* a, u64* out, ScalarPairs sp, int L, const u64* qtab, int logN) {
    pdl_begin();
    const Row<W> r(logN);
    const int i = (int)(r.row % (uint32_t)L);
    const u64 q = qtab[i], w = sp.w[i], ws = sp.ws[i];
    Words<W> t = load_words<W>(a + r.off);
#pragma unroll
    for (int j = 0; j < W; ++j) t.v[j] = shoup(t.v[j], w, ws, q);
    store_words<W>(out + r.off, t);
}

// Listing 5: r = v[s-1]; r += r + v[i], i = s-2 .. 0
template <int W>
__global__ void __launch_bounds__(256) k_horner(const u64* bits, uint32_t s, u64* out, size_t words, int L, const u64* qtab,
                                                int logN) {
    pdl_begin();
    const Row<W> r(logN);
    const u64 q = qtab[r.row % (uint32_t)L];
    const u64* p = bits + (size_t)(s - 1) * words + r.off;
    Words<W> acc = load_words<W>(p);
#pragma unroll (W == 2 ? 8 : 4)
    for (int i = (int)s - 2; i >= 0; --i) {
        p -= words;
        const Words<W> t = load_words<W>(p);
#pragma unroll
        for (int w = 0; w < W; ++w) acc.v[w] = add_mod(acc.v[w], add_mod(acc.v[w], t.v[w], q), q);
    }
    store_words<W>(out + r.off, acc);
}

// gather gate operands: A[g] = wires[x], B[g] = wires[y] (MUX: wires[y] - wires[z]); rows: gate, then the wire's limbs
template <int W>
__global__ void __launch_bounds__(256) k_gather_ops(u64* A, u64* B, const u64* wires, uint32_t rows, const int32_t* table, int L,
                                                    const u64* qtab, int logN) {
    pdl_begin();
    const Row<W> r(logN);
    const uint32_t g = r.row / rows, lr = r.row - g * rows;
    const size_t ctw = (size_t)rows << logN, o = ((size_t)lr << logN) + r.k;
    const int32_t* e = table + 5 * g;
    store_words<W>(A + r.off, load_words<W>(wires + (size_t)e[1] * ctw + o));
    Words<W> y = load_words<W>(wires + (size_t)e[2] * ctw + o);
    if ((e[0] & 0xff) == BFHE_MUX) {
        const u64 q = qtab[lr % (uint32_t)L];
        const Words<W> z = load_words<W>(wires + (size_t)e[3] * ctw + o);
#pragma unroll
        for (int w = 0; w < W; ++w) y.v[w] = sub_mod(y.v[w], z.v[w], q);
    }
    store_words<W>(B + r.off, y);
}

// gate epilogue: wires[out] = lin(op)(x, y, z, prod[g]); entries g >= n_mul have no product
template <int W>
__global__ void __launch_bounds__(256) k_gate_epilogue(u64* wires, uint32_t rows, const int32_t* table, int n_mul, const u64* prod,
                                                       int L, const u64* qtab, const u64* delta, int logN) {
    pdl_begin();
    const Row<W> r(logN);
    const uint32_t g = r.row / rows, lr = r.row - g * rows;
    const size_t ctw = (size_t)rows << logN, o = ((size_t)lr << logN) + r.k;
    const int32_t* e = table + 5 * g;
    int cc, cx, cy, cz, cp;
    gate_coefs(e[0], cc, cx, cy, cz, cp);
    if ((int)g >= n_mul) cp = 0;
    const uint32_t h = lr / (uint32_t)L;
    const int i = (int)(lr - h * L);
    const u64* x = wires + (size_t)e[1] * ctw;
    const u64* y = wires + (size_t)e[2] * ctw;
    const u64* z = wires + (size_t)e[3] * ctw;
    const u64* p = (int)g < n_mul ? prod + (size_t)g * ctw : nullptr;
    store_words<W>(wires + (size_t)e[4] * ctw + o,
                   lin_words<W>(cc, cx, cy, cz, cp, 1, x, y, z, p, o, (h & 1) == 0 && r.k == 0, qtab[i], delta[i], delta[L + i]));
}

// encrypt epilogue: ct[c][0] += Delta m + e1, ct[c][1] += e2; one block row per limb of c0, which does both components
template <int W>
__global__ void __launch_bounds__(256) k_enc_finish(u64* ct, const u64* M, const i64* e1, const i64* e2, int L, const u64* qtab,
                                                    const u64* delta, int logN, u64 t, uint32_t* flags) {
    pdl_begin();
    const Row<W> r(logN);
    const uint32_t c = r.row / (uint32_t)L, i = r.row - c * L;
    const u64 q = qtab[i];
    const size_t po = ((size_t)c << logN) + r.k;
    const Words<W> m = load_words<W>(M + po);
    const Words<W> a = load_words<W>(reinterpret_cast<const u64*>(e1) + po), b = load_words<W>(reinterpret_cast<const u64*>(e2) + po);
    u64* p0 = ct + ((size_t)(2 * c * L + i) << logN) + r.k;
    u64* p1 = p0 + ((size_t)L << logN);
    Words<W> v0 = load_words<W>(p0), v1 = load_words<W>(p1);
#pragma unroll
    for (int w = 0; w < W; ++w) {
        if (i == 0 && m.v[w] >= t) atomicOr(flags, BFHE_FLAG_PLAINTEXT);   // plaintext coefficients must be < t
        const i64 x = (i64)a.v[w], y = (i64)b.v[w];
        u64 v = add_mod(v0.v[w], shoup(m.v[w], delta[i], delta[L + i], q), q);
        v0.v[w] = x >= 0 ? add_mod(v, (u64)x, q) : sub_mod(v, (u64)(-x), q);
        v1.v[w] = y >= 0 ? add_mod(v1.v[w], (u64)y, q) : sub_mod(v1.v[w], (u64)(-y), q);
    }
    store_words<W>(p0, v0);
    store_words<W>(p1, v1);
}

// integer-pipe probe: 8 independent lazy Shoup chains per thread
__global__ void k_probe_modmul(u64* out, uint32_t iters, u64 q, u64 w, u64 ws) {
    pdl_begin();
    u64 x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = (u64)threadIdx.x * 977u + (u64)blockIdx.x * 131u + (u64)i;
    for (uint32_t it = 0; it < iters; ++it) {
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = shoup_lazy(x[i], w, ws, q);
    }
    u64 s = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) s ^= x[i];
    out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = s;
}

// trivial ciphertexts (Delta bit_k(c_base + c), 0), layout [s][C][n][2][L][N]
template <int W>
__global__ void __launch_bounds__(256) k_trivial_bits(u64* out, u64 c_base, const u64* cbp, uint32_t C, uint32_t n, int L,
                                                      const u64* delta, int logN) {
    pdl_begin();
    const Row<W> r(logN);
    if (cbp) c_base = *cbp;
    const uint32_t h = r.row / (uint32_t)L, i = r.row - h * L;   // h: (bit, c, n, component)
    const uint32_t cn = (h >> 1) / n, kbit = cn / C, c = cn - kbit * C;
    Words<W> t{};
    if ((h & 1) == 0 && r.k == 0 && (((c_base + c) >> kbit) & 1)) t.v[0] = delta[i];
    store_words<W>(out + r.off, t);
}

// bits[k][i] += sum over c of src (PAPER: src [s][C][n]; SELECT: src [C][n], only if bit k of c)
template <int W>
__global__ void __launch_bounds__(256) k_accumulate(u64* bits, const u64* src, uint32_t rows, u64 c_base, const u64* cbp, int C,
                                                    int select, int L, const u64* qtab, int logN) {
    pdl_begin();
    const Row<W> r(logN);
    if (cbp) c_base = *cbp;
    const uint32_t kbit = r.row / rows, lr = r.row - kbit * rows;
    const size_t words = (size_t)rows << logN, w0 = ((size_t)lr << logN) + r.k;
    const u64 q = qtab[lr % (uint32_t)L];
    Words<W> acc = load_words<W>(bits + r.off);
    const u64* p = src + w0 + (select ? 0 : (size_t)kbit * C * words);
#pragma unroll 4
    for (int c = 0; c < C; ++c, p += words) {
        if (select && !(((c_base + c) >> kbit) & 1)) continue;
        const Words<W> t = load_words<W>(p);
#pragma unroll
        for (int w = 0; w < W; ++w) acc.v[w] = add_mod(acc.v[w], t.v[w], q);
    }
    store_words<W>(bits + r.off, acc);
}

// out[c][i] = x[i] - (c_base + c)   (layout [C][n])
template <int W>
__global__ void __launch_bounds__(256) k_sub_const_chains(const u64* x, u64* out, uint32_t rows, u64 c_base, const u64* cbp, int L,
                                                          const u64* qtab, const u64* delta, u64 t, int logN) {
    pdl_begin();
    const Row<W> r(logN);
    if (cbp) c_base = *cbp;
    const uint32_t c = r.row / rows, lr = r.row - c * rows;
    const uint32_t h = lr / (uint32_t)L, i = lr - h * L;
    Words<W> v = load_words<W>(x + ((size_t)lr << logN) + r.k);
    if ((h & 1) == 0 && r.k == 0) {
        const u64 q = qtab[i];
        v.v[0] = sub_mod(v.v[0], shoup((c_base + c) % t, delta[i], delta[L + i], q), q);
    }
    store_words<W>(out + r.off, v);
}

// one device word (the candidate base read by a replayed mod_to_bits tile)
__global__ void k_set_word(u64* w, u64 v) { pdl_begin(); *w = v; }

}  // namespace

// ================================================================== launchers
#define LAUNCH(kern, work, ...)                                                   \
    do {                                                                          \
        auto* _kfn = kern;                                                        \
        BFHE_CUDA(launch_kernel(_kfn, dim3(grid_for(work)), dim3(TPB), 0, st, 1, __VA_ARGS__)); \
        BFHE_LAUNCH_CHECK(#kern);                                                \
    } while (0)

int launch_sample_uniform(const bfhe_ctx* ctx, u64* out, int n_polys, int n_limbs, LimbMap map, u64 seed,
                          u64 purpose, u64 poly_base, cudaStream_t st) {
    LAUNCH(k_sample_uniform, (size_t)n_polys * n_limbs * ctx->N / 2, out, n_polys, n_limbs, map, ctx->tab, ctx->d_R2,
           seed, purpose, poly_base, (int)ctx->N);
    return BFHE_OK;
}

int launch_sample_small(const bfhe_ctx* ctx, i64* out, int n_polys, u64 seed, u64 purpose, u64 poly_base, int cbd,
                        cudaStream_t st) {
    LAUNCH(k_sample_small, (size_t)n_polys * ctx->N / 4, out, n_polys, seed, purpose, poly_base, cbd, (int)ctx->N);
    return BFHE_OK;
}

int launch_spread(const bfhe_ctx* ctx, const i64* in, u64* out, int n_polys, int n_limbs, LimbMap map,
                  cudaStream_t st) {
    LAUNCH(k_spread, (size_t)n_polys * n_limbs * ctx->N, in, out, n_polys, n_limbs, map, ctx->tab, (int)ctx->N);
    return BFHE_OK;
}

int launch_pointwise(const bfhe_ctx* ctx, const u64* A, const u64* B, u64* out, int n, int polys, int n_limbs,
                     LimbMap map, PwStrides s, cudaStream_t st) {
    LAUNCH(k_pointwise, (size_t)n * polys * n_limbs * ctx->N, A, B, out, n, polys, n_limbs, map, ctx->tab, s,
           (int)ctx->N);
    return BFHE_OK;
}

int launch_tensor(const bfhe_ctx* ctx, u64* X, int n, int square, cudaStream_t st) {
    // per word of Q u B: 4 read, 3 written (squaring: 2 read)
    ProfScope ps(ctx, BFHE_K_TENSOR, st, 4.0 * n * (ctx->L + ctx->K) * ctx->N,
                 (square ? 40.0 : 56.0) * n * (ctx->L + ctx->K) * ctx->N);
    const int LK = (int)(ctx->L + ctx->K);
    if (ctx->pm_ext) {
        const dim3 grid((unsigned)((size_t)n * LK << (ctx->logN - 9)));
        BFHE_CUDA(launch_kernel(square ? k_tensor_pm<true> : k_tensor_pm<false>, grid, dim3(256), 0, st, 1, X, LK, ctx->mapQB(),
                                ctx->tab, (int)ctx->logN, (int)ctx->prime_bits));
        BFHE_LAUNCH_CHECK("k_tensor_pm");
        return BFHE_OK;
    }
    if (square)
        LAUNCH(k_tensor_sq, (size_t)n * LK * ctx->N / 2, X, n, LK, ctx->mapQB(), ctx->tab, (int)ctx->N);
    else
        LAUNCH(k_tensor, (size_t)n * LK * ctx->N / 2, X, n, LK, ctx->mapQB(), ctx->tab, (int)ctx->N);
    return BFHE_OK;
}

template <int L>
int run_inner(const bfhe_ctx* ctx, const u64* Dg, u64* W, int n, cudaStream_t st) {
    const int QP = (int)(ctx->L + ctx->alpha);
    // The key is read once per group of ciphertexts: as few groups as give four waves of two blocks per SM.  (A fixed four
    // read the 151 MB key of N = 32768, L = 16 four times, half of the kernel's traffic: 236 -> 175 us for 8 ciphertexts;
    // N = 4096, L = 2 left half of the SMs idle: 13 -> 12 us for 64.)
    const size_t plane = (size_t)QP * ctx->N, want = (size_t)4 * 152 * 2 * TPB;
    const int groups = (int)std::min<size_t>((size_t)n, std::max<size_t>(1, (want + plane - 1) / plane));
    const int cpg = (n + groups - 1) / groups;
    const size_t work = plane * ((n + cpg - 1) / cpg);
    if (ctx->pm_ext)
        LAUNCH(k_inner_pm<L>, work, Dg, ctx->d_rlk_ntt, W, n, QP, cpg, ctx->tab, (int)ctx->logN, (int)ctx->prime_bits);
    else if (ctx->prime_bits <= 50)   // digits below 64q < 2^56 (lazy transforms), key words below 2^50
        LAUNCH((k_inner<L, true>), work, Dg, ctx->d_rlk_ntt, W, n, QP, cpg, ctx->tab, (int)ctx->N);
    else
        LAUNCH((k_inner<L, false>), work, Dg, ctx->d_rlk_ntt, W, n, QP, cpg, ctx->tab, (int)ctx->N);
    return BFHE_OK;
}

#define SWITCH_L(Lv, FN, ...)                                                                                  \
    switch (Lv) {                                                                                              \
        case 1: return FN<1>(__VA_ARGS__);                                                                     \
        case 2: return FN<2>(__VA_ARGS__);                                                                     \
        case 3: return FN<3>(__VA_ARGS__);                                                                     \
        case 4: return FN<4>(__VA_ARGS__);                                                                     \
        case 5: return FN<5>(__VA_ARGS__);                                                                     \
        case 6: return FN<6>(__VA_ARGS__);                                                                     \
        case 7: return FN<7>(__VA_ARGS__);                                                                     \
        case 8: return FN<8>(__VA_ARGS__);                                                                     \
        case 9: return FN<9>(__VA_ARGS__);                                                                     \
        case 10: return FN<10>(__VA_ARGS__);                                                                   \
        case 11: return FN<11>(__VA_ARGS__);                                                                   \
        case 12: return FN<12>(__VA_ARGS__);                                                                   \
        case 13: return FN<13>(__VA_ARGS__);                                                                   \
        case 14: return FN<14>(__VA_ARGS__);                                                                   \
        case 15: return FN<15>(__VA_ARGS__);                                                                   \
        case 16: return FN<16>(__VA_ARGS__);                                                                   \
        default: break;                                                                                        \
    }

int launch_inner(const bfhe_ctx* ctx, const u64* Dg, u64* W, int n, cudaStream_t st) {
    // per word of Q u P: L digits read and 2 words written per ciphertext, the key's 2L words once
    ProfScope ps(ctx, BFHE_K_INNER, st, 2.0 * ctx->L * n * (ctx->L + ctx->alpha) * ctx->N,
                 8.0 * (ctx->L + ctx->alpha) * ctx->N * ((double)n * (ctx->L + 2) + 2.0 * ctx->L));
    SWITCH_L(ctx->L, run_inner, ctx, Dg, W, n, st)
    if (ctx->L > BFHE_MAX_L) return set_error(BFHE_EINVAL, "unsupported number of data primes");
    const int QP = (int)(ctx->L + ctx->alpha);
    LAUNCH(k_inner_n, (size_t)QP * ctx->N * n, Dg, ctx->d_rlk_ntt, W, n, QP, (int)ctx->L, ctx->tab, (int)ctx->N);
    return BFHE_OK;
}

int launch_permute(const bfhe_ctx* ctx, const u64* in, u64* out, int n, int scatter, cudaStream_t st) {
    LAUNCH(k_permute, (size_t)n * ctx->N, in, out, ctx->d_brv, n, scatter, (int)ctx->N, ctx->t, ctx->d_flags);
    return BFHE_OK;
}

// one block per 256 W words of each row; two words per thread when every buffer is 16-byte aligned
#define LAUNCH_ROWS(kern, wide, rows, ...)                                                                     \
    do {                                                                                                       \
        const size_t _rows = (rows);                                                                           \
        if (wide)                                                                                              \
            BFHE_CUDA(launch_kernel(kern<2>, dim3((unsigned)(_rows << (ctx->logN - 9))), dim3(TPB), 0, st, 1, __VA_ARGS__)); \
        else                                                                                                   \
            BFHE_CUDA(launch_kernel(kern<1>, dim3((unsigned)(_rows << (ctx->logN - 8))), dim3(TPB), 0, st, 1, __VA_ARGS__)); \
        BFHE_LAUNCH_CHECK(#kern);                                                                              \
    } while (0)

int launch_enc_finish(const bfhe_ctx* ctx, u64* ct, const u64* M, const i64* e1, const i64* e2, int n,
                      cudaStream_t st) {
    LAUNCH_ROWS(k_enc_finish, aligned16(ct) && aligned16(M) && aligned16(e1) && aligned16(e2), (size_t)n * ctx->L, ct, M, e1,
                e2, (int)ctx->L, ctx->tab.q, ctx->d_delta_q, (int)ctx->logN, ctx->t, ctx->d_flags);
    return BFHE_OK;
}

int launch_neg_add_small(const bfhe_ctx* ctx, const u64* as, const i64* e, u64* out, int n_polys, int n_limbs,
                         LimbMap map, const u64* s2, int gadget, cudaStream_t st) {
    LAUNCH(k_neg_add_small, (size_t)n_polys * n_limbs * ctx->N, as, e, out, n_polys, n_limbs, map, ctx->tab, s2,
           gadget, ctx->d_P_q, (int)ctx->L, (int)ctx->N);
    return BFHE_OK;
}

int launch_lincomb(const bfhe_ctx* ctx, u64* out, const u64* x, const u64* y, const u64* z, const u64* p,
                   LinCoef cf, u64 cval, size_t n, cudaStream_t st) {
    const bool wide = aligned16(out) && (!cf.cx || aligned16(x)) && (!cf.cy || aligned16(y)) && (!cf.cz || aligned16(z)) &&
                      (!cf.cp || aligned16(p));
    LAUNCH_ROWS(k_lincomb, wide, n * 2 * ctx->L, out, x, y, z, p, cf, cval, (int)ctx->L, ctx->tab.q, ctx->d_delta_q,
                (int)ctx->logN);
    return BFHE_OK;
}

int launch_mul_scalar(const bfhe_ctx* ctx, const u64* a, u64 c, u64* out, size_t n, cudaStream_t st) {
    ScalarPairs sp;
    for (uint32_t i = 0; i < ctx->L; ++i) {
        const u64 q = ctx->primes[i];
        const u64 w = c % q;
        sp.w[i] = w;
        sp.ws[i] = (u64)(((u128)w << 64) / q);
    }
    LAUNCH_ROWS(k_mul_scalar, aligned16(a) && aligned16(out), n * 2 * ctx->L, a, out, sp, (int)ctx->L, ctx->tab.q,
                (int)ctx->logN);
    return BFHE_OK;
}

int launch_horner(const bfhe_ctx* ctx, const u64* bits, uint32_t s, u64* out, size_t n, cudaStream_t st) {
    LAUNCH_ROWS(k_horner, aligned16(bits) && aligned16(out), n * 2 * ctx->L, bits, s, out, n * ctx->ct_words(), (int)ctx->L,
                ctx->tab.q, (int)ctx->logN);
    return BFHE_OK;
}

int launch_gather(const bfhe_ctx* ctx, u64* dst, const u64* wires, size_t n, const int32_t* table, int n_gates,
                  cudaStream_t st) {
    // dst holds A then B ([2][n_gates][n] ciphertexts)
    const size_t ctw = n * ctx->ct_words();
    LAUNCH_ROWS(k_gather_ops, aligned16(dst) && aligned16(wires), (size_t)n_gates * n * 2 * ctx->L, dst,
                dst + (size_t)n_gates * ctw, wires, (uint32_t)(n * 2 * ctx->L), table, (int)ctx->L, ctx->tab.q,
                (int)ctx->logN);
    return BFHE_OK;
}

int launch_gate_epilogue(const bfhe_ctx* ctx, u64* wires, size_t n, const int32_t* table, int n_gates,
                         const u64* prod, int n_mul, cudaStream_t st) {
    LAUNCH_ROWS(k_gate_epilogue, aligned16(wires) && aligned16(prod), (size_t)n_gates * n * 2 * ctx->L, wires,
                (uint32_t)(n * 2 * ctx->L), table, n_mul, prod, (int)ctx->L, ctx->tab.q, ctx->d_delta_q, (int)ctx->logN);
    return BFHE_OK;
}

int launch_trivial_bits(const bfhe_ctx* ctx, u64* out, uint32_t s, u64 c_base, const u64* cbp, int C, size_t n,
                        cudaStream_t st) {
    LAUNCH_ROWS(k_trivial_bits, aligned16(out), (size_t)s * C * n * 2 * ctx->L, out, c_base, cbp, (uint32_t)C, (uint32_t)n,
                (int)ctx->L, ctx->d_delta_q, (int)ctx->logN);
    return BFHE_OK;
}

int launch_accumulate(const bfhe_ctx* ctx, u64* bits, const u64* src, uint32_t s, u64 c_base, const u64* cbp, int C,
                      size_t n, int select, cudaStream_t st) {
    LAUNCH_ROWS(k_accumulate, aligned16(bits) && aligned16(src), (size_t)s * n * 2 * ctx->L, bits, src,
                (uint32_t)(n * 2 * ctx->L), c_base, cbp, C, select, (int)ctx->L, ctx->tab.q, (int)ctx->logN);
    return BFHE_OK;
}

int launch_sub_const_chains(const bfhe_ctx* ctx, const u64* x, u64* out, u64 c_base, const u64* cbp, int C, size_t n,
                            cudaStream_t st) {
    LAUNCH_ROWS(k_sub_const_chains, aligned16(x) && aligned16(out), (size_t)C * n * 2 * ctx->L, x, out,
                (uint32_t)(n * 2 * ctx->L), c_base, cbp, (int)ctx->L, ctx->tab.q, ctx->d_delta_q, ctx->t, (int)ctx->logN);
    return BFHE_OK;
}

int launch_set_word(u64* w, u64 v, cudaStream_t st) {
    BFHE_CUDA(launch_kernel(k_set_word, dim3(1), dim3(1), 0, st, 1, w, v));
    BFHE_LAUNCH_CHECK("k_set_word");
    return BFHE_OK;
}

int launch_probe_modmul(u64* out, int blocks, int threads, uint32_t iters, u64 q, u64 w, u64 ws, cudaStream_t st) {
    BFHE_CUDA(launch_kernel(k_probe_modmul, dim3(blocks), dim3(threads), 0, st, 1, out, iters, q, w, ws));
    BFHE_LAUNCH_CHECK("k_probe_modmul");
    return BFHE_OK;
}

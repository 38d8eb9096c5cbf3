// ext.cu -- exact base extensions of the multiply and of decryption.
//
// The multiply lifts each input coefficient to the centred range and extends
// it exactly to the auxiliary base (k_modup); scale-and-round computes
// round(t d / Q) as y = (t d - r) / Q with r the centred residue of t d mod Q,
// by two exact extensions (Q -> B for r, B -> Q for y; k_scale); mod-down
// extends the special-prime part to Q (k_moddown); decryption extends to t
// (k_dec_finish).  Extensions run Garner's mixed-radix conversion, or, when
// the context enables it, the guarded fast conversion (a fixed-point overflow
// count with a mixed-radix fallback near the rounding boundary).  Both give
// the same integers.  Contexts with moduli 2^b - d of 45 to 55 bits and at most
// 16 data primes take ext_pm.cu instead, and k_moddown_pm here.
#include "ext_device.cuh"
#include "rows.cuh"

namespace {

// The guarded fast extension's per-source factors and 26-bit limb pairs for NS sources and ND targets, passed by
// value as a kernel parameter (it sits in the constant bank): with the loops over sources and targets unrolled,
// every factor is an operand of the multiply-add that uses it, with no load instruction.
template <int NS, int ND>
struct FastTab {
    uint2 c[ND][NS];        // (low, high) 26-bit limbs of [(S/s_i) 2^64]_{T_j}
    u64 qh[NS], qhs[NS];    // [(S/s_i)^-1]_{s_i} and its Shoup companion
    u64 ghi[NS], glo[NS];   // floor(2^128 / s_i): high and low words
};

template <int NS, int ND>
FastTab<NS, ND> fast_tab(const ExtHost& h) {
    FastTab<NS, ND> t{};
    if (h.n != NS || h.m != ND) return t;   // only the instances the launchers use are ever filled
    for (int j = 0; j < ND; ++j)
        for (int i = 0; i < NS; ++i) t.c[j][i] = make_uint2(h.c26[((size_t)j * NS + i) * 2], h.c26[((size_t)j * NS + i) * 2 + 1]);
    for (int i = 0; i < NS; ++i) {
        t.qh[i] = h.qhinv[i];
        t.qhs[i] = h.qhinv_s[i];
        t.ghi[i] = h.g_hi[i];
        t.glo[i] = h.g_lo[i];
    }
    return t;
}

// Guarded fast exact extension (all moduli below 2^50), first half: y_i = [x_i (S/s_i)^-1]_{s_i} split
// into 26-bit limbs, and v = round(sum_i y_i / s_i) from the 64.64 fixed-point sum of
// floor(y_i floor(2^128/s_i) / 2^64) (each term at most 2 units below y_i 2^64 / s_i).  Returns false
// when the fraction lies within 2n + 2 units of 1/2: then the caller takes the exact mixed-radix path.
template <int NS, int ND>
__device__ __forceinline__ bool fast_prep(const u64 (&x)[NS], const ExtDesc& d, const FastTab<NS, ND>& ft,
                                          uint32_t (&y0)[NS], uint32_t (&y1)[NS], int& v) {
    u64 lo = 0, hi = 0;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const u64 s = d.src_q[i];
        const u64 y = shoup(x[i], ft.qh[i], ft.qhs[i], s);
        y0[i] = (uint32_t)(y & 0x3FFFFFFull);
        y1[i] = (uint32_t)(y >> 26);
        const u64 term = y * ft.ghi[i] + __umul64hi(y, ft.glo[i]);
        lo += term;
        hi += lo < term ? 1ull : 0ull;
    }
    const u64 half = 1ull << 63;
    if (lo > half) {
        v = (int)hi + 1;
        return true;
    }
    if (lo + (u64)(2 * NS + 2) <= half) {
        v = (int)hi;
        return true;
    }
    return false;
}

// second half: sum_i y_i [(S/s_i) 2^64]_{T_j} with the 26-bit limb products accumulated in four 64-bit
// words (no carries below 2^13 sources), one Montgomery reduction, minus [v S]_{T_j}; canonical result
template <int NS, int ND>
__device__ __forceinline__ u64 fast_eval(const uint32_t (&y0)[NS], const uint32_t (&y1)[NS], int v, const ExtDesc& d,
                                         const FastTab<NS, ND>& ft, int j) {
    u64 p00 = 0, p01 = 0, p10 = 0, p11 = 0;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const uint32_t c0 = ft.c[j][i].x, c1 = ft.c[j][i].y;
        p00 += (u64)y0[i] * c0;
        p01 += (u64)y0[i] * c1;
        p10 += (u64)y1[i] * c0;
        p11 += (u64)y1[i] * c1;
    }
    const u64 mid = p01 + p10;                       // weight 2^26
    u64 lo = p00 + (mid << 26);
    u64 hi = (mid >> 38) + (lo < p00 ? 1ull : 0ull);
    const u64 top = p11 << 52;                       // weight 2^52
    lo += top;
    hi += (p11 >> 12) + (lo < top ? 1ull : 0ull);
    const u64 T = d.dst_q[j];
    return sub_mod(redc(hi, lo, T, d.dst_qinv[j]), d.vS[(size_t)j * (NS + 1) + v], T);
}

// the same sum with three limb products per term (Karatsuba): the weight-2^26 part is
// sum (y0 + y1)(c0 + c1) - sum y0 c0 - sum y1 c1, the same integer (every factor below 2^27, every product
// below 2^54, so each sum fits 64 bits for fewer than 2^10 sources); scale-and-round takes this form, the base
// extension of the multiply's inputs keeps four products (fewer registers)
template <int NS, int ND>
__device__ __forceinline__ u64 fast_eval3(const uint32_t (&y0)[NS], const uint32_t (&y1)[NS], int v, const ExtDesc& d,
                                          const FastTab<NS, ND>& ft, int j) {
    static_assert(NS < 1024, "the three-product sums are bounded for fewer than 2^10 sources");
    u64 p00 = 0, pm = 0, p11 = 0;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const uint32_t c0 = ft.c[j][i].x, c1 = ft.c[j][i].y;
        p00 += (u64)y0[i] * c0;
        p11 += (u64)y1[i] * c1;
        pm += (u64)(y0[i] + y1[i]) * (c0 + c1);
    }
    const u64 mid = pm - p00 - p11;                  // weight 2^26
    u64 lo = p00 + (mid << 26);
    u64 hi = (mid >> 38) + (lo < p00 ? 1ull : 0ull);
    const u64 top = p11 << 52;                       // weight 2^52
    lo += top;
    hi += (p11 >> 12) + (lo < top ? 1ull : 0ull);
    const u64 T = d.dst_q[j];
    return sub_mod(redc(hi, lo, T, d.dst_qinv[j]), d.vS[(size_t)j * (NS + 1) + v], T);
}

// B limbs of X[c][slot] (slots a0 a1 b0 b1; only a0 a1 when squaring): the centred extension
template <int NS, bool FAST>
__global__ void __launch_bounds__(256, NS <= 8 ? 4 : 2) k_modup(const u64* A, const u64* B, u64* X, int n, int slots, int K, ExtDesc ext, int N,
                        uint32_t* flags, FastTab<FAST ? NS : 1, FAST ? NS + 1 : 1> ft) {
    pdl_begin();
    const size_t total = (size_t)n * slots * N;
    const int LK = NS + K;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(idx % N);
        const size_t pp = idx / N;
        const size_t c = pp / slots;
        const int slot = (int)(pp % slots);
        const u64* src = (slot < 2 ? A : B) + (c * 2 + (slot & 1)) * (size_t)NS * N + k;
        u64* dst = X + (c * 4 + slot) * (size_t)LK * N + k;
        u64 x[NS];
        bool bad = false;
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            x[i] = src[(size_t)i * N];
            bad |= x[i] >= ext.src_q[i];
        }
        if (bad) atomicOr(flags, BFHE_FLAG_RESIDUE);
        if constexpr (FAST) {
            uint32_t y0[NS], y1[NS];
            int vv = 0;
            if (fast_prep<NS, NS + 1>(x, ext, ft, y0, y1, vv)) {   // the fast path has K = NS + 1 targets
#pragma unroll
                for (int j = 0; j < NS + 1; ++j)
                    dst[(size_t)(NS + j) * N] = fast_eval<NS, NS + 1>(y0, y1, vv, ext, ft, j);
                continue;
            }
        }
        u64 v[NS];
        const bool neg = garner<NS>(x, ext, v);
        for (int j = 0; j < K; ++j) dst[(size_t)(NS + j) * N] = ext_eval<NS, false>(v, neg, ext, j);
    }
}

// scale-and-round of the tensor (X slots 0..2, Q u B limbs) into C3 [n][3][L][N].  The inverse transforms
// leave the tensor untwisted: the first product of each limb, by t, also carries the twist N^-1 psi^-k R.
// PM: moduli 2^bits - d (mixed radix alone, where the caller has switched the guarded form off); a choice at run time
// between the two products costs every instance 10 to 20% (64 pairs at N = 16384, L = 8: 613 -> 717 us at 40 bits, 860 -> 940 at 56).
template <int NS, int KS, bool FAST, bool PM>
__global__ void __launch_bounds__(256, 2) k_scale(const u64* X, u64* C3, int n, ExtDesc eQB, ExtDesc eBQ, const u64* twist, int nP,
                        const u64* Qinv_b, const u64* bq, int N, int bits, FastTab<FAST ? NS : 1, FAST ? KS : 1> fq,
                        FastTab<FAST ? KS : 1, FAST ? NS : 1> fb) {
    pdl_begin();
    static_assert(!(FAST && PM), "moduli 2^b - d have a guarded form of their own");
    if (!PM) bits = 0;
    const size_t total = (size_t)n * 3 * N;
    constexpr int LK = NS + KS;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(idx % N);
        const size_t cp = idx / N;
        const size_t c = cp / 3;
        const int comp = (int)(cp % 3);
        const u64* d = X + (c * 4 + comp) * (size_t)LK * N + k;
        u64 r[NS];
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            const u64 qi = eQB.src_q[i];
            const ulonglong2 f = twist_at(twist, i, 2, k, N);
            r[i] = twist_mul(d[(size_t)i * N], f, qi, bits);   // [t d]_{q_i}, < 2 q_i
        }
        // r -> B (centred), then y = (t d - r) / Q in B
        u64 y[KS];
        {
            uint32_t r0[NS], r1[NS];
            int vv = 0;
            bool fast = false;
            if constexpr (FAST) fast = fast_prep<NS, KS>(r, eQB, fq, r0, r1, vv);
            u64 v[NS];
            bool neg = false;
            if (!fast) neg = garner<NS>(r, eQB, v);
#pragma unroll
            for (int j = 0; j < KS; ++j) {
                const u64 bj = bq[j];
                const int pj = NS + (nP - 1 - NS - KS) + j;                      // prime index of b_j
                const ulonglong2 f = twist_at(twist, pj, 2, k, N);
                const u64 td = twist_mul(d[(size_t)(NS + j) * N], f, bj, bits);   // [t d]_{b_j}, < 2 b_j
                u64 rb;
                if constexpr (FAST)
                    rb = fast ? fast_eval3<NS, KS>(r0, r1, vv, eQB, fq, j) : ext_eval<NS, false>(v, neg, eQB, j);
                else rb = ext_eval<NS, false>(v, neg, eQB, j);
                y[j] = shoup_lazy(td + bj - rb, Qinv_b[j], Qinv_b[KS + j], bj);  // (t d - r) / Q, < 2 b_j
            }
        }
        // y -> Q (centred)
        u64* o = C3 + cp * (size_t)NS * N + k;
        if constexpr (FAST) {
            uint32_t y0[KS], y1[KS];
            int vy = 0;
            if (fast_prep<KS, NS>(y, eBQ, fb, y0, y1, vy)) {
#pragma unroll
                for (int i = 0; i < NS; ++i) o[(size_t)i * N] = fast_eval3<KS, NS>(y0, y1, vy, eBQ, fb, i);
                continue;
            }
        }
        u64 w[KS];
        const bool negy = garner<KS>(y, eBQ, w);
#pragma unroll
        for (int i = 0; i < NS; ++i) o[(size_t)i * N] = ext_eval<KS, false>(w, negy, eBQ, i);
    }
}

// Scale-and-round in two passes (fast path, 10 or more data primes, where the one-pass kernel needs more than
// 128 registers and runs one CTA per SM), so that each pass holds one extension's digits in registers:
// pass A writes y = (t d - r) / Q over B (words below 2 b_j) to Yt [n][3][KS][N]; pass B extends y to Q.
// Measured at N = 32768, L = 16: mul_relin +10.6%, squarings +12.1%; at L = 8 the one-pass kernel is 1% faster.
template <int NS, int KS>
__global__ void __launch_bounds__(256, 2) k_scale_a(const u64* X, u64* Yt, int n, ExtDesc eQB, const u64* twist, int nP,
                                                    const u64* Qinv_b, const u64* bq, int N, FastTab<NS, KS> fq) {
    pdl_begin();
    const size_t total = (size_t)n * 3 * N;
    constexpr int LK = NS + KS;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(idx % N);
        const size_t cp = idx / N;
        const size_t c = cp / 3;
        const int comp = (int)(cp % 3);
        const u64* d = X + (c * 4 + comp) * (size_t)LK * N + k;
        u64* yo = Yt + cp * (size_t)KS * N + k;
        uint32_t r0[NS], r1[NS];
        int vv = 0;
        bool fast;
        {
            u64 r[NS];
#pragma unroll
            for (int i = 0; i < NS; ++i) {
                const ulonglong2 f = twist_at(twist, i, 2, k, N);
                r[i] = twist_mul(d[(size_t)i * N], f, eQB.src_q[i], 0);
            }
            fast = fast_prep<NS, KS>(r, eQB, fq, r0, r1, vv);
        }
        if (!fast) {
            // the exact mixed-radix path near the rounding boundary (rare): recompute r from memory
            u64 r[NS], v[NS];
#pragma unroll
            for (int i = 0; i < NS; ++i) {
                const ulonglong2 f = twist_at(twist, i, 2, k, N);
                r[i] = twist_mul(d[(size_t)i * N], f, eQB.src_q[i], 0);
            }
            const bool neg = garner<NS>(r, eQB, v);
            for (int j = 0; j < KS; ++j) {
                const u64 bj = bq[j];
                const int pj = NS + (nP - 1 - NS - KS) + j;
                const ulonglong2 f = twist_at(twist, pj, 2, k, N);
                const u64 td = twist_mul(d[(size_t)(NS + j) * N], f, bj, 0);
                const u64 rb = ext_eval<NS, false>(v, neg, eQB, j);
                yo[(size_t)j * N] = shoup_lazy(td + bj - rb, Qinv_b[j], Qinv_b[KS + j], bj);
            }
            continue;
        }
#pragma unroll 1
        for (int j = 0; j < KS; ++j) {
            const u64 bj = bq[j];
            const int pj = NS + (nP - 1 - NS - KS) + j;
            const ulonglong2 f = twist_at(twist, pj, 2, k, N);
            const u64 td = twist_mul(d[(size_t)(NS + j) * N], f, bj, 0);
            const u64 rb = fast_eval3<NS, KS>(r0, r1, vv, eQB, fq, j);
            yo[(size_t)j * N] = shoup_lazy(td + bj - rb, Qinv_b[j], Qinv_b[KS + j], bj);
        }
    }
}

template <int NS, int KS>
__global__ void __launch_bounds__(256, 2) k_scale_b(const u64* Yt, u64* C3, int n, ExtDesc eBQ, int N,
                                                    FastTab<KS, NS> fb) {
    pdl_begin();
    const size_t total = (size_t)n * 3 * N;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(idx % N);
        const size_t cp = idx / N;
        const u64* yi = Yt + cp * (size_t)KS * N + k;
        u64 y[KS];
#pragma unroll
        for (int j = 0; j < KS; ++j) y[j] = yi[(size_t)j * N];
        u64* o = C3 + cp * (size_t)NS * N + k;
        uint32_t y0[KS], y1[KS];
        int vy = 0;
        if (fast_prep<KS, NS>(y, eBQ, fb, y0, y1, vy)) {
#pragma unroll
            for (int i = 0; i < NS; ++i) o[(size_t)i * N] = fast_eval3<KS, NS>(y0, y1, vy, eBQ, fb, i);
            continue;
        }
        u64 w[KS];
        const bool negy = garner<KS>(y, eBQ, w);
#pragma unroll
        for (int i = 0; i < NS; ++i) o[(size_t)i * N] = ext_eval<KS, false>(w, negy, eBQ, i);
    }
}

// out[c][comp] = C3[c][comp] + round(W / P) mod Q, W over Q u P (coefficient form, untwisted: each word is
// first multiplied by the twist N^-1 psi^-k R that the inverse transform left out)
template <int NA>
__global__ void k_moddown(const u64* W, const u64* C3, u64* out, int n, int L, ExtDesc ePQ, const u64* Pinv,
                          const u64* qtab, const u64* twist, int N, int bits) {
    pdl_begin();
    // two consecutive coefficients per thread (N is even, every limb starts 16-byte aligned): 16-byte accesses
    const size_t half = (size_t)N >> 1;
    const size_t total = (size_t)n * 2 * half;
    const int QP = L + NA;
    const ulonglong2* tw2 = reinterpret_cast<const ulonglong2*>(twist);
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(idx % half) * 2;
        const size_t cp = idx / half;
        const size_t c = cp >> 1;
        const int comp = (int)(cp & 1);
        const u64* w = W + cp * (size_t)QP * N + k;
        u64 x0[NA], x1[NA], v0[NA], v1[NA];
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            const ulonglong2 ww = *reinterpret_cast<const ulonglong2*>(w + (size_t)(L + a) * N);
            const ulonglong2* f = tw2 + ((size_t)(L + a) * 3 + 1) * N + k;
            const ulonglong2 f0 = __ldg(f), f1 = __ldg(f + 1);
            x0[a] = twist_mul(ww.x, f0, ePQ.src_q[a], bits);   // < 2 p_a
            x1[a] = twist_mul(ww.y, f1, ePQ.src_q[a], bits);
        }
        const bool neg0 = garner<NA>(x0, ePQ, v0), neg1 = garner<NA>(x1, ePQ, v1);
        const u64* cin = C3 + (c * 3 + comp) * (size_t)L * N + k;
        u64* o = out + cp * (size_t)L * N + k;
        for (int i = 0; i < L; ++i) {
            const u64 qi = qtab[i], pw = Pinv[i], pws = Pinv[L + i];
            const ulonglong2* f = tw2 + ((size_t)i * 3 + 1) * N + k;
            const ulonglong2 f0 = __ldg(f), f1 = __ldg(f + 1);
            const ulonglong2 ww = *reinterpret_cast<const ulonglong2*>(w + (size_t)i * N);
            const ulonglong2 cc = *reinterpret_cast<const ulonglong2*>(cin + (size_t)i * N);
            const u64 w0 = twist_mul(ww.x, f0, qi, bits), w1 = twist_mul(ww.y, f1, qi, bits);   // < 2 q_i
            const u64 y0 = shoup(sub_mod(w0, ext_eval<NA, false>(v0, neg0, ePQ, i), qi), pw, pws, qi);
            const u64 y1 = shoup(sub_mod(w1, ext_eval<NA, false>(v1, neg1, ePQ, i), qi), pw, pws, qi);
            *reinterpret_cast<ulonglong2*>(o + (size_t)i * N) = make_ulonglong2(add_mod(cc.x, y0, qi), add_mod(cc.y, y1, qi));
        }
    }
}

// The same for moduli 2^b - d, W of plain residues: with v the canonical digits of the special part x (v = x for one
// special prime), neg its sign and P^-1 folded into the data primes' twist, the result is c + w twist - v P^-1 (- v1 p_0
// P^-1) + neg, one folded sum per word (10 wide multiplies against 16 and two more reductions: 64
// ciphertexts at N = 16384, L = 8 90 -> 72 us between events, 5.3 TB/s; 62 us by its own counters, 93% of the copy rate,
// and 98% between events at 468 ciphertexts).
__device__ __forceinline__ void mul28(u64 w, const ulonglong2& e, u64& P, u64& Q) {
    P = mad_wide_u((uint32_t)w, (uint32_t)e.x, P);
    Q = mad_wide_u((uint32_t)w, (uint32_t)(e.x >> 32), Q);
    P = mad_wide_s((int)(w >> 32), (int)(uint32_t)e.y, P);
    Q = mad_wide_s((int)(w >> 32), (int)(e.y >> 32), Q);
}
__device__ __forceinline__ u64 fold28(u64 P, u64 Q, int b, uint32_t d) {
    const int k = b - 28;
    const uint32_t ql = (uint32_t)Q;
    return mad_wide_s((int)(Q >> 32), (int)(d << 4), add64(P, ((u64)(ql >> (32 - k)) << 32) | (ql << k)));
}

template <int NA, bool EPI>
__global__ void __launch_bounds__(256) k_moddown_pm(const u64* W, const u64* C3, u64* out,
                                                    int L, ExtDesc ePQ, const ulonglong2* __restrict__ mtw,
                                                    const ulonglong2* __restrict__ mpc, const u64* __restrict__ qtab, int logN, int b,
                                                    MulEpilogue epi, const u64* __restrict__ delta) {
    pdl_next();
    // a block takes 512 coefficients of one polynomial
    const int sh = logN - 9;
    const uint32_t cp = blockIdx.x >> sh, c = cp >> 1, comp = cp & 1;
    const int k = (int)((blockIdx.x & ((1u << sh) - 1u)) * 512 + threadIdx.x * 2);
    const u64* w = W + ((size_t)cp * (L + NA) << logN) + k;
    pdl_wait();
    u64 x0[NA], x1[NA], v0[NA], v1[NA];
#pragma unroll
    for (int a = 0; a < NA; ++a) {
        const ulonglong2 ww = *reinterpret_cast<const ulonglong2*>(w + ((size_t)(L + a) << logN));
        const ulonglong2* f = mtw + ((size_t)(L + a) << logN) + k;
        const u64 p = ePQ.src_q[a];
        const uint32_t d = (uint32_t)(((u64)1 << b) - p);
        u64 P = 0, Q = 0;
        mul28(ww.x, __ldg(f), P, Q);
        x0[a] = pm_canon(fold28(P, Q, b, d), p, b, d);
        P = Q = 0;
        mul28(ww.y, __ldg(f + 1), P, Q);
        x1[a] = pm_canon(fold28(P, Q, b, d), p, b, d);
    }
    const u64 neg0 = garner<NA>(x0, ePQ, v0) ? 1 : 0, neg1 = garner<NA>(x1, ePQ, v1) ? 1 : 0;
    const u64* cin = C3 + ((size_t)(c * 3 + comp) * L << logN) + k;
    u64* o = out + ((size_t)cp * L << logN) + k;
    // EPI: the operands' words sit where the product's would, shifted to their wires for a table entry
    LinCoef cf{};
    const u64 *ex = nullptr, *ey = nullptr, *ez = nullptr;
    if constexpr (EPI) {
        const uint32_t cg = epi.c0 + c;
        if (epi.kind == 1) {
            cf = epi.cf;
            const size_t at = ((size_t)(2 * cg + comp) * L << logN) + k;
            ex = epi.x + at;
            ey = epi.y + at;
            ez = epi.z + at;
        } else {
            const uint32_t g = cg / epi.n, ci = cg - g * epi.n;
            const int32_t* t = epi.table + 5 * g;
            gate_coefs(t[0], cf.cc, cf.cx, cf.cy, cf.cz, cf.cp);
            const size_t ctw = (size_t)epi.n * 2 * L << logN, at = ((size_t)(2 * ci + comp) * L << logN) + k;
            ex = epi.wires + (size_t)t[1] * ctw + at;
            ey = epi.wires + (size_t)t[2] * ctw + at;
            ez = epi.wires + (size_t)t[3] * ctw + at;
            o = epi.wires + (size_t)t[4] * ctw + at;
        }
    }
#pragma unroll 4
    for (int i = 0; i < L; ++i) {
        const u64 q = qtab[i];
        const uint32_t d = (uint32_t)(((u64)1 << b) - q);
        const ulonglong2* f = mtw + ((size_t)i << logN) + k;
        const ulonglong2 ww = *reinterpret_cast<const ulonglong2*>(w + ((size_t)i << logN));
        const ulonglong2 cc = *reinterpret_cast<const ulonglong2*>(cin + ((size_t)i << logN));
        u64 P0 = cc.x + neg0, Q0 = 0, P1 = cc.y + neg1, Q1 = 0;
        mul28(ww.x, __ldg(f), P0, Q0);
        mul28(ww.y, __ldg(f + 1), P1, Q1);
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            const ulonglong2 e = __ldg(mpc + i * NA + a);
            mul28(v0[a], e, P0, Q0);
            mul28(v1[a], e, P1, Q1);
        }
        u64 r0 = pm_canon(fold28(P0, Q0, b, d), q, b, d), r1 = pm_canon(fold28(P1, Q1, b, d), q, b, d);
        const size_t l = (size_t)i << logN;
        if constexpr (EPI) {
            Words<2> acc{};
            if (cf.cc && comp == 0 && k == 0) acc.v[0] = apply(0, delta[i], cf.cc, q);   // the constant 1
            auto term = [&](const u64* s, int m) {
                const Words<2> t = load_words<2>(s);
                acc.v[0] = apply(acc.v[0], t.v[0], m, q);
                acc.v[1] = apply(acc.v[1], t.v[1], m, q);
            };
            if (cf.cx) term(ex + l, cf.cx);
            if (cf.cy) term(ey + l, cf.cy);
            if (cf.cz) term(ez + l, cf.cz);
            r0 = apply(acc.v[0], r0, cf.cp, q);
            r1 = apply(acc.v[1], r1, cf.cp, q);
        }
        *reinterpret_cast<ulonglong2*>(o + l) = make_ulonglong2(r0, r1);
    }
}

// decrypt: m = [-r Q^-1]_t with r the centred [t (c0 + c1 s)]_Q
template <int NS>
__global__ void k_dec_finish(const u64* V, const u64* ct, u64* M, int n, ExtDesc eQt, const u64* tmod, int nP,
                             u64 Qinv_t, int N, uint32_t* flags) {
    pdl_begin();
    const size_t total = (size_t)n * N;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(idx % N);
        const size_t c = idx / N;
        u64 r[NS], v[NS];
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            const u64 qi = eQt.src_q[i];
            const u64 c0 = ct[(c * 2 * NS + i) * N + k];
            if (c0 >= qi) atomicOr(flags, BFHE_FLAG_RESIDUE);
            const u64 vi = add_mod(V[(c * NS + i) * N + k], c0, qi);
            r[i] = shoup(vi, tmod[i], tmod[nP + i], qi);
        }
        const bool neg = garner<NS>(r, eQt, v);
        const u64 t = eQt.dst_q[0];
        const u64 rho = ext_eval<NS, true>(v, neg, eQt, 0);        // [r]_t
        const u64 mneg = rho == 0 ? 0 : t - rho;
        M[idx] = (mneg * Qinv_t) % t;
    }
}

// ---------------------------------------------------------------- more than 16 data primes
// The insecure test-only parameter sets with 17..BFHE_MAX_L data primes run the same exact arithmetic with
// sizes known only at run time (digits in local memory, loops not unrolled), so that they need no template
// instance per size; the guarded fast extension is not offered there.
__global__ void k_modup_n(const u64* A, const u64* B, u64* X, int n, int slots, int K, ExtDesc ext, int N,
                          uint32_t* flags) {
    pdl_begin();
    const int ns = ext.n_src;
    const size_t total = (size_t)n * slots * N;
    const int LK = ns + K;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(idx % N);
        const size_t pp = idx / N;
        const size_t c = pp / slots;
        const int slot = (int)(pp % slots);
        const u64* src = (slot < 2 ? A : B) + (c * 2 + (slot & 1)) * (size_t)ns * N + k;
        u64* dst = X + (c * 4 + slot) * (size_t)LK * N + k;
        u64 x[NMAX], v[NMAX];
        bool bad = false;
        for (int i = 0; i < ns; ++i) {
            x[i] = src[(size_t)i * N];
            bad |= x[i] >= ext.src_q[i];
        }
        if (bad) atomicOr(flags, BFHE_FLAG_RESIDUE);
        const bool neg = garner_n(x, ext, v, ns);
        for (int j = 0; j < K; ++j) dst[(size_t)(ns + j) * N] = ext_eval_n(v, neg, ext, j, ns, false);
    }
}

__global__ void k_scale_n(const u64* X, u64* C3, int n, ExtDesc eQB, ExtDesc eBQ, const u64* twist, int nP,
                          const u64* Qinv_b, const u64* bq, int N, int bits) {
    pdl_begin();
    const int ns = eQB.n_src, ks = eBQ.n_src, LK = ns + ks;
    const size_t total = (size_t)n * 3 * N;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(idx % N);
        const size_t cp = idx / N;
        const size_t c = cp / 3;
        const int comp = (int)(cp % 3);
        const u64* d = X + (c * 4 + comp) * (size_t)LK * N + k;
        u64 r[NMAX], v[NMAX], y[NMAX];
        for (int i = 0; i < ns; ++i) {
            const ulonglong2 f = twist_at(twist, i, 2, k, N);
            r[i] = twist_mul(d[(size_t)i * N], f, eQB.src_q[i], bits);
        }
        const bool neg = garner_n(r, eQB, v, ns);
        for (int j = 0; j < ks; ++j) {
            const u64 bj = bq[j];
            const int pj = ns + (nP - 1 - ns - ks) + j;
            const ulonglong2 f = twist_at(twist, pj, 2, k, N);
            const u64 td = twist_mul(d[(size_t)(ns + j) * N], f, bj, bits);
            const u64 rb = ext_eval_n(v, neg, eQB, j, ns, false);
            y[j] = shoup_lazy(td + bj - rb, Qinv_b[j], Qinv_b[ks + j], bj);
        }
        const bool negy = garner_n(y, eBQ, v, ks);
        u64* o = C3 + cp * (size_t)ns * N + k;
        for (int i = 0; i < ns; ++i) o[(size_t)i * N] = ext_eval_n(v, negy, eBQ, i, ks, false);
    }
}

__global__ void k_dec_finish_n(const u64* V, const u64* ct, u64* M, int n, ExtDesc eQt, const u64* tmod, int nP,
                               u64 Qinv_t, int N, uint32_t* flags) {
    pdl_begin();
    const int ns = eQt.n_src;
    const size_t total = (size_t)n * N;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(idx % N);
        const size_t c = idx / N;
        u64 r[NMAX], v[NMAX];
        for (int i = 0; i < ns; ++i) {
            const u64 qi = eQt.src_q[i];
            const u64 c0 = ct[(c * 2 * ns + i) * N + k];
            if (c0 >= qi) atomicOr(flags, BFHE_FLAG_RESIDUE);
            r[i] = shoup(add_mod(V[(c * ns + i) * N + k], c0, qi), tmod[i], tmod[nP + i], qi);
        }
        const bool neg = garner_n(r, eQt, v, ns);
        const u64 t = eQt.dst_q[0];
        const u64 rho = ext_eval_n(v, neg, eQt, 0, ns, true);
        const u64 mneg = rho == 0 ? 0 : t - rho;
        M[idx] = (mneg * Qinv_t) % t;
    }
}

}  // namespace

// ================================================================== launchers
template <int NS>
int run_modup(const bfhe_ctx* ctx, const u64* A, const u64* B, u64* X, int n, int slots, cudaStream_t st) {
    const size_t work = (size_t)n * slots * ctx->N;
    if (ctx->fast_ext && ctx->ext_QB.fast_ok && (int)ctx->K == NS + 1)
        LAUNCH((k_modup<NS, true>), work, A, B, X, n, slots, (int)ctx->K, ctx->ext_QB, (int)ctx->N, ctx->d_flags,
               fast_tab<NS, NS + 1>(ctx->exth_QB));
    else
        LAUNCH((k_modup<NS, false>), work, A, B, X, n, slots, (int)ctx->K, ctx->ext_QB, (int)ctx->N, ctx->d_flags,
               FastTab<1, 1>{});
    return BFHE_OK;
}

template <int NS>
int run_scale(const bfhe_ctx* ctx, const u64* X, u64* C3, int n, cudaStream_t st, u64* tmp) {
    const size_t work = (size_t)n * 3 * ctx->N;
    const u64* bq = ctx->tab.q + ctx->L + ctx->alpha;
    if (ctx->pm) {   // the extension switched off, which is possible where it is on by default
        if constexpr (NS >= 8) {
            LAUNCH((k_scale<NS, NS + 1, false, true>), work, X, C3, n, ctx->ext_QB, ctx->ext_BQ, ctx->tab.twist, (int)ctx->nP,
                   ctx->d_Qinv_b, bq, (int)ctx->N, ctx->pm_bits(), FastTab<1, 1>{}, FastTab<1, 1>{});
            return BFHE_OK;
        }
        return set_error(BFHE_EINVAL, "no mixed-radix scale-and-round for these moduli");
    }
    const bool fast = ctx->fast_ext && ctx->ext_QB.fast_ok && ctx->ext_BQ.fast_ok;
    if constexpr (NS >= 10) {
        if (tmp && fast) {
            LAUNCH((k_scale_a<NS, NS + 1>), work, X, tmp, n, ctx->ext_QB, ctx->tab.twist, (int)ctx->nP,
                   ctx->d_Qinv_b, bq, (int)ctx->N, fast_tab<NS, NS + 1>(ctx->exth_QB));
            LAUNCH((k_scale_b<NS, NS + 1>), work, tmp, C3, n, ctx->ext_BQ, (int)ctx->N,
                   fast_tab<NS + 1, NS>(ctx->exth_BQ));
            return BFHE_OK;
        }
    }
    if (fast)
        LAUNCH((k_scale<NS, NS + 1, true, false>), work, X, C3, n, ctx->ext_QB, ctx->ext_BQ, ctx->tab.twist, (int)ctx->nP,
               ctx->d_Qinv_b, bq, (int)ctx->N, 0, fast_tab<NS, NS + 1>(ctx->exth_QB),
               fast_tab<NS + 1, NS>(ctx->exth_BQ));
    else
        LAUNCH((k_scale<NS, NS + 1, false, false>), work, X, C3, n, ctx->ext_QB, ctx->ext_BQ, ctx->tab.twist, (int)ctx->nP,
               ctx->d_Qinv_b, bq, (int)ctx->N, 0, FastTab<1, 1>{}, FastTab<1, 1>{});
    return BFHE_OK;
}

template <int NS>
int run_dec_finish(const bfhe_ctx* ctx, const u64* V, const u64* ct, u64* M, int n, cudaStream_t st) {
    const size_t work = (size_t)n * ctx->N;
    LAUNCH(k_dec_finish<NS>, work, V, ct, M, n, ctx->ext_Qt, ctx->d_tmod, (int)ctx->nP, ctx->Qinv_t, (int)ctx->N,
           ctx->d_flags);
    return BFHE_OK;
}

int launch_modup(const bfhe_ctx* ctx, const u64* A, const u64* B, u64* X, int n, int slots, cudaStream_t st) {
    const double L_ = ctx->L, K_ = ctx->K;
    // counted as a whole lift, L limbs read and L + K written per coefficient of each input poly (the kernels write the
    // K new limbs; the transform reads the L others from the inputs)
    ProfScope ps(ctx, BFHE_K_MODUP, st, (double)slots * n * ctx->N * (L_ * (L_ - 1) / 2 + K_ * (L_ - 1)),
                 8.0 * slots * n * ctx->N * (2 * L_ + K_));
    if (ctx->use_pm_ext()) return launch_modup_pm(ctx, A, B, X, n, slots, st);
    SWITCH_L(ctx->L, run_modup, ctx, A, B, X, n, slots, st)
    if (ctx->L > BFHE_MAX_L) return set_error(BFHE_EINVAL, "unsupported number of data primes");
    LAUNCH(k_modup_n, (size_t)n * slots * ctx->N, A, B, X, n, slots, (int)ctx->K, ctx->ext_QB, (int)ctx->N,
           ctx->d_flags);
    return BFHE_OK;
}

int launch_scale(const bfhe_ctx* ctx, const u64* X, u64* C3, int n, cudaStream_t st, u64* tmp) {
    if (ctx->K != ctx->L + 1) return set_error(BFHE_EINVAL, "auxiliary base must have L+1 primes");
    const double L_ = ctx->L, K_ = ctx->K;
    // per coefficient of each of 3 polys: L + K limbs read, L written
    ProfScope ps(ctx, BFHE_K_SCALE, st,
                 3.0 * n * ctx->N * (2 * L_ + 3 * K_ + L_ * (L_ - 1) / 2 + K_ * (L_ - 1) + K_ * (K_ - 1) / 2 + L_ * (K_ - 1)),
                 24.0 * n * ctx->N * (2 * L_ + K_));
    if (ctx->use_pm_ext()) return launch_scale_pm(ctx, X, C3, n, st, tmp);
    SWITCH_L(ctx->L, run_scale, ctx, X, C3, n, st, tmp)
    if (ctx->L > BFHE_MAX_L) return set_error(BFHE_EINVAL, "unsupported number of data primes");
    LAUNCH(k_scale_n, (size_t)n * 3 * ctx->N, X, C3, n, ctx->ext_QB, ctx->ext_BQ, ctx->tab.twist, (int)ctx->nP,
           ctx->d_Qinv_b, ctx->tab.q + ctx->L + ctx->alpha, (int)ctx->N, ctx->pm_bits());
    return BFHE_OK;
}

int launch_moddown(const bfhe_ctx* ctx, const u64* W, const u64* C3, u64* out, int n, cudaStream_t st,
                   const MulEpilogue* epi) {
    if (epi && !ctx->pm_ext) return set_error(BFHE_EINVAL, "no fused gate equation for these moduli");
    const double A_ = ctx->alpha;
    // work: the rounding division by P, plus the twist the inverse transform left to this kernel
    // per coefficient of each of 2 polys: L + alpha words of W and L of C3 read, L written
    ProfScope ps(ctx, BFHE_K_MODDOWN, st, 2.0 * n * ctx->N * (A_ * (A_ - 1) / 2 + ctx->L * A_ + ctx->L + A_),
                 16.0 * n * ctx->N * (3.0 * ctx->L + A_));
    const size_t work = (size_t)n * ctx->N;   // two coefficients per thread
    if (ctx->pm_ext) {
        const dim3 grid((unsigned)((size_t)n * 2 << (ctx->logN - 9)));
        auto* kern = epi ? (ctx->alpha == 1 ? k_moddown_pm<1, true> : k_moddown_pm<2, true>)
                         : (ctx->alpha == 1 ? k_moddown_pm<1, false> : k_moddown_pm<2, false>);
        BFHE_CUDA(launch_kernel(kern, grid, dim3(256), 0, st, 1, W, C3, out, (int)ctx->L, ctx->ext_PQ, ctx->d_mtw, ctx->d_mpc,
                                ctx->tab.q, (int)ctx->logN, (int)ctx->prime_bits, epi ? *epi : MulEpilogue{},
                                ctx->d_delta_q));
        BFHE_LAUNCH_CHECK("k_moddown_pm");
        return BFHE_OK;
    }
    if (ctx->alpha == 1)
        LAUNCH(k_moddown<1>, work, W, C3, out, n, (int)ctx->L, ctx->ext_PQ, ctx->d_Pinv_q, ctx->tab.q, ctx->tab.twist,
               (int)ctx->N, ctx->pm_bits());
    else if (ctx->alpha == 2)
        LAUNCH(k_moddown<2>, work, W, C3, out, n, (int)ctx->L, ctx->ext_PQ, ctx->d_Pinv_q, ctx->tab.q, ctx->tab.twist,
               (int)ctx->N, ctx->pm_bits());
    else
        return set_error(BFHE_EINVAL, "alpha must be 1 or 2");
    return BFHE_OK;
}

int launch_dec_finish(const bfhe_ctx* ctx, const u64* V, const u64* ct, u64* M, int n, cudaStream_t st) {
    // (64-bit sums of 26-bit words mod t)
    if (ctx->use_pm_ext() && ctx->t < ((u64)1 << 26)) return launch_dec_pm(ctx, V, ct, M, n, st);
    SWITCH_L(ctx->L, run_dec_finish, ctx, V, ct, M, n, st)
    if (ctx->L > BFHE_MAX_L) return set_error(BFHE_EINVAL, "unsupported number of data primes");
    LAUNCH(k_dec_finish_n, (size_t)n * ctx->N, V, ct, M, n, ctx->ext_Qt, ctx->d_tmod, (int)ctx->nP, ctx->Qinv_t,
           (int)ctx->N, ctx->d_flags);
    return BFHE_OK;
}


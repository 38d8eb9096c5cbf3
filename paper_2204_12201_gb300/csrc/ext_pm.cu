// ext_pm.cu -- the multiply's exact base extensions for moduli 2^b - d (contexts with pm set, at most 16 data primes).
//
// The guarded fast conversion of ext.cu with other arithmetic: y_i = [x_i (S/s_i)^-1]_{s_i} (any representative),
// x = sum_i y_i (S/s_i) - v S with v the integer nearest to sum_i y_i / s_i.  Three things follow from s_i = 2^b - d_i:
//  - sum_i y_i / s_i is sum_i y_i / 2^b up to a relative d/2^b (below 2^-18): v is the rounded top of the plain sum
//    of the y_i, without a multiply; the exact mixed-radix path runs when the sum lies within `guard` (the bound of
//    that error, times 2^b) of a half, 2^-19 to 2^-26 of the coefficients;
//  - a sum of products is folded once: each y is cut at bit hs = (b+2)/2, y = y1 2^hs + y0, and takes two constants c and
//    2^hs c mod T, each cut at bit k = b - 28, so that sum y c = P + 2^k Q with P, Q sums of 32 x 32 -> 64-bit
//    multiply-adds; with Q = qh 2^32 + ql it is P + 2^k ql + 16d qh (2^(b+4) = 16d mod T), one multiply;
//  - the product of a tensor word by the inverse transform's twist has the same form, so it joins the sum.
// Scale-and-round computes round(t d / Q) = (t d - r) / Q, r the centred [t d]_Q: the constants t, (Q/q_i)^-1, 1/Q and
// the second extension's (B/b_j)^-1 are all folded into the twist tables (xtw) and the sums' constants, so that its
// intermediate words are the second extension's digits themselves.
//
// All of it is bound by the multiplier pipe (a wide multiply-add takes it four cycles per warp and scheduler).  Wide
// multiplies per coefficient at L = 8: base extension 40 + 9 x 35 = 355, scale-and-round 48 + 9 x 40 + 8 x 40 = 728.
// 64 pairs at N = 16384, L = 8 (GB300): lift 372 -> 197 us (89% of the pipe), scale-and-round 612 -> 343 us (70%: two
// CTAs of 256 threads per SM); N = 8192, L = 4: 97 -> 46 and 146 -> 76 us against mixed radix.
//
// The instances compile as five objects (BFHE_EXT_PM_PART) in parallel.
#include "ext_device.cuh"

#ifndef BFHE_EXT_PM_PART
#define BFHE_EXT_PM_PART 0
#endif

namespace {

// constants of one extension sum from NS sources to ND targets: c[j][i] = (l, h) of c and (l, h) of 2^hs c, cv the
// constant that the overflow count v multiplies, d16 = 16 d of the target
template <int NS, int ND>
struct SumTab {
    uint4 c[ND][NS];
    uint2 cv[ND];
    uint32_t d16[ND];
    u64 guard;
};

template <int NS, int ND>
SumTab<NS, ND> sum_tab(const PmSum& h) {
    SumTab<NS, ND> t{};
    if (h.n != NS || h.m != ND) return t;   // only the instances the launchers use are ever filled
    for (int j = 0; j < ND; ++j) {
        for (int i = 0; i < NS; ++i) {
            const uint32_t* w = &h.c[((size_t)j * NS + i) * 4];
            t.c[j][i] = make_uint4(w[0], w[1], w[2], w[3]);
        }
        t.cv[j] = make_uint2(h.cv[2 * j], h.cv[2 * j + 1]);
        t.d16[j] = h.d[j] << 4;
    }
    t.guard = h.guard;
    return t;
}

template <int NS>
struct PrepTab {
    uint4 w[NS];      // (l, h) of (S/s_i)^-1 and (l, h) of 2^hs times it
    u64 q[NS];
    uint32_t d[NS];
};

template <int NS>
PrepTab<NS> prep_tab(const PmSum& h) {
    PrepTab<NS> t{};
    if (h.n != NS) return t;
    for (int i = 0; i < NS; ++i) {
        t.w[i] = make_uint4(h.w[4 * i], h.w[4 * i + 1], h.w[4 * i + 2], h.w[4 * i + 3]);
        t.q[i] = h.q[i];
        t.d[i] = h.dsrc[i];
    }
    return t;
}

// 2^k w as a pair of words
__device__ __forceinline__ u64 shl_word(uint32_t w, int k) { return ((u64)(w >> (32 - k)) << 32) | (w << k); }

// P + 2^k Q folded at bit b + 4
__device__ __forceinline__ u64 fold_sum(u64 P, u64 Q, int k, uint32_t d16) {
    return mad_wide_s((int)(Q >> 32), (int)d16, add64(P, shl_word((uint32_t)Q, k)));
}

// the integer v nearest to sum / 2^b; false within `guard` of a half
__device__ __forceinline__ bool round_sum(i64 sum, int b, u64 guard, int& v) {
    const u64 one = (u64)1 << b, z = (u64)sum + (one >> 1);
    v = (int)((i64)z >> b);
    return (z & (one - 1)) - guard < one - 2 * guard;
}

// the digits of one extension's sources
template <int NS>
struct Digits {
    uint32_t y0[NS];
    int y1[NS];
    i64 sum;
    __device__ __forceinline__ void set(int i, u64 y, int hs) {
        y0[i] = (uint32_t)y & ((1u << hs) - 1u);
        y1[i] = (int)__funnelshift_r((uint32_t)y, (uint32_t)(y >> 32), hs);
        sum = (i64)add64((u64)sum, y);
    }
    __device__ __forceinline__ bool round(int b, u64 guard, int& v) const { return round_sum(sum, b, guard, v); }
};

template <int NS, int ND>
__device__ __forceinline__ void sum_terms(const Digits<NS>& g, int v, const SumTab<NS, ND>& t, int j, u64& P, u64& Q) {
    P = mad_wide_s(v, (int)t.cv[j].x, P);
    Q = mad_wide_s(v, (int)t.cv[j].y, Q);
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        P = mad_wide_u(g.y0[i], t.c[j][i].x, P);
        Q = mad_wide_u(g.y0[i], t.c[j][i].y, Q);
        P = mad_wide_s(g.y1[i], (int)t.c[j][i].z, P);
        Q = mad_wide_s(g.y1[i], (int)t.c[j][i].w, Q);
    }
}

// the exact paths of one coefficient (mixed radix, as the kernels of more than 16 data primes): near a half only
__device__ __noinline__ void modup_exact(const u64* src, u64* dst, int N, int K, ExtDesc ext) {
    const int ns = ext.n_src;
    u64 x[NMAX], v[NMAX];
    for (int i = 0; i < ns; ++i) x[i] = src[(size_t)i * N];
    const bool neg = garner_n(x, ext, v, ns);
    for (int j = 0; j < K; ++j) dst[(size_t)(ns + j) * N] = ext_eval_n(v, neg, ext, j, ns, false);
}

struct ExactScale {
    ExtDesc eQB, eBQ;
    const u64 *twist, *Qinv_b, *bq;
    int nP;
};

__device__ __noinline__ void scale_exact(const u64* d, u64* o, int k, int N, int bits, ExactScale e) {
    const int ns = e.eQB.n_src, ks = e.eBQ.n_src;
    u64 r[NMAX], v[NMAX], y[NMAX];
    for (int i = 0; i < ns; ++i)
        r[i] = twist_mul(d[(size_t)i * N], twist_at(e.twist, i, 2, k, N), e.eQB.src_q[i], bits);
    const bool neg = garner_n(r, e.eQB, v, ns);
    for (int j = 0; j < ks; ++j) {
        const u64 bj = e.bq[j];
        const int pj = ns + (e.nP - 1 - ns - ks) + j;
        const u64 td = twist_mul(d[(size_t)(ns + j) * N], twist_at(e.twist, pj, 2, k, N), bj, bits);
        const u64 rb = ext_eval_n(v, neg, e.eQB, j, ns, false);
        y[j] = shoup_lazy(td + bj - rb, e.Qinv_b[j], e.Qinv_b[ks + j], bj);
    }
    const bool negy = garner_n(y, e.eBQ, v, ks);
    for (int i = 0; i < ns; ++i) o[(size_t)i * N] = ext_eval_n(v, negy, e.eBQ, i, ks, false);
}

// B limbs of X[c][slot]: the centred extension, not canonical (the forward transform reduces): below 2^60 up to 52 bits,
// folded below 2^(b+1) above
template <int NS>
__global__ void __launch_bounds__(256, NS <= 8 ? 4 : 2)
    k_modup_pm(const u64* A, const u64* B, u64* X, int n, int slots, int logN, int b,
               ExtDesc ext, uint32_t* flags, const __grid_constant__ PrepTab<NS> p,
               const __grid_constant__ SumTab<NS, NS + 1> t) {
    pdl_begin();
    constexpr int KS = NS + 1, LK = NS + KS;
    const int N = 1 << logN, k = b - 28, hs = (b + 2) >> 1;
    const size_t total = (size_t)n * slots << logN;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int kk = (int)(idx & (N - 1));
        const uint32_t pp = (uint32_t)(idx >> logN);
        const uint32_t c = slots == 4 ? pp >> 2 : pp >> 1;   // 4 (a0 a1 b0 b1) or 2 (squaring)
        const int slot = (int)(pp & (slots - 1));
        const u64* src = (slot < 2 ? A : B) + ((size_t)(c * 2 + (slot & 1)) * NS << logN) + kk;
        u64* dst = X + ((size_t)(c * 4 + slot) * LK << logN) + kk;
        u64 x[NS];
#pragma unroll
        for (int i = 0; i < NS; ++i) x[i] = src[(size_t)i << logN];
        Digits<NS> g;
        g.sum = 0;
        bool bad = false;
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            bad |= x[i] >= p.q[i];
            // x cut at bit hs; folded at bit b: below 2^b + 2^(hs+1) d + 2^(hs+k+1)
            const uint32_t x0 = (uint32_t)x[i] & ((1u << hs) - 1u);
            const uint32_t x1 = __funnelshift_r((uint32_t)x[i], (uint32_t)(x[i] >> 32), hs);
            u64 Q = (u64)x0 * p.w[i].y;
            Q = mad_wide_u(x1, p.w[i].w, Q);
            u64 y = shl_word((uint32_t)Q & 0xFFFFFFFu, k);
            y = mad_wide_u(x0, p.w[i].x, y);
            y = mad_wide_u(x1, p.w[i].z, y);
            y = mad_wide_u(__funnelshift_r((uint32_t)Q, (uint32_t)(Q >> 32), 28), p.d[i], y);
            g.set(i, y, hs);
        }
        if (bad) atomicOr(flags, BFHE_FLAG_RESIDUE);
        int v;
        if (!g.round(b, t.guard, v)) {
            modup_exact(src, dst, N, KS, ext);
            continue;
        }
#pragma unroll 1
        for (int j = 0; j < KS; ++j) {
            u64 P = 0, Q = 0;
            sum_terms<NS, KS>(g, v, t, j, P, Q);
            u64 r = fold_sum(P, Q, k, t.d16[j]);
            if (b > 52) r = pm_fold(r, b, t.d16[j] >> 4);
            dst[(size_t)(NS + j) << logN] = r;
        }
    }
}

// y_i of scale-and-round's first extension from the untwisted tensor words d (signed, below 2^63 in magnitude)
template <int NS>
__device__ __forceinline__ void scale_digits(const u64* d, const ulonglong2* f, int logN, int b, const uint32_t (&d16)[NS],
                                             Digits<NS>& g) {
    const int k = b - 28, hs = (b + 2) >> 1;
    u64 w[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) w[i] = d[(size_t)i << logN];
    g.sum = 0;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const ulonglong2 e = __ldg(f + ((size_t)i << logN));
        const uint32_t a0 = (uint32_t)w[i];
        const int a1 = (int)(w[i] >> 32);
        u64 Q = (u64)a0 * (uint32_t)(e.x >> 32);
        Q = mad_wide_s(a1, (int)(e.y >> 32), Q);
        u64 P = shl_word((uint32_t)Q, k);
        P = mad_wide_u(a0, (uint32_t)e.x, P);
        P = mad_wide_s(a1, (int)(uint32_t)e.y, P);
        P = mad_wide_s((int)(Q >> 32), (int)d16[i], P);
        g.set(i, pm_fold(P, b, d16[i] >> 4), hs);
    }
}

// the digit z_j = [(t d - r) / Q (B/b_j)^-1]_{b_j}: the tensor word w times its twist entry, and the sum over y
template <int NS>
__device__ __forceinline__ u64 scale_term(u64 w, const ulonglong2& e, const Digits<NS>& g, int v,
                                          const SumTab<NS, NS + 1>& t, int j, int b) {
    const uint32_t a0 = (uint32_t)w;
    const int a1 = (int)(w >> 32);
    u64 P = (u64)a0 * (uint32_t)e.x, Q = (u64)a0 * (uint32_t)(e.x >> 32);
    P = mad_wide_s(a1, (int)(uint32_t)e.y, P);
    Q = mad_wide_s(a1, (int)(e.y >> 32), Q);
    sum_terms<NS, NS + 1>(g, v, t, j, P, Q);
    return pm_fold(fold_sum(P, Q, b - 28, t.d16[j]), b, t.d16[j] >> 4);
}

template <int NS>
__device__ __forceinline__ u64 scale_out(const Digits<NS + 1>& z, int v, const SumTab<NS + 1, NS>& t, int i, int b) {
    u64 P = 0, Q = 0;
    sum_terms<NS + 1, NS>(z, v, t, i, P, Q);
    const uint32_t d = t.d16[i] >> 4;
    return pm_canon(fold_sum(P, Q, b - 28, t.d16[i]), ((u64)1 << b) - d, b, d);
}

// scale-and-round of the untwisted tensor (X slots 0..2, signed words over Q u B) into C3 [n][3][L][N], one pass: every
// loop unrolled, so that the constants are operands and the digits stay in registers
template <int NS>
__global__ void __launch_bounds__(256, 2)
    k_scale_pm(const u64* X, u64* C3, int n, int logN, int b, const ulonglong2* __restrict__ xtw,
               const __grid_constant__ SumTab<NS, NS + 1> tq, const __grid_constant__ SumTab<NS + 1, NS> tb,
               const __grid_constant__ ExactScale ex) {
    pdl_begin();
    constexpr int KS = NS + 1, LK = NS + KS;
    const int N = 1 << logN, hs = (b + 2) >> 1;
    const size_t total = (size_t)n * 3 << logN;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int kk = (int)(idx & (N - 1));
        const uint32_t cp = (uint32_t)(idx >> logN);
        const uint32_t c = cp / 3, comp = cp - 3 * c;
        const u64* d = X + ((size_t)(c * 4 + comp) * LK << logN) + kk;
        u64* o = C3 + ((size_t)cp * NS << logN) + kk;
        const ulonglong2* f = xtw + kk;
        Digits<NS> g;
        scale_digits<NS>(d, f, logN, b, tb.d16, g);
        int v;
        bool ok = g.round(b, tq.guard, v);
        Digits<KS> z;
        z.sum = 0;
#pragma unroll
        for (int j = 0; j < KS; ++j) {
            const size_t l = (size_t)(NS + j) << logN;
            z.set(j, scale_term<NS>(d[l], __ldg(f + l), g, v, tq, j, b), hs);
        }
        ok = z.round(b, tb.guard, v) && ok;
        if (!ok) {
            scale_exact(d, o, kk, N, b, ex);
            continue;
        }
#pragma unroll
        for (int i = 0; i < NS; ++i) o[(size_t)i << logN] = scale_out<NS>(z, v, tb, i, b);
    }
}

// The same in two passes above 8 data primes, where one pass needs more registers than two CTAs per SM have: pass A
// writes the digits z to Z [n][3][K][N], pass B extends them.  Near a half pass A leaves z_0 = 2^62, which pass B takes
// as the mark for the exact path.  (8 squarings at N = 32768, L = 16: 256 us; loops over the targets at run time, whose
// constants then take a load each, 360; one pass that sums each digit into all targets 297.)
constexpr u64 Z_EXACT = (u64)1 << 62;

template <int NS>
__global__ void __launch_bounds__(256, 2)
    k_scale_pm_a(const u64* X, u64* Z, int n, int logN, int b, const ulonglong2* __restrict__ xtw,
                 const __grid_constant__ SumTab<NS, NS + 1> tq, const __grid_constant__ SumTab<NS + 1, NS> tb) {
    pdl_begin();
    constexpr int KS = NS + 1, LK = NS + KS;
    const int N = 1 << logN;
    const size_t total = (size_t)n * 3 << logN;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int kk = (int)(idx & (N - 1));
        const uint32_t cp = (uint32_t)(idx >> logN);
        const uint32_t c = cp / 3, comp = cp - 3 * c;
        const u64* d = X + ((size_t)(c * 4 + comp) * LK << logN) + kk;
        u64* zo = Z + ((size_t)cp * KS << logN) + kk;
        const ulonglong2* f = xtw + kk;
        Digits<NS> g;
        scale_digits<NS>(d, f, logN, b, tb.d16, g);
        int v;
        if (!g.round(b, tq.guard, v)) {
            zo[0] = Z_EXACT;
            continue;
        }
        u64 next = d[(size_t)NS << logN];   // a word ahead: a load does not pass the store of the word before it
#pragma unroll
        for (int j = 0; j < KS; ++j) {
            const size_t l = (size_t)(NS + j) << logN;
            const u64 w = next;
            if (j + 1 < KS) next = d[(size_t)(NS + j + 1) << logN];
            zo[(size_t)j << logN] = scale_term<NS>(w, __ldg(f + l), g, v, tq, j, b);
        }
    }
}

template <int NS>
__global__ void __launch_bounds__(256, 2)
    k_scale_pm_b(const u64* X, const u64* Z, u64* C3, int n, int logN, int b,
                 const __grid_constant__ SumTab<NS + 1, NS> tb, const __grid_constant__ ExactScale ex) {
    pdl_begin();
    constexpr int KS = NS + 1, LK = NS + KS;
    const int N = 1 << logN, hs = (b + 2) >> 1;
    const size_t total = (size_t)n * 3 << logN;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int kk = (int)(idx & (N - 1));
        const uint32_t cp = (uint32_t)(idx >> logN);
        const uint32_t c = cp / 3, comp = cp - 3 * c;
        const u64* zi = Z + ((size_t)cp * KS << logN) + kk;
        u64* o = C3 + ((size_t)cp * NS << logN) + kk;
        u64 w[KS];
#pragma unroll
        for (int j = 0; j < KS; ++j) w[j] = zi[(size_t)j << logN];
        Digits<KS> z;
        z.sum = 0;
#pragma unroll
        for (int j = 0; j < KS; ++j) z.set(j, w[j], hs);
        int v;
        if (w[0] == Z_EXACT || !z.round(b, tb.guard, v)) {
            scale_exact(X + ((size_t)(c * 4 + comp) * LK << logN) + kk, o, kk, N, b, ex);
            continue;
        }
#pragma unroll
        for (int i = 0; i < NS; ++i) o[(size_t)i << logN] = scale_out<NS>(z, v, tb, i, b);
    }
}

// decryption's last step for t < 2^26: with y_i = [t (c0 + c1 s) (Q/q_i)^-1]_{q_i} and v nearest to sum y_i / q_i, the
// centred [t x]_Q is sum y_i (Q/q_i) - v Q and the plaintext -[t x]_Q / Q = v - sum y_i / q_i mod t.
template <int NS>
struct DecTab {
    uint4 w[NS];
    u64 q[NS];
    uint32_t d[NS], c[NS], c2[NS];
    u64 guard, t, mu, Qinv_t;
};

__device__ __noinline__ u64 dec_exact(const u64* V, const u64* c0, int N, ExtDesc e, const u64* tmod, int nP, u64 Qinv_t) {
    const int ns = e.n_src;
    u64 r[NMAX], v[NMAX];
    for (int i = 0; i < ns; ++i)
        r[i] = shoup(add_mod(V[(size_t)i * N], c0[(size_t)i * N], e.src_q[i]), tmod[i], tmod[nP + i], e.src_q[i]);
    const bool neg = garner_n(r, e, v, ns);
    const u64 t = e.dst_q[0], rho = ext_eval_n(v, neg, e, 0, ns, true);
    return ((rho == 0 ? 0 : t - rho) * Qinv_t) % t;
}

template <int NS>
__global__ void __launch_bounds__(256, 4)
    k_dec_pm(const u64* V, const u64* ct, u64* M, int n, int logN, int b, ExtDesc ext,
             const u64* tmod, int nP, uint32_t* flags, const __grid_constant__ DecTab<NS> p) {
    pdl_begin();
    const int k = b - 28, hs = (b + 2) >> 1;
    const size_t total = (size_t)n << logN;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int kk = (int)(idx & ((1u << logN) - 1u));
        const size_t c = idx >> logN;
        const u64* vp = V + (c * NS << logN) + kk;
        const u64* cp = ct + (c * 2 * NS << logN) + kk;
        u64 x[NS];
        bool bad = false;
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            const u64 c0 = cp[(size_t)i << logN];
            bad |= c0 >= p.q[i];
            x[i] = vp[(size_t)i << logN] + c0;
        }
        if (bad) atomicOr(flags, BFHE_FLAG_RESIDUE);
        i64 sum = 0;
        u64 z = p.t << 26;   // the digits may be slightly negative
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            const uint32_t a0 = (uint32_t)x[i];
            const int a1 = (int)(x[i] >> 32);
            u64 Q = (u64)a0 * p.w[i].y;
            Q = mad_wide_s(a1, (int)p.w[i].w, Q);
            u64 P = shl_word((uint32_t)Q, k);
            P = mad_wide_u(a0, p.w[i].x, P);
            P = mad_wide_s(a1, (int)p.w[i].z, P);
            P = mad_wide_s((int)(Q >> 32), (int)(p.d[i] << 4), P);
            const u64 y = pm_fold(P, b, p.d[i]);
            sum = (i64)add64((u64)sum, y);
            z = mad_wide_u((uint32_t)y & ((1u << hs) - 1u), p.c[i], z);
            z = mad_wide_s((int)__funnelshift_r((uint32_t)y, (uint32_t)(y >> 32), hs), (int)p.c2[i], z);
        }
        int v;
        if (!round_sum(sum, b, p.guard, v)) {
            M[idx] = dec_exact(vp, cp, 1 << logN, ext, tmod, nP, p.Qinv_t);
            continue;
        }
        M[idx] = reduce64((u64)((i64)v + (i64)(64 * p.t) - (i64)reduce64(z, p.t, p.mu)), p.t, p.mu);
    }
}

template <int NS>
int run_dec_pm(const bfhe_ctx* ctx, const u64* V, const u64* ct, u64* M, int n, cudaStream_t st) {
    const PmDec& h = ctx->pm_dec;
    DecTab<NS> t{};
    for (int i = 0; i < NS; ++i) {
        t.w[i] = make_uint4(h.w[4 * i], h.w[4 * i + 1], h.w[4 * i + 2], h.w[4 * i + 3]);
        t.q[i] = h.q[i];
        t.d[i] = h.d[i];
        t.c[i] = h.c[i];
        t.c2[i] = h.c2[i];
    }
    t.guard = h.guard;
    t.t = ctx->t;
    t.mu = (u64)(((u128)1 << 64) / ctx->t);
    t.Qinv_t = ctx->Qinv_t;
    LAUNCH(k_dec_pm<NS>, (size_t)n * ctx->N, V, ct, M, n, (int)ctx->logN, (int)ctx->prime_bits, ctx->ext_Qt, ctx->d_tmod,
           (int)ctx->nP, ctx->d_flags, t);
    return BFHE_OK;
}

template <int NS>
int run_modup_pm(const bfhe_ctx* ctx, const u64* A, const u64* B, u64* X, int n, int slots, cudaStream_t st) {
    LAUNCH(k_modup_pm<NS>, (size_t)n * slots * ctx->N, A, B, X, n, slots, (int)ctx->logN, (int)ctx->prime_bits,
           ctx->ext_QB, ctx->d_flags, prep_tab<NS>(ctx->pm_up), (sum_tab<NS, NS + 1>(ctx->pm_up)));
    return BFHE_OK;
}

template <int NS>
int run_scale_pm(const bfhe_ctx* ctx, const u64* X, u64* C3, int n, cudaStream_t st, u64* tmp) {
    const ExactScale ex{ctx->ext_QB, ctx->ext_BQ, ctx->tab.twist, ctx->d_Qinv_b, ctx->tab.q + ctx->L + ctx->alpha,
                        (int)ctx->nP};
    const size_t work = (size_t)n * 3 * ctx->N;
    const int logN = (int)ctx->logN, b = (int)ctx->prime_bits;
    if constexpr (NS <= 8) {
        LAUNCH(k_scale_pm<NS>, work, X, C3, n, logN, b, ctx->d_xtw, (sum_tab<NS, NS + 1>(ctx->pm_toB)),
               (sum_tab<NS + 1, NS>(ctx->pm_toQ)), ex);
    } else {
        if (!tmp) return set_error(BFHE_EINVAL, "no room for the two-pass scale-and-round");
        LAUNCH(k_scale_pm_a<NS>, work, X, tmp, n, logN, b, ctx->d_xtw, (sum_tab<NS, NS + 1>(ctx->pm_toB)),
               (sum_tab<NS + 1, NS>(ctx->pm_toQ)));
        LAUNCH(k_scale_pm_b<NS>, work, X, tmp, C3, n, logN, b, (sum_tab<NS + 1, NS>(ctx->pm_toQ)), ex);
    }
    return BFHE_OK;
}

}  // namespace

// one part's numbers of data primes
#if BFHE_EXT_PM_PART == 0
#define PM_CASES(FN, ...)                                                                          \
    case 1: return FN<1>(__VA_ARGS__);                                                             \
    case 2: return FN<2>(__VA_ARGS__);                                                             \
    case 3: return FN<3>(__VA_ARGS__);                                                             \
    case 4: return FN<4>(__VA_ARGS__);                                                             \
    case 5: return FN<5>(__VA_ARGS__);                                                             \
    case 6: return FN<6>(__VA_ARGS__);                                                             \
    case 7: return FN<7>(__VA_ARGS__);                                                             \
    case 8: return FN<8>(__VA_ARGS__);
#define PM_NAME(f) f##_0
#elif BFHE_EXT_PM_PART == 1
#define PM_CASES(FN, ...)                                                                          \
    case 9: return FN<9>(__VA_ARGS__);                                                             \
    case 10: return FN<10>(__VA_ARGS__);                                                           \
    case 11: return FN<11>(__VA_ARGS__);                                                           \
    case 12: return FN<12>(__VA_ARGS__);
#define PM_NAME(f) f##_1
#elif BFHE_EXT_PM_PART == 2
#define PM_CASES(FN, ...)                                                                          \
    case 13: return FN<13>(__VA_ARGS__);                                                           \
    case 14: return FN<14>(__VA_ARGS__);
#define PM_NAME(f) f##_2
#elif BFHE_EXT_PM_PART == 3
#define PM_CASES(FN, ...) \
    case 15: return FN<15>(__VA_ARGS__);
#define PM_NAME(f) f##_3
#else
#define PM_CASES(FN, ...) \
    case 16: return FN<16>(__VA_ARGS__);
#define PM_NAME(f) f##_4
#endif

int PM_NAME(modup_pm)(const bfhe_ctx* ctx, const u64* A, const u64* B, u64* X, int n, int slots, cudaStream_t st) {
    switch (ctx->L) {
        PM_CASES(run_modup_pm, ctx, A, B, X, n, slots, st)
        default: return set_error(BFHE_EINVAL, "unsupported number of data primes");
    }
}

int PM_NAME(scale_pm)(const bfhe_ctx* ctx, const u64* X, u64* C3, int n, cudaStream_t st, u64* tmp) {
    switch (ctx->L) {
        PM_CASES(run_scale_pm, ctx, X, C3, n, st, tmp)
        default: return set_error(BFHE_EINVAL, "unsupported number of data primes");
    }
}

int PM_NAME(dec_pm)(const bfhe_ctx* ctx, const u64* V, const u64* ct, u64* M, int n, cudaStream_t st) {
    switch (ctx->L) {
        PM_CASES(run_dec_pm, ctx, V, ct, M, n, st)
        default: return set_error(BFHE_EINVAL, "unsupported number of data primes");
    }
}

#if BFHE_EXT_PM_PART == 0
#define PM_DECLARE(p)                                                                                               \
    int modup_pm_##p(const bfhe_ctx* ctx, const u64* A, const u64* B, u64* X, int n, int slots, cudaStream_t st);  \
    int scale_pm_##p(const bfhe_ctx* ctx, const u64* X, u64* C3, int n, cudaStream_t st, u64* tmp);                 \
    int dec_pm_##p(const bfhe_ctx* ctx, const u64* V, const u64* ct, u64* M, int n, cudaStream_t st);
PM_DECLARE(1) PM_DECLARE(2) PM_DECLARE(3) PM_DECLARE(4)

static int pm_part(uint32_t L) { return L <= 8 ? 0 : L <= 12 ? 1 : L <= 14 ? 2 : L == 15 ? 3 : 4; }

int launch_modup_pm(const bfhe_ctx* ctx, const u64* A, const u64* B, u64* X, int n, int slots, cudaStream_t st) {
    switch (pm_part(ctx->L)) {
        case 0: return modup_pm_0(ctx, A, B, X, n, slots, st);
        case 1: return modup_pm_1(ctx, A, B, X, n, slots, st);
        case 2: return modup_pm_2(ctx, A, B, X, n, slots, st);
        case 3: return modup_pm_3(ctx, A, B, X, n, slots, st);
        default: return modup_pm_4(ctx, A, B, X, n, slots, st);
    }
}

int launch_scale_pm(const bfhe_ctx* ctx, const u64* X, u64* C3, int n, cudaStream_t st, u64* tmp) {
    switch (pm_part(ctx->L)) {
        case 0: return scale_pm_0(ctx, X, C3, n, st, tmp);
        case 1: return scale_pm_1(ctx, X, C3, n, st, tmp);
        case 2: return scale_pm_2(ctx, X, C3, n, st, tmp);
        case 3: return scale_pm_3(ctx, X, C3, n, st, tmp);
        default: return scale_pm_4(ctx, X, C3, n, st, tmp);
    }
}

int launch_dec_pm(const bfhe_ctx* ctx, const u64* V, const u64* ct, u64* M, int n, cudaStream_t st) {
    switch (pm_part(ctx->L)) {
        case 0: return dec_pm_0(ctx, V, ct, M, n, st);
        case 1: return dec_pm_1(ctx, V, ct, M, n, st);
        case 2: return dec_pm_2(ctx, V, ct, M, n, st);
        case 3: return dec_pm_3(ctx, V, ct, M, n, st);
        default: return dec_pm_4(ctx, V, ct, M, n, st);
    }
}
#endif

// common.cuh -- shared definitions of the bfhe CUDA library (sm_103a).
//
// Exact 64-bit modular arithmetic for RNS BFV on the integer pipe: for moduli
// 2^b - d of 45 to 55 bits, products and sums of products folded by 2^b = d;
// otherwise Shoup products for multiplications by precomputed constants
// (twiddles, CRT constants) and Montgomery reduction (REDC) for products of
// two runtime values and for lazily accumulated sums of them.  Every modulus
// is an odd prime below 2^60.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/bfhe.h"

typedef uint64_t u64;
typedef int64_t i64;
typedef unsigned __int128 u128;

// up to 16 data primes every kernel has a compiled instance per size; 17..32 (insecure, test-only
// parameter sets for deep circuits) run runtime-size variants of the base extensions and the inner product
#define BFHE_MAX_L 32
#define BFHE_MAX_L_UNROLLED 16
#define BFHE_MAX_ALPHA 2
#define BFHE_MAX_PRIMES 80
#define BFHE_MAX_DEVICES 64

// ------------------------------------------------------------------ device modular arithmetic
__host__ __device__ __forceinline__ u64 mulhi64(u64 a, u64 b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (u64)(((u128)a * b) >> 64);
#endif
}

__host__ __device__ __forceinline__ u64 add_mod(u64 a, u64 b, u64 q) {
    u64 s = a + b;
    return s >= q ? s - q : s;
}

__host__ __device__ __forceinline__ u64 sub_mod(u64 a, u64 b, u64 q) { return a >= b ? a - b : a + q - b; }

// a * w mod q in [0, 2q) for any a < 2^64, w < q, ws = floor(w 2^64 / q) (Shoup).
__host__ __device__ __forceinline__ u64 shoup_lazy(u64 a, u64 w, u64 ws, u64 q) {
    return a * w - mulhi64(a, ws) * q;
}

// a * w mod q in [0, 4q) for a < 2^64: the quotient estimate keeps a1 w1 and the high
// halves of the two cross products a1 w0, a0 w1 (their low halves and a0 w0 together are
// below 3 2^64), so it is floor(a ws / 2^64) minus 0, 1 or 2, and Shoup's own estimate
// is the true quotient or one less.  The modulus is passed negated (nq = 2^64 - q):
// r = a w + h nq mod 2^64, written in 32-bit pieces so that each partial product is one
// multiply-add (the low word of a0 w0 + h0 nq0 as one wide multiply-add, the high word as
// four narrow ones).
__device__ __forceinline__ u64 shoup_lazy4n(u64 a, u64 w, u64 ws, u64 nq) {
    const uint32_t a0 = (uint32_t)a, a1 = (uint32_t)(a >> 32), s0 = (uint32_t)ws, s1 = (uint32_t)(ws >> 32);
    u64 h = (u64)a1 * s1 + __umulhi(a1, s0);
    h += __umulhi(a0, s1);
    const uint32_t h0 = (uint32_t)h, h1 = (uint32_t)(h >> 32);
    const uint32_t w0 = (uint32_t)w, w1 = (uint32_t)(w >> 32), n0 = (uint32_t)nq, n1 = (uint32_t)(nq >> 32);
    u64 r = (u64)a0 * w0;
    r += (u64)h0 * n0;
    const uint32_t rh = (uint32_t)(r >> 32) + a0 * w1 + a1 * w0 + h0 * n1 + h1 * n0;
    return ((u64)rh << 32) | (uint32_t)r;
}

__host__ __device__ __forceinline__ u64 shoup(u64 a, u64 w, u64 ws, u64 q) {
    u64 r = shoup_lazy(a, w, ws, q);
    return r >= q ? r - q : r;
}

// Montgomery reduction: z = hi 2^64 + lo < q 2^64, qinv = -q^-1 mod 2^64;
// returns z 2^-64 mod q in [0, q).
__host__ __device__ __forceinline__ u64 redc(u64 hi, u64 lo, u64 q, u64 qinv) {
    u64 m = lo * qinv;
    u64 t = hi + mulhi64(m, q) + (lo != 0 ? 1ull : 0ull);
    return t >= q ? t - q : t;
}

// 128-bit accumulate of a * b
__host__ __device__ __forceinline__ void mac128(u64& hi, u64& lo, u64 a, u64 b) {
    u64 l = a * b;
    u64 h = mulhi64(a, b);
    lo += l;
    hi += h + (lo < l ? 1ull : 0ull);
}

// x mod q for any 64-bit x, mu = floor(2^64 / q).
__host__ __device__ __forceinline__ u64 reduce64(u64 x, u64 q, u64 mu) {
    u64 r = x - mulhi64(x, mu) * q;
    return r >= q ? r - q : r;
}

// ------------------------------------------------------------------ products modulo q = 2^b - d
// The parameter rule scans downwards from 2^b, so every modulus is q = 2^b - d with d below 2^27, and 2^(b+2) = 4d
// (mod q).  A product by a constant w takes the table entry e of w: with v = 2^32 w mod q and both cut at bit
// k = b - 30, e.x = wl | wh << 32, e.y = vl | vh << 32 (wl, vl < 2^k; wh, vh < 2^30).  For a = a1 2^32 + a0 (a signed
// 64-bit word, a0 its unsigned low half)
//   a w = a0 w + a1 v = P + 2^k Q,   P = a0 wl + a1 vl,   Q = a0 wh + a1 vh = qh 2^32 + ql,
//   pm_mul = P + 2^k ql + 4d qh,
// signed, congruent to a w and below 3 2^29 4d + 2^(b+3.4) in magnitude for |a| < 2^63: five 32 x 32 -> 64-bit
// multiply-adds and two shifts.  Shoup's product above takes five wide and four narrow ones; on this chip a wide
// multiply holds the multiplier pipe four cycles per warp and scheduler, a narrow one or any other operation two, so the
// pipe is the bound of every transform: 9.7 -> 7.0 SM cycles per warp butterfly (registers only, GB300).
__device__ __forceinline__ u64 mad_wide_u(uint32_t a, uint32_t b, u64 c) {
    // as a carry pair: one wide multiply-add (the 64-bit form compiles to a multiply, an add and a move)
    uint32_t lo = (uint32_t)c, hi = (uint32_t)(c >> 32);
    asm("mad.lo.cc.u32 %0, %2, %3, %0;\n\tmadc.hi.u32 %1, %2, %3, %1;" : "+r"(lo), "+r"(hi) : "r"(a), "r"(b));
    return ((u64)hi << 32) | lo;
}
__device__ __forceinline__ u64 mad_wide_s(int a, int b, u64 c) {
    uint32_t lo = (uint32_t)c, hi = (uint32_t)(c >> 32);
    asm("mad.lo.cc.s32 %0, %2, %3, %0;\n\tmadc.hi.s32 %1, %2, %3, %1;" : "+r"(lo), "+r"(hi) : "r"(a), "r"(b));
    return ((u64)hi << 32) | lo;
}
__device__ __forceinline__ u64 add64(u64 a, u64 b) {
    uint32_t lo, hi;
    asm("add.cc.u32 %0, %2, %4;\n\taddc.u32 %1, %3, %5;"
        : "=r"(lo), "=r"(hi)
        : "r"((uint32_t)a), "r"((uint32_t)(a >> 32)), "r"((uint32_t)b), "r"((uint32_t)(b >> 32)));
    return ((u64)hi << 32) | lo;
}
__device__ __forceinline__ u64 sub64(u64 a, u64 b) {
    uint32_t lo, hi;
    asm("sub.cc.u32 %0, %2, %4;\n\tsubc.u32 %1, %3, %5;"
        : "=r"(lo), "=r"(hi)
        : "r"((uint32_t)a), "r"((uint32_t)(a >> 32)), "r"((uint32_t)b), "r"((uint32_t)(b >> 32)));
    return ((u64)hi << 32) | lo;
}
__device__ __forceinline__ u64 pm_mul(u64 a, ulonglong2 e, int k, uint32_t d4) {
    const uint32_t a0 = (uint32_t)a;
    const int a1 = (int)(a >> 32);
    u64 Q = (u64)a0 * (uint32_t)(e.x >> 32);
    Q = mad_wide_s(a1, (int)(e.y >> 32), Q);
    const uint32_t ql = (uint32_t)Q;
    u64 T = ((u64)(ql >> (32 - k)) << 32) | (ql << k);
    T = mad_wide_u(a0, (uint32_t)e.x, T);
    T = mad_wide_s(a1, (int)(uint32_t)e.y, T);
    return mad_wide_s((int)(Q >> 32), (int)d4, T);
}
// signed x = h 2^b + l (0 <= l < 2^b) to the congruent h d + l, above -2^(63-b) d and below 2^b + 2^(63-b) d
__device__ __forceinline__ u64 pm_fold(u64 x, int b, uint32_t d) {
    const int xh = (int)(x >> 32);
    const u64 l = ((u64)((uint32_t)xh & ((1u << (b - 32)) - 1u)) << 32) | (uint32_t)x;
    return mad_wide_s(xh >> (b - 32), (int)d, l);
}
// a signed 64-bit word to its residue below 2^b + 2^(63-b) d < 2q (non-negative)
__device__ __forceinline__ u64 pm_lazy(u64 x, u64 q, int b, uint32_t d) {
    const u64 y = pm_fold(x, b, d);
    return add64(y, (u64)((i64)y >> 63) & q);
}
// to the canonical residue
__device__ __forceinline__ u64 pm_canon(u64 x, u64 q, int b, uint32_t d) {
    const u64 y = pm_lazy(x, q, b, d);
    return y >= q ? y - q : y;
}
// Sums of products of run-time factors x, y cut at bit hs = (b + 2) / 2 (x = x1 2^hs + x0): p00, pm, p11 the sums of
// x0 y0, x0 y1 + x1 y0, x1 y1, below 2^61 and p11 2^(2 hs - b) below 2^60.  With H = floor(pm / 2^(b - hs)) +
// p11 2^(2 hs - b) the sum is p00 + (pm mod 2^(b - hs)) 2^hs + H 2^b, folded by H 2^b = H d twice: signed, below 2^62.
__device__ __forceinline__ u64 pm_fold3(u64 p00, u64 pm, u64 p11, int b, uint32_t d) {
    const int hs = (b + 2) >> 1, s = b - 32;
    const u64 H = (pm >> (b - hs)) + (p11 << (2 * hs - b));
    const u64 g = (u64)(uint32_t)(H >> 32) * d;   // weight 2^32
    u64 r = p00 + ((pm & (((u64)1 << (b - hs)) - 1)) << hs) + ((u64)((uint32_t)g & ((1u << s) - 1u)) << 32);
    r = mad_wide_u((uint32_t)H, d, r);
    return mad_wide_u((uint32_t)(g >> s), d, r);
}
// a b mod q, canonical, for two run-time factors below 2^(bits+1): the 128-bit product folded three times (eight wide
// multiplies against Montgomery's ten and their carries)
__device__ __forceinline__ u64 pm_mul_var(u64 a, u64 b, u64 q, int bits, uint32_t d) {
    const uint32_t a0 = (uint32_t)a, a1 = (uint32_t)(a >> 32), b0 = (uint32_t)b, b1 = (uint32_t)(b >> 32);
    const u64 lo = (u64)a0 * b0;
    u64 m = mad_wide_u(a1, b0, lo >> 32);      // below 2^57 + 2^32
    m = mad_wide_u(a0, b1, m);
    const u64 top = mad_wide_u(a1, b1, m >> 32);
    const int s = bits - 32;
    // product = H 2^bits + (m mod 2^s) 2^32 + lo: H = h1 2^32 + h0
    const uint32_t h0 = __funnelshift_r((uint32_t)m, (uint32_t)top, s), h1 = (uint32_t)(top >> s);
    const u64 g = (u64)h1 * d;                 // weight 2^32: g = (g >> s) 2^s + f, 2^(s + 32) = 2^bits
    u64 r = ((u64)(((uint32_t)m & ((1u << s) - 1u))) << 32) | (uint32_t)lo;
    r += (u64)((uint32_t)g & ((1u << s) - 1u)) << 32;
    r = mad_wide_u(h0, d, r);
    r = mad_wide_u((uint32_t)(g >> s), d, r);  // below 2^60
    return pm_canon(r, q, bits, d);
}
// host: x mod q for q = 2^b - d with d below 2^27 and x below 2^(2b) (folds; a 128-bit division takes several times longer
// and a context's tables need one per entry)
inline u64 pm_reduce(u128 x, u64 q) {
    const int b = 64 - __builtin_clzll(q);
    const u64 d = ((u64)1 << b) - q, mask = ((u64)1 << b) - 1;
    while (x >> b) x = (x >> b) * d + ((u64)x & mask);
    u64 r = (u64)x;
    while (r >= q) r -= q;
    return r;
}
// host: the table entry of w, cut at bit k (b - 30 for pm_mul)
inline void pm_entry(u64 w, u64 q, int k, u64* x, u64* y) {
    const u64 m = ((u64)1 << k) - 1, v = pm_reduce((u128)w << 32, q);
    *x = (w & m) | ((w >> k) << 32);
    *y = (v & m) | ((v >> k) << 32);
}

// ------------------------------------------------------------------ exact base extension tables
// Centred extension of an integer given by residues modulo the source primes
// s_0..s_{n-1} (S = prod s_i) to target primes T_0..T_{m-1}: Garner's mixed
// radix digits v_i, a lexicographic compare of (v_{n-1}..v_0) against the
// digits of (S-1)/2 to decide x > S/2, Horner evaluation mod T_j and a
// subtraction of [S]_{T_j} for the negative half.
struct ExtDesc {
    int n_src, n_dst;
    const u64* src_q;    // [n_src]
    const u64* ginv;     // [n_src][n_src]: (i, j<i) -> s_j^-1 mod s_i   (Shoup pair w, ws)
    const u64* ginv_s;
    const u64* hdig;     // [n_src] mixed-radix digits of (S-1)/2
    const u64* dst_q;    // [n_dst]
    const u64* dst_mu;   // [n_dst] floor(2^64 / T_j)
    const u64* radix;    // [n_dst][n_src]: [s_i]_{T_j} (Shoup pair)
    const u64* radix_s;
    const u64* smod;     // [n_dst]: [S]_{T_j}
    // guarded fast path (all moduli < 2^50): x = sum_i y_i (S/s_i) - v S with y_i = [x_i (S/s_i)^-1]_{s_i}
    // and v = round(sum_i y_i / s_i) from a 64.64 fixed-point sum, unless that sum lies within
    // 2 n_src + 2 units of 1/2 (then the exact mixed-radix path decides)
    const u64* qhinv;    // [n_src] [(S/s_i)^-1]_{s_i} (Shoup pair)
    const u64* qhinv_s;
    const u64* g_hi;     // [n_src] floor(2^128 / s_i) >> 64
    const u64* g_lo;     // [n_src] floor(2^128 / s_i) mod 2^64
    const uint32_t* c26; // [n_dst][n_src][2] 26-bit limbs (low, high) of [(S/s_i) 2^64]_{T_j}
    const u64* dst_qinv; // [n_dst] -T_j^-1 mod 2^64
    const u64* vS;       // [n_dst][n_src + 1] [v S]_{T_j}
    int fast_ok;         // all moduli < 2^50: the fast path's tables are valid
};

// Host copies of the guarded fast extension's per-source tables and 26-bit limb pairs: the kernels take them
// as a kernel parameter (constant bank), so that the inner products read their factors without a load
struct ExtHost {
    int n = 0, m = 0;
    std::vector<uint32_t> c26;                       // [m][n][2]
    std::vector<u64> qhinv, qhinv_s, g_hi, g_lo;     // [n]
};

// Host constants of an extension sum for moduli 2^b - d (ext_pm.cu): words cut at bit k = b - 28
struct PmSum {
    int n = 0, m = 0;
    std::vector<uint32_t> c;          // [m][n][4] (l, h) of the constant and of 2^hs times it, hs = (b + 2) / 2
    std::vector<uint32_t> cv, d;      // [m][2] the overflow count's constant, [m] d of the target
    std::vector<uint32_t> w, dsrc;    // [n][4] (S/s_i)^-1 in the same form, [n] d of the source
    std::vector<u64> q;               // [n]
    u64 guard = 0;                    // bound of 2^b |sum y_i / s_i - sum y_i / 2^b|
};

// Host constants of decryption's last step in the same arithmetic, for t below 2^26: t (Q/q_i)^-1 mod q_i as (l, h) of it
// and of 2^32 times it, 1/q_i and 2^hs/q_i mod t
struct PmDec {
    std::vector<uint32_t> w, d, c, c2;   // [n][4], [n], [n], [n]
    std::vector<u64> q;
    u64 guard = 0;
};

// Device-side prime tables of a context, by prime index
// (0..L-1 data, L..L+alpha-1 special, L+alpha..L+alpha+K-1 auxiliary, last: t).  The pairs of tw, twl, itw and
// twist are pm_mul's entries for the moduli of a context with pm set, (w, Shoup(w)) otherwise and always for t.
struct PrimeTab {
    const u64* q;        // modulus
    const u64* qinv;     // -q^-1 mod 2^64
    const u64* mu;       // floor(2^64 / q)
    const u64* tw;       // [nP][N][2] psi^brv(k)                         forward twiddles
    const u64* twl;      // [nP][3][N][2] the same, stages b < le regrouped per le = 3, 4, 5 (forward last pass)
    const u64* itw;      // [nP][N][2] inverse (DIT) twiddles: entry 2^b + j = omega^-(N/2^(b+1)) j, omega = psi^2
    const u64* twist;    // [nP][3][N][2] output twist N^-1 psi^-m (plain; times R = 2^64; times t R), mod q
};

// limb -> prime index map of a polynomial base: limb < split ? limb : limb + off
struct LimbMap {
    int split, off;
    __host__ __device__ __forceinline__ int operator()(int limb) const { return limb < split ? limb : limb + off; }
};

// ------------------------------------------------------------------ context
struct bfhe_ctx {
    int device = 0;
    uint32_t N = 0, logN = 0, L = 0, alpha = 0, K = 0, nP = 0, prime_bits = 0;
    u64 t = 0;
    bool pm = false;        // the moduli's products run as pm_mul: 45 to 55 bits, transforms bounded below 2^63
    bool batching = true;   // t = 1 mod 2N: slot encoding; t = 2: coefficient encoding only
    std::vector<u64> primes;     // nP: Q, P, B, t
    std::vector<uint32_t> brv;   // host copy of bit reversal (N)

    void* d_arena = nullptr;     // all constant tables
    size_t arena_bytes = 0;
    PrimeTab tab{};
    uint32_t* d_brv = nullptr;   // [N] storage position of slot j's evaluation
    ExtDesc ext_QB{}, ext_BQ{}, ext_PQ{}, ext_Qt{};
    ExtHost exth_QB, exth_BQ;
    // pm contexts of at most 16 data primes: the input extension, scale-and-round's two sums and its twist table
    // [L + K][N] (data: t R N^-1 psi^-k (Q/q_i)^-1; auxiliary: t R N^-1 psi^-k Q^-1 (B/b_j)^-1; words cut at b - 28)
    PmSum pm_up, pm_toB, pm_toQ;
    PmDec pm_dec;
    const ulonglong2* d_xtw = nullptr;
    // the same contexts' rounding division by P: twists N^-1 psi^-k P^-1 (data) and N^-1 psi^-k (special) [L + alpha][N],
    // and the constants of the special digits [L][alpha]: -P^-1, then -p_0 P^-1 (words cut at b - 28).  Their tensor and
    // key-switch inner product leave plain residues (no Montgomery factor).
    const ulonglong2 *d_mtw = nullptr, *d_mpc = nullptr;
    // Shoup pair tables: p[i] = w_i, p[n + i] = ws_i
    const u64* d_tmod = nullptr;    // [nP] [t]_{prime}
    const u64* d_delta_q = nullptr; // [L]  [Delta]_{q_i}
    const u64* d_Qinv_b = nullptr;  // [K]  [Q^-1]_{b_j}
    const u64* d_Pinv_q = nullptr;  // [L]  [P^-1]_{q_i}
    const u64* d_P_q = nullptr;     // [L]  [P]_{q_i}
    const u64* d_R2 = nullptr;      // [nP] 2^128 mod prime (Montgomery R^2)
    u64 Qinv_t = 0;                 // [Q^-1]_t
    u64 delta_t = 0;

    // keys
    bool have_keys = false;
    i64* d_sk = nullptr;         // [N]
    u64* d_sk_ntt = nullptr;     // [L+alpha][N]
    u64* d_pk = nullptr;         // [2][L][N] coefficient form
    u64* d_pk_ntt = nullptr;     // [2][L][N]
    u64* d_rlk_ntt = nullptr;    // [L][2][L+alpha][N]

    // input-range flags raised by kernels (BFHE_FLAG_*), read and cleared by bfhe_check
    uint32_t* d_flags = nullptr;

    // scratch
    void* scratch = nullptr;
    size_t scratch_bytes = 0;
    uint64_t scratch_gen = 0;    // arenas so far: kernels recorded in a CUDA graph hold the address of one
    size_t reserve_n = 0;

    uint64_t counts[4] = {0, 0, 0, 0};
    bool fast_ext = false;       // guarded fast base extension in the multiply (bfhe_set_fast_extension)
    bool fast_default = false;   // its setting when the context is made
    bool exact_ext = false;      // the caller has switched off a setting that is on by default: mixed radix everywhere
    bool pm_ext = false;         // the extensions of ext_pm.cu are available (at most 16 primes, pm)
    bool use_pm_ext() const { return pm_ext && !exact_ext; }

    // mod_to_bits tiles replayed from a CUDA graph (bfhe_set_graph_tiles): the tile is captured once on a
    // context-owned stream and replayed with its candidate base in the device word d_cbase; the
    // instantiated graph is kept for later calls with the same buffers and shape (key)
    bool graph_tiles = false;
    bool capturing = false;      // inside a stream capture: no profiling events
    cudaStream_t cap_stream = nullptr;
    cudaEvent_t cap_in = nullptr, cap_out = nullptr;
    u64* d_cbase = nullptr;
    cudaGraphExec_t tile_exec = nullptr;
    std::vector<u64> tile_key;
    uint64_t tile_counts[4] = {0, 0, 0, 0};   // op counts of one captured tile
    uint64_t tile_launches = 0;                // kernels in the captured tile

    // launch timing (measurement only): pending (class, start, stop) event triples
    struct ProfRec {
        int cls;
        double work, bytes;
        cudaEvent_t a, b;
    };
    mutable bool prof_on = false;
    mutable std::vector<ProfRec> prof_pending;
    mutable std::vector<cudaEvent_t> prof_pool;

    int pm_bits() const { return pm ? (int)prime_bits : 0; }
    LimbMap mapQ() const { return LimbMap{(int)L, 0}; }
    LimbMap mapQP() const { return LimbMap{(int)(L + alpha), 0}; }
    LimbMap mapQB() const { return LimbMap{(int)L, (int)alpha}; }
    LimbMap mapT() const { return LimbMap{0, (int)(L + alpha + K)}; }
    size_t ct_words() const { return (size_t)2 * L * N; }
};

// ------------------------------------------------------------------ host helpers (host.cu)
bool pm_bounded(uint32_t bits, uint32_t logN, u64 d);   // bfhe_ctx::pm of moduli 2^bits - d at ring degree 2^logN
int set_error(int code, const std::string& msg);
// process-wide count of kernel launches made by this library (measurement)
void count_launch();
void count_launches(uint64_t n);   // kernels launched by a graph replay
int cuda_check(cudaError_t e, const char* where);
#define BFHE_CUDA(call)                                          \
    do {                                                         \
        cudaError_t _e = (call);                                 \
        if (_e != cudaSuccess) return cuda_check(_e, #call);     \
    } while (0)
#define BFHE_LAUNCH_CHECK(where)                                 \
    do {                                                         \
        count_launch();                                          \
        cudaError_t _e = cudaGetLastError();                     \
        if (_e != cudaSuccess) return cuda_check(_e, where);     \
    } while (0)

// Every kernel of the library starts with pdl_begin and is launched with launch_kernel: the launch of a kernel, its
// blocks' arrival and its reads of constant tables overlap the tail of the one before it on the stream (programmatic
// dependent launch), and nothing that an earlier kernel writes, or still reads, is touched before pdl_wait returns, which
// is when that kernel has completed.  A kernel's buffers therefore change while it is resident: only the tables made with
// the context are read through __restrict__ or __ldg, whose loads the wait need not order; ciphertexts, scratch and keys
// (which key generation's kernels write) are plain pointers.  Measured on GB300, calls one after another: a multiply of one pair at N = 16384,
// L = 8 102 -> 81 us, of 64 pairs at N = 4096, L = 2 159 -> 145 us, of 64 at N = 16384 2510 -> 2491 us; one XOR gate at
// N = 4096 53 -> 37 us.  Inside a CUDA graph the plain dependency is the cheaper one (16-bit comparator at N = 4096
// replayed: 263 us, with programmatic edges 286), so a launch on a capturing stream leaves the attribute out.
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_begin() {
    pdl_next();
    pdl_wait();
}
template <class... P, class... A>
cudaError_t launch_kernel(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cluster_y, A&&... a) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const bool plain = cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone;
    at[0].val.programmaticStreamSerializationAllowed = plain ? 0 : 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = 1;
    at[1].val.clusterDim.y = cluster_y;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster_y > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(a)...);
}

// scratch arena: returns a pointer to at least `bytes` bytes (grows, syncing the device)
int ctx_scratch(bfhe_ctx* ctx, size_t bytes, void** out);
// bytes of scratch one mul_relin of n ciphertexts needs
size_t mul_scratch_bytes(const bfhe_ctx* ctx, size_t n);

// RAII bracket of one launcher's kernels by CUDA events when profiling is on
// (work = the launch's algorithmic 64-bit modular multiplies)
// work: algorithmic modmuls of the launch; bytes: its algorithmic DRAM bytes (each operand read and each
// result written once; tables that stay in L2 not counted)
struct ProfScope {
    const bfhe_ctx* c;
    int cls;
    double work, bytes;
    cudaStream_t st;
    cudaEvent_t a = nullptr, b = nullptr;
    ProfScope(const bfhe_ctx* ctx, int k, cudaStream_t s, double w, double by);
    ~ProfScope();
};

// ------------------------------------------------------------------ kernel launchers (ntt.cu)
// In/out-of-place negacyclic NTT over n_polys x n_limbs limbs.
// Poly p of a launch is (outer, inner) = (p / n_inner, p % n_inner); a limb's
// words start at base + outer*os + inner*is + limb*ls (strides in words).
struct NttIO {
    const u64* in;
    u64* out;
    int n_inner;
    size_t in_os, in_is, in_ls;
    size_t out_os, out_is, out_ls;
    bool natural = false;   // the evaluation side in bit-reversed index order (bfhe_ntt) rather than the storage order
    // forward only: limbs below src_limbs of poly (outer, inner) are read from src[inner >> 1], ciphertexts
    // [outer][2][src_limbs][N] of which inner & 1 selects the polynomial (the multiply's inputs, which need no copy)
    const u64* src[2] = {nullptr, nullptr};
    int src_limbs = 0;
    // inverse only, pm contexts, canonical outputs: every input word is first multiplied by the word of the same limb
    // and index of mul (poly (outer, inner) at outer mul_os + inner mul_is, limbs N words apart); factors below 2q
    const u64* mul = nullptr;
    size_t mul_os = 0, mul_is = 0;
};
// contiguous [n_polys][n_limbs][N] in and out
inline NttIO ntt_io(const u64* in, u64* out, size_t n_limbs, size_t N) {
    NttIO io;
    io.in = in;
    io.out = out;
    io.n_inner = 1;
    io.in_os = io.out_os = n_limbs * N;
    io.in_is = io.out_is = 0;
    io.in_ls = io.out_ls = N;
    return io;
}
// lazy_out: outputs left below 2q (pm contexts) or 64q (others, only taken when every prime is below 2^50) for
// consumers that multiply them in Montgomery form; otherwise canonical
int launch_ntt_fwd(const bfhe_ctx* ctx, NttIO io, int n_polys, int n_limbs, LimbMap map, cudaStream_t st,
                   int lazy_out = 0);
// mont != 0: the final scale is N^-1 R (undoes one Montgomery factor R^-1 of the inputs)
// lazy_out: 0 canonical; 2 no twist at all (words below 61q, or signed words below 2^63 in a pm context; from inputs
// below q) for consumers that fold the twist into a product of their own (scale-and-round, mod-down)
int launch_ntt_inv(const bfhe_ctx* ctx, NttIO io, int n_polys, int n_limbs, LimbMap map, int mont,
                   cudaStream_t st, int lazy_out = 0);
// shape of a launch of `limbs` limbs; pm: products modulo 2^b - d
int ntt_config(int logN, int inverse, bool pm, size_t limbs, int* log_m, int* log_e);

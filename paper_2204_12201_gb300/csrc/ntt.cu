// ntt.cu -- negacyclic NTT / INTT over Z_q[X]/(X^N + 1) per RNS prime.
//
// Forward: Cooley-Tukey with merged psi twiddles (natural order in, bit-
// reversed evaluation order out); butterfly on bit b of the index with
// twiddle psi^brv((N + j) >> (b + 1)) and one Shoup product.  The forward
// butterfly (X, Y) -> (X + T, X - T + 4q), T = Shoup(Y) in [0, 4q) (the
// quotient estimate may be up to three short, see shoup_lazy4n), grows the
// bound by 4q per stage and is never reduced in between: from inputs < 4q,
// 15 stages stay below 64q <= 2^64 for q < 2^58, and one Barrett-style
// reduction at the end makes the output canonical.  Moduli q = 2^b - d of a context with pm set (common.cuh) take
// the product pm_mul instead: T signed and the butterfly (X + T, X - T), from canonical inputs below 2^63 in
// magnitude after 15 stages (checked when the context is made).  Inverse: a_m = N^-1 psi^-m sum_k a^_k
// omega^-km (omega = psi^2) -- a cyclic decimation-in-time transform on the
// bit-reversed input with the same reduction-free butterfly, then one twist
// product by N^-1 psi^-m per word (times R = 2^64 when the inputs carry a
// Montgomery factor), which also makes the output canonical; the butterflies whose twiddle is 1 for every thread
// (r = 0 in the first pass: 31 of 80 at 32 words per thread, 15 of 32 at 16) are additions only.  Twiddles are
// stored as (w, Shoup(w)) pairs, or pm_mul's entries, and fetched as one 16-byte load; the forward's
// last pass reads a copy regrouped so that a warp's loads are contiguous.
//
// One CTA transforms a block of M = 2^LOG_M words of a limb held in shared
// memory; each thread keeps E = 2^LOG_E words in registers and runs up to
// LOG_E radix-2 stages on them per pass, with one padded shared-memory
// exchange (one pad word per 16, conflict-free for every window) and one
// barrier between passes (of the warp where the exchange stays inside it).  The first pass reads global memory directly
// (coalesced: lanes differ in the low index bits) and the last pass writes it
// directly (forward: E consecutive words per thread as 16-byte stores in
// the order of eval_pos; inverse: coalesced).
//
// When N = 2M a limb is split over two CTAs (so that two of them share an SM
// at N = 16384), launched as a thread-block cluster of two so they are always
// co-resident.  Forward: the outermost stage pairs word j of the first half
// with word j of the second; each CTA reads both halves in its first pass and
// keeps the output of its own half, so the stage costs no extra pass; a
// cluster barrier after those reads keeps an in-place transform from
// overwriting words the partner has not read yet.
// Inverse: the two CTAs form a thread-block cluster; after the inner stages
// the outermost stage pairs word j of the first half with word j of the
// second: CTA 0 takes the pairs with j < M/2, CTA 1 the others, each reading
// the partner's word of its pairs through distributed shared memory, making
// the pair's one product and writing both outputs (and the twist).
#include <cooperative_groups.h>

#include <atomic>
#include <cstdlib>

#include "common.cuh"

namespace cg = cooperative_groups;

#ifndef BFHE_NTT_PART
#define BFHE_NTT_PART 0
#endif

struct NttArgs {
    const u64* in;
    u64* out;
    int n_inner;
    size_t in_os, in_is, in_ls, out_os, out_is, out_ls;
    const u64 *src0, *src1;   // limbs below src_limbs come from here (NttIO::src)
    const u64* mul;           // the inverse's second factor (NttIO::mul)
    size_t mul_os, mul_is;
    int src_limbs;
    int n_limbs;
    LimbMap map;
    PrimeTab tab;
    int N, logN;
    bool natural;   // the evaluation side lies in index order (bfhe_ntt), not in eval_pos order
    int bits;   // the moduli are 2^bits - d (pm kernels)
    int mont;   // inverse: inputs carry a Montgomery factor
    int lazy;   // host side only: forward outputs not canonical (selects the template)
    int device; // host side only: the context's device (function attributes are per device)
};

namespace {

__device__ __forceinline__ int phys(int j) { return j + (j >> 4); }

// padded offset of word base + (e << W_LO) relative to phys(base): no carry crosses bit 4
// when e << W_LO is added to a pass's base (checked for every shape on the host), so the
// offset is a compile-time constant per e
template <int W_LO>
__device__ __forceinline__ constexpr int poff(int e) { return (e << W_LO) + ((e << W_LO) >> 4); }


// Barrier between two passes.  A pass whose words' low window is at most 5 bits gives each warp the 32 2^LOG_E
// consecutive words of its own threads, so an exchange between two such passes stays inside the warp.
template <int W_A, int W_B>
__device__ __forceinline__ void exchange_sync() {
    if constexpr (W_A <= 5 && W_B <= 5) __syncwarp();
    else __syncthreads();
}

// Storage order of the evaluation domain: index w (bit-reversed order) lies at eval_pos(w), which exchanges bits 1-4
// and 5-9 of w.  A thread of the forward's last and the inverse's first pass holds 2^LOG_E consecutive indices, pair e
// of them at eval_pos(base) + 64 e, so that the lanes of a warp access 512, 2 x 256 or 4 x 128 contiguous bytes (at 32,
// 16, 8 words per thread) instead of 32 half-used sectors.
__device__ __forceinline__ int eval_pos(int w) {
    return (w & ~1022) | ((w & 30) << 5) | ((w >> 4) & 62);
}

// a 16-byte load that the compiler issues where it stands: all of a thread's first-pass words are then in flight
// before its first butterfly (left to itself it sinks half of them between the butterflies, which a thread of the
// inverse's first pass, mostly additions, then waits for: 511 -> 479 us for 4352 limbs at N = 16384)
__device__ __forceinline__ ulonglong2 load_now(const ulonglong2* p) {
    ulonglong2 v;
    asm volatile("ld.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p));
    return v;
}

struct LimbPtrs {
    const u64* in;   // limb start
    u64* out;        // limb start
    const u64* mul;  // limb start
    int p;
};

template <bool FWD>
__device__ __forceinline__ LimbPtrs limb_ptrs(const NttArgs& a, int bx) {
    const int limb = bx % a.n_limbs;
    const int poly = bx / a.n_limbs;
    const int outer = poly / a.n_inner, inner = poly % a.n_inner;
    LimbPtrs r;
    r.in = FWD && limb < a.src_limbs
               ? (inner < 2 ? a.src0 : a.src1) + ((size_t)(2 * outer + (inner & 1)) * a.src_limbs + limb) * a.N
               : a.in + outer * a.in_os + inner * a.in_is + limb * a.in_ls;
    r.out = a.out + outer * a.out_os + inner * a.out_is + limb * a.out_ls;
    r.mul = FWD ? nullptr : a.mul + outer * a.mul_os + inner * a.mul_is + (size_t)limb * a.N;
    r.p = a.map(limb);
    return r;
}

// one limb's modulus: what the butterfly's product needs
template <bool PM>
struct Mod {
    u64 q;
    int b;         // PM: q = 2^b - d
    uint32_t d;
    __device__ __forceinline__ Mod(u64 q_, int bits) : q(q_), b(bits), d(PM ? (uint32_t)(((u64)1 << bits) - q_) : 0) {}
    // x, y <- x + w y, x - w y (lazily; without PM the difference is raised by 4q)
    __device__ __forceinline__ void butterfly(u64& x, u64& y, const ulonglong2& w) const {
        const u64 X = x;
        const u64 T = product(y, w);
        combine(X, T, x, y);
    }
    __device__ __forceinline__ void trivial(u64& x, u64& y) const {   // w = 1
        const u64 X = x;
        combine(X, y, x, y);
    }
    __device__ __forceinline__ u64 product(u64 y, const ulonglong2& w) const {
        if constexpr (PM) return pm_mul(y, w, b - 30, d << 2);
        else return shoup_lazy4n(y, w.x, w.y, 0 - q);
    }
    __device__ __forceinline__ u64 sum(u64 X, u64 T) const { return PM ? add64(X, T) : X + T; }
    __device__ __forceinline__ u64 diff(u64 X, u64 T) const { return PM ? sub64(X, T) : X + 4 * q - T; }
    __device__ __forceinline__ void combine(u64 X, u64 T, u64& x, u64& y) const {
        x = sum(X, T);
        y = diff(X, T);
    }
};

// ---------------------------------------------------------------- forward stages
// The last pass (W_LO = 0: E consecutive words per thread) takes its twiddles from the regrouped table:
// twc is this thread's column there, and its g-th twiddle of stage b sits (N >> (b+1)) + g (N / E) entries
// further, so lanes read consecutive 16-byte entries (the standard table gives each lane its own run of
// E >> (b+1) entries: 32 sectors per warp load instead of 16 contiguous).
template <bool PM, int LOG_N, int LOG_E, int W_LO, int HI, int LO>
__device__ __forceinline__ void fwd_stages(u64 (&x)[1 << LOG_E], u64 jb, const ulonglong2* __restrict__ tw,
                                           const ulonglong2* __restrict__ twc, const Mod<PM>& m) {
    constexpr int E = 1 << LOG_E;
#pragma unroll
    for (int st = 0; st <= HI - LO; ++st) {
        const int b = HI - st;
        const int h = b - W_LO;
        const u64 base = jb >> (b + 1);
#pragma unroll
        for (int g = 0; g < (E >> (h + 1)); ++g) {
            const ulonglong2 wp = W_LO == 0 ? __ldg(twc + ((1 << LOG_N) >> (b + 1)) + g * (1 << (LOG_N - LOG_E)))
                                            : __ldg(tw + base + g);
#pragma unroll
            for (int r = 0; r < (1 << h); ++r) {
                const int e = (g << (h + 1)) | r;
                m.butterfly(x[e], x[e | (1 << h)], wp);
            }
        }
    }
}

// TOP: this CTA is half `half` of a limb of N = 2M words and first applies the
// outermost stage (twiddle psi^brv(1)) to the pairs (j, j + M) it reads.
template <bool PM, int LOG_M, int LOG_E, int P, bool TOP, bool LAZY>
__device__ __forceinline__ void fwd_pass(u64 (&x)[1 << LOG_E], u64* sm, int tid, u64 jglob, const ulonglong2* tw,
                                         const ulonglong2* twl, const Mod<PM>& m, u64 mu, const u64* in, u64* out,
                                         int half, bool natural) {
    constexpr int E = 1 << LOG_E;
    constexpr int M = 1 << LOG_M;
    constexpr int NPASS = (LOG_M + LOG_E - 1) / LOG_E;
    constexpr int HI = LOG_M - 1 - P * LOG_E;
    constexpr int LO = (HI - LOG_E + 1) > 0 ? (HI - LOG_E + 1) : 0;
    constexpr int W_LO = LO;
    const int base = (tid & ((1 << W_LO) - 1)) | ((tid >> W_LO) << (W_LO + LOG_E));
    const int pb = phys(base);
    if (P == 0) {
        if (TOP) {
            const ulonglong2 w1 = __ldg(tw + 1);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const u64 X = in[base + (e << W_LO)];
                const u64 T = m.product(in[M + base + (e << W_LO)], w1);
                x[e] = half ? m.diff(X, T) : m.sum(X, T);
            }
            // both halves of the limb are read before either CTA writes (in-place transforms)
            cg::this_cluster().sync();
        } else {
#pragma unroll
            for (int e = 0; e < E; ++e) x[e] = in[base + (e << W_LO)];
        }
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) x[e] = sm[pb + poff<W_LO>(e)];
    }
    // the compiler does not move the first butterflies up between the loads (516 -> 504 us for 4352 limbs, N = 16384)
    if (P == 0 && !TOP) __syncwarp();
    constexpr int LOG_N = TOP ? LOG_M + 1 : LOG_M;
    // thread index over the whole limb (last pass): (jglob - N + base) / E
    const ulonglong2* twc = W_LO == 0 ? twl + ((((u64)half << LOG_M) + base) >> LOG_E) : twl;
    fwd_stages<PM, LOG_N, LOG_E, W_LO, HI, LO>(x, jglob + base, tw, twc, m);
    if constexpr (P + 1 < NPASS) {
#pragma unroll
        for (int e = 0; e < E; ++e) sm[pb + poff<W_LO>(e)] = x[e];
        constexpr int W_NEXT = LO - LOG_E > 0 ? LO - LOG_E : 0;
        exchange_sync<W_LO, W_NEXT>();
        fwd_pass<PM, LOG_M, LOG_E, P + 1, TOP, LAZY>(x, sm, tid, jglob, tw, twl, m, mu, in, out, half, natural);
    } else {
        // W_LO == 0 here: E consecutive words per thread; values < 64q -> canonical unless the
        // consumer takes lazy words (Montgomery products of operands < 64q, q < 2^50; PM: below 2q)
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if constexpr (PM) x[e] = LAZY ? pm_lazy(x[e], m.q, m.b, m.d) : pm_canon(x[e], m.q, m.b, m.d);
            else if constexpr (!LAZY) x[e] = reduce64(x[e], m.q, mu);
        }
        if (!LAZY && natural) {   // bfhe_ntt
            ulonglong2* o2 = reinterpret_cast<ulonglong2*>(out + base);
#pragma unroll
            for (int e = 0; e < E / 2; ++e) o2[e] = make_ulonglong2(x[2 * e], x[2 * e + 1]);
        } else {
            ulonglong2* o2 = reinterpret_cast<ulonglong2*>(out + eval_pos(base));
#pragma unroll
            for (int e = 0; e < E / 2; ++e) o2[e * 32] = make_ulonglong2(x[2 * e], x[2 * e + 1]);
        }
    }
}

template <bool PM, int LOG_M, int LOG_E, bool TOP, bool LAZY>
__global__ void __launch_bounds__(1 << (LOG_M - LOG_E), (LOG_M < 14 && LOG_M - LOG_E <= 8 ? 2 : 1)) k_ntt_fwd(NttArgs a) {
    extern __shared__ u64 sm[];
    const LimbPtrs lp = limb_ptrs<true>(a, blockIdx.x);
    const int half = blockIdx.y;
    const Mod<PM> m(a.tab.q[lp.p], a.bits);
    const u64 mu = PM ? 0 : a.tab.mu[lp.p];
    const ulonglong2* tw = reinterpret_cast<const ulonglong2*>(a.tab.tw) + (size_t)lp.p * a.N;
    const ulonglong2* twl = reinterpret_cast<const ulonglong2*>(a.tab.twl) + ((size_t)lp.p * 3 + (LOG_E - 3)) * a.N;
    const u64 jglob = (u64)a.N + ((u64)half << LOG_M);
    const u64* in = TOP ? lp.in : lp.in + ((size_t)half << LOG_M);
    u64 x[1 << LOG_E];
    pdl_begin();
    fwd_pass<PM, LOG_M, LOG_E, 0, TOP, LAZY>(x, sm, threadIdx.x, jglob, tw, twl, m, mu, in,
                                             lp.out + ((size_t)half << LOG_M), half, a.natural);
}

// ---------------------------------------------------------------- inverse stages
// Decimation in time on the bit-reversed input with inverse roots: the butterfly on
// bit b at lower index x is (U, V) -> (U + T, U - T + 4q), T = V omega^-(N/2^(b+1)) (x mod 2^b)
// (table entry 2^b + (x mod 2^b)); bounds grow by 4q per stage, as in the forward.  In the first pass a thread holds
// consecutive words, so r = 0 is the twiddle omega^0 = 1 in each of its stages: sums of inputs, below 2^LOG_E q.
// The natural-order output is then multiplied by the twist N^-1 psi^-m.
template <bool PM, int LOG_E, int W_LO, int LO, int HI>
__device__ __forceinline__ void inv_stages(u64 (&x)[1 << LOG_E], int base, const ulonglong2* __restrict__ itw,
                                           const Mod<PM>& m) {
    constexpr int E = 1 << LOG_E;
#pragma unroll
    for (int st = 0; st <= HI - LO; ++st) {
        const int b = LO + st;
        const int h = b - W_LO;
        const int tbase = (1 << b) + (base & ((1 << b) - 1));
#pragma unroll
        for (int r = 0; r < (1 << h); ++r) {
            if (PM && W_LO == 0 && r == 0) {
#pragma unroll
                for (int g = 0; g < (E >> (h + 1)); ++g) m.trivial(x[g << (h + 1)], x[(g << (h + 1)) | (1 << h)]);
                continue;
            }
            const ulonglong2 wp = __ldg(itw + tbase + (r << W_LO));
#pragma unroll
            for (int g = 0; g < (E >> (h + 1)); ++g) {
                const int e = (g << (h + 1)) | r;
                m.butterfly(x[e], x[e | (1 << h)], wp);
            }
        }
    }
}

// MODE 1: the block is the whole limb; MODE 2: half `half` of a limb of N = 2M words,
// whose outermost stage pairs with the partner CTA of the cluster.
// OUT 0: twisted, canonical; 1: the same, of the input times the words of mul (an evaluation-domain product that would
// otherwise be a kernel and a round trip through memory of its own); 2: not twisted (the consumer multiplies by the twist, folded into a product it makes
// anyway): from inputs below q, 15 stages leave words below 61q < 2^64, or signed words below 2^63 (PM).
template <bool PM>
__device__ __forceinline__ u64 twisted(u64 x, const ulonglong2& t, const Mod<PM>& m) {
    if constexpr (PM) return pm_canon(m.product(x, t), m.q, m.b, m.d);
    else return shoup(x, t.x, t.y, m.q);
}

template <bool PM, int LOG_M, int LOG_E, int P, int MODE, int OUT>
__device__ __forceinline__ void inv_pass(u64 (&x)[1 << LOG_E], u64* sm, int tid, const ulonglong2* itw,
                                         const ulonglong2* twist, const Mod<PM>& m, const u64* in, u64* out, const u64* mul,
                                         int half, bool natural) {
    constexpr int E = 1 << LOG_E;
    constexpr int M = 1 << LOG_M;
    constexpr int NPASS = (LOG_M + LOG_E - 1) / LOG_E;
    constexpr int LO = P * LOG_E;
    constexpr int HI = (LO + LOG_E - 1) < (LOG_M - 1) ? (LO + LOG_E - 1) : (LOG_M - 1);
    constexpr int W_LO = (HI - LO + 1 == LOG_E) ? LO : (LOG_M - LOG_E);
    const int base = (tid & ((1 << W_LO) - 1)) | ((tid >> W_LO) << (W_LO + LOG_E));
    const int pb = phys(base);
    if (P == 0) {
        // W_LO == 0: E consecutive words per thread
        if (OUT == 0 && natural) {   // bfhe_ntt
            const ulonglong2* i2 = reinterpret_cast<const ulonglong2*>(in + base);
#pragma unroll
            for (int e = 0; e < E / 2; ++e) {
                const ulonglong2 v = load_now(i2 + e);
                x[2 * e] = v.x;
                x[2 * e + 1] = v.y;
            }
        } else {
            const ulonglong2* i2 = reinterpret_cast<const ulonglong2*>(in + eval_pos(base));
#pragma unroll
            for (int e = 0; e < E / 2; ++e) {
                const ulonglong2 v = load_now(i2 + e * 32);
                x[2 * e] = v.x;
                x[2 * e + 1] = v.y;
            }
        }
        if constexpr (OUT == 1) {
            const ulonglong2* m2 = reinterpret_cast<const ulonglong2*>(mul + eval_pos(base));
#pragma unroll
            for (int e = 0; e < E / 2; ++e) {
                const ulonglong2 v = m2[e * 32];
                x[2 * e] = pm_mul_var(x[2 * e], v.x, m.q, m.b, m.d);
                x[2 * e + 1] = pm_mul_var(x[2 * e + 1], v.y, m.q, m.b, m.d);
            }
        }
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) x[e] = sm[pb + poff<W_LO>(e)];
    }
    constexpr bool LAST = (P + 1 == NPASS);
    inv_stages<PM, LOG_E, W_LO, LO, HI>(x, base, itw, m);
    if constexpr (!LAST) {
#pragma unroll
        for (int e = 0; e < E; ++e) sm[pb + poff<W_LO>(e)] = x[e];
        constexpr int W_NEXT = LO + 2 * LOG_E <= LOG_M ? LO + LOG_E : LOG_M - LOG_E;
        exchange_sync<W_LO, W_NEXT>();
        inv_pass<PM, LOG_M, LOG_E, P + 1, MODE, OUT>(x, sm, tid, itw, twist, m, in, out, mul, half, natural);
    } else if constexpr (MODE == 2) {
        // outermost stage across the halves, pairs (j, j + M): the top bit of e is bit LOG_M - 1 of j, so
        // CTA 0 takes the pairs with j < M/2 and CTA 1 those with j >= M/2; each publishes the words of the
        // other set, reads the partner's word of each pair it takes through distributed shared memory,
        // makes the pair's one product and writes both outputs (the limb's positions j and j + M)
        cg::cluster_group cl = cg::this_cluster();
        constexpr int EH = E / 2;
        // (register indices stay compile-time: the half selects between two words)
#pragma unroll
        for (int e = 0; e < EH; ++e) {
            const u64 v = half ? x[e] : x[e + EH];   // the set the partner takes
            sm[pb + (half ? poff<W_LO>(e) : poff<W_LO>(e + EH))] = v;
        }
        cl.sync();
        const u64* peer = cl.map_shared_rank(sm, cl.block_rank() ^ 1u);
        u64* o = out - (size_t)half * M;        // limb start
#pragma unroll
        for (int e = 0; e < EH; ++e) {
            const u64 mine = half ? x[e + EH] : x[e];
            const int off = half ? poff<W_LO>(e + EH) : poff<W_LO>(e);
            const int j = base + ((half ? e + EH : e) << W_LO);
            const u64 other = peer[pb + off];
            const u64 U = half ? other : mine, V = half ? mine : other;
            const ulonglong2 wp = __ldg(itw + M + j);
            const u64 T = m.product(V, wp);
            const u64 y0 = m.sum(U, T), y1 = m.diff(U, T);
            if constexpr (OUT == 2) {
                o[j] = y0;
                o[j + M] = y1;
            } else {
                const ulonglong2 t0 = __ldg(twist + j), t1 = __ldg(twist + j + M);
                o[j] = twisted<PM>(y0, t0, m);
                o[j + M] = twisted<PM>(y1, t1, m);
            }
        }
        cl.sync();   // the partner has finished reading this CTA's shared memory
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int j = base + (e << W_LO);
            if constexpr (OUT == 2) {
                out[j] = x[e];
            } else {
                out[j] = twisted<PM>(x[e], __ldg(twist + j), m);
            }
        }
    }
}

template <bool PM, int LOG_M, int LOG_E, int MODE, int OUT>
__global__ void __launch_bounds__(1 << (LOG_M - LOG_E), (LOG_M < 14 && LOG_M - LOG_E <= 8 ? 2 : 1)) k_ntt_inv(NttArgs a) {
    extern __shared__ u64 sm[];
    const LimbPtrs lp = limb_ptrs<false>(a, blockIdx.x);
    const int half = blockIdx.y;
    const Mod<PM> m(a.tab.q[lp.p], a.bits);
    const ulonglong2* itw = reinterpret_cast<const ulonglong2*>(a.tab.itw) + (size_t)lp.p * a.N;
    const ulonglong2* twist = reinterpret_cast<const ulonglong2*>(a.tab.twist) + ((size_t)lp.p * 3 + (a.mont ? 1 : 0)) * a.N;
    u64 x[1 << LOG_E];
    pdl_begin();
    inv_pass<PM, LOG_M, LOG_E, 0, MODE, OUT>(x, sm, threadIdx.x, itw, twist, m, lp.in + ((size_t)half << LOG_M),
                                             lp.out + ((size_t)half << LOG_M), lp.mul + ((size_t)half << LOG_M), half,
                                             a.natural);
}

template <int LOG_M, int LOG_E>
constexpr size_t smem_bytes() {
    return (LOG_M + LOG_E - 1) / LOG_E > 1 ? (size_t)((1 << LOG_M) + ((1 << LOG_M) >> 4)) * 8 : 0;
}

template <bool PM, int LOG_M, int LOG_E, bool TOP, bool LAZY>
int run_fwd(const NttArgs& a, int blocks, cudaStream_t st) {
    constexpr int T = 1 << (LOG_M - LOG_E);
    const size_t smem = smem_bytes<LOG_M, LOG_E>();
    static std::atomic<uint64_t> attr{0};   // devices whose function attribute is set
    const int dev = a.device;
    if (!(attr.load() >> dev & 1)) {
        BFHE_CUDA(cudaFuncSetAttribute(k_ntt_fwd<PM, LOG_M, LOG_E, TOP, LAZY>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem));
        attr.fetch_or(1ull << dev);
    }
    BFHE_CUDA(launch_kernel(k_ntt_fwd<PM, LOG_M, LOG_E, TOP, LAZY>, dim3(blocks, TOP ? 2 : 1), dim3(T), smem, st, TOP ? 2 : 1, a));
    BFHE_LAUNCH_CHECK("k_ntt_fwd");
    return BFHE_OK;
}

template <bool PM, int LOG_M, int LOG_E, int MODE, int OUT>
int run_inv(const NttArgs& a, int blocks, cudaStream_t st) {
    constexpr int T = 1 << (LOG_M - LOG_E);
    // the cluster exchange needs the shared buffer even for a single pass
    const size_t smem = MODE == 2 ? (size_t)((1 << LOG_M) + ((1 << LOG_M) >> 4)) * 8 : smem_bytes<LOG_M, LOG_E>();
    static std::atomic<uint64_t> attr{0};   // devices whose function attribute is set
    const int dev = a.device;
    if (!(attr.load() >> dev & 1)) {
        BFHE_CUDA(cudaFuncSetAttribute(k_ntt_inv<PM, LOG_M, LOG_E, MODE, OUT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem));
        attr.fetch_or(1ull << dev);
    }
    BFHE_CUDA(launch_kernel(k_ntt_inv<PM, LOG_M, LOG_E, MODE, OUT>, dim3(blocks, (MODE == 2) ? 2 : 1), dim3(T), smem, st, (MODE == 2) ? 2 : 1, a));
    BFHE_LAUNCH_CHECK("k_ntt_inv");
    return BFHE_OK;
}

template <bool PM, int LM, int LE>
int fwd_shape(const NttArgs& a, int blocks, cudaStream_t st, bool top) {
    if (top)
        return a.lazy ? run_fwd<PM, LM, LE, true, true>(a, blocks, st) : run_fwd<PM, LM, LE, true, false>(a, blocks, st);
    return a.lazy ? run_fwd<PM, LM, LE, false, true>(a, blocks, st) : run_fwd<PM, LM, LE, false, false>(a, blocks, st);
}

template <int LM, int LE>
int inv_mul_shape(const NttArgs& a, int blocks, cudaStream_t st, bool split) {
    return split ? run_inv<true, LM, LE, 2, 1>(a, blocks, st) : run_inv<true, LM, LE, 1, 1>(a, blocks, st);
}

template <bool PM, int LM, int LE>
int inv_shape(const NttArgs& a, int blocks, cudaStream_t st, bool split) {
    if (split)
        return a.lazy ? run_inv<PM, LM, LE, 2, 2>(a, blocks, st) : run_inv<PM, LM, LE, 2, 0>(a, blocks, st);
    return a.lazy ? run_inv<PM, LM, LE, 1, 2>(a, blocks, st) : run_inv<PM, LM, LE, 1, 0>(a, blocks, st);
}

}  // namespace

#define NTT_SHAPES(CASE)                          \
    CASE(10, 3) CASE(10, 4) CASE(10, 5)           \
    CASE(11, 3) CASE(11, 4) CASE(11, 5)           \
    CASE(12, 3) CASE(12, 4) CASE(12, 5)           \
    CASE(13, 3) CASE(13, 4) CASE(13, 5)           \
    CASE(14, 4) CASE(14, 5)
#define FWD_CASE(LM, LE) \
    if (log_m == LM && log_e == LE) return fwd_shape<PM, LM, LE>(a, blocks, st, split);
#define INV_CASE(LM, LE) \
    if (log_m == LM && log_e == LE) return inv_shape<PM, LM, LE>(a, blocks, st, split);
#define INV_MUL_CASE(LM, LE) \
    if (log_m == LM && log_e == LE) return inv_mul_shape<LM, LE>(a, blocks, st, split);

// The shapes' kernels are compiled as five objects of this file (BFHE_NTT_PART: forward and inverse, without and with
// pm, and the inverse of a product), in parallel; part 0 also holds the host side.
int ntt_fwd_any(const NttArgs& a, int log_m, int log_e, int blocks, bool split, cudaStream_t st);
int ntt_fwd_any_pm(const NttArgs& a, int log_m, int log_e, int blocks, bool split, cudaStream_t st);
int ntt_inv_any(const NttArgs& a, int log_m, int log_e, int blocks, bool split, cudaStream_t st);
int ntt_inv_any_pm(const NttArgs& a, int log_m, int log_e, int blocks, bool split, cudaStream_t st);
int ntt_inv_mul_any_pm(const NttArgs& a, int log_m, int log_e, int blocks, bool split, cudaStream_t st);

#if BFHE_NTT_PART == 0
int ntt_fwd_any(const NttArgs& a, int log_m, int log_e, int blocks, bool split, cudaStream_t st) {
    constexpr bool PM = false;
    NTT_SHAPES(FWD_CASE)
    return set_error(BFHE_EINVAL, "no NTT configuration for this ring degree");
}
#elif BFHE_NTT_PART == 1
int ntt_fwd_any_pm(const NttArgs& a, int log_m, int log_e, int blocks, bool split, cudaStream_t st) {
    constexpr bool PM = true;
    NTT_SHAPES(FWD_CASE)
    return set_error(BFHE_EINVAL, "no NTT configuration for this ring degree");
}
#elif BFHE_NTT_PART == 2
int ntt_inv_any(const NttArgs& a, int log_m, int log_e, int blocks, bool split, cudaStream_t st) {
    constexpr bool PM = false;
    NTT_SHAPES(INV_CASE)
    return set_error(BFHE_EINVAL, "no NTT configuration for this ring degree");
}
#elif BFHE_NTT_PART == 3
int ntt_inv_any_pm(const NttArgs& a, int log_m, int log_e, int blocks, bool split, cudaStream_t st) {
    constexpr bool PM = true;
    NTT_SHAPES(INV_CASE)
    return set_error(BFHE_EINVAL, "no NTT configuration for this ring degree");
}
#elif BFHE_NTT_PART == 4
int ntt_inv_mul_any_pm(const NttArgs& a, int log_m, int log_e, int blocks, bool split, cudaStream_t st) {
    NTT_SHAPES(INV_MUL_CASE)
    return set_error(BFHE_EINVAL, "no NTT configuration for this ring degree");
}
#endif

#if BFHE_NTT_PART == 0
namespace {

NttArgs make_args(const bfhe_ctx* ctx, const NttIO& io, int n_limbs, LimbMap map, int mont, int lazy) {
    NttArgs a;
    a.in = io.in;
    a.out = io.out;
    a.n_inner = io.n_inner > 0 ? io.n_inner : 1;
    a.in_os = io.in_os;
    a.in_is = io.in_is;
    a.in_ls = io.in_ls;
    a.out_os = io.out_os;
    a.out_is = io.out_is;
    a.out_ls = io.out_ls;
    a.n_limbs = n_limbs;
    a.map = map;
    a.tab = ctx->tab;
    a.N = (int)ctx->N;
    a.logN = (int)ctx->logN;
    a.src0 = io.src[0];
    a.src1 = io.src[1];
    a.src_limbs = io.src_limbs;
    a.mul = io.mul;
    a.mul_os = io.mul_os;
    a.mul_is = io.mul_is;
    a.natural = io.natural;
    a.bits = (int)ctx->prime_bits;
    a.mont = mont;
    a.lazy = lazy;
    a.device = ctx->device < 64 ? ctx->device : 63;
    return a;
}

int env_int(const char* name) {
    const char* s = getenv(name);
    return s ? atoi(s) : 0;
}

}  // namespace

// Block size and registers per thread.  Defaults (measured on GB300 inside the multiply, pm products, us per
// launch class, forward / inverse): N <= 4096 in one block of 16 words per thread (64 pairs at N = 4096, L = 2: 52 / 41;
// 32 words 61 / 87, halves 54 / 53).  N = 8192 in one block of 32 words, two blocks per SM (64 pairs, L = 4: 196 / 137;
// 16 words 233 / 151).  N = 16384 in one block of 32 words (64 pairs, L = 8: 1017 / 515; halves 1029 / 559).  N = 32768
// as two 16384-word halves, 32 words (8 pairs, L = 16: 887 / 347; 16 words 949 / 471).  A launch whose halves fit the 152
// SMs at one CTA each takes halves at 16 words, which puts twice the threads on each limb: at N = 16384 (72 limbs: 14 / 15
// against 19 / 19) and for the forward at N = 8192 (8.3 against 12.5); the inverse there takes one block of 16 words
// (up to 152 limbs: 10.4 to 11.7 against 12.4; halves 10.3).  The Shoup products' kernels take the same shapes (64 pairs
// at N = 8192, L = 4, 40 bits: 219 / 162, 16 words 266 / 193) but for the forward at N = 16384, in halves of 32 words (64
// pairs, L = 8: 1139 against 1188 us at 40 bits, 1301 against 1358 at 56).  bfhe_ntt_config (the autotuner) or BFHE_NTT_LOG_M /
// BFHE_NTT_LOG_E override the defaults.
int g_cfg[16][2][2] = {};   // [logN][inverse] -> (log_m, log_e), 0 = default

int ntt_config(int logN, int inverse, bool pm, size_t limbs, int* log_m, int* log_e) {
    static const int env_m = env_int("BFHE_NTT_LOG_M");
    static const int env_e = env_int("BFHE_NTT_LOG_E");
    int m = logN <= 14 ? logN : logN - 1;
    int e = logN >= 13 ? 5 : 4;
    if (logN == 14 && !inverse && !pm) m = 13;
    if ((logN == 14 || (logN == 13 && !inverse)) && 2 * limbs <= 152) {
        m = logN - 1;
        e = 4;
    }
    if (logN == 13 && inverse && limbs <= 152) e = 4;
    if (env_m >= logN - 1 && env_m <= logN && env_m >= 10 && env_m <= 14) m = env_m;
    if (env_e >= 3 && env_e <= 5) e = env_e;
    if (logN >= 0 && logN < 16 && g_cfg[logN][inverse ? 1 : 0][0]) {
        m = g_cfg[logN][inverse ? 1 : 0][0];
        e = g_cfg[logN][inverse ? 1 : 0][1];
    }
    if (m == 14 && e < 4) e = 4;
    *log_m = m;
    *log_e = e;
    return BFHE_OK;
}

extern "C" int bfhe_ntt_config(uint32_t logN, int inverse, uint32_t log_m, uint32_t log_e, uint32_t* cur_m,
                               uint32_t* cur_e) {
    if (logN < 10 || logN > 15) return set_error(BFHE_EINVAL, "logN must be in [10, 15]");
    if (log_m != 0) {
        if (log_m > logN || log_m + 1 < logN || log_m < 10 || log_m > 14 || log_e < 3 || log_e > 5 ||
            (log_m == 14 && log_e < 4))
            return set_error(BFHE_EINVAL, "unsupported NTT block configuration");
        // the shape that large launches take anyway is no override: small launches keep theirs
        int dm, de;
        g_cfg[logN][inverse ? 1 : 0][0] = 0;
        ntt_config((int)logN, inverse, true, (size_t)1 << 30, &dm, &de);
        if ((int)log_m != dm || (int)log_e != de) {
            g_cfg[logN][inverse ? 1 : 0][0] = (int)log_m;
            g_cfg[logN][inverse ? 1 : 0][1] = (int)log_e;
        }
    }
    int m, e;
    ntt_config((int)logN, inverse, true, (size_t)1 << 30, &m, &e);   // the shape of a large launch of the default moduli
    if (cur_m) *cur_m = (uint32_t)m;
    if (cur_e) *cur_e = (uint32_t)e;
    return BFHE_OK;
}

int launch_ntt_fwd(const bfhe_ctx* ctx, NttIO io, int n_polys, int n_limbs, LimbMap map, cudaStream_t st,
                   int lazy_out) {
    if (n_polys <= 0 || n_limbs <= 0) return BFHE_OK;
    ProfScope ps(ctx, BFHE_K_NTT_FWD, st, (double)n_polys * n_limbs * (ctx->N / 2) * ctx->logN,
                 16.0 * n_polys * n_limbs * ctx->N);
    // the slot modulus t (prime index nP - 1) is not of the form 2^b - d
    const bool pm = ctx->pm && map(0) != (int)ctx->nP - 1;
    int log_m, log_e;
    ntt_config((int)ctx->logN, 0, pm, (size_t)n_polys * n_limbs, &log_m, &log_e);
    NttArgs a = make_args(ctx, io, n_limbs, map, 0, lazy_out && (pm || ctx->prime_bits <= 50) ? 1 : 0);
    const int blocks = n_polys * n_limbs;
    const int subs = (int)(ctx->N >> log_m);
    if (subs != 1 && subs != 2) return set_error(BFHE_EINVAL, "unsupported ring degree");
    return pm ? ntt_fwd_any_pm(a, log_m, log_e, blocks, subs == 2, st)
              : ntt_fwd_any(a, log_m, log_e, blocks, subs == 2, st);
}

int launch_ntt_inv(const bfhe_ctx* ctx, NttIO io, int n_polys, int n_limbs, LimbMap map, int mont,
                   cudaStream_t st, int lazy_out) {
    if (n_polys <= 0 || n_limbs <= 0) return BFHE_OK;
    ProfScope ps(ctx, BFHE_K_NTT_INV, st, (double)n_polys * n_limbs * (ctx->N / 2) * ctx->logN,
                 16.0 * n_polys * n_limbs * ctx->N);
    const bool pm = ctx->pm && map(0) != (int)ctx->nP - 1;
    int log_m, log_e;
    ntt_config((int)ctx->logN, 1, pm, (size_t)n_polys * n_limbs, &log_m, &log_e);
    NttArgs a = make_args(ctx, io, n_limbs, map, mont, lazy_out);
    const int blocks = n_polys * n_limbs;
    const int subs = (int)(ctx->N >> log_m);
    if (subs != 1 && subs != 2) return set_error(BFHE_EINVAL, "unsupported ring degree");
    if (lazy_out != 0 && lazy_out != 2) return set_error(BFHE_EINVAL, "bad inverse output form");
    if (io.mul) {
        if (!pm || lazy_out) return set_error(BFHE_EINVAL, "the inverse of a product needs moduli 2^b - d");
        return ntt_inv_mul_any_pm(a, log_m, log_e, blocks, subs == 2, st);
    }
    return pm ? ntt_inv_any_pm(a, log_m, log_e, blocks, subs == 2, st)
              : ntt_inv_any(a, log_m, log_e, blocks, subs == 2, st);
}
#endif

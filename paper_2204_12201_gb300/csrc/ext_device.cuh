// ext_device.cuh -- device and launch helpers shared by the base-extension kernels (ext.cu, ext_pm.cu).
#pragma once
#include "kernels.cuh"

namespace {

constexpr int TPB = 256;

inline int grid_for(size_t work) {
    size_t b = (work + TPB - 1) / TPB;
    if (b > (size_t)1 << 30) b = (size_t)1 << 30;
    return (int)(b ? b : 1);
}

// ---------------------------------------------------------------- exact base extension
// Inputs x_i may be lazy (< 2 s_i); digits come out canonical.  Inner steps keep
// u in [0, 2 s_i): u + s_i - v_j < 3 s_i goes straight into a lazy Shoup product.
template <int NS>
__device__ __forceinline__ bool garner(const u64 (&x)[NS], const ExtDesc& d, u64 (&v)[NS]) {
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const u64 si = d.src_q[i];
        u64 u = x[i];
#pragma unroll
        for (int j = 0; j < i; ++j) {
            u64 vj = v[j];
            vj = vj >= si ? vj - si : vj;
            u = shoup_lazy(u + si - vj, d.ginv[i * NS + j], d.ginv_s[i * NS + j], si);
        }
        u = u >= si ? u - si : u;
        v[i] = u;
    }
    int state = 0;
#pragma unroll
    for (int i = NS - 1; i >= 0; --i) {
        const u64 h = d.hdig[i];
        if (state == 0) state = v[i] > h ? 1 : (v[i] < h ? -1 : 0);
    }
    return state > 0;   // x > (S-1)/2: the centred value is x - S
}

// value mod T_j of the centred integer with digits v (SMALL: T may be far below the sources).
// Without SMALL every digit is < 2 T_j, so Horner runs lazily below 4 T_j.
template <int NS, bool SMALL>
__device__ __forceinline__ u64 ext_eval(const u64 (&v)[NS], bool neg, const ExtDesc& d, int j) {
    const u64 T = d.dst_q[j];
    u64 acc;
    if (SMALL) {
        const u64 mu = d.dst_mu[j];
        acc = reduce64(v[NS - 1], T, mu);
#pragma unroll
        for (int i = NS - 2; i >= 0; --i) {
            acc = shoup(acc, d.radix[j * NS + i], d.radix_s[j * NS + i], T);
            acc = add_mod(acc, reduce64(v[i], T, mu), T);
        }
    } else {
        acc = v[NS - 1];
#pragma unroll
        for (int i = NS - 2; i >= 0; --i)
            acc = shoup_lazy(acc, d.radix[j * NS + i], d.radix_s[j * NS + i], T) + v[i];
        const u64 T2 = T << 1;
        acc = acc >= T2 ? acc - T2 : acc;
        acc = acc >= T ? acc - T : acc;
    }
    if (neg) acc = sub_mod(acc, d.smod[j], T);
    return acc;
}

// pair (w, Shoup(w)) of the twist table row f of prime p at coefficient k: f = 1 is N^-1 psi^-k R,
// f = 2 is t N^-1 psi^-k R (mod the prime)
__device__ __forceinline__ ulonglong2 twist_at(const u64* twist, int p, int f, int k, int N) {
    return __ldg(reinterpret_cast<const ulonglong2*>(twist) + ((size_t)p * 3 + f) * N + k);
}

// a word times a twist entry, in [0, 2q): Shoup pairs, or pm_mul's entries when the moduli are 2^bits - d (bits > 0)
__device__ __forceinline__ u64 twist_mul(u64 w, const ulonglong2& f, u64 q, int bits) {
    if (bits) {
        const uint32_t d = (uint32_t)(((u64)1 << bits) - q);
        return pm_lazy(pm_mul(w, f, bits - 30, d << 2), q, bits, d);
    }
    return shoup_lazy(w, f.x, f.y, q);
}

// sizes known only at run time (digits in local memory, loops not unrolled): the sets of more than 16 data primes and
// the rare exact path of ext_pm.cu
constexpr int NMAX = BFHE_MAX_L + 1;

__device__ bool garner_n(const u64* x, const ExtDesc& d, u64* v, int ns) {
#pragma unroll 1
    for (int i = 0; i < ns; ++i) {
        const u64 si = d.src_q[i];
        u64 u = x[i];
#pragma unroll 1
        for (int j = 0; j < i; ++j) {
            u64 vj = v[j];
            vj = vj >= si ? vj - si : vj;
            u = shoup_lazy(u + si - vj, d.ginv[i * ns + j], d.ginv_s[i * ns + j], si);
        }
        v[i] = u >= si ? u - si : u;
    }
    int state = 0;
#pragma unroll 1
    for (int i = ns - 1; i >= 0 && state == 0; --i) {
        const u64 h = d.hdig[i];
        state = v[i] > h ? 1 : (v[i] < h ? -1 : 0);
    }
    return state > 0;
}

__device__ u64 ext_eval_n(const u64* v, bool neg, const ExtDesc& d, int j, int ns, bool small) {
    const u64 T = d.dst_q[j];
    u64 acc;
    if (small) {
        const u64 mu = d.dst_mu[j];
        acc = reduce64(v[ns - 1], T, mu);
#pragma unroll 1
        for (int i = ns - 2; i >= 0; --i) {
            acc = shoup(acc, d.radix[j * ns + i], d.radix_s[j * ns + i], T);
            acc = add_mod(acc, reduce64(v[i], T, mu), T);
        }
    } else {
        acc = v[ns - 1];
#pragma unroll 1
        for (int i = ns - 2; i >= 0; --i) acc = shoup_lazy(acc, d.radix[j * ns + i], d.radix_s[j * ns + i], T) + v[i];
        const u64 T2 = T << 1;
        acc = acc >= T2 ? acc - T2 : acc;
        acc = acc >= T ? acc - T : acc;
    }
    if (neg) acc = sub_mod(acc, d.smod[j], T);
    return acc;
}

}  // namespace

#define LAUNCH(kern, work, ...)                                                   \
    do {                                                                          \
        auto* _kfn = kern;                                                        \
        BFHE_CUDA(launch_kernel(_kfn, dim3(grid_for(work)), dim3(TPB), 0, st, 1, __VA_ARGS__)); \
        BFHE_LAUNCH_CHECK(#kern);                                                \
    } while (0)

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


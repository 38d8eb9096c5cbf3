// rows.cuh -- linear combinations and accesses over whole limbs, shared by the row kernels (kernels.cu) and the multiply's
// last kernel (ext.cu).
#pragma once
#include "kernels.cuh"

namespace {

// ---------------------------------------------------------------- linear ops
__device__ __forceinline__ u64 apply(u64 acc, u64 v, int c, u64 q) {
    switch (c) {
        case 1: return add_mod(acc, v, q);
        case 2: return add_mod(add_mod(acc, v, q), v, q);
        case -1: return sub_mod(acc, v, q);
        case -2: return sub_mod(sub_mod(acc, v, q), v, q);
        default: return acc;
    }
}

__constant__ int c_gate_coef[8][5] = {
    // cc  cx  cy  cz  cp
    {0, 0, 0, 0, 1},     // AND  = xy
    {0, 1, 1, 0, -1},    // OR   = x + y - xy
    {0, 1, 1, 0, -2},    // XOR  = x + y - 2xy
    {1, 0, 0, 0, -1},    // NAND = 1 - xy
    {1, -1, -1, 0, 1},   // NOR  = 1 - (x + y - xy)
    {1, -1, -1, 0, 2},   // XNOR = 1 - (x + y - 2xy)
    {1, -1, 0, 0, 0},    // NOT  = 1 - x
    {0, 0, 0, 1, 1},     // MUX  = x (y - z) + z
};

// coefficients of a table entry's operation
__device__ __forceinline__ void gate_coefs(int code0, int& cc, int& cx, int& cy, int& cz, int& cp) {
    const int op = code0 & 0xff;
    if (op == BFHE_OP_MUL) {
        cc = cx = cy = cz = 0;
        cp = 1;
    } else if (op == BFHE_OP_LIN) {
        const int code = code0 >> 8;
        cc = code / 125 - 2;
        cx = (code / 25) % 5 - 2;
        cy = (code / 5) % 5 - 2;
        cz = code % 5 - 2;
        cp = 0;
    } else {
        const int* cf = c_gate_coef[op & 7];
        cc = cf[0];
        cx = cf[1];
        cy = cf[2];
        cz = cf[3];
        cp = cf[4];
    }
}

// ---- rows: a kernel over whole limbs.  A block of 256 threads takes 256 W consecutive words of one limb (row), W = 2 as
// one 16-byte access per thread, W = 1 where a caller's buffer is only 8-byte aligned, so that the limb, its modulus
// and everything that hangs on them are computed once per block and not by divisions per word (bound: HBM; the genotype
// dot product's additions of 48 ciphertexts at N = 16384, L = 8: 86 -> 47 us, 6.5 TB/s; a level of 31 gates at N = 8192,
// L = 4: gather 16 -> 10, epilogue 17 -> 9 us).
template <int W>
struct Words {
    u64 v[W];
};
template <int W>
__device__ __forceinline__ Words<W> load_words(const u64* p) {
    Words<W> r;
    if constexpr (W == 2) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p);
        r.v[0] = t.x;
        r.v[1] = t.y;
    } else {
        r.v[0] = *p;
    }
    return r;
}
template <int W>
__device__ __forceinline__ void store_words(u64* p, const Words<W>& r) {
    if constexpr (W == 2) *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(r.v[0], r.v[1]);
    else *p = r.v[0];
}
// row of this block and the thread's first word in it
template <int W>
struct Row {
    uint32_t row;
    int k;
    size_t off;   // row N + k
    __device__ __forceinline__ explicit Row(int logN) {
        const int sh = logN - (W == 2 ? 9 : 8);   // N >= 1024
        row = blockIdx.x >> sh;
        k = (int)(((blockIdx.x & ((1u << sh) - 1u)) * 256 + threadIdx.x) * W);
        off = ((size_t)row << logN) + k;
    }
};
inline bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

// linear combinations, W words (coefficient k onwards of limb i; the constant sits at coefficient 0 of c0)
template <int W>
__device__ __forceinline__ Words<W> lin_words(int cc, int cx, int cy, int cz, int cp, u64 cval, const u64* x, const u64* y,
                                              const u64* z, const u64* p, size_t o, bool first, u64 q, u64 dw, u64 dws) {
    Words<W> acc{};
    if (cc != 0 && first) acc.v[0] = apply(0, shoup(cval, dw, dws, q), cc, q);
    auto term = [&](const u64* s, int c) {
        const Words<W> t = load_words<W>(s + o);
#pragma unroll
        for (int w = 0; w < W; ++w) acc.v[w] = apply(acc.v[w], t.v[w], c, q);
    };
    if (cx) term(x, cx);
    if (cy) term(y, cy);
    if (cz) term(z, cz);
    if (cp) term(p, cp);
    return acc;
}

}  // namespace

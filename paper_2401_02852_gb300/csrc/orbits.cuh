// Device building blocks of the kernels that keep amplitudes in shared memory
// and butterfly them in rounds of a few generators (small.cu, mid.cu).
//
// A round takes orbits of K generators (2^K amplitudes) into registers.  An orbit
// is enumerated by its representative z0, whose K acting bits are zero; every
// other member's index is z0 XOR a constant of the round, so any set of
// generators with independent acting bits fits the same code.  The layout permutes
// the low index bits by XOR with higher ones (linear over XOR, so a member's
// address is the representative's XOR a constant), which spreads every round's
// accesses over the banks.
#pragma once

#include "pass_common.cuh"
#include "qaoa_internal.cuh"

namespace qaoa {

// One layer's coefficients, 32 bytes in complex128 and double-float.  sigma^2 is FP64,
// or a double-float pair for complex64.
template <typename R>
struct SmallCoef {
    R A, B;
    int unit_a;
    typename std::conditional<sizeof(R) == 4, dfloat, double>::type sigma2;
};
static_assert(sizeof(SmallCoef<double>) == 32 && sizeof(SmallCoef<dfloat>) == 32, "one stride for complex128");

// Bytes of p layers' tables, up to the coefficients behind them.
__host__ __device__ inline size_t small_table_bytes(size_t entry, int p, int m) {
    return (entry * (size_t)p * (size_t)(m + 1) + 15) & ~(size_t)15;
}

template <typename V>
__device__ __forceinline__ uint32_t swz(uint32_t i) {
    return sizeof(V) == 8 ? i ^ ((i >> 4) & 15u) : i ^ ((i >> 3) & 7u) ^ ((i >> 6) & 7u);
}

// An amplitude in FP64.
__device__ __forceinline__ double2 amp_f64(float2 v) { return make_double2(v.x, v.y); }
__device__ __forceinline__ double2 amp_f64(double2 v) { return v; }
__device__ __forceinline__ double2 amp_f64(float4 v) { return make_double2((double)v.x + v.y, (double)v.z + v.w); }

// Calls f(byte offsets of the 2^K members, representative) for this thread's
// orbits in 2^lb amplitudes of shared memory: acting bits [j, j + K), the lowest
// of them standing for the complement when `mir`.
template <typename V, int K, class F>
__device__ __forceinline__ void orbits(int lb, int j, bool mir, const F &f) {
    const uint32_t L = 1u << lb;
    uint32_t m[K];
#pragma unroll
    for (int q = 0; q < K; ++q) m[q] = swz<V>(q == 0 && mir ? L - 1u : 1u << (j + q)) * (uint32_t)sizeof(V);
    for (uint32_t g = threadIdx.x; g < L >> K; g += blockDim.x) {
        const uint32_t z0 = ((g >> j) << (j + K)) | (g & ((1u << j) - 1u));
        uint32_t off[1 << K];
        off[0] = swz<V>(z0) * (uint32_t)sizeof(V);
#pragma unroll
        for (int q = 0; q < K; ++q)
#pragma unroll
            for (int r = 0; r < (1 << q); ++r) off[r | (1 << q)] = off[r] ^ m[q];
        f(off, z0);
    }
}

template <typename V>
__device__ __forceinline__ V &at(V *s, uint32_t off) {
    return *reinterpret_cast<V *>(reinterpret_cast<char *>(s) + off);
}

// The costs of 2^K consecutive amplitudes (sc aligned to them).
template <int K>
struct CostBytes {
    uint32_t w[K > 2 ? 1 << (K - 2) : 1];
    __device__ __forceinline__ explicit CostBytes(const uint8_t *sc) {
        if constexpr (K == 1) {
            w[0] = *reinterpret_cast<const uint16_t *>(sc);
        } else if constexpr (K == 2) {
            w[0] = *reinterpret_cast<const uint32_t *>(sc);
        } else if constexpr (K == 3) {
            const uint2 t = *reinterpret_cast<const uint2 *>(sc);
            w[0] = t.x, w[1] = t.y;
        } else {
            const uint4 t = *reinterpret_cast<const uint4 *>(sc);
            w[0] = t.x, w[1] = t.y, w[2] = t.z, w[3] = t.w;
        }
    }
    __device__ __forceinline__ uint32_t operator[](int r) const { return (w[r >> 2] >> (8 * (r & 3))) & 0xFFu; }
};

// K butterflies on an orbit.
template <bool UA, int K, typename V, typename R>
__device__ __forceinline__ void orbit_bfly(V *v, R A, R B) {
#pragma unroll
    for (int q = 0; q < K; ++q)
#pragma unroll
        for (int i = 0; i < (1 << K); ++i)
            if (!(i & (1 << q))) bfly<UA>(v[i], v[i | (1 << q)], A, B);
}

// The phase table of one layer, fetched ahead into registers (entries tid + k
// blockDim) and put into shared memory later; entries above m are zero.
constexpr int TAB_REGS = MAX_TABLE / 128;  // at least 128 threads
template <typename V>
struct TabAhead {
    V e[TAB_REGS];
    __device__ __forceinline__ void fetch(const V *tb, int m, bool last = false) {
#pragma unroll
        for (int k = 0; k < TAB_REGS; ++k) {
            const int c = (int)(threadIdx.x + k * blockDim.x);
            memset(&e[k], 0, sizeof(V));
            if (c < MAX_TABLE && (c <= m || last)) e[k] = tb[c <= m ? c : m];
        }
    }
    __device__ __forceinline__ void put(V *stab) const {
#pragma unroll
        for (int k = 0; k < TAB_REGS; ++k) {
            const int c = (int)(threadIdx.x + k * blockDim.x);
            if (c < MAX_TABLE) stab[c] = e[k];
        }
    }
};

}  // namespace qaoa

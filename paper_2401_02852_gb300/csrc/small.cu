// K6: whole evolutions and gradients of small instances, state resident in
// shared memory, one thread-block cluster per instance.
//
// The 2^nb amplitudes (nb = n, or n - 1 when the cost table is flip-symmetric,
// C(x) = C(not x): then psi(x) = psi(not x) and only the x with bit n-1 clear
// are held) are spread over the 2^CB CTAs of a cluster by their top CB index
// bits.  A layer is a sequence of rounds: each thread takes whole orbits of K
// generators (2^K amplitudes) into registers, butterflies them and puts them
// back, in place, with a barrier between rounds.  The generators are the
// factors X_j, j < nb, each flipping one index bit, and for a halved state
// X_{n-1}, which there maps index z to its complement (flips every bit).  An
// orbit is enumerated by its representative z0, whose K acting bits are zero;
// every other member's index is z0 XOR a constant of the round, so any set of
// generators with independent acting bits fits the same code.  Local rounds
// cover the CTA's own bits; with CB > 0 one remote round per layer covers the
// CTA bits and the complement through distributed shared memory.
//
// The layout permutes the low index bits by XOR with higher ones (linear over
// XOR, so a member's address is the representative's XOR a constant), which
// spreads every round's accesses over the banks.
//
// FP64 instances are bound by the FP64 pipe (2 FMA per SM and clock: 2 FMA per
// amplitude and generator), the others by the rounds' latency (shared memory,
// address arithmetic, barriers; about 0.5 us a round).  Before (one CTA per
// instance on the full state, radix-4 passes over shared memory, FP64 tables):
// n = 12, p = 5, 100 instances FP64 172 -> 86 us, double-float 83 -> 45,
// complex64 45 -> 24; one FP64 instance 171 -> 49 us (a cluster of 8); 400 x n =
// 13, p = 10 complex64 291 -> 102 us.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "orbits.cuh"
#include "pass_common.cuh"
#include "qaoa_internal.cuh"

namespace qaoa {

namespace cg = cooperative_groups;

constexpr int SMALL_PT = 256;     // threads of a CTA that is alone
constexpr int SMALL_PT_CL = 128;  // ... in a cluster
constexpr int SMALL_SYM_N = 6;    // smallest n held as a half

// Where a CTA's part of the state lies and how its orbits are addressed.
template <typename V, int CB>
struct Part {
    int lb;          // log2 amplitudes of this CTA
    uint32_t rank;   // its place in the cluster: the top CB index bits
    bool sym;        // halved state
    // local rounds of a layer: the first `bigger` of `rounds` take `k` + 1
    // generators, the others k; the last one of a halved state ends with the
    // complement (CB = 0)
    int rounds, k, bigger;
    // At most 4 generators per round, and at least 128 orbits (FP64, whose
    // pipes want a warp on each quarter of the SM) or 256 (the rest).
    __device__ __forceinline__ void plan(bool fp64) {
        const int G = lb + (sym && CB == 0 ? 1 : 0);
        const int kmax = fp64 ? max(1, min(4, lb - 7)) : max(2, min(4, lb - 8));
        rounds = (G + kmax - 1) / kmax;
        k = G / rounds;
        bigger = G - k * rounds;
    }
    __device__ __forceinline__ V *peer(V *s, uint32_t r) const {
        if constexpr (CB == 0)
            return s;
        else
            return cg::this_cluster().map_shared_rank(s, r);
    }
};

// The same for remote round i: generators 2 i and 2 i + 1 of [the complement
// (halved states), CTA bit 0, CTA bit 1, ...].  The complement's acting bit is
// the CTA's top local bit; with it or without, the members of an orbit lie at
// one or two local indices of 2^K or 2^(K-1) CTAs.  The orbits are split evenly
// over the cluster.
template <typename V, int K, bool MIR, int CB, class F>
__device__ __forceinline__ void remote_orbits(const Part<V, CB> &pt, int bit, const F &f) {
    constexpr uint32_t C = 1u << CB;
    constexpr int KR = MIR ? K - 1 : K;  // CTA bits [bit, bit + KR) of this round
    const uint32_t L = 1u << pt.lb, per = L >> K;
    const int gl = MIR ? pt.lb - 1 : pt.lb;  // representative: gl local bits, then the other CTA bits
    for (uint32_t i = threadIdx.x; i < per; i += blockDim.x) {
        const uint32_t g = pt.rank * per + i, loc = g & ((1u << gl) - 1u), hi = g >> gl;
        const uint32_t rk0 = ((hi >> bit) << (bit + KR)) | (hi & ((1u << bit) - 1u));
        const uint32_t at = swz<V>(loc), atm = swz<V>(loc ^ (L - 1u));
        f([&](V *s, int r) {
            const bool m = MIR && (r & 1);
            const uint32_t rk = rk0 ^ ((uint32_t)(MIR ? r >> 1 : r) << bit) ^ (m ? C - 1u : 0u);
            return pt.peer(s, rk) + (m ? atm : at);
        });
    }
}

// The remote rounds of a layer, f(integral_constant<K>, bool_constant<MIR>, bit):
// two generators each, so that the orbits keep every warp busy.
template <int CB, class F>
__device__ __forceinline__ void remote_rounds(bool sym, const F &f) {
    if constexpr (CB > 0) {
        int bit = 0;
        if (sym) {
            f(std::integral_constant<int, 2>{}, std::true_type{}, 0);
            bit = 1;
        }
        for (; bit < CB; bit += 2) {
            if (bit + 1 < CB)
                f(std::integral_constant<int, 2>{}, std::false_type{}, bit);
            else
                f(std::integral_constant<int, 1>{}, std::false_type{}, bit);
        }
    }
}

// The local rounds of a layer, f(integral_constant<K>, j, mir, first, last).
template <typename V, int CB, class F>
__device__ __forceinline__ void local_rounds(const Part<V, CB> &pt, const F &f) {
    int j = 0;
    for (int i = 0; i < pt.rounds; ++i) {
        const int k = pt.k + (i < pt.bigger ? 1 : 0);
        const bool first = i == 0, last = i == pt.rounds - 1, mir = CB == 0 && pt.sym && last;
        const int jj = mir ? pt.lb - k : j;
        if (k == 4)
            f(std::integral_constant<int, 4>{}, jj, mir, first, last);
        else if (k == 3)
            f(std::integral_constant<int, 3>{}, jj, mir, first, last);
        else if (k == 2)
            f(std::integral_constant<int, 2>{}, jj, mir, first, last);
        else
            f(std::integral_constant<int, 1>{}, jj, mir, first, last);
        j += k;
    }
}

template <int CB>
__device__ __forceinline__ void barrier(bool wide) {
    if constexpr (CB > 0) {
        if (wide) {
            cg::this_cluster().sync();
            return;
        }
    }
    __syncthreads();
}

// The inverse butterflies with B = 1, (a, b) <- (A a - i b, A b - i a).
template <int K, typename V, typename R>
__device__ __forceinline__ void inv_orbit(V *v, R A) {
#pragma unroll
    for (int q = 0; q < K; ++q)
#pragma unroll
        for (int i = 0; i < (1 << K); ++i) {
            if (i & (1 << q)) continue;
            V &a = v[i], &b = v[i | (1 << q)];
            const V x = a;
            a.x = fma(A, x.x, b.y);
            a.y = fma(A, x.y, -b.x);
            const V y = b;
            b.x = fma(A, y.x, x.y);
            b.y = fma(A, y.y, -x.x);
        }
}

// Is the instance's table flip-symmetric?  Each CTA reads its share of the
// table (16 bytes at a time when the table is aligned); a verdict over the
// cluster.
template <int CB>
__device__ __forceinline__ bool table_symmetric(const uint8_t *cost, int n, uint32_t rank, int *s_bad) {
    if (n < SMALL_SYM_N) return false;
    const uint32_t N = 1u << n, nt = blockDim.x << CB, t = rank * blockDim.x + threadIdx.x;
    uint32_t bad = 0;
    if ((reinterpret_cast<uintptr_t>(cost) & 15u) == 0) {
        const uint4 *c = reinterpret_cast<const uint4 *>(cost);
        for (uint32_t w = t; w < N / 32; w += nt) {
            const uint4 a = c[w], b = c[N / 16 - 1 - w];
            bad |= (a.x ^ __byte_perm(b.w, 0, 0x0123)) | (a.y ^ __byte_perm(b.z, 0, 0x0123)) |
                   (a.z ^ __byte_perm(b.y, 0, 0x0123)) | (a.w ^ __byte_perm(b.x, 0, 0x0123));
        }
    } else {
        for (uint32_t x = t; x < N / 2; x += nt) bad |= (uint32_t)(cost[x] ^ cost[N - 1 - x]);
    }
    int any = __syncthreads_or(bad != 0);
    if constexpr (CB > 0) {
        cg::cluster_group cl = cg::this_cluster();
        if (threadIdx.x == 0) *s_bad = any;
        cl.sync();
        any = 0;
        for (uint32_t r = 0; r < (1u << CB); ++r) any |= *cl.map_shared_rank(s_bad, r);
    }
    return any == 0;
}

// This CTA's cost bytes, by local index.
__device__ __forceinline__ void load_costs(uint8_t *sc, const uint8_t *cost, uint32_t z0, uint32_t L) {
    const uint8_t *c = cost + z0;
    if (L >= 16 && (reinterpret_cast<uintptr_t>(c) & 15u) == 0) {
        for (uint32_t i = threadIdx.x; i < L / 16; i += blockDim.x)
            reinterpret_cast<uint4 *>(sc)[i] = reinterpret_cast<const uint4 *>(c)[i];
    } else {
        for (uint32_t i = threadIdx.x; i < L; i += blockDim.x) sc[i] = c[i];
    }
}

// p >= 1 layers forward from |+>; s holds the CTA's part afterwards.  tb0, cf0:
// the layers' tables [p][m + 1] and coefficients [p].  LAST: a cost above m takes
// the phase of m (gradients do, as their phase terms' weights).  On return the last
// layer's table is in stab + ((p - 1) & 1) MAX_TABLE and the state is visible to
// the whole cluster.
template <typename R, int CB, bool LAST, typename V>
__device__ __forceinline__ void forward_layers(const Part<V, CB> &pt, V *s, V *stab, const uint8_t *sc, int m, int p,
                                               const V *tb0, const SmallCoef<R> *cf0) {
    TabAhead<V> ahead;
    ahead.fetch(tb0, m, LAST);
    SmallCoef<R> cf = cf0[0];
    ahead.put(stab);
    __syncthreads();
    for (int l = 0; l < p; ++l) {
        const V *tab = stab + (l & 1) * MAX_TABLE;
        const R A = cf.A, B = cf.B;
        const bool ua = cf.unit_a != 0, next = l + 1 < p;
        if (next) {
            ahead.fetch(tb0 + (size_t)(l + 1) * (m + 1), m, LAST);
            cf = cf0[l + 1];
        }
        local_rounds(pt, [&](auto kc, int j, bool mir, bool first, bool last) {
            constexpr int K = decltype(kc)::value;
            orbits<V, K>(pt.lb, j, mir, [&](const uint32_t(&off)[1 << K], uint32_t z0) {
                V v[1 << K];
                if (first) {  // j = 0: the members are consecutive
                    const CostBytes<K> c(sc + z0);
                    if (l == 0) {
#pragma unroll
                        for (int r = 0; r < (1 << K); ++r) v[r] = tab[c[r]];
                    } else {
#pragma unroll
                        for (int r = 0; r < (1 << K); ++r) v[r] = cmul(at(s, off[r]), tab[c[r]]);
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < (1 << K); ++r) v[r] = at(s, off[r]);
                }
                if (ua)
                    orbit_bfly<true, K>(v, A, B);
                else
                    orbit_bfly<false, K>(v, A, B);
#pragma unroll
                for (int r = 0; r < (1 << K); ++r) at(s, off[r]) = v[r];
            });
            if (last && next) ahead.put(stab + ((l + 1) & 1) * MAX_TABLE);
            barrier<CB>(last);
        });
        remote_rounds<CB>(pt.sym, [&](auto kc, auto mc, int bit) {
            constexpr int K = decltype(kc)::value;
            remote_orbits<V, K, decltype(mc)::value, CB>(pt, bit, [&](auto where) {
                V v[1 << K];
#pragma unroll
                for (int r = 0; r < (1 << K); ++r) v[r] = *where(s, r);
                if (ua)
                    orbit_bfly<true, K>(v, A, B);
                else
                    orbit_bfly<false, K>(v, A, B);
#pragma unroll
                for (int r = 0; r < (1 << K); ++r) *where(s, r) = v[r];
            });
            barrier<CB>(true);
        });
    }
}

// One cluster of 2^CB CTAs per job: the whole evolution.  complex128 runs in
// FP64, or with QAOA_DF64 in double-float arithmetic (float4 amplitudes in
// shared memory, FP64 (re, im) written out).  Tables [p][m+1] and coefficients
// [p] are in the kernel's own types: converting FP64 ones here took a third of
// the FP64 pipe in complex64 evolutions.
//
// With jobs == nullptr cluster i evolves the batch's instance i of `all`, and
// the tables and coefficients lie in `prm` (kernel parameters) when they fit.
constexpr int SMALL_PRM = 3840;  // bytes: with the other arguments under 4 KiB
struct alignas(16) SmallPrm {
    char x[SMALL_PRM];
};
template <typename R, int CB>
__global__ void __launch_bounds__(CB == 0 ? SMALL_PT : SMALL_PT_CL, CB == 0 ? 2 : 4)
    small_kernel(const SmallJob *jobs, const __grid_constant__ SmallJob all, const void *tables, const void *coefs,
                 int max_n, const __grid_constant__ SmallPrm prm) {
    using V = typename VecOf<R>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_bad;
    __shared__ double s_sum[2];
    pdl_wait();
    SmallJob jb = all;
    if (jobs) {
        jb = jobs[blockIdx.x >> CB];
    } else {
        const size_t i = blockIdx.x >> CB;
        jb.cost += i << jb.n;
        if (jb.state) jb.state = reinterpret_cast<char *>(jb.state) + ((i << jb.n) * (sizeof(R) == 4 ? 8 : 16));
        if (jb.result) jb.result += 2 * i;
    }
    const int n = jb.n;
    V *s = reinterpret_cast<V *>(smem_raw);
    V *stab = s + ((1u << max_n) >> CB);
    uint8_t *sc = reinterpret_cast<uint8_t *>(stab + 2 * MAX_TABLE);
    Part<V, CB> pt;
    pt.rank = CB > 0 ? blockIdx.x & ((1u << CB) - 1u) : 0u;
    pt.sym = table_symmetric<CB>(jb.cost, n, pt.rank, &s_bad);
    pt.lb = (pt.sym ? n - 1 : n) - CB;
    pt.plan(std::is_same<R, double>::value);
    const uint32_t L = 1u << pt.lb, z0 = pt.rank << pt.lb;
    load_costs(sc, jb.cost, z0, L);
    const V *tb = tables ? reinterpret_cast<const V *>(tables) + jb.table_off : reinterpret_cast<const V *>(prm.x);
    const SmallCoef<R> *cf = coefs ? reinterpret_cast<const SmallCoef<R> *>(coefs) + jb.coef_off
                                   : reinterpret_cast<const SmallCoef<R> *>(
                                         prm.x + small_table_bytes(sizeof(V), max(jb.p, 1), jb.m));
    if (jb.p > 0) {
        forward_layers<R, CB, false>(pt, s, stab, sc, jb.m, jb.p, tb, cf);
    } else {  // |+>: the table of "layer 0" holds the amplitude
        const V z = tb[0];
        for (uint32_t i = threadIdx.x; i < L; i += blockDim.x) s[i] = z;
        barrier<CB>(true);
    }
    double acc[2] = {0.0, 0.0};
    double2 *out2 = reinterpret_cast<double2 *>(jb.state);
    V *out = reinterpret_cast<V *>(jb.state);
    for (uint32_t i = threadIdx.x; i < L; i += blockDim.x) {
        const V v = s[swz<V>(i)];
        const double2 d = amp_f64(v);
        const double w = d.x * d.x + d.y * d.y;
        const uint32_t z = z0 + i, zc = (1u << n) - 1u - z;
        if (jb.state) {
            if constexpr (std::is_same<R, dfloat>::value) {
                out2[z] = d;
                if (pt.sym) out2[zc] = d;
            } else {
                out[z] = v;
                if (pt.sym) out[zc] = v;
            }
        }
        acc[1] += w;
        if (sc[i] == 0) acc[0] += w;
    }
    if (!jb.result) return;  // no other CTA reads this one's shared memory from here on
    block_sum<2, CB == 0 ? SMALL_PT : SMALL_PT_CL>(acc);
    const double f = pt.sym ? 2.0 : 1.0;  // each amplitude stands for its complement too
    if constexpr (CB > 0) {
        cg::cluster_group cl = cg::this_cluster();
        if (threadIdx.x == 0) s_sum[0] = acc[0], s_sum[1] = acc[1];
        cl.sync();
        if (pt.rank == 0 && threadIdx.x == 0) {
            double a = 0.0, b = 0.0;
            for (uint32_t r = 0; r < (1u << CB); ++r) {
                const double *q = cl.map_shared_rank(s_sum, r);
                a += q[0];
                b += q[1];
            }
            jb.result[0] = f * a;
            jb.result[1] = f * b;
        }
        cl.sync();  // the sums stay until they are read
    } else if (threadIdx.x == 0) {
        jb.result[0] = f * acc[0];
        jb.result[1] = f * acc[1];
    }
}

// ---------------------------------------------------------------------------
// Gradient of small instances: forward as above, then the reverse sweep on psi
// and lam = P psi (see adjoint.cu), both states resident.
//
// The inverse layers run in the factored form too: M_l^dagger = sigma^n prod_j
// [A I - i B X_j], so a round that starts after g generators holds both states
// times sigma^-g each, and its pair terms Im(conj(lam_x) psi_(x^j) + ...) count
// with sigma^(2 g).  Every X_j commutes with the inverse butterflies, so the
// terms of a round's K generators are taken together at its start, two
// generators at a time: for the four amplitudes 00, 01, 10, 11 of a pair of
// generators they sum to Im[conj(l00 + l11)(p01 + p10) + conj(l01 + l10)(p00 +
// p11)], 12 operations instead of 16.  sigma^n and the phase are undone with the
// forward table's conjugate, at the start of the next layer's first round
// (local, like the cost bytes).  In complex64 the sums of p_succ and the norm are FP64
// and the powers of sigma double-float products (32 x n = 12, p = 4, beta derivatives'
// error against 80 bits 9.2e-8 with FP32 ones, 6.2e-8 with these; 100 x n = 12, p = 16 147
// and 143 us).  Two passes of FP64 work per layer and amplitude:
// 2 n + 4 operations forward, about 5.5 n + 11 backward.  (100 instances of n =
// 12, p = 16 in FP64: 3.50 ms with one CTA per instance on the full states and
// normalised radix-2 butterflies, 1.05 ms here; the operations alone take 0.83
// ms on 100 SMs, 0.55 on all.)

// Im of the sum over generators q of conj(l_r) p_(r ^ 2^q), r over the orbit.
template <int K, typename V, typename R>
__device__ __forceinline__ R pair_terms(const V *p, const V *l, R t) {
#pragma unroll
    for (int q = 0; q + 1 < K; q += 2)
#pragma unroll
        for (int r = 0; r < (1 << K); ++r) {
            if ((r >> q) & 3) continue;
            const int r1 = r | (1 << q), r2 = r | (2 << q), r3 = r | (3 << q);
            const R px = p[r1].x + p[r2].x, py = p[r1].y + p[r2].y, qx = p[r].x + p[r3].x, qy = p[r].y + p[r3].y;
            const R lx = l[r].x + l[r3].x, ly = l[r].y + l[r3].y, mx = l[r1].x + l[r2].x, my = l[r1].y + l[r2].y;
            t = fma(lx, py, t);
            t = fma(-ly, px, t);
            t = fma(mx, qy, t);
            t = fma(-my, qx, t);
        }
    if constexpr (K & 1) {
        constexpr int q = K - 1;
#pragma unroll
        for (int r = 0; r < (1 << q); ++r) {
            const int r1 = r | (1 << q);
            t = fma(l[r].x, p[r1].y, t);
            t = fma(-l[r].y, p[r1].x, t);
            t = fma(l[r1].x, p[r].y, t);
            t = fma(-l[r1].y, p[r].x, t);
        }
    }
    return t;
}

// The weight sigma^(2 g) of a round after g generators, w sigma^(2 K) after the next: in
// complex64 a double-float product, of which a round takes the nearest float.
__device__ __forceinline__ double one_weight(double) { return 1.0; }
__device__ __forceinline__ dfloat one_weight(dfloat) { return dfloat{1.f, 0.f}; }
__device__ __forceinline__ double weight_of(double w) { return w; }
__device__ __forceinline__ float weight_of(dfloat w) { return w.hi; }
template <int K>
__device__ __forceinline__ double weigh(double w, double s2) {
#pragma unroll
    for (int q = 0; q < K; ++q) w *= s2;
    return w;
}
template <int K>
__device__ __forceinline__ dfloat weigh(dfloat w, dfloat s2) {
#pragma unroll
    for (int q = 0; q < K; ++q) w = df_mul(w, s2.hi, s2.lo);
    return w;
}

// out: [instance][CTA of its cluster][1 + p][2]: the CTA's share of (p_succ,
// norm), then of (mixer term, phase term) of each layer.
template <typename R, int CB>
__global__ void __launch_bounds__(CB == 0 ? SMALL_PT : SMALL_PT_CL, CB == 0 ? 1 : 2)
    small_grad_kernel(const uint8_t *costs, int n, int m, int p, const void *tables, const void *coefs, double *out) {
    using V = typename VecOf<R>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_bad;
    __shared__ double2 s_red[CB == 0 ? SMALL_PT : SMALL_PT_CL];
    pdl_wait();
    const uint8_t *cost = costs + ((size_t)(blockIdx.x >> CB) << n);
    V *s = reinterpret_cast<V *>(smem_raw);
    V *sl = s + ((1u << n) >> CB);
    V *stab = sl + ((1u << n) >> CB);
    uint8_t *sc = reinterpret_cast<uint8_t *>(stab + 2 * MAX_TABLE);
    Part<V, CB> pt;
    pt.rank = CB > 0 ? blockIdx.x & ((1u << CB) - 1u) : 0u;
    pt.sym = table_symmetric<CB>(cost, n, pt.rank, &s_bad);
    pt.lb = (pt.sym ? n - 1 : n) - CB;
    pt.plan(std::is_same<R, double>::value);
    const uint32_t L = 1u << pt.lb;
    load_costs(sc, cost, pt.rank << pt.lb, L);
    const V *tb = reinterpret_cast<const V *>(tables);
    const SmallCoef<R> *cfs = reinterpret_cast<const SmallCoef<R> *>(coefs);
    forward_layers<R, CB, true>(pt, s, stab, sc, m, p, tb, cfs);
    double *o = out + (size_t)blockIdx.x * 2 * (1 + p);
    const double f = pt.sym ? 2.0 : 1.0;  // each amplitude stands for its complement too
    // The threads' shares of output row i, summed by the first warp: written
    // before a barrier, summed after it (and before the next row's).
    auto share = [&](double a, double b) { s_red[threadIdx.x] = make_double2(a, b); };
    auto emit = [&](int i) {
        if (threadIdx.x < 32) {
            double x[2] = {0.0, 0.0};
            for (int w = threadIdx.x; w < (int)blockDim.x; w += 32) x[0] += s_red[w].x, x[1] += s_red[w].y;
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) {
                x[0] += __shfl_xor_sync(0xFFFFFFFFu, x[0], d);
                x[1] += __shfl_xor_sync(0xFFFFFFFFu, x[1], d);
            }
            if (threadIdx.x == 0) {
                o[2 * i] = f * x[0];
                o[2 * i + 1] = f * x[1];
            }
        }
    };
    TabAhead<V> ahead;
    SmallCoef<R> cf = cfs[p - 1];
    double prev_term = 0.0, prev_w = 0.0;  // of layer l + 1: its mixer term, sigma^(2 n)
    for (int l = p - 1; l >= 0; --l) {
        // the table of layer l + 1 (whose phase this layer's first round undoes)
        // is in buffer (l + 1) & 1; layer l's goes into the other
        const V *tab = stab + ((l + 1) & 1) * MAX_TABLE;
        const R A = cf.unit_a ? (R)1 : cf.A, B = cf.unit_a ? -cf.B : (R)-1;
        const bool ua = cf.unit_a != 0, seed = l == p - 1;
        const auto sg2 = cf.sigma2;
        if (!seed) ahead.fetch(tb + (size_t)l * (m + 1), m, true);
        if (l > 0) cf = cfs[l - 1];
        R term = 0;
        auto w = one_weight(sg2);
        local_rounds(pt, [&](auto kc, int j, bool mir, bool first, bool last) {
            constexpr int K = decltype(kc)::value;
            R t = 0, g = 0;
            double q0 = 0.0, q1 = 0.0;
            orbits<V, K>(pt.lb, j, mir, [&](const uint32_t(&off)[1 << K], uint32_t z0) {
                V v[1 << K], u[1 << K];
#pragma unroll
                for (int r = 0; r < (1 << K); ++r) v[r] = at(s, off[r]);
                if (first && seed) {  // lam = P psi, and p_succ, norm
                    const CostBytes<K> c(sc + z0);
#pragma unroll
                    for (int r = 0; r < (1 << K); ++r) {
                        const bool sol = c[r] == 0;
                        double2 d;
                        if constexpr (sizeof(R) == 4)
                            d = make_double2(widen(v[r].x), widen(v[r].y));
                        else
                            d = amp_f64(v[r]);
                        const double q = d.x * d.x + d.y * d.y;
                        q1 += q;
                        if (sol) q0 += q;
                        u[r].x = sol ? v[r].x : (R)0;
                        u[r].y = sol ? v[r].y : (R)0;
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < (1 << K); ++r) u[r] = at(sl, off[r]);
                    if (first) {  // layer l + 1: phase term, then D^dagger sigma^n
                        const CostBytes<K> c(sc + z0);
#pragma unroll
                        for (int r = 0; r < (1 << K); ++r) {
                            const int cst = min((int)c[r], m);
                            g += (R)cst * (u[r].x * v[r].y - u[r].y * v[r].x);
                            V ph = tab[cst];
                            ph.y = -ph.y;
                            v[r] = cmul(v[r], ph);
                            u[r] = cmul(u[r], ph);
                        }
                    }
                }
                t = pair_terms<K>(v, u, t);
                if (ua) {
                    orbit_bfly<true, K>(v, A, B);
                    orbit_bfly<true, K>(u, A, B);
                } else {
                    inv_orbit<K>(v, A);
                    inv_orbit<K>(u, A);
                }
#pragma unroll
                for (int r = 0; r < (1 << K); ++r) {
                    at(s, off[r]) = v[r];
                    at(sl, off[r]) = u[r];
                }
            });
            term = fma(weight_of(w), t, term);
            w = weigh<K>(w, sg2);
            if (first) {  // (p_succ, norm), or layer l + 1 done
                if (seed)
                    share(q0, q1);
                else
                    share(prev_term, prev_w * (double)g);
            }
            if (last && !seed) ahead.put(stab + (l & 1) * MAX_TABLE);
            barrier<CB>(last);
            if (first) {
                emit(seed ? 0 : l + 2);
                if (first && last) barrier<CB>(false);  // one round: the next row's shares wait for this sum
            }
        });
        remote_rounds<CB>(pt.sym, [&](auto kc, auto mc, int bit) {
            constexpr int K = decltype(kc)::value;
            R t = 0;
            remote_orbits<V, K, decltype(mc)::value, CB>(pt, bit, [&](auto where) {
                V v[1 << K], u[1 << K];
#pragma unroll
                for (int r = 0; r < (1 << K); ++r) {
                    v[r] = *where(s, r);
                    u[r] = *where(sl, r);
                }
                t = pair_terms<K>(v, u, t);
                if (ua) {
                    orbit_bfly<true, K>(v, A, B);
                    orbit_bfly<true, K>(u, A, B);
                } else {
                    inv_orbit<K>(v, A);
                    inv_orbit<K>(u, A);
                }
#pragma unroll
                for (int r = 0; r < (1 << K); ++r) {
                    *where(s, r) = v[r];
                    *where(sl, r) = u[r];
                }
            });
            term = fma(weight_of(w), t, term);
            w = weigh<K>(w, sg2);
            barrier<CB>(true);
        });
        prev_term = (double)term;
        prev_w = (double)weight_of(w);
    }
    // layer 0's phase term
    R g = 0;
    for (uint32_t i = threadIdx.x; i < L; i += blockDim.x) {
        const V v = s[swz<V>(i)], u = sl[swz<V>(i)];
        g += (R)min((int)sc[i], m) * (u.x * v.y - u.y * v.x);
    }
    share(prev_term, prev_w * (double)g);
    __syncthreads();
    emit(1);
}

int small_n_limit(int dtype) { return dtype == QAOA_C64 ? T_C64 : T_C128; }
int small_n_pack_limit(int dtype) { return dtype == QAOA_C64 ? 14 : 13; }

// Dynamic shared memory of one CTA: `states` parts of the state (the whole one,
// as an asymmetric table needs it), two phase tables, the cost bytes.
static size_t small_smem(int dtype, int max_n, int cb, int states) {
    const size_t es = dtype == QAOA_C64 ? sizeof(float2) : sizeof(double2), L = (size_t(1) << max_n) >> cb;
    return es * (states * L + 2 * MAX_TABLE) + ((L + 15) & ~(size_t)15);
}

static int launch_clusters(const void *kernel, int n_clusters, int cb, int threads, size_t smem, cudaStream_t stream,
                           void **args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_clusters << cb);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = 1u << cb;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cb > 0 ? 2 : 1;
    QAOA_CUDA_TRY(cudaLaunchKernelExC(&cfg, kernel, args));
    return QAOA_OK;
}

// Cluster size (log2) for `count` FP64 evolutions of n qubits: the least of
//   ceil(count 2^cb / SMs) W / 2^cb + V(cb)
// with W the FP64 clocks of one layer on one SM (2 FMA per clock) and V the
// clocks a layer takes beside them, measured on one n = 12 instance: 4, 6.5, 8.7
// and 11.6 thousand for clusters of 1, 2, 4 and 8 (barriers and distributed
// shared memory; per layer 15.8, 10.1, 7.7 and 7.4 us).  From one instance per SM
// on the pipe is busy anyway (500 x n = 10, p = 10: 0.17 ms alone, 0.26 in pairs).
// The other arithmetics are not bound by their pipe and take one CTA.
static int small_cluster(int n, int count, int sms) {
    if (n < 10 || count >= sms) return 0;
    const double W = std::ldexp(1.0, n - 1) * (2 * n + 4) / 2, V[4] = {4.0e3, 6.5e3, 8.7e3, 11.6e3};
    int best = 0;
    double least = 0.0;
    for (int cb = 0; cb < 4; ++cb) {
        const double waves = std::ceil((double)count * (1 << cb) / sms), t = waves * W / (1 << cb) + V[cb];
        if (cb == 0 || t < least) best = cb, least = t;
    }
    return best;
}

// Kernel attributes once per device.
template <class F>
static int once_per_device(int *state, std::mutex &mu, const F &set) {
    const int dev = current_device_slot();
    if (dev < 0) return QAOA_ECUDA;
    std::lock_guard<std::mutex> lk(mu);
    if (!state[dev]) {
        const cudaError_t e = set();
        if (e != cudaSuccess) return cuda_error(e, "small-n kernel attributes");
        state[dev] = 1;
    }
    return QAOA_OK;
}

static int small_launch(int dtype, int flags, int count, const SmallJob *d_jobs, const SmallJob &all,
                        const void *d_tables, const void *d_coefs, int max_n, const SmallPrm &prm, int cb,
                        cudaStream_t stream) {
    static std::mutex mu;
    static int state[MAX_DEVICES] = {};
    static const void *kd[4] = {(const void *)small_kernel<double, 0>, (const void *)small_kernel<double, 1>,
                                (const void *)small_kernel<double, 2>, (const void *)small_kernel<double, 3>};
    static const void *kf = (const void *)small_kernel<float, 0>, *kx = (const void *)small_kernel<dfloat, 0>;
    int rc = once_per_device(state, mu, [&] {
        const int bf = (int)small_smem(QAOA_C64, small_n_pack_limit(QAOA_C64), 0, 1);
        cudaError_t e = cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, bf);
        for (int c = 0; c < 4 && e == cudaSuccess; ++c) {
            const int bd = (int)small_smem(QAOA_C128, small_n_pack_limit(QAOA_C128), c, 1);
            e = cudaFuncSetAttribute(kd[c], cudaFuncAttributeMaxDynamicSharedMemorySize, bd);
            if (c == 0 && e == cudaSuccess) e = cudaFuncSetAttribute(kx, cudaFuncAttributeMaxDynamicSharedMemorySize, bd);
        }
        return e;
    });
    if (rc) return rc;
    const int threads = cb == 0 ? SMALL_PT : SMALL_PT_CL;
    void *args[] = {(void *)&d_jobs, (void *)&all, (void *)&d_tables, (void *)&d_coefs, (void *)&max_n, (void *)&prm};
    const void *k = dtype == QAOA_C64 ? kf : ((flags & QAOA_DF64) ? kx : kd[cb]);
    profile_before(K_SMALL_N, stream);
    rc = launch_clusters(k, count, cb, threads, small_smem(dtype, max_n, cb, 1), stream, args);
    if (rc) return rc;
    return profile_after(K_SMALL_N, stream);
}

int launch_small_batch(int dtype, int n_jobs, const SmallJob *d_jobs, const void *d_tables, const void *d_coefs,
                       int max_n, int flags, cudaStream_t stream) {
    static const SmallPrm none{};
    return small_launch(dtype, flags, n_jobs, d_jobs, SmallJob{}, d_tables, d_coefs, max_n, none, 0, stream);
}

// One layer's table and coefficients in the kernel's types.
template <typename R>
static void fill_layer(int n, int m, double gamma, double beta, bool layer, bool first, int sign, int arith, void *tab,
                       void *coef) {
    using V = typename VecOf<R>::type;
    const LayerCoef k = layer ? layer_coef(beta, sign, arith) : LayerCoef{1.0, 1.0, 0.0, true};
    double scale = layer_scale(k, n);
    if (first) scale *= std::pow(2.0, -0.5 * n);
    double re[MAX_TABLE], im[MAX_TABLE];
    phase_table(layer ? gamma : 0.0, scale, m, arith, re, im);
    V *t = reinterpret_cast<V *>(tab);
    for (int c = 0; c <= m; ++c) {
        if constexpr (std::is_same<R, dfloat>::value) {
            const float rh = (float)re[c], ih = (float)im[c];
            t[c] = make_float4(rh, (float)(re[c] - (double)rh), ih, (float)(im[c] - (double)ih));
        } else {
            t[c].x = (R)re[c];
            t[c].y = (R)im[c];
        }
    }
    SmallCoef<R> *q = reinterpret_cast<SmallCoef<R> *>(coef);
    q->unit_a = k.unit_a ? 1 : 0;
    const double s2 = layer_sigma2(k);
    if constexpr (sizeof(R) == 4)
        q->sigma2 = dfloat{(float)s2, (float)(s2 - (double)(float)s2)};
    else
        q->sigma2 = s2;
    if constexpr (std::is_same<R, dfloat>::value) {
        const float a = (float)k.A, b = (float)k.B;
        q->A = dfloat{a, (float)(k.A - (double)a)};
        q->B = dfloat{b, (float)(k.B - (double)b)};
    } else {
        q->A = (R)k.A;
        q->B = (R)k.B;
    }
}

size_t small_entry_bytes(int dtype) { return dtype == QAOA_C64 ? sizeof(float2) : sizeof(double2); }
size_t small_coef_bytes(int dtype) { return dtype == QAOA_C64 ? sizeof(SmallCoef<float>) : sizeof(SmallCoef<double>); }

void small_fill_layers(int dtype, int flags, int n, int m, int p, const double *gamma, const double *beta, void *tab,
                       void *coef) {
    const int sign = (flags & QAOA_MIXER_RX2B) ? -1 : 1, arith = arith_of(dtype, flags), pl = p > 0 ? p : 1;
    char *t = reinterpret_cast<char *>(tab), *c = reinterpret_cast<char *>(coef);
    for (int l = 0; l < pl; ++l) {
        const double g = p > 0 ? gamma[l] : 0.0, b = p > 0 ? beta[l] : 0.0;
        if (dtype == QAOA_C64)
            fill_layer<float>(n, m, g, b, p > 0, l == 0, sign, arith, t, c);
        else if (flags & QAOA_DF64)
            fill_layer<dfloat>(n, m, g, b, p > 0, l == 0, sign, arith, t, c);
        else
            fill_layer<double>(n, m, g, b, p > 0, l == 0, sign, arith, t, c);
        t += small_entry_bytes(dtype) * (size_t)(m + 1);
        c += small_coef_bytes(dtype);
    }
}

size_t small_stage_bytes(int dtype, int m, int p) {
    const int pl = p > 0 ? p : 1;
    const size_t b = small_table_bytes(small_entry_bytes(dtype), pl, m) + small_coef_bytes(dtype) * (size_t)pl;
    return b <= (size_t)SMALL_PRM ? 0 : b;
}

int evolve_small(const EvolveReq &r, void *h_stage, void *d_stage, cudaStream_t stream) {
    const size_t bytes = small_stage_bytes(r.dtype, r.m, r.p);
    const size_t tab = small_table_bytes(small_entry_bytes(r.dtype), r.p > 0 ? r.p : 1, r.m);
    SmallPrm prm;
    char *h = bytes ? reinterpret_cast<char *>(h_stage) : prm.x;
    small_fill_layers(r.dtype, r.flags, r.n, r.m, r.p, r.gamma, r.beta, h, h + tab);
    const char *d_tab = nullptr;
    if (bytes) {
        QAOA_CUDA_TRY(cudaMemcpyAsync(d_stage, h_stage, bytes, cudaMemcpyHostToDevice, stream));
        d_tab = reinterpret_cast<const char *>(d_stage);
    }
    const SmallJob all{r.cost, r.state, r.d_result, r.n, r.m, r.p, 0, 0};
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc) return rc;
    const int cb = r.dtype == QAOA_C128 && !(r.flags & QAOA_DF64) ? small_cluster(r.n, r.batch, di.sms) : 0;
    rc = small_launch(r.dtype, r.flags, r.batch, nullptr, all, d_tab, d_tab ? d_tab + tab : nullptr, r.n, prm, cb,
                      stream);
    if (rc) return rc;
    // the pinned staging block is reused by the next call on this stream, and the
    // results are the caller's to read
    if (bytes || r.d_result) QAOA_CUDA_TRY(cudaStreamSynchronize(stream));
    return QAOA_OK;
}

template <typename R>
static int grad_small_impl(int batch, int n, const uint8_t *cost, int m, int p, const double *gamma, const double *beta,
                           int dtype, int flags, cudaStream_t stream, double *p_succ, double *dgamma, double *dbeta) {
    static std::mutex mu;
    static int state[MAX_DEVICES] = {};
    constexpr int CBS = std::is_same<R, double>::value ? 3 : 0;  // clusters up to 2^CBS (small_cluster)
    static const void *ks[4] = {(const void *)small_grad_kernel<R, 0>, (const void *)small_grad_kernel<R, CBS < 1 ? 0 : 1>,
                                (const void *)small_grad_kernel<R, CBS < 2 ? 0 : 2>,
                                (const void *)small_grad_kernel<R, CBS < 3 ? 0 : 3>};
    int rc = once_per_device(state, mu, [&] {
        cudaError_t e = cudaSuccess;
        for (int c = 0; c <= CBS && e == cudaSuccess; ++c)
            e = cudaFuncSetAttribute(ks[c], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)small_smem(dtype, small_n_limit(dtype), c, 2));
        return e;
    });
    if (rc) return rc;
    DeviceInfo di;
    if ((rc = device_info(&di))) return rc;
    const int cb = CBS > 0 ? small_cluster(n, batch, di.sms) : 0;
    const size_t tab = small_table_bytes(small_entry_bytes(dtype), p, m);
    const size_t in = (tab + small_coef_bytes(dtype) * (size_t)p + 255) & ~(size_t)255;
    Scratch *sc = nullptr;
    if ((rc = scratch_for(stream, in, in + (((size_t)batch << cb) * 2 * (1 + p)) * sizeof(double), &sc))) return rc;
    char *h = reinterpret_cast<char *>(sc->host), *d = reinterpret_cast<char *>(sc->dev);
    small_fill_layers(dtype, flags, n, m, p, gamma, beta, h, h + tab);
    QAOA_CUDA_TRY(cudaMemcpyAsync(d, h, tab + small_coef_bytes(dtype) * (size_t)p, cudaMemcpyHostToDevice, stream));
    // the kernel writes its sums into the pinned block itself
    double *h_out = reinterpret_cast<double *>(h + in);
    const char *d_tab = d, *d_coef = d + tab;
    void *args[] = {(void *)&cost, (void *)&n, (void *)&m, (void *)&p, (void *)&d_tab, (void *)&d_coef, (void *)&h_out};
    profile_before(K_SMALL_N, stream);
    rc = launch_clusters(ks[cb], batch, cb, cb == 0 ? SMALL_PT : SMALL_PT_CL, small_smem(dtype, n, cb, 2), stream, args);
    if (rc) return rc;
    if ((rc = profile_after(K_SMALL_N, stream))) return rc;
    QAOA_CUDA_TRY(cudaStreamSynchronize(stream));
    const int sign = (flags & QAOA_MIXER_RX2B) ? -1 : 1;
    for (int b = 0; b < batch; ++b)
        for (int i = 0; i <= p; ++i) {
            double x = 0.0, y = 0.0;  // over the cluster, in order
            for (int r = 0; r < (1 << cb); ++r) {
                const double *o = h_out + 2 * ((((size_t)b << cb) + r) * (1 + p) + i);
                x += o[0];
                y += o[1];
            }
            if (i == 0) {
                if (p_succ) p_succ[b] = x;
            } else {
                dbeta[(size_t)b * p + i - 1] = -2.0 * sign * x;
                dgamma[(size_t)b * p + i - 1] = 2.0 * y;
            }
        }
    return QAOA_OK;
}

int grad_small(int batch, int n, const uint8_t *cost, int m, int p, const double *gamma, const double *beta, int dtype,
               int flags, cudaStream_t stream, double *p_succ, double *dgamma, double *dbeta) {
    return dtype == QAOA_C64 ? grad_small_impl<float>(batch, n, cost, m, p, gamma, beta, dtype, flags, stream, p_succ,
                                                      dgamma, dbeta)
                             : grad_small_impl<double>(batch, n, cost, m, p, gamma, beta, dtype, flags, stream, p_succ,
                                                       dgamma, dbeta);
}

}  // namespace qaoa

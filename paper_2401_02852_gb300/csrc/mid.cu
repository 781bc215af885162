// Whole evolutions of mid-sized states (n = 13 or 14 .. 20) in one cooperative
// launch.
//
// The HBM passes of these sizes are short: a state of n = 16 is a handful of the
// passes' 64 KiB tiles, so a few SMs work while the others idle, a pass takes the
// latency of one tile (5 us in complex64, 25 to 30 us in FP64 or double-float
// arithmetic) and a layer one and a half launches.  Here a tile has 2^T amplitudes
// with T just large enough for two groups of qubits to cover the state, so there
// are up to a few hundred tiles, one CTA each, and the CTAs of an instance pass a
// grid barrier between passes.  Pass i (i = 0 .. p) works on the low group (i
// even) or the high group (i odd): it finishes layer i - 1, whose other group the
// pass before did, applies layer i's phase and butterflies layer i on its group:
// p + 1 passes for p layers.  Between passes the state lies in the caller's buffer
// (in L2); within one it is butterflied in shared-memory rounds (orbits.cuh), down
// from the tile's top bits to its bottom ones and back up, so that both the loads
// and the stores run along consecutive amplitudes and the phase is taken in the
// registers of the turning round.
//
// Bound by latency: a pass takes about 6 us (barrier 1.3, loads from L2, two runs
// of rounds) in complex64; FP64 by its pipe from n = 18 on.  One instance, p = 10,
// per call, passes / this: n = 16 complex64 140 / 109 us, FP64 906 / 167,
// double-float (n = 17) 344 / 166; n = 13 FP64 449 / 149.
//
// As in mixer.cu a flip-symmetric table is evolved on half of its amplitudes; the
// check is the launch's first phase.
//
// Barriers: the CTAs of an instance are resident together (cooperative launch),
// every wait has a limit after which the kernel records the failure, skips the
// remaining waits and ends.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "orbits.cuh"
#include "pass_common.cuh"
#include "qaoa_internal.cuh"

namespace qaoa {

constexpr int MID_PT = 128;         // threads per CTA
constexpr int MID_ROW = 2;          // high tiles: rows of 4 amplitudes (32 or 64 bytes, whole sectors)
constexpr int MID_N_MAX = 20;       // largest n (see evolve_mid)
constexpr int MID_T_MIN = 9, MID_T_MAX = (MID_N_MAX + MID_ROW + 1) / 2;
constexpr unsigned MID_SPINS = 1u << 21;  // about a second of polls

template <typename R>
struct MidArgs {
    const uint8_t *cost;
    typename VecOf<R>::type *state;
    const typename VecOf<R>::type *tab;  // [p][m + 1]
    const SmallCoef<R> *coef;            // [p]
    double *partials;                    // [batch][G][2]
    double *result;                      // nullable: [batch][2]
    int *slots;                          // [batch][G] verdicts of the flip-symmetry check
    unsigned *bar;                       // [batch][2]: arrivals, phase (uploaded as zeros)
    int *failed;                         // the stream's fault word: set when a wait ran out
    int n, m, p, T;
    int G;     // CTAs per instance
    int kmax;  // most generators per round
    int half;  // the caller's halved state and table
};

// All CTAs of an instance arrive; the last one resets the count and flips the
// phase the others wait for.
__device__ __forceinline__ void instance_barrier(unsigned *bar, unsigned G, bool &dead, int *failed) {
    __syncthreads();
    if (threadIdx.x == 0 && !dead) {
        volatile unsigned *phase = bar + 1;
        const unsigned was = *phase;
        __threadfence();
        if (atomicAdd(bar, 1u) == G - 1) {
            atomicExch(bar, 0u);
            __threadfence();
            atomicExch(bar + 1, was ^ 1u);
        } else {
            unsigned i = 0;
            for (; i < MID_SPINS; ++i) {
                unsigned now;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(bar + 1) : "memory");
                if (now != was) break;
            }
            if (i == MID_SPINS) {
                dead = true;
                *failed = 1;
            }
        }
        __threadfence();
    }
    __syncthreads();
}

// The rounds of a group: generators on tile bits [T - bits, T), at most kmax per
// round; the first `bigger` rounds from the top take k + 1, the others k.
struct MidRounds {
    int count, k, bigger, T;
    __device__ __forceinline__ MidRounds(int bits, int kmax, int T_) : T(T_) {
        count = (bits + kmax - 1) / kmax;
        k = bits / count;
        bigger = bits - k * count;
    }
    __device__ __forceinline__ int size(int r) const { return k + (r < bigger ? 1 : 0); }
    __device__ __forceinline__ int pos(int r) const { return T - (r + 1) * k - min(r + 1, bigger); }
};

__device__ __forceinline__ float2 stored(float2 v) { return v; }
__device__ __forceinline__ double2 stored(double2 v) { return v; }
__device__ __forceinline__ float4 stored(float4 v) { return df_renorm(v); }

template <typename R>
__global__ void __launch_bounds__(MID_PT, 4) mid_kernel(const __grid_constant__ MidArgs<R> a) {
    using V = typename VecOf<R>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int T = a.T;
    const uint32_t L = 1u << T;
    V *s = reinterpret_cast<V *>(smem_raw);
    V *stab = s + L;
    uint8_t *scs = reinterpret_cast<uint8_t *>(stab + MAX_TABLE);  // cost bytes of the low and of the high tile
    const uint32_t G = (uint32_t)a.G, inst = blockIdx.x / G, c = blockIdx.x % G;
    constexpr uint32_t nt = MID_PT;
    const int sbits = a.half ? a.n - 1 : a.n;
    V *st = a.state + ((size_t)inst << sbits);
    const uint8_t *cost = a.cost + ((size_t)inst << sbits);
    unsigned *bar = a.bar + 2 * inst;
    bool dead = false;
    TabAhead<V> ahead;
    ahead.fetch(a.tab, a.m);
    SmallCoef<R> up = a.coef[0], down = up;
    bool half = a.half != 0;
    if (!half) {
        const uint4 *w4 = reinterpret_cast<const uint4 *>(cost);
        const uint32_t W = 1u << (a.n - 4);
        uint32_t bad = 0;
        for (uint32_t w = c * nt + threadIdx.x; w < W / 2; w += G * nt) {
            const uint4 x = w4[w], y = w4[W - 1 - w];
            bad |= (x.x ^ __byte_perm(y.w, 0, 0x0123)) | (x.y ^ __byte_perm(y.z, 0, 0x0123)) |
                   (x.z ^ __byte_perm(y.y, 0, 0x0123)) | (x.w ^ __byte_perm(y.x, 0, 0x0123));
        }
        const int any = __syncthreads_or(bad != 0);
        if (threadIdx.x == 0) a.slots[inst * G + c] = any;
        instance_barrier(bar, G, dead, a.failed);
        int v = 0;
        for (uint32_t i = threadIdx.x; i < G; i += nt) v |= __ldcg(a.slots + inst * G + i);
        half = !__syncthreads_or(v);
    }
    const int nb = half ? a.n - 1 : a.n;             // index bits worked on
    const int low_bits = half ? T - 1 : T;           // of which the low group covers these (and the mirror)
    const int glo = nb - (T - MID_ROW);              // the high tiles' strided bits [glo, nb)
    const uint32_t tiles = 1u << (nb - T), M = (1u << nb) - 1u, H = L / 2;
    const bool once = tiles <= G;                    // one tile per group and CTA: its costs are read once
    const MidRounds rl(T, a.kmax, T), rh(nb - low_bits, a.kmax, T);
    double acc[2] = {0.0, 0.0};
    for (int i = 0; i <= a.p; ++i) {
        const bool low = (i & 1) == 0, init = i == 0, last = i == a.p;
        const MidRounds &rr = low ? rl : rh;
        if (!last) ahead.put(stab);
        __syncthreads();
        for (uint32_t t = c; t < tiles; t += G) {
            uint8_t *sc = scs + (low ? 0u : L);
            const uint32_t base = low ? (half ? t << (T - 1) : t << T) : tile_base32(t, MID_ROW, glo, T);
            // state index of tile element u (low group of a halved state: the upper
            // half of the tile mirrors the lower)
            auto index = [&](uint32_t u) -> uint32_t {
                if (!low) return base + elem_offset32(u, MID_ROW, glo);
                return half && (u & H) ? M - base - (u & (H - 1)) : base + u;
            };
            if (!once || i < 2) {
                for (uint32_t w = threadIdx.x; w < L / 4; w += nt) {  // four bytes at a time, reversed in the mirror
                    const uint32_t u = 4 * w;
                    const bool mir = low && half && (u & H);
                    const uint32_t x = mir ? index(u) - 3 : index(u);
                    const uint32_t v = *reinterpret_cast<const uint32_t *>(cost + x);
                    reinterpret_cast<uint32_t *>(sc)[w] = mir ? __byte_perm(v, 0, 0x0123) : v;
                }
                if (init || rr.count == 1) __syncthreads();
            }
            // round r of the group; which layers' butterflies it does, whether the
            // phase lies between them, where its amplitudes come from and go
            auto round = [&](int r, bool gload, bool dn, bool ph, bool u_, bool gstore) {
                const int j = rr.pos(r);
                auto body = [&](auto kc) {
                    constexpr int K = decltype(kc)::value;
                    orbits<V, K>(T, j, false, [&](const uint32_t(&off)[1 << K], uint32_t z0) {
                        V v[1 << K];
                        if (ph && init) {
#pragma unroll
                            for (int q = 0; q < (1 << K); ++q) v[q] = stab[sc[z0 | (uint32_t)q << j]];
                        } else if (gload) {
#pragma unroll
                            for (int q = 0; q < (1 << K); ++q) v[q] = __ldcg(st + index(z0 | (uint32_t)q << j));
                        } else {
#pragma unroll
                            for (int q = 0; q < (1 << K); ++q) v[q] = at(s, off[q]);
                        }
                        if (dn) {
                            if (down.unit_a)
                                orbit_bfly<true, K>(v, down.A, down.B);
                            else
                                orbit_bfly<false, K>(v, down.A, down.B);
                        }
                        if (ph && !init) {
#pragma unroll
                            for (int q = 0; q < (1 << K); ++q) v[q] = cmul(v[q], stab[sc[z0 | (uint32_t)q << j]]);
                        }
                        if (u_) {
                            if (up.unit_a)
                                orbit_bfly<true, K>(v, up.A, up.B);
                            else
                                orbit_bfly<false, K>(v, up.A, up.B);
                        }
                        if (gstore) {
#pragma unroll
                            for (int q = 0; q < (1 << K); ++q) st[index(z0 | (uint32_t)q << j)] = stored(v[q]);
                        } else {
#pragma unroll
                            for (int q = 0; q < (1 << K); ++q) at(s, off[q]) = v[q];
                        }
                    });
                };
                switch (rr.size(r)) {
                    case 4: body(std::integral_constant<int, 4>{}); break;
                    case 3: body(std::integral_constant<int, 3>{}); break;
                    case 2: body(std::integral_constant<int, 2>{}); break;
                    default: body(std::integral_constant<int, 1>{}); break;
                }
                __syncthreads();
            };
            const int bot = rr.count - 1;
            if (!init)
                for (int r = 0; r < bot; ++r) round(r, r == 0, true, false, false, false);
            round(bot, !init && bot == 0, !init, !last, !last, !last && bot == 0);
            if (!last) {
                for (int r = bot - 1; r >= 0; --r) round(r, false, false, false, true, r == 0);
                continue;
            }
            // the result, in index order, with its sums (complex64: four terms in
            // FP32, everything above in FP64)
            V *exp = half && !a.half ? st + (2 * (size_t)M + 1) : nullptr;  // a full buffer's other half
            for (uint32_t u0 = threadIdx.x; u0 < L; u0 += 4 * nt) {
                decltype(amp_prob(V{})) w[4], ws[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t u = u0 + q * nt;
                    w[q] = ws[q] = 0;
                    if (u < L) {
                        const V v = s[swz<V>(u)];
                        const uint32_t x = index(u);
                        w[q] = amp_prob(v);
                        ws[q] = sc[u] == 0 ? w[q] : 0;
                        if constexpr (std::is_same<R, dfloat>::value) {
                            const double2 d = amp_f64(v);
                            reinterpret_cast<double2 *>(st)[x] = d;
                            if (exp) reinterpret_cast<double2 *>(exp)[-(int64_t)x] = d;
                        } else {
                            st[x] = v;
                            if (exp) exp[-(int64_t)x] = v;
                        }
                    }
                }
                acc[0] += (double)((ws[0] + ws[1]) + (ws[2] + ws[3]));
                acc[1] += (double)((w[0] + w[1]) + (w[2] + w[3]));
            }
            __syncthreads();
        }
        if (!last) {
            down = up;
            if (i + 1 < a.p) {
                ahead.fetch(a.tab + (size_t)(i + 1) * (a.m + 1), a.m);
                up = a.coef[i + 1];
            }
            instance_barrier(bar, G, dead, a.failed);
        }
    }
    if (!a.result) return;
    block_sum<2, MID_PT>(acc);
    if (threadIdx.x == 0) {
        a.partials[2 * blockIdx.x] = acc[0];
        a.partials[2 * blockIdx.x + 1] = acc[1];
    }
    instance_barrier(bar, G, dead, a.failed);
    if (c != 0) return;
    acc[0] = acc[1] = 0.0;
    for (uint32_t i = threadIdx.x; i < G; i += nt) {
        acc[0] += __ldcg(a.partials + 2 * (inst * G + i));
        acc[1] += __ldcg(a.partials + 2 * (inst * G + i) + 1);
    }
    block_sum<2, MID_PT>(acc);
    if (threadIdx.x == 0) {
        const double f = half && !a.half ? 2.0 : 1.0;  // the caller of a halved state doubles its results itself
        a.result[2 * inst] = f * acc[0];
        a.result[2 * inst + 1] = f * acc[1];
    }
}

// Tile bits for n qubits (at least 13): two groups cover the state, T + (T - MID_ROW) >= n.
static int mid_tile(int n) { return std::max(MID_T_MIN, (n + MID_ROW + 1) / 2); }

template <typename R>
static size_t mid_smem(int T) {
    return sizeof(typename VecOf<R>::type) * ((size_t(1) << T) + MAX_TABLE) + 2 * (size_t(1) << T);
}

// CTAs of tile size T that the device holds at once.
template <typename R>
static int mid_capacity(int T, const DeviceInfo &di, int *out) {
    static std::mutex mu;
    static int cap[MAX_DEVICES][MID_T_MAX + 1] = {};
    const int dev = current_device_slot();
    if (dev < 0) return QAOA_ECUDA;
    std::lock_guard<std::mutex> lk(mu);
    if (!cap[dev][T]) {
        QAOA_CUDA_TRY(cudaFuncSetAttribute(mid_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)mid_smem<R>(MID_T_MAX)));
        int per = 0;
        QAOA_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, mid_kernel<R>, MID_PT, mid_smem<R>(T)));
        cap[dev][T] = std::max(1, per * di.sms);
    }
    *out = cap[dev][T];
    return QAOA_OK;
}

template <typename R>
static int mid_run(const EvolveReq &r, cudaStream_t stream, double *h_result, bool *taken) {
    using V = typename VecOf<R>::type;
    const int T = mid_tile(r.n), G = 1 << (r.n - 1 - T);
    DeviceInfo di;
    int rc = device_info(&di), cap = 0;
    if (rc) return rc;
    if ((rc = mid_capacity<R>(T, di, &cap))) return rc;
    if ((int64_t)r.batch * G > cap) return QAOA_OK;
    const size_t tab = small_table_bytes(sizeof(V), r.p, r.m), cof = sizeof(SmallCoef<R>) * (size_t)r.p;
    const size_t bar = (tab + cof + 15) & ~(size_t)15, sent = bar + 2 * sizeof(unsigned) * (size_t)r.batch;
    const size_t part = sizeof(double) * 2 * (size_t)r.batch * G, slot = sizeof(int) * (size_t)r.batch * G;
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    Scratch *sc = nullptr;
    if ((rc = scratch_for(stream, al(sent) + al(part) + slot, 2 * sizeof(double) * (size_t)r.batch, &sc))) return rc;
    int *failed = nullptr;
    if ((rc = fault_word(stream, &failed))) return rc;
    char *d = reinterpret_cast<char *>(sc->dev);
    double *result = reinterpret_cast<double *>(sc->host);
    // the tables, and the barrier words as zeros: whatever a launch before left
    Upload *up = nullptr;
    if ((rc = upload_buffer(sc, sent, &up))) return rc;
    char *h = reinterpret_cast<char *>(up->host);
    small_fill_layers(r.dtype, r.flags, r.n, r.m, r.p, r.gamma, r.beta, h, h + tab);
    memset(h + bar, 0, sent - bar);
    QAOA_CUDA_TRY(cudaMemcpyAsync(d, h, sent, cudaMemcpyHostToDevice, stream));
    // a call with results waits for the stream, its upload included (the event's record
    // takes 3 to 4 us of such a call)
    if (!h_result && (rc = upload_sent(up, stream))) return rc;
    MidArgs<R> a;
    a.cost = r.cost;
    a.state = reinterpret_cast<V *>(r.state);
    a.tab = reinterpret_cast<const V *>(d);
    a.coef = reinterpret_cast<const SmallCoef<R> *>(d + tab);
    a.partials = reinterpret_cast<double *>(d + al(sent));
    a.result = h_result ? result : nullptr;
    a.slots = reinterpret_cast<int *>(d + al(sent) + al(part));
    a.bar = reinterpret_cast<unsigned *>(d + bar);
    a.failed = failed;
    a.n = r.n;
    a.m = r.m;
    a.p = r.p;
    a.T = T;
    a.G = G;
    // one orbit per thread; FP64 takes smaller ones in small tiles, whose warps
    // then feed every quarter of the SM
    a.kmax = std::min(4, std::is_same<R, double>::value ? T - 7 : std::max(3, T - 7));
    a.half = (r.flags & QAOA_Z2_HALF) ? 1 : 0;
    void *args[] = {(void *)&a};
    profile_before(K_MID, stream);
    const cudaError_t e = cudaLaunchCooperativeKernel((const void *)mid_kernel<R>, dim3((unsigned)(r.batch * G)),
                                                      dim3(MID_PT), args, mid_smem<R>(T), stream);
    if (e == cudaErrorCooperativeLaunchTooLarge) {  // e.g. fewer SMs than the device's (a partition)
        cudaGetLastError();
        return h_result ? upload_sent(up, stream) : QAOA_OK;
    }
    if ((rc = profile_after(K_MID, stream))) {
        if (h_result) cudaStreamSynchronize(stream);
        return rc;
    }
    *taken = true;
    if (!h_result) return QAOA_OK;
    QAOA_CUDA_TRY(cudaStreamSynchronize(stream));
    if ((rc = stream_fault(stream))) return rc;
    memcpy(h_result, result, 2 * sizeof(double) * (size_t)r.batch);
    return QAOA_OK;
}

int evolve_mid(const EvolveReq &r, cudaStream_t stream, double *h_result, bool *taken) {
    *taken = false;
    // Where the passes' tiles fill the device they are the better ones: n = 21, p =
    // 7 complex64 115 us against 138 here.  n = 20, p = 10: 157 / 148 us, in FP64
    // 1274 / 586, in double-float 372 / 286.  One complex64 layer is two passes
    // either way (n = 14: 49 / 53 us).
    if (r.p < 1 || r.n > MID_N_MAX || (r.dtype == QAOA_C64 && r.p < 2)) return QAOA_OK;
    if ((reinterpret_cast<uintptr_t>(r.cost) | reinterpret_cast<uintptr_t>(r.state)) & 15u) return QAOA_OK;
    // a captured copy would read its host source again at every replay
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    QAOA_CUDA_TRY(cudaStreamIsCapturing(stream, &cap));
    if (cap != cudaStreamCaptureStatusNone) return QAOA_OK;
    if (r.dtype == QAOA_C64) return mid_run<float>(r, stream, h_result, taken);
    return (r.flags & QAOA_DF64) ? mid_run<dfloat>(r, stream, h_result, taken)
                                 : mid_run<double>(r, stream, h_result, taken);
}

}  // namespace qaoa

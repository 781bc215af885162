// K1: the NAE cost table C(x) (Eq. for C^NAE, Sec. "Problem Hamiltonian"; its
// De Morgan form in Appendix A.2: a clause is violated when its literals are
// all false or all true).
//
// Bit-sliced design.  A thread owns one 32-bit word of assignments,
// x = 32 X + b for b = 0..31.  Variables 0..4 vary inside the word, variables
// >= 5 are constant across it.  Per clause the host precomputes
//   hi_mask / hi_neg : the clause's variables >= 5 and their negations,
//   all_true  : bit b set iff every literal on a variable < 5 is true at b,
//   all_false : bit b set iff every such literal is false at b.
// With t = ((32 X) ^ hi_neg) & hi_mask (the literal values on the high
// variables) the clause's violation word is
//   V = (t == 0 ? all_false : 0) | (t == hi_mask ? all_true : 0),
// i.e. all literals false, or all true.  The 32 per-x counts are kept as
// bit planes by a carry-save (Harley-Seal) adder over chunks of 16 clauses,
// then transposed to bytes with 8x8 bit-matrix transposes.  The records that a
// block counts sit in shared memory (one broadcast 16-byte load per clause) and
// each thread counts two words per record load.  The number of solutions (count
// 0) and the largest count come out of the same pass.
//
// Large clause counts.  The records are staged CT_CHUNK at a time: the block
// filters and counts one chunk, then the next, accumulating into the same
// counters.  Up to 1023 clauses 10 bit planes count exactly; beyond that 13
// planes do (m <= 8191).  Only the counts <= 255 go into the table; a larger
// one makes the call fail with the exact maximum.
//
// Global-flip symmetry.  Flipping every bit of x flips every literal, so a
// clause's literals stay all equal or not: C(not x) = C(x) (Sec. 2.2).  The
// complement of x = 32 X + b is 32 (W - 1 - X) + (31 - b) (W = 2^(n - 5)
// words), so a full table is counted on its lower half only: each counted
// word is written twice, the second time byte-reversed at word W - 1 - X.
//
// Clause filtering.  A block takes 512 consecutive words at a time (256 for small
// tables), so the variables >= 14 (13) are constant over them.  A clause whose
// literals on those variables are neither all true nor all false is violated
// nowhere in the block; the block first keeps only the others, each reduced to
// its remaining variables and to the one or two patterns still possible (for
// random 5-literal clauses over 30 variables about 40% survive), then counts
// against that list (long lists: against each warp's part of it).  Counts are sums
// of 0/1 terms, so the list order is immaterial.
#include <cuda_runtime.h>

#include <cstring>

#include "qaoa_internal.cuh"

namespace qaoa {

constexpr int CT_THREADS = 256;
constexpr int CT_CHUNK = 1024;     // clause records staged in shared memory at a time
constexpr int CT_PARAM_M = 1023;   // largest m passed as kernel parameters
constexpr int CT_PARAM_S = 240;    // ... in 4 KiB of them (13 us of host time a call, 22 with 16 KiB and the stats' memset)
constexpr size_t ENCODE_MIN_LITS = 1 << 15;  // batches encoded on the device
constexpr int NPL_SMALL = 10;      // bit planes for m <= 1023
constexpr int NPL_LARGE = 13;      // bit planes for m <= 8191
static_assert(QAOA_MAX_M < (1 << NPL_LARGE), "counts must fit the planes");

template <int CAP>
struct CostParams {
    int n, m;
    int mirror;  // count the lower half, write both (full tables, n >= 6)
    ClauseRec rec[CAP];
};

__device__ __forceinline__ void csa(uint32_t &h, uint32_t &l, uint32_t a, uint32_t b, uint32_t c) {
    const uint32_t u = a ^ b;
    h = (a & b) | (u & c);
    l = u ^ c;
}

__device__ __forceinline__ uint32_t violation_word(uint32_t xh, const ClauseRec &r) {
    const uint32_t t = (xh ^ r.hi_neg) & r.hi_mask;
    return (t == 0u ? r.all_false : 0u) | (t == r.hi_mask ? r.all_true : 0u);
}

// Carry-save counter of the violated clauses of one 32-assignment word:
// bit plane q holds bit q of every count (q = 0..NPL-1, counts < 2^NPL).
template <int NPL>
struct WordCounter {
    uint32_t ones = 0, twos = 0, fours = 0, eights = 0;
    uint32_t up[NPL - 4] = {};
    // Adds 16 violation words (a Harley-Seal chunk).
    __device__ __forceinline__ void add16(const uint32_t v[16]) {
        uint32_t twosA, twosB, foursA, foursB, eightsA, eightsB, sixteens;
        csa(twosA, ones, ones, v[0], v[1]);
        csa(twosB, ones, ones, v[2], v[3]);
        csa(foursA, twos, twos, twosA, twosB);
        csa(twosA, ones, ones, v[4], v[5]);
        csa(twosB, ones, ones, v[6], v[7]);
        csa(foursB, twos, twos, twosA, twosB);
        csa(eightsA, fours, fours, foursA, foursB);
        csa(twosA, ones, ones, v[8], v[9]);
        csa(twosB, ones, ones, v[10], v[11]);
        csa(foursA, twos, twos, twosA, twosB);
        csa(twosA, ones, ones, v[12], v[13]);
        csa(twosB, ones, ones, v[14], v[15]);
        csa(foursB, twos, twos, twosA, twosB);
        csa(eightsB, fours, fours, foursA, foursB);
        csa(sixteens, eights, eights, eightsA, eightsB);
        uint32_t carry = sixteens;
#pragma unroll
        for (int q = 0; q < NPL - 4; ++q) {
            const uint32_t t = up[q] & carry;
            up[q] ^= carry;
            carry = t;
        }
    }
    __device__ __forceinline__ void planes(uint32_t p[NPL]) const {
        p[0] = ones;
        p[1] = twos;
        p[2] = fours;
        p[3] = eights;
#pragma unroll
        for (int q = 0; q < NPL - 4; ++q) p[4 + q] = up[q];
    }
};

// Adds to c0 (and, with WPT = 2, c1) the counts of words X0 (and X1) against the clause records in
// shared memory (m16 = record count rounded up to 16; the padding records are
// all zero, which are never violated: t = 0 = hi_mask selects
// all_false | all_true = 0).
template <int NPL, int WPT>
__device__ __forceinline__ void count_words(uint32_t X0, uint32_t X1, int m16, const uint4 *srec,
                                            WordCounter<NPL> &c0, WordCounter<NPL> &c1) {
    const uint32_t xh0 = X0 << 5, xh1 = X1 << 5;
    for (int i0 = 0; i0 < m16; i0 += 16) {
        uint32_t v0[16], v1[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const uint4 r4 = srec[i0 + j];
            const ClauseRec r{r4.x, r4.y, r4.z, r4.w};
            v0[j] = violation_word(xh0, r);
            if (WPT == 2) v1[j] = violation_word(xh1, r);
        }
        c0.add16(v0);
        if (WPT == 2) c1.add16(v1);
    }
}

// 8x8 bit transpose of a 64-bit word (byte j = row j, bit i = column i).
__device__ __forceinline__ uint64_t transpose8(uint64_t w) {
    uint64_t t;
    t = (w ^ (w >> 7)) & 0x00AA00AA00AA00AAull;
    w ^= t ^ (t << 7);
    t = (w ^ (w >> 14)) & 0x0000CCCC0000CCCCull;
    w ^= t ^ (t << 14);
    t = (w ^ (w >> 28)) & 0x00000000F0F0F0F0ull;
    w ^= t ^ (t << 28);
    return w;
}

// Byte b of the result (b = 0..31) = bits 0..7 of the count of x = 32 X + b.
__device__ __forceinline__ void planes_to_bytes(const uint32_t *planes, uint32_t out[8]) {
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        // row j of the 8x8 block = byte g of plane j
        const uint32_t lo = __byte_perm(__byte_perm(planes[0], planes[1], 0x0040 + g * 0x0011),
                                        __byte_perm(planes[2], planes[3], 0x0040 + g * 0x0011), 0x5410);
        const uint32_t hi = __byte_perm(__byte_perm(planes[4], planes[5], 0x0040 + g * 0x0011),
                                        __byte_perm(planes[6], planes[7], 0x0040 + g * 0x0011), 0x5410);
        const uint64_t w = transpose8(((uint64_t)hi << 32) | lo);
        out[2 * g] = (uint32_t)w;
        out[2 * g + 1] = (uint32_t)(w >> 32);
    }
}

// Writes the 32 counts of word X (bytes) and folds its solution count and max.
// With `mirror` (n >= 6) the same counts also go, byte-reversed, to the
// complement word W - 1 - X, and they count twice.
template <int NPL>
__device__ __forceinline__ void emit_word(int n, uint64_t X, const uint32_t planes[NPL], uint8_t *cost,
                                          unsigned long long &nsol, uint32_t &mx, bool mirror) {
    const uint32_t valid = n >= 5 ? 0xFFFFFFFFu : ((1u << (1u << n)) - 1u);
    uint32_t bytes[8];
    planes_to_bytes(planes, bytes);
    uint32_t any = 0;
    uint32_t over = 0;
#pragma unroll
    for (int q = 0; q < NPL; ++q) {
        any |= planes[q];
        if (q >= 8) over |= planes[q];
    }
    nsol += (mirror ? 2u : 1u) * __popc(~any & valid);
    over &= valid;
    uint32_t bm = 0;
    if (n >= 5) {
#pragma unroll
        for (int q = 0; q < 8; ++q) bm = __vmaxu4(bm, bytes[q]);
        bm = max(max(bm & 0xFF, (bm >> 8) & 0xFF), max((bm >> 16) & 0xFF, bm >> 24));
    } else {
        for (uint32_t b = 0; b < (1u << n); ++b) bm = max(bm, (bytes[b >> 2] >> (8 * (b & 3))) & 0xFFu);
    }
    if (over) {  // some count >= 256: take those lanes exactly
        for (uint32_t b = 0; b < 32; ++b)
            if ((over >> b) & 1u) {
                uint32_t c = 0;
                for (int q = 0; q < NPL; ++q) c |= ((planes[q] >> b) & 1u) << q;
                bm = max(bm, c);
            }
    }
    mx = max(mx, bm);
    if (n >= 5) {
        uint4 *dst = reinterpret_cast<uint4 *>(cost + 32 * X);
        dst[0] = make_uint4(bytes[0], bytes[1], bytes[2], bytes[3]);
        dst[1] = make_uint4(bytes[4], bytes[5], bytes[6], bytes[7]);
        if (mirror) {  // byte 31 - b of the complement word holds the count of byte b
            const uint64_t Xm = (1ull << (n - 5)) - 1ull - X;
            uint4 *dm = reinterpret_cast<uint4 *>(cost + 32 * Xm);
            dm[0] = make_uint4(__byte_perm(bytes[7], 0, 0x0123), __byte_perm(bytes[6], 0, 0x0123),
                               __byte_perm(bytes[5], 0, 0x0123), __byte_perm(bytes[4], 0, 0x0123));
            dm[1] = make_uint4(__byte_perm(bytes[3], 0, 0x0123), __byte_perm(bytes[2], 0, 0x0123),
                               __byte_perm(bytes[1], 0, 0x0123), __byte_perm(bytes[0], 0, 0x0123));
        }
    } else {
        for (uint32_t b = 0; b < (1u << n); ++b) cost[b] = (uint8_t)((bytes[b >> 2] >> (8 * (b & 3))) & 0xFFu);
    }
}

// A block step takes WPT words per thread, WPT * CT_THREADS = 256 or 512 words:
// variables >= 13 or 14 (sub_bits) are constant over it.  Two words per thread
// share each record load and each filter; one word per thread gives small tables
// twice the blocks and half the chain of clauses each, so it is taken while the
// blocks of two do not fill the device twice (tables one after the other, with
// their launches: n = 21, m = 168 20.3 -> 14.6 us, n = 23, m = 184 21.9 -> 14.5).
template <int WPT>
constexpr int sub_bits() {
    return WPT == 2 ? 14 : 13;
}

// Keeps the clauses of recs[0, m) (m <= CT_CHUNK; shared or global memory)
// that can be violated somewhere in the step's words from base on, reduced to
// variables 5 .. sub_bits - 1, in alive[0, *count), zero-padded to a multiple
// of 16, and alive[that count] all zero too.  Called by all threads of the block.
template <int WPT>
__device__ __forceinline__ int filter_clauses(uint32_t base, int m, const uint4 *recs, uint4 *alive, int *count) {
    constexpr uint32_t MID = (1u << sub_bits<WPT>()) - 32u;
    const uint32_t xu = base << 5;  // the constant x bits of the step (the others are zero)
    if (threadIdx.x == 0) *count = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int i0 = 0; i0 < m; i0 += CT_THREADS) {
        const int i = i0 + threadIdx.x;
        uint4 r = make_uint4(0, 0, 0, 0);
        bool keep = false;
        if (i < m) {
            r = recs[i];
            const uint32_t umask = r.x & ~MID & ~31u;
            const uint32_t tu = (xu ^ r.y) & umask;
            const bool at = tu == umask, af = tu == 0u;  // uniform literals all true / all false
            keep = at || af;
            r = make_uint4(r.x & MID, r.y & MID, at ? r.z : 0u, af ? r.w : 0u);
        }
        const uint32_t ballot = __ballot_sync(0xFFFFFFFFu, keep);
        int pos = 0;
        if (lane == 0 && ballot) pos = atomicAdd(count, __popc(ballot));
        pos = __shfl_sync(0xFFFFFFFFu, pos, 0) + __popc(ballot & ((1u << lane) - 1u));
        if (keep) alive[pos] = r;
    }
    __syncthreads();
    const int c = *count, c16 = (c + 15) & ~15;
    for (int i = c + threadIdx.x; i <= c16; i += CT_THREADS) alive[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    return c16;
}

// Long lists are filtered once more, by each warp for its own 32 WPT consecutive
// words, over which three more variables are constant (x bits 11..13 or 10..12):
// of a block's list of 9-literal clauses about 0.4 remain.  wl receives the
// remaining clauses' places in alive, padded to a multiple of 16 with that of a
// record that is never violated; the counts then read their records through it.
// For short lists (under WARP_FILTER_MIN) the pass and the indirection cost what
// they save.  256 x (n = 17, k = 9, about 3000 clauses): 545 -> 273 us; 128 x (n =
// 19, k = 7, 830 clauses): 272 -> 181; 256 x (n = 15, k = 7, 660): 51 -> 38.
constexpr int WARP_FILTER_MIN = 256;
template <int WPT>
__device__ __forceinline__ int warp_filter(uint32_t X, int c16, const uint4 *alive, uint16_t *wl) {
    constexpr uint32_t MASK = WPT == 2 ? 7u << 11 : 7u << 10;
    const uint32_t lane = threadIdx.x & 31, xw = X << 5;
    int cnt = 0;
    for (int i0 = 0; i0 < c16; i0 += 32) {
        const int i = i0 + (int)lane;
        const uint4 r = i < c16 ? alive[i] : make_uint4(0, 0, 0, 0);
        const uint32_t um = r.x & MASK, tu = (xw ^ r.y) & um;
        const bool keep = (r.z != 0u && tu == um) || (r.w != 0u && tu == 0u);
        const uint32_t ballot = __ballot_sync(0xFFFFFFFFu, keep);
        if (keep) wl[cnt + __popc(ballot & ((1u << lane) - 1u))] = (uint16_t)i;
        cnt += __popc(ballot);
    }
    const int w16 = (cnt + 15) & ~15;
    if (cnt + (int)lane < w16) wl[cnt + lane] = (uint16_t)c16;
    __syncwarp();
    return w16;
}

// count_words over the listed records.
template <int NPL, int WPT>
__device__ __forceinline__ void count_listed(uint32_t X0, uint32_t X1, int w16, const uint4 *alive, const uint16_t *wl,
                                             WordCounter<NPL> &c0, WordCounter<NPL> &c1) {
    const uint32_t xh0 = X0 << 5, xh1 = X1 << 5;
    for (int i0 = 0; i0 < w16; i0 += 16) {
        const uint4 a = *reinterpret_cast<const uint4 *>(wl + i0), b = *reinterpret_cast<const uint4 *>(wl + i0 + 8);
        const uint32_t ix[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        uint32_t v0[16], v1[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const uint4 r4 = alive[(j & 1) ? ix[j / 2] >> 16 : ix[j / 2] & 0xFFFFu];
            const ClauseRec r{r4.x, r4.y, r4.z, r4.w};
            v0[j] = violation_word(xh0, r);
            if (WPT == 2) v1[j] = violation_word(xh1, r);
        }
        c0.add16(v0);
        if (WPT == 2) c1.add16(v1);
    }
}

// One table: each block steps through WPT * CT_THREADS consecutive words at a
// time; a warp takes 32 WPT consecutive ones, lane t of it the t-th and, with WPT
// = 2, the (32 + t)-th.  wl: null, or CT_CHUNK places per warp for the second
// filter.  stats may be null.  recs holds the m records (shared or global
// memory), taken CT_CHUNK at a time.
template <int NPL, int WPT>
__device__ __forceinline__ void cost_table_body(int n, int m, const uint4 *recs, uint4 *alive, int *acount,
                                                uint8_t *cost, unsigned long long *stats, bool mirror,
                                                uint16_t *wl) {
    constexpr int SUB_WORDS = WPT * CT_THREADS;
    mirror = mirror && n >= 6;  // the lower half is then a whole number of words
    const uint64_t words = n >= 5 ? (1ull << (n - 5)) >> (mirror ? 1 : 0) : 1ull;  // words counted
    const uint64_t steps = (words + SUB_WORDS - 1) / SUB_WORDS;
    unsigned long long nsol = 0;
    uint32_t mx = 0;
    for (uint64_t sb = blockIdx.x; sb < steps; sb += gridDim.x) {
        const uint32_t base = (uint32_t)(sb * SUB_WORDS);
        const uint32_t Xw = base + (threadIdx.x >> 5) * (32 * WPT);  // the warp's first word
        const uint64_t X0 = Xw + (threadIdx.x & 31), X1 = X0 + 32;
        WordCounter<NPL> c0, c1;
        for (int k0 = 0; k0 < m || k0 == 0; k0 += CT_CHUNK) {
            const int mc = m - k0 < CT_CHUNK ? m - k0 : CT_CHUNK;
            const int c16 = filter_clauses<WPT>(base, mc, recs + k0, alive, acount);
            const uint32_t X1c = (uint32_t)(X1 < words ? X1 : X0);
            if (wl && c16 >= WARP_FILTER_MIN) {
                uint16_t *mine = wl + (threadIdx.x >> 5) * CT_CHUNK;
                const int w16 = warp_filter<WPT>(Xw, c16, alive, mine);
                if (X0 < words) count_listed<NPL, WPT>((uint32_t)X0, X1c, w16, alive, mine, c0, c1);
            } else if (X0 < words) {
                count_words<NPL, WPT>((uint32_t)X0, X1c, c16, alive, c0, c1);
            }
            __syncthreads();  // the list is rebuilt for the next chunk or step
        }
        if (X0 < words) {
            uint32_t p0[NPL], p1[NPL];
            c0.planes(p0);
            emit_word<NPL>(n, X0, p0, cost, nsol, mx, mirror);
            if (WPT == 2 && X1 < words) {
                c1.planes(p1);
                emit_word<NPL>(n, X1, p1, cost, nsol, mx, mirror);
            }
        }
    }
    if (!stats) return;
    // warp then block reduction, one atomic pair per block
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        nsol += __shfl_xor_sync(0xFFFFFFFFu, nsol, o);
        mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
    }
    __shared__ unsigned long long s_sol[CT_THREADS / 32];
    __shared__ uint32_t s_max[CT_THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        s_sol[wid] = nsol;
        s_max[wid] = mx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long a = 0;
        uint32_t b = 0;
        for (int w = 0; w < CT_THREADS / 32; ++w) {
            a += s_sol[w];
            b = max(b, s_max[w]);
        }
        if (a) atomicAdd(&stats[0], a);
        atomicMax(&stats[1], (unsigned long long)b);
    }
}

// One table, m <= CT_PARAM_M, the records passed as kernel parameters and
// copied to shared memory once.
template <int CAP, int WPT>
__global__ void __launch_bounds__(CT_THREADS) cost_table_kernel(const __grid_constant__ CostParams<CAP> prm,
                                                                uint8_t *cost, unsigned long long *stats) {
    __shared__ uint4 srec[CAP];
    __shared__ uint4 alive[CAP + 16];
    __shared__ int acount;
    for (int i = threadIdx.x; i < prm.m; i += CT_THREADS) {
        const ClauseRec r = prm.rec[i];
        srec[i] = make_uint4(r.hi_mask, r.hi_neg, r.all_true, r.all_false);
    }
    __syncthreads();
    pdl_wait();
    cost_table_body<NPL_SMALL, WPT>(prm.n, prm.m, srec, alive, &acount, cost, stats, prm.mirror != 0, nullptr);
}

// Batched tables.  With ns == nullptr every instance has n qubits and its table
// at costs + inst 2^n; otherwise instance inst has ns[inst] qubits and its table
// at costs + offs[inst].  The records are read from global memory (each once per
// block step) CT_CHUNK at a time.
// `bad` (nullable): set when the encoder found an invalid literal; nothing is
// written then.
template <int NPL, int WPT>
__global__ void __launch_bounds__(CT_THREADS) cost_table_batch_kernel(int n, const int *ns, const uint64_t *offs,
                                                                      const ClauseRec *recs, const int *ms,
                                                                      int m_stride, uint8_t *costs,
                                                                      unsigned long long *stats, int mirror,
                                                                      const unsigned long long *bad) {
    static_assert(sizeof(ClauseRec) == sizeof(uint4), "a clause record is one 16-byte load");
    __shared__ uint4 alive[CT_CHUNK + 16];
    __shared__ __align__(16) uint16_t wl[(CT_THREADS / 32) * CT_CHUNK];
    __shared__ int acount;
    pdl_wait();
    if (bad && *bad) return;
    const int inst = blockIdx.y;
    const int m = ms[inst];
    const uint4 *src = reinterpret_cast<const uint4 *>(recs + (size_t)inst * m_stride);
    const int ni = ns ? ns[inst] : n;
    uint8_t *dst = ns ? costs + offs[inst] : costs + ((size_t)inst << n);
    cost_table_body<NPL, WPT>(ni, m, src, alive, &acount, dst, stats + 2 * inst, mirror != 0, wl);
}

// Clause records of a batch, one clause per thread, from the literals in host
// memory (HostLits: the caller's own arrays where the device can read pageable
// memory through the host's page tables, a pinned copy elsewhere), with the
// checks of validate_instance: *bad is set when a variable is outside [0, n), a
// negation flag is not 0 or 1, or a variable is repeated.
//
// Bound by the reads over the chip-to-chip link.  The host's own loop over the
// literals took 21 ms for 256 instances of about 3000 9-literal clauses (35 MB).
struct HostLits {
    const int32_t *var;
    const uint8_t *neg;
    int32_t m, k;
};
__global__ void __launch_bounds__(CT_THREADS) encode_kernel(int n, const HostLits *lits, int m_stride, ClauseRec *recs,
                                                            unsigned long long *bad) {
    pdl_wait();
    const HostLits h = lits[blockIdx.y];
    const int i = blockIdx.x * CT_THREADS + threadIdx.x;
    bool wrong = false;
    if (i < h.m) {
        const int32_t *var = h.var + (size_t)i * h.k;
        const uint8_t *neg = h.neg + (size_t)i * h.k;
        uint32_t mask = 0, negp = 0, at = 0xFFFFFFFFu, af = 0xFFFFFFFFu;
        for (int j = 0; j < h.k; ++j) {
            const uint32_t v = (uint32_t)var[j], s = neg[j];
            wrong |= v >= (uint32_t)n || s > 1u || ((mask >> (v & 31u)) & 1u);
            mask |= 1u << (v & 31u);
            negp |= (s & 1u) << (v & 31u);
            if (v < 5) {  // bit b of the column: the literal is true at b
                const uint32_t col = v == 0   ? 0xAAAAAAAAu
                                     : v == 1 ? 0xCCCCCCCCu
                                     : v == 2 ? 0xF0F0F0F0u
                                     : v == 3 ? 0xFF00FF00u
                                              : 0xFFFF0000u;
                const uint32_t lit = s ? ~col : col;
                at &= lit;
                af &= ~lit;
            }
        }
        *reinterpret_cast<uint4 *>(recs + (size_t)blockIdx.y * m_stride + i) =
            make_uint4(mask & ~31u, negp & ~31u, at, af);
    }
    if (__syncthreads_or(wrong) && threadIdx.x == 0) *bad = 1;
}

// ---------------------------------------------------------------------------
// The sizes and pointers of an instance; its literals are checked apart.
static int valid_sizes(const naesat_instance *inst) {
    if (!inst) return set_error(QAOA_EINVAL, "instance is NULL");
    const int n = inst->n, m = inst->m, k = inst->k;
    if (n < 1 || n > QAOA_MAX_N) return set_error(QAOA_ERANGE, "n=%d outside [1, %d]", n, QAOA_MAX_N);
    if (m < 0 || m > QAOA_MAX_M) return set_error(QAOA_ERANGE, "m=%d outside [0, %d]", m, QAOA_MAX_M);
    if (m == 0) return QAOA_OK;
    if (k < 1 || k > n) return set_error(QAOA_ERANGE, "k=%d outside [1, n=%d]", k, n);
    if (!inst->var || !inst->neg) return set_error(QAOA_EINVAL, "var/neg is NULL");
    return QAOA_OK;
}

int validate_instance(const naesat_instance *inst) {
    const int rc = valid_sizes(inst);
    if (rc) return rc;
    const int n = inst->n, m = inst->m, k = inst->k;
    for (int i = 0; i < m; ++i) {
        uint64_t seen = 0;
        for (int j = 0; j < k; ++j) {
            const int v = inst->var[(size_t)i * k + j];
            const int s = inst->neg[(size_t)i * k + j];
            if (v < 0 || v >= n) return set_error(QAOA_EINVAL, "clause %d: variable %d outside [0, %d)", i, v, n);
            if (s != 0 && s != 1) return set_error(QAOA_EINVAL, "clause %d: negation flag %d not 0/1", i, s);
            if ((seen >> v) & 1ull) return set_error(QAOA_EINVAL, "clause %d: variable %d repeated", i, v);
            seen |= 1ull << v;
        }
    }
    return QAOA_OK;
}

int encode_instance(const naesat_instance *inst, ClauseRec *out) {
    // bit b of COL[v] = bit v of b: the value of variable v < 5 at x = b (mod 32)
    static const uint32_t COL[5] = {0xAAAAAAAAu, 0xCCCCCCCCu, 0xF0F0F0F0u, 0xFF00FF00u, 0xFFFF0000u};
    const int m = inst->m, k = inst->k;
    for (int i = 0; i < m; ++i) {
        uint32_t mask = 0, negp = 0, at = 0xFFFFFFFFu, af = 0xFFFFFFFFu;
        for (int j = 0; j < k; ++j) {
            const int v = inst->var[(size_t)i * k + j];
            const uint32_t s = inst->neg[(size_t)i * k + j];
            mask |= 1u << v;
            negp |= s << v;
            if (v < 5) {
                const uint32_t lit = s ? ~COL[v] : COL[v];  // bit b: the literal is true at b
                at &= lit;
                af &= ~lit;
            }
        }
        out[i] = ClauseRec{mask & ~31u, negp & ~31u, at, af};
    }
    return QAOA_OK;
}

// Blocks per table, and the words per thread (see sub_bits).
static int grid_for(uint64_t words, int batch, int *wpt) {
    DeviceInfo di;
    if (device_info(&di)) return -1;
    const uint64_t two = (words + 2 * CT_THREADS - 1) / (2 * CT_THREADS);
    *wpt = two * (uint64_t)batch >= 2 * (uint64_t)di.sms ? 2 : 1;
    const uint64_t need = *wpt == 2 ? two : (words + CT_THREADS - 1) / CT_THREADS;
    uint64_t cap = (uint64_t)di.sms * 8 * 4;
    cap = cap / (uint64_t)batch + 1;
    return (int)(need < cap ? need : cap);
}

int launch_cost_table_batch(int batch, int n, const int *d_ns, const uint64_t *d_offs, const ClauseRec *d_recs,
                            const int *d_m, int m_stride, uint8_t *d_costs, unsigned long long *d_stats,
                            cudaStream_t stream, bool mirror, const unsigned long long *d_bad) {
    const uint64_t words = n >= 5 ? (1ull << (n - 5)) >> (mirror && n >= 6 ? 1 : 0) : 1ull;
    int wpt = 2;
    const int gx = grid_for(words, batch, &wpt);
    if (gx < 0) return QAOA_ECUDA;
    const int mi = mirror ? 1 : 0;
    auto launch = [&](auto kernel) {
        launch_pdl(kernel, dim3(gx, batch), dim3(CT_THREADS), 0, stream, n, d_ns, d_offs, d_recs, d_m, m_stride, d_costs,
                   d_stats, mi, d_bad);
    };
    profile_before(K_COST_TABLE, stream);
    if (m_stride <= CT_PARAM_M)
        wpt == 2 ? launch(cost_table_batch_kernel<NPL_SMALL, 2>) : launch(cost_table_batch_kernel<NPL_SMALL, 1>);
    else
        wpt == 2 ? launch(cost_table_batch_kernel<NPL_LARGE, 2>) : launch(cost_table_batch_kernel<NPL_LARGE, 1>);
    return profile_after(K_COST_TABLE, stream);
}

// One table whose records travel as kernel parameters.
template <int CAP>
static int launch_params(const naesat_instance *inst, int n, bool half, uint8_t *d_cost, unsigned long long *d_stats,
                         cudaStream_t stream) {
    CostParams<CAP> prm;
    prm.n = n;
    prm.m = inst->m;
    prm.mirror = (!half && n >= 6) ? 1 : 0;  // a full table: count its lower half
    encode_instance(inst, prm.rec);
    const uint64_t words = prm.n >= 5 ? (1ull << (prm.n - 5)) >> prm.mirror : 1ull;
    int wpt = 2;
    const int gx = grid_for(words, 1, &wpt);
    if (gx < 0) return QAOA_ECUDA;
    profile_before(K_COST_TABLE, stream);
    launch_pdl(wpt == 2 ? cost_table_kernel<CAP, 2> : cost_table_kernel<CAP, 1>, dim3(gx), dim3(CT_THREADS), 0, stream,
               prm, d_cost, d_stats);
    return profile_after(K_COST_TABLE, stream);
}

int launch_cost_table_one(const naesat_instance *inst, uint8_t *d_cost, unsigned long long *d_stats,
                          cudaStream_t stream, bool half, void *d_big, void *h_big) {
    // the kernel uses n only for the number of assignments: the half table is
    // the first 2^(n-1) of them (variable n - 1 is 0 there)
    const int n = half ? inst->n - 1 : inst->n;
    if (inst->m > CT_PARAM_M) {
        // records in global memory: d_big holds the m records then the count, from h_big
        if (!d_big || !h_big) return set_error(QAOA_EINVAL, "m=%d needs space for the clause records", inst->m);
        ClauseRec *d_rec = reinterpret_cast<ClauseRec *>(d_big), *h_rec = reinterpret_cast<ClauseRec *>(h_big);
        int *d_m = reinterpret_cast<int *>(d_rec + inst->m);
        encode_instance(inst, h_rec);
        *reinterpret_cast<int *>(h_rec + inst->m) = inst->m;
        QAOA_CUDA_TRY(cudaMemcpyAsync(d_rec, h_rec, cost_table_big_bytes(inst->m), cudaMemcpyHostToDevice, stream));
        return launch_cost_table_batch(1, n, nullptr, nullptr, d_rec, d_m, inst->m, d_cost, d_stats, stream, !half);
    }
    return inst->m <= CT_PARAM_S ? launch_params<CT_PARAM_S>(inst, n, half, d_cost, d_stats, stream)
                                 : launch_params<CT_PARAM_M>(inst, n, half, d_cost, d_stats, stream);
}

size_t cost_table_big_bytes(int m) { return m > CT_PARAM_M ? (size_t)m * sizeof(ClauseRec) + 16 : 0; }

}  // namespace qaoa

using namespace qaoa;

static int cost_table_common(const naesat_instance *inst, uint8_t *d_cost, uint64_t *n_sol, uint32_t *max_cost,
                             void *stream_, bool half) {
    int rc = validate_instance(inst);
    if (rc) return rc;
    if (!d_cost) return set_error(QAOA_EINVAL, "d_cost is NULL");
    if (half && inst->n < 6) return set_error(QAOA_ERANGE, "half table needs n >= 6 (n=%d)", inst->n);
    cudaStream_t stream = (cudaStream_t)stream_;
    Scratch *sc = nullptr;
    rc = scratch_for(stream, 256 + cost_table_big_bytes(inst->m), 256 + cost_table_big_bytes(inst->m), &sc);
    if (rc) return rc;
    // the counts are needed for the results, and for the range check when a count
    // may exceed the uint8 table
    const bool want = n_sol || max_cost || inst->m > 255;
    unsigned long long *d_stats = want ? reinterpret_cast<unsigned long long *>(sc->dev) : nullptr;
    if (want) QAOA_CUDA_TRY(cudaMemsetAsync(d_stats, 0, 2 * sizeof(unsigned long long), stream));
    rc = launch_cost_table_one(inst, d_cost, d_stats, stream, half, reinterpret_cast<char *>(sc->dev) + 256,
                               reinterpret_cast<char *>(sc->host) + 256);
    if (rc) return rc;
    if (!want) return QAOA_OK;
    unsigned long long *h = reinterpret_cast<unsigned long long *>(sc->host);
    QAOA_CUDA_TRY(cudaMemcpyAsync(h, d_stats, 2 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, stream));
    QAOA_CUDA_TRY(cudaStreamSynchronize(stream));
    if (n_sol) *n_sol = half ? 2 * h[0] : h[0];  // C(not x) = C(x): each half solution has its complement
    if (max_cost) *max_cost = (uint32_t)h[1];
    if (h[1] > 255) return set_error(QAOA_ERANGE, "max C = %llu does not fit the uint8 table", h[1]);
    return QAOA_OK;
}

extern "C" int naesat_cost_table(const naesat_instance *inst, uint8_t *d_cost, uint64_t *n_sol, uint32_t *max_cost,
                                 void *stream) {
    return cost_table_common(inst, d_cost, n_sol, max_cost, stream, false);
}

extern "C" int naesat_cost_table_half(const naesat_instance *inst, uint8_t *d_cost_half, uint64_t *n_sol,
                                      uint32_t *max_cost, void *stream) {
    return cost_table_common(inst, d_cost_half, n_sol, max_cost, stream, true);
}

extern "C" int naesat_cost_table_batch(int batch, const naesat_instance *insts, uint8_t *d_costs, uint64_t *n_sol,
                                       uint32_t *max_cost, void *stream_) {
    if (batch < 1 || !insts || !d_costs) return set_error(QAOA_EINVAL, "batch/insts/d_costs");
    const int n = insts[0].n;
    int m_stride = 1;
    size_t lits = 0;  // literals of the batch
    bool aligned = true;
    for (int b = 0; b < batch; ++b) {
        int rc = valid_sizes(&insts[b]);
        if (rc) return rc;
        if (insts[b].n != n) return set_error(QAOA_EINVAL, "batch instances differ in n");
        m_stride = insts[b].m > m_stride ? insts[b].m : m_stride;
        if (insts[b].m > 0) {
            lits += (size_t)insts[b].m * insts[b].k;
            aligned = aligned && (reinterpret_cast<uintptr_t>(insts[b].var) % sizeof(int32_t)) == 0;
        }
    }
    // Short batches are checked and encoded here (about 3 ns a literal), without
    // the encoder's launch and its first touch of the caller's memory; so are arrays at
    // odd addresses (a record's field, say), which the host reads and the device cannot.
    const bool on_device = lits >= ENCODE_MIN_LITS && batch <= 65535 && aligned;
    if (!on_device)
        for (int b = 0; b < batch; ++b) {
            int rc = validate_instance(&insts[b]);
            if (rc) return rc;
        }
    cudaStream_t stream = (cudaStream_t)stream_;
    DeviceInfo di;
    int rc = device_info(&di);
    if (rc) return rc;
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    // device: records, clause counts, stats [batch][2] and the encoder's verdict,
    // then its descriptors; host: the same, and a copy of the literals where the
    // device cannot read them in place
    const size_t rec_bytes = al((size_t)batch * m_stride * sizeof(ClauseRec));
    const size_t m_bytes = al((size_t)batch * sizeof(int));
    const size_t desc_bytes = on_device ? al((size_t)batch * sizeof(HostLits)) : 0;
    const size_t stat_bytes = ((size_t)batch * 2 + 1) * sizeof(unsigned long long);
    const bool copy = on_device && !di.pageable;
    const size_t host_recs = on_device ? 0 : rec_bytes, copy_bytes = copy ? al(lits * 4) + lits : 0;
    Scratch *sc = nullptr;
    rc = scratch_for(stream, rec_bytes + m_bytes + desc_bytes + stat_bytes,
                     host_recs + m_bytes + desc_bytes + al(stat_bytes) + copy_bytes, &sc);
    if (rc) return rc;
    char *hbase = reinterpret_cast<char *>(sc->host);
    char *dbase = reinterpret_cast<char *>(sc->dev);
    ClauseRec *d_recs = reinterpret_cast<ClauseRec *>(dbase);
    int *d_m = reinterpret_cast<int *>(dbase + rec_bytes);
    HostLits *d_lits = reinterpret_cast<HostLits *>(dbase + rec_bytes + m_bytes);
    unsigned long long *d_stats = reinterpret_cast<unsigned long long *>(dbase + rec_bytes + m_bytes + desc_bytes);
    unsigned long long *d_bad = on_device ? d_stats + 2 * (size_t)batch : nullptr;
    char *h_up = hbase + host_recs;  // clause counts and descriptors, uploaded together
    int *h_m = reinterpret_cast<int *>(h_up);
    HostLits *h_lits = reinterpret_cast<HostLits *>(h_up + m_bytes);
    unsigned long long *h_stats = reinterpret_cast<unsigned long long *>(h_up + m_bytes + desc_bytes);
    char *h_copy = h_up + m_bytes + desc_bytes + al(stat_bytes);
    size_t off = 0;
    for (int b = 0; b < batch; ++b) {
        const naesat_instance &q = insts[b];
        h_m[b] = q.m;
        if (!on_device) {
            encode_instance(&q, reinterpret_cast<ClauseRec *>(hbase) + (size_t)b * m_stride);
            continue;
        }
        HostLits &l = h_lits[b];
        l = HostLits{q.var, q.neg, q.m, q.k};
        if (copy && q.m > 0) {
            const size_t c = (size_t)q.m * q.k;
            int32_t *v = reinterpret_cast<int32_t *>(h_copy) + off;
            uint8_t *g = reinterpret_cast<uint8_t *>(h_copy + al(lits * 4)) + off;
            std::memcpy(v, q.var, c * sizeof(int32_t));
            std::memcpy(g, q.neg, c);
            l.var = v;
            l.neg = g;
            off += c;
        }
    }
    QAOA_CUDA_TRY(cudaMemsetAsync(d_stats, 0, stat_bytes, stream));
    if (on_device) {
        QAOA_CUDA_TRY(cudaMemcpyAsync(d_m, h_up, m_bytes + desc_bytes, cudaMemcpyHostToDevice, stream));
        profile_before(K_ENCODE, stream);
        launch_pdl(encode_kernel, dim3((m_stride + CT_THREADS - 1) / CT_THREADS, batch), dim3(CT_THREADS), 0, stream, n,
                   (const HostLits *)d_lits, m_stride, d_recs, d_bad);
        if ((rc = profile_after(K_ENCODE, stream))) return rc;
    } else {
        QAOA_CUDA_TRY(cudaMemcpyAsync(dbase, hbase, rec_bytes + m_bytes, cudaMemcpyHostToDevice, stream));
    }
    rc = launch_cost_table_batch(batch, n, nullptr, nullptr, d_recs, d_m, m_stride, d_costs, d_stats, stream, true, d_bad);
    if (rc) return rc;
    QAOA_CUDA_TRY(cudaMemcpyAsync(h_stats, d_stats, stat_bytes, cudaMemcpyDeviceToHost, stream));
    QAOA_CUDA_TRY(cudaStreamSynchronize(stream));  // the pinned staging block is reused by the next call
    if (on_device && h_stats[2 * (size_t)batch]) {  // name the first invalid literal
        for (int b = 0; b < batch; ++b) {
            rc = validate_instance(&insts[b]);
            if (rc) return rc;
        }
        return set_error(QAOA_EINVAL, "a literal changed during the call");
    }
    int status = QAOA_OK;
    for (int b = 0; b < batch; ++b) {
        if (n_sol) n_sol[b] = h_stats[2 * b];
        if (max_cost) max_cost[b] = (uint32_t)h_stats[2 * b + 1];
        if (h_stats[2 * b + 1] > 255 && status == QAOA_OK)
            status = set_error(QAOA_ERANGE, "instance %d: max C = %llu does not fit the uint8 table", b, h_stats[2 * b + 1]);
    }
    return status;
}

// ga_mrca.cu -- pairwise MRCA bounds over sampled end-state agents (post hoc relatedness
// estimation from hstrat markers, Fig. 1 caption of the paper).
//
// Synchronous runs (one counter T) take two launches, pack_kernel and pair_kernel; asynchronous
// ones (counters differ) two others, mixed_table_kernel and mixed_pair_kernel (each described
// there).  The second kernel of each pair is in flight while the first still writes what it reads, and
// the first may be while an earlier launch writes the population: inputs are read with plain loads
// behind the wait, not as constant data (__ldg, const __restrict__), which a compiler may move.
#include "ga_device.cuh"
#include "ga_internal.h"

#include <type_traits>

namespace ga {

namespace {

constexpr uint32_t kPackWords = 8;  // 256-bit rank-ordered strings
size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Scratch of a synchronous call: the bounds by first differing bit, then the sampled agents'
// strings of 2 or 8 words (S b <= 64; up to 256 bits).
constexpr size_t kTableBytes = 257 * sizeof(uint2) + 248;  // padded to 256 bytes
static_assert(kTableBytes % 256 == 0, "strings aligned");
uint32_t string_words(uint32_t sites, uint32_t bits) { return sites * bits <= 64u ? 2u : 8u; }
size_t sync_scratch_bytes(uint32_t sites, uint32_t bits, uint32_t n)
{
    return kTableBytes + static_cast<size_t>(n) * string_words(sites, bits) * 4u;
}

// ---------------------------------------------------------------------------------------
// Ranks retained at count T (ranks 0..T-1 deposited), without replaying them.
//
// Steady, S = 2^s sites: while T <= S every rank below T is held.  Otherwise let t >= 1 be
// the epoch of rank T - 1 (bit length minus s) and P = 2^(s+t-1) its first rank.  At P the
// surface holds exactly the ranks below P whose hanoi value is at least t - 1: the S/2 with
// hanoi >= t (rank + 1 = 2^t q, q = 1..S/2) and the S/2 with hanoi exactly t - 1 (rank + 1 =
// 2^(t-1) (2m + 1), m = 0..S/2-1).  Each of the c = T / 2^t - S/2 ranks of epoch t stored so
// far (hanoi >= t: rank + 1 = 2^t (S/2 + 1), 2^t (S/2 + 2), ...) replaced the oldest remaining
// rank of hanoi t - 1, so those m < c are gone.  Retained rank q (0 <= q < S), as rank + 1:
// q < S/2: 2^t (q + 1); S/2 <= q < S - c: 2^(t-1) (2 (c + q - S/2) + 1); else 2^t (S/2 + 1 +
// q - (S - c)).  A rank never moves, so its site is the closed-form site of the rank itself.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t steady_retained(uint32_t s, uint32_t T, uint32_t q)
{
    const uint32_t S = 1u << s;
    if (T <= S) return q < T ? q + 1u : 0u;
    const uint32_t t = 32u - __clz(T - 1u) - s;
    const uint32_t half = S >> 1;
    const uint32_t c = (T >> t) - half;
    uint64_t r1;
    if (q < half) r1 = static_cast<uint64_t>(q + 1u) << t;
    else if (q < S - c) r1 = static_cast<uint64_t>(2u * (c + q - half) + 1u) << (t - 1u);
    else r1 = static_cast<uint64_t>(half + 1u + q - (S - c)) << t;
    return static_cast<uint32_t>(r1);
}

// Tilted, S sites in L = S/2 levels: site k = 2h + p.  Below the top level (h < L - 1) the
// site holds the newest rank < T whose hanoi value is exactly h -- rank + 1 = 2^h (2m + 1) --
// with m of parity p; the top level the newest whose hanoi value is at least L - 1 -- rank + 1
// = 2^(L-1) m', m' >= 1 -- with m' - 1 of parity p.  Returns rank + 1, or 0 for an empty site.
__device__ __forceinline__ uint32_t tilted_holder(uint32_t S, uint32_t T, uint32_t k)
{
    const uint32_t L = S >> 1, h = k >> 1, p = k & 1u;
    if (h + 1u < L) {
        if (h >= 32u || static_cast<uint64_t>(T) < (1ull << h)) return 0u;
        const uint64_t mmax = (static_cast<uint64_t>(T) - (1ull << h)) >> (h + 1u);
        const int64_t m = (mmax & 1u) == p ? static_cast<int64_t>(mmax) : static_cast<int64_t>(mmax) - 1;
        if (m < 0) return 0u;
        return static_cast<uint32_t>(static_cast<uint64_t>(2 * m + 1) << h);
    }
    const uint32_t e = L - 1u;
    if (e >= 32u) return 0u;
    const int64_t mpmax = static_cast<int64_t>(static_cast<uint64_t>(T) >> e);
    const int64_t mp = ((mpmax - 1) & 1) == static_cast<int64_t>(p) ? mpmax : mpmax - 1;
    if (mp < 1) return 0u;
    return static_cast<uint32_t>(static_cast<uint64_t>(mp) << e);
}

// Retained entry q of the surface at count T (q < S): its site and rank + 1 (0: none).
// Hybrid: q < S/2 are the steady half's retained ranks over the even ranks (local count
// ceil(T/2), global rank 2 x local), q >= S/2 the tilted half's sites over the odd ranks
// (local count floor(T/2), global rank 2 x local + 1).
__device__ __forceinline__ uint32_t retained_entry(uint32_t policy, uint32_t s, uint32_t S,
                                                   uint32_t T, uint32_t q, uint32_t &site)
{
    if (policy == kSteady) {
        const uint32_t r1 = steady_retained(s, T, q);
        site = r1 ? static_cast<uint32_t>(steady_site(s, r1 - 1u)) : 0u;
        return r1;
    }
    if (policy == kTilted) {
        site = q;
        return tilted_holder(S, T, q);
    }
    const uint32_t half = S >> 1;
    if (q < half) {
        const uint32_t Te = static_cast<uint32_t>((static_cast<uint64_t>(T) + 1u) >> 1);
        const uint32_t r1 = steady_retained(s - 1u, Te, q);
        site = r1 ? static_cast<uint32_t>(steady_site(s - 1u, r1 - 1u)) : 0u;
        return r1 ? 2u * (r1 - 1u) + 1u : 0u;
    }
    site = q;
    const uint32_t r1 = tilted_holder(half, T >> 1, q - half);
    return r1 ? 2u * r1 : 0u;
}

// 32 x 32 bit transposes across a warp: bit (r, c) -- lane r's bit c -- moves to (c, r), in five
// exchanges of half-width blocks.  The lane's masks, byte selectors and rotations are made once.
struct Transpose32 {
    uint32_t select16, select8, keep[3], turn[3];
    __device__ __forceinline__ explicit Transpose32(uint32_t lane)
    {
        select16 = (lane & 16u) ? 0x3276u : 0x5410u;
        select8 = (lane & 8u) ? 0x3715u : 0x6240u;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t j = 4u >> k, low = k == 0 ? 0x0F0F0F0Fu : k == 1 ? 0x33333333u : 0x55555555u;
            keep[k] = (lane & j) ? ~low : low;
            turn[k] = (lane & j) ? 32u - j : j;
        }
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t x) const
    {
        x = __byte_perm(x, __shfl_xor_sync(0xffffffffu, x, 16), select16);
        x = __byte_perm(x, __shfl_xor_sync(0xffffffffu, x, 8), select8);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            uint32_t y = __shfl_xor_sync(0xffffffffu, x, 4 >> k);
            y = __funnelshift_l(y, y, turn[k]);
            x = (x & keep[k]) | (y & ~keep[k]);
        }
        return x;
    }
};

uint32_t margin(uint32_t bits)
{
    // smallest K with 2^(-bits*K) < 0.05, i.e. bits*K > log2(20) = 4.32
    uint32_t K = 1;
    while (bits * K <= 4u) ++K;
    return K;
}

// ---------------------------------------------------------------------------------------
// One counter T.  With r_0 < ... < r_{m-1} the ranks retained at T and i* the first rank index
// at which two agents' differentiae differ: hi = r_{i*} and lo = r_{i*-K} + 1 (0 if i* < K);
// with no mismatch hi = T and lo = r_{m-K} + 1 (0 if m < K).
//   1. pack_kernel: 256 agents per block.  The rank order at T in closed form, in every block:
//      thread k < S finds retained entry k and puts it at its site; the occupied sites are sorted
//      by counting smaller ranks (block 0 writes the table of both bounds by first differing
//      bit).  Each warp packs 32 agents into strings with differentia index i in bits
//      [i b, i b + b), each word bit-reversed so that the first differing bit of a pair is the
//      highest of the first words that differ.  The permutation from site order to rank order
//      moves bit planes: a 32 x 32 bit transpose turns 32 agents' words into one word per surface
//      bit, which are read back in rank order and transposed again.  Bound by two dependent reads,
//      ids and records.
//   2. pair_kernel: one thread per pair in output order, each warp a contiguous stretch of whole
//      128-byte lines; lane t takes pairs base + t, base + t + 32, ... and steps 32 columns at a
//      time, reloading row i's string only when a step carries it into the next rows.  Per pair one
//      string load (8 bytes; 32 where S b > 64), a find-highest-bit and one table read.  Bound by
//      the bounds it writes, 8 bytes per pair: a plain fill of the same 67 MB takes 12.5 us.
// Slower: rows taken whole by a warp, whose ends leave part of a line to the next row (16.5 us
// for the call of 4,096 agents, 17.8 unrolled by four); 4-byte string and table reads (20.2 us);
// one launch in which a block packs the agents of its own tile of pairs (17 to 24 us).
// The call (with the order, now found while the previous grid drains, and the bit-by-bit gather it
// took 4 us before the pair kernel): 4,096 agents with 64 sites (8.4M pairs) 14.1 us, 18.3 before;
// 3,000 agents with 256 sites 16.3 us, 28.5 before; 300 agents 5.5 and 7.2 us, 7.9 and 10.7 before.
// ---------------------------------------------------------------------------------------
constexpr uint32_t kPairThreads = 256;

// Table entry of a pair: 32 W less the index of the first bit in which its strings of W words
// differ, 0 for none.  Words are bit-reversed: the first differing bit is the highest of the first
// words that differ.
__device__ __forceinline__ uint32_t highest_bit(uint32_t x)
{
    uint32_t at;
    asm("bfind.u32 %0, %1;" : "=r"(at) : "r"(x));  // ~0 for 0
    return at;
}
__device__ __forceinline__ uint32_t pair_entry(uint2 a, uint2 b)
{
    const uint32_t x0 = a.x ^ b.x, x1 = a.y ^ b.y;
    return highest_bit(x0 != 0u ? x0 : x1) + (x0 != 0u ? 33u : 1u);
}
struct String8 {
    uint4 h[2];
};
__device__ __forceinline__ uint32_t pair_entry(const String8 &a, const String8 &b)
{
    const uint32_t x[8] = {a.h[0].x ^ b.h[0].x, a.h[0].y ^ b.h[0].y, a.h[0].z ^ b.h[0].z, a.h[0].w ^ b.h[0].w,
                           a.h[1].x ^ b.h[1].x, a.h[1].y ^ b.h[1].y, a.h[1].z ^ b.h[1].z, a.h[1].w ^ b.h[1].w};
    const bool f = (x[0] | x[1] | x[2] | x[3]) != 0u;
    const uint32_t y0 = f ? x[0] : x[4], y1 = f ? x[1] : x[5], y2 = f ? x[2] : x[6], y3 = f ? x[3] : x[7];
    const bool g = (y0 | y1) != 0u;
    const uint32_t z0 = g ? y0 : y2, z1 = g ? y1 : y3;
    const bool k = z0 != 0u;
    return highest_bit(k ? z0 : z1) + 1u + (f ? 128u : 0u) + (g ? 64u : 0u) + (k ? 32u : 0u);
}
// The string of sampled agent a of n: W = 2, an 8-byte word each; W = 8, two arrays of 16 bytes.
__device__ __forceinline__ void read_string(const void *packed, uint32_t, uint32_t a, uint2 &v)
{
    v = static_cast<const uint2 *>(packed)[a];
}
__device__ __forceinline__ void read_string(const void *packed, uint32_t n, uint32_t a, String8 &v)
{
    v.h[0] = static_cast<const uint4 *>(packed)[a];
    v.h[1] = static_cast<const uint4 *>(packed)[n + a];
}

// W: words of a string (2: S b <= 64; 8: up to 256 bits).
template <uint32_t W>
__global__ void __launch_bounds__(256)
pack_kernel(const uint4 *pop, uint32_t record_quads, uint32_t n_agents,
            const uint32_t *ids, uint32_t n, uint32_t policy, uint32_t log2_sites,
            uint32_t log2_bits, uint32_t K, uint32_t T, uint2 *__restrict__ tab,
            void *__restrict__ packed, int *__restrict__ status)
{
    constexpr uint32_t kEmpty = 0xFFFFFFFFu;          // ranks are below a counter
    __shared__ __align__(16) uint32_t held[32 * W];  // by site: its rank
    __shared__ uint32_t rank_s[32 * W], place[32 * W];  // by rank index: rank, site bit
    __shared__ uint32_t plane[8][32u * W];
    const uint32_t k = threadIdx.x, warp = k >> 5, lane = k & 31u;
    const uint32_t a = blockIdx.x * 256u + k;
    const uint32_t sites = 1u << log2_sites, bits = 1u << log2_bits;
    const uint32_t words = (sites * bits + 31u) >> 5;
    // the rank order needs nothing from the grid before
    if (k < 32u * W) held[k] = kEmpty;
    __syncthreads();
    if (k < sites) {
        uint32_t site = 0;
        const uint32_t r1 = retained_entry(policy, log2_sites, sites, T, k, site);
        if (r1 != 0u && in_bounds(site < sites, status)) held[site] = r1 - 1u;
    }
    __syncthreads();
    const uint32_t mine = k < sites ? held[k] : kEmpty;
    const uint32_t m = static_cast<uint32_t>(__syncthreads_count(mine != kEmpty));
    if (mine != kEmpty) {
        uint32_t pos = 0;
        for (uint32_t q = 0; q < sites; q += 4u) {
            const uint4 v = *reinterpret_cast<const uint4 *>(&held[q]);
            pos += (v.x < mine) + (v.y < mine) + (v.z < mine) + (v.w < mine);
        }
        rank_s[pos] = mine;
        place[pos] = k << log2_bits;
    }
    // the previous grid may still be writing the population (or reading what this call
    // overwrites); the pair kernel may start its set-up
    wait_previous_grid();
    release_next_grid();
    uint32_t w[W];
#pragma unroll
    for (uint32_t e = 0; e < W; ++e) w[e] = 0u;
    if (a < n) {
        const uint32_t id = ids[a];
        if (id >= n_agents) {
            atomicCAS(status, GA_OK, GA_EINVAL);
        } else {
            const uint4 *r = pop + static_cast<size_t>(id) * record_quads;
            const uint4 q0 = r[0];
            w[0] = q0.z;
            w[1] = words > 1u ? q0.w : 0u;
            if constexpr (W > 2u) {  // records of 32 or 48 bytes
                const uint4 q1 = r[1];
                w[2] = q1.x;
                w[3] = words > 3u ? q1.y : 0u;
                w[4] = words > 4u ? q1.z : 0u;
                w[5] = words > 5u ? q1.w : 0u;
                if (record_quads > 2u) {
                    const uint4 q2 = r[2];
                    w[6] = words > 6u ? q2.x : 0u;
                    w[7] = words > 7u ? q2.y : 0u;
                }
            }
            if (q0.y != T) atomicCAS(status, GA_OK, GA_ESTATE);
        }
    }
    __syncthreads();
    if (blockIdx.x == 0)
        for (uint32_t c = k; c <= 32u * W; c += 256u) {  // c: first differing bit, 32 W: none
            const uint32_t r = min(c >> log2_bits, m);
            tab[32u * W - c] = make_uint2(r >= K ? rank_s[r - K] + 1u : 0u, r < m ? rank_s[r] : T);
        }
    if (blockIdx.x * 256u + 32u * warp >= n) return;  // whole warps
    const Transpose32 transpose(lane);
#pragma unroll
    for (uint32_t e = 0; e < W; ++e)
        if (e < words) plane[warp][32u * e + lane] = transpose(w[e]);
    __syncwarp();
#pragma unroll
    for (uint32_t e = 0; e < W; ++e) {
        w[e] = 0u;
        if (e < words) {
            const uint32_t q = 32u * e + lane, i = q >> log2_bits;
            w[e] = __brev(transpose(i < m ? plane[warp][place[i] + (q & (bits - 1u))] : 0u));
        }
    }
    if (a >= n) return;
    if constexpr (W == 2u) {
        static_cast<uint2 *>(packed)[a] = make_uint2(w[0], w[1]);
    } else {
        static_cast<uint4 *>(packed)[a] = make_uint4(w[0], w[1], w[2], w[3]);
        static_cast<uint4 *>(packed)[static_cast<size_t>(n) + a] = make_uint4(w[4], w[5], w[6], w[7]);
    }
}

// Row and column of pair p in output order: row i holds pairs off(i) <= p < off(i + 1) with
// off(i) = i (2n - i - 1) / 2.  A single-precision root of i^2 - (2n - 1) i + 2p = 0 from the
// exact 64-bit discriminant is within one row; integer comparisons correct it.
__device__ __forceinline__ void first_pair(uint32_t n, uint32_t p, uint32_t &i, uint32_t &j)
{
    const unsigned long long b = 2ull * n - 1ull;  // off(r) = r (b - r) / 2
    const float est = (static_cast<float>(b) - sqrtf(static_cast<float>(b * b - 8ull * p))) * 0.5f;
    i = est > 0.0f ? static_cast<uint32_t>(est) : 0u;
    if (i > n - 2u) i = n - 2u;
    while (i > 0u && static_cast<unsigned long long>(i) * (b - i) / 2ull > p) --i;
    while (i + 2u < n && static_cast<unsigned long long>(i + 1u) * (b - i - 1u) / 2ull <= p) ++i;
    j = i + 1u + static_cast<uint32_t>(p - static_cast<unsigned long long>(i) * (b - i) / 2ull);
}

template <uint32_t W>
__global__ void __launch_bounds__(kPairThreads)
pair_kernel(const void *packed, uint32_t n, const uint2 *tab_g,
            uint32_t per_warp, uint32_t *__restrict__ lo, uint32_t *__restrict__ hi, int *__restrict__ status)
{
    __shared__ uint2 tab[32 * W + 1];
    // pairs [warp * per_warp, (warp + 1) * per_warp) of n (n - 1) / 2 (fewer than 2^31)
    const uint32_t n_pairs = static_cast<uint32_t>(static_cast<unsigned long long>(n) * (n - 1u) / 2ull);
    const uint32_t warp = (blockIdx.x * kPairThreads + threadIdx.x) >> 5;
    const unsigned long long w_end = static_cast<unsigned long long>(warp + 1u) * per_warp;
    const uint32_t p_end = w_end < n_pairs ? static_cast<uint32_t>(w_end) : n_pairs;
    const unsigned long long p0 = static_cast<unsigned long long>(warp) * per_warp + (threadIdx.x & 31u);
    const bool active = p0 < p_end;
    uint32_t q = active ? static_cast<uint32_t>(p0) : 0u;
    uint32_t i = 0, j = 1;
    first_pair(n, q, i, j);

    wait_previous_grid();  // the table and the strings come from pack_kernel
    for (uint32_t c = threadIdx.x; c <= 32u * W; c += kPairThreads) tab[c] = tab_g[c];
    __syncthreads();
    if (!active || !in_bounds(i < j && j < n, status)) return;

    std::conditional_t<W == 2u, uint2, String8> row, other;
    read_string(packed, n, i, row);
    for (;;) {
        read_string(packed, n, j, other);
        const uint2 bound = tab[pair_entry(row, other)];
        __stcs(lo + q, bound.x);
        __stcs(hi + q, bound.y);
        q += 32u;
        if (q >= p_end) break;
        j += 32u;
        if (j >= n) {  // past the end of row i: pair (i + 1, i + 2) follows (i, n - 1)
            do {
                j = j - n + i + 2u;
                ++i;
            } while (j >= n);
            if (!in_bounds(i < j, status)) break;
            read_string(packed, n, i, row);
        }
    }
}

// Both launches of one synchronous MRCA call (shared by the allocating and the fixed-scratch
// entry points).
cudaError_t launch_sync_mrca(const void *pop, uint32_t record_bytes, uint32_t n_agents, const uint32_t *d_ids,
                             uint32_t n, void *scratch, uint32_t policy, uint32_t log2_sites, uint32_t sites,
                             uint32_t bits, uint32_t T, uint32_t *d_lo, uint32_t *d_hi, int *status,
                             cudaStream_t stream)
{
    const uint32_t log2_bits = bits == 1u ? 0u : bits == 2u ? 1u : bits == 4u ? 2u : 3u;
    const bool narrow = string_words(sites, bits) == 2u;
    uint2 *tab = static_cast<uint2 *>(scratch);
    void *packed = static_cast<uint8_t *>(scratch) + kTableBytes;
    cudaError_t e = launch_dependent(narrow ? pack_kernel<2> : pack_kernel<8>, (n + 255u) / 256u, 256, stream,
                                     static_cast<const uint4 *>(pop), record_bytes / 16u, n_agents, d_ids, n,
                                     policy, log2_sites, log2_bits, margin(bits), T, tab, packed, status);
    if (e != cudaSuccess) return e;
    // enough blocks for the whole GPU (8 resident on each of 152 SMs), each warp then sweeping a
    // contiguous stretch of whole lines
    const unsigned long long pairs = static_cast<unsigned long long>(n) * (n - 1u) / 2ull;
    const unsigned long long want = (pairs + kPairThreads - 1u) / kPairThreads;
    const uint32_t grid = static_cast<uint32_t>(want < 1216u ? want : 1216u);
    const unsigned long long warps = static_cast<unsigned long long>(grid) * (kPairThreads / 32u);
    const uint32_t per_warp = static_cast<uint32_t>(((pairs + warps - 1ull) / warps + 31ull) / 32ull * 32ull);
    return launch_dependent(narrow ? pair_kernel<2> : pair_kernel<8>, grid, kPairThreads, stream,
                            static_cast<const void *>(packed), n, static_cast<const uint2 *>(tab), per_warp, d_lo, d_hi, status);
}

// ---------------------------------------------------------------------------------------
// Mixed counters (asynchronous runs): agents i and j may hold different counters Ti, Tj.  A
// rank, once deposited, stays at its own site until overwritten, and what is dropped never
// comes back.  So with Ta <= Tb the ranks retained at both counters are exactly those of b's
// holder table that are below Ta: in b's rank order the common ranks are a prefix, and one
// binary search (or the rank at the first mismatch itself) finds its end.
//   1. mixed_table_kernel: each sampled agent's counter, surface words and, in closed form at
//                      its own counter, its sites sorted by retained rank.
//   2. mixed_pair_kernel: a tile of 32 x 64 pairs per block; every pair is done by the warp
//                      that holds its larger-counter agent b (rank order uniform in the warp)
//                      with the smaller-counter agents a in the lanes.  The agents' surfaces
//                      lie transposed in shared memory (one word per surface bit, one bit per
//                      agent), so lane l looks up the mismatches of all 32 agents at b's l-th
//                      rank in one word, and a 32 x 32 bit transpose hands every lane its own
//                      agent's mismatches in b's rank order: the first set bit is the answer.
// Issue-bound: 215 warp-instructions per 32 pairs (the tables 25 more), against 2,757 for one thread per pair
// walking both agents' sites twice.  The whole call for 3,001 agents with 64 sites (4.5M pairs, 36
// MB of bounds): 47 us, 376 us before; 2,816 agents with 256 sites 122 us, 1,371 before.
// ---------------------------------------------------------------------------------------
constexpr uint32_t kMixRows = 32, kMixCols = 64;
constexpr uint32_t kMixPad = kMixCols + 1;  // staged bounds: row stride without bank conflicts

struct MixedLayout {
    uint32_t *cnt;     // [n] counters of the sampled agents
    uint32_t *held;    // [n] retained ranks m of each
    uint32_t *surf;    // [n][W] surface words
    uint32_t *ranks;   // [n][S] retained ranks, ascending (m of them)
    uint8_t *order;    // [n][S] their sites
};

uint32_t surface_words(uint32_t S, uint32_t bits) { return (S * bits + 31u) / 32u; }

// Carves the scratch at `scratch` (null: only the size is wanted) and returns its bytes.
size_t carve_mixed(void *scratch, uint32_t S, uint32_t bits, uint32_t n, MixedLayout &l)
{
    uint8_t *p = static_cast<uint8_t *>(scratch);
    const size_t agents = n;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        uint8_t *at = p ? p + off : nullptr;
        off += align_up(bytes, 256);
        return at;
    };
    l.cnt = reinterpret_cast<uint32_t *>(take(agents * 4u));
    l.held = reinterpret_cast<uint32_t *>(take(agents * 4u));
    l.surf = reinterpret_cast<uint32_t *>(take(agents * surface_words(S, bits) * 4u));
    l.ranks = reinterpret_cast<uint32_t *>(take(agents * S * 4u));
    l.order = take(agents * S);
    return off;
}

// 256 / S agents per block, S threads each: thread (agent, k) finds retained entry k of the
// agent's counter and puts it at its site, then sorts site k among the occupied ones by
// counting the smaller ranks.
__global__ void __launch_bounds__(256)
mixed_table_kernel(const uint32_t *pop, uint32_t record_words, uint32_t n_agents,
                   const uint32_t *ids, uint32_t n, uint32_t policy,
                   uint32_t log2_sites, uint32_t words, uint32_t *__restrict__ cnt,
                   uint32_t *__restrict__ held, uint32_t *__restrict__ surf,
                   uint32_t *__restrict__ ranks, uint8_t *__restrict__ order,
                   int *__restrict__ status)
{
    constexpr uint32_t kEmpty = 0xFFFFFFFFu;  // no rank reaches it: ranks are below a counter
    __shared__ __align__(16) uint32_t h[256];
    release_next_grid();
    const uint32_t sites = 1u << log2_sites;
    const uint32_t base = threadIdx.x & ~(sites - 1u), k = threadIdx.x & (sites - 1u);
    const uint32_t a = (blockIdx.x * 256u + threadIdx.x) >> log2_sites;
    const uint32_t id = a < n ? ids[a] : 0u;
    const bool ok = a < n && id < n_agents;
    const uint32_t *rec = pop + static_cast<size_t>(ok ? id : 0u) * record_words;
    const uint32_t T = ok ? rec[1] : 0u;
    if (a < n && k < words) surf[static_cast<size_t>(a) * words + k] = ok ? rec[2u + k] : 0u;
    h[threadIdx.x] = kEmpty;
    __syncthreads();
    uint32_t site = 0;
    const uint32_t r1 = retained_entry(policy, log2_sites, sites, T, k, site);
    if (r1 != 0u && in_bounds(site < sites, status)) h[base + site] = r1 - 1u;
    __syncthreads();
    const uint32_t mine = h[threadIdx.x];
    uint32_t pos = 0, m = 0;
    for (uint32_t q = 0; q < sites; q += 4u) {
        const uint4 v = *reinterpret_cast<const uint4 *>(&h[base + q]);
        pos += (v.x < mine) + (v.y < mine) + (v.z < mine) + (v.w < mine);
        m += (v.x != kEmpty) + (v.y != kEmpty) + (v.z != kEmpty) + (v.w != kEmpty);
    }
    if (a >= n) return;
    if (mine != kEmpty) {
        ranks[static_cast<size_t>(a) * sites + pos] = mine;
        order[static_cast<size_t>(a) * sites + pos] = static_cast<uint8_t>(k);
    }
    if (k == 0u) {
        if (!ok) atomicCAS(status, GA_OK, GA_EINVAL);
        cnt[a] = T;
        held[a] = m;
    }
}

// Block (x, y): rows i in [32 y, 32 y + 32), columns j in [64 x, 64 x + 64), pairs i < j.  THREADS:
// 256, or 1,024 where there are fewer tiles than two for each SM (a tile's 128 steps then take a
// quarter of the time: 249 agents 12.6 us, 20 with 256).  BIT: one-bit differentiae.
template <uint32_t THREADS, bool BIT>
__global__ void __launch_bounds__(THREADS)
mixed_pair_kernel(uint32_t n, uint32_t sites, uint32_t words, uint32_t bits, uint32_t K,
                  const uint32_t *cnt, const uint32_t *held,
                  const uint32_t *surf, const uint32_t *ranks,
                  const uint8_t *order, uint32_t *__restrict__ lo,
                  uint32_t *__restrict__ hi, int *__restrict__ status)
{
    constexpr uint32_t kNone = 0xFFFFFFFFu;
    // groups of 32 agents: 0 the tile's rows, 1 and 2 its columns; word q of a group: bit q of
    // the 32 agents' surfaces
    __shared__ uint32_t plane[3][32u * kPackWords];
    __shared__ uint32_t count[3][32];
    __shared__ uint32_t held_s[3][32];
    __shared__ uint32_t s_lo[kMixRows][kMixPad], s_hi[kMixRows][kMixPad];
    const uint32_t i0 = blockIdx.y * kMixRows, j0 = blockIdx.x * kMixCols;
    if (j0 + kMixCols <= i0 + 1u) return;  // whole tile on or below the diagonal
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    const Transpose32 transpose(lane);
    auto first_of = [&](uint32_t g) { return g == 0u ? i0 : j0 + 32u * (g - 1u); };
    wait_previous_grid();
    for (uint32_t t = warp; t < 3u * words; t += THREADS / 32u) {
        const uint32_t g = t / words, w = t - g * words;
        const uint32_t a = first_of(g) + lane;
        const uint32_t v = a < n ? surf[static_cast<size_t>(a) * words + w] : 0u;
        plane[g][32u * w + lane] = transpose(v);
    }
    if (threadIdx.x < 96u) {
        const uint32_t g = threadIdx.x >> 5, a = first_of(g) + lane;
        count[g][lane] = a < n ? cnt[a] : 0u;
        held_s[g][lane] = a < n ? held[a] : 0u;
    }
    __syncthreads();

    // The pairs of agent b (lane bl of group gb, index nb in the sample) with the agents of NG
    // groups from ga on (one per lane each, counters at most b's where `active`): bounds of each
    // lane's pairs.  site0: b's site at rank index `lane`, read a step ahead.
    auto pairs_of = [&](auto groups, uint32_t gb, uint32_t bl, uint32_t nb, uint32_t ga, uint32_t site0,
                        const uint32_t *Ta, const bool *active, uint32_t *l, uint32_t *h) {
        constexpr int NG = decltype(groups)::value;
        const uint32_t m = held_s[gb][bl];
        const uint32_t *rk = ranks + static_cast<size_t>(nb) * sites;
        const uint8_t *od = order + static_cast<size_t>(nb) * sites;
        uint32_t first[NG];  // first index in b's rank order whose differentiae differ
        bool open[NG], any = false;
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            first[g] = kNone;
            open[g] = active[g];
        }
        for (uint32_t c0 = 0; c0 < m; c0 += 32u) {
            uint32_t differ[NG];  // bit a: agent a differs from b at b's (c0 + lane)-th rank
#pragma unroll
            for (int g = 0; g < NG; ++g) differ[g] = 0u;
            if (c0 + lane < m) {
                const uint32_t q0 = (c0 == 0u ? site0 : od[c0 + lane]) * (BIT ? 1u : bits);
                if (in_bounds(q0 + bits <= 32u * words, status)) {
                    for (uint32_t q = q0; q < q0 + (BIT ? 1u : bits); ++q) {
                        const uint32_t mine = 0u - ((plane[gb][q] >> bl) & 1u);
#pragma unroll
                        for (int g = 0; g < NG; ++g) differ[g] |= plane[ga + g][q] ^ mine;
                    }
                }
            }
            any = false;
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                const uint32_t x = transpose(differ[g]);
                if (open[g] && x != 0u) {
                    first[g] = c0 + static_cast<uint32_t>(__ffs(static_cast<int>(x))) - 1u;
                    open[g] = false;
                }
                any = any || open[g];
            }
            if (!__any_sync(0xffffffffu, any)) break;
        }
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            if (!active[g]) continue;
            // a mismatch at a rank not below Ta lies past the common prefix
            const uint32_t fr = first[g] != kNone ? rk[first[g]] : kNone;
            const uint32_t fl = first[g] != kNone && first[g] >= K ? rk[first[g] - K] + 1u : 0u;
            h[g] = fr;
            l[g] = fl;
            if (fr >= Ta[g]) {  // no common rank differs: the prefix ends at the first rank >= Ta
                uint32_t below = 0, above = m;
                while (below < above) {
                    const uint32_t mid = (below + above) >> 1;
                    if (rk[mid] < Ta[g]) below = mid + 1u;
                    else above = mid;
                }
                h[g] = Ta[g];
                l[g] = below >= K ? rk[below - K] + 1u : 0u;
            }
        }
    };
    // the site at rank index `lane` of sampled agent a (0 where there is none)
    auto first_site = [&](uint32_t a) {
        return a < n && lane < sites ? static_cast<uint32_t>(order[static_cast<size_t>(a) * sites + lane]) : 0u;
    };

    // pairs whose row agent holds the larger counter (or the same): b = row, lanes = columns
    uint32_t ahead = first_site(i0 + warp);
    for (uint32_t r = warp; r < kMixRows; r += THREADS / 32u) {
        const uint32_t i = i0 + r, Tb = count[0][r], site0 = ahead;
        if (r + THREADS / 32u < kMixRows) ahead = first_site(i + THREADS / 32u);
        uint32_t Ta[2], l[2], h[2];
        bool active[2];
#pragma unroll
        for (uint32_t g = 0; g < 2u; ++g) {
            const uint32_t j = j0 + 32u * g + lane;
            Ta[g] = count[1u + g][lane];
            active[g] = i < j && j < n && Ta[g] <= Tb;
        }
        if (!__any_sync(0xffffffffu, active[0] || active[1])) continue;
        pairs_of(std::integral_constant<int, 2>(), 0u, r, i, 1u, site0, Ta, active, l, h);
#pragma unroll
        for (uint32_t g = 0; g < 2u; ++g)
            if (active[g]) {
                s_lo[r][32u * g + lane] = l[g];
                s_hi[r][32u * g + lane] = h[g];
            }
    }
    // pairs whose column agent holds the larger counter: b = column, lanes = rows
    ahead = first_site(j0 + warp);
    for (uint32_t c = warp; c < kMixCols; c += THREADS / 32u) {
        const uint32_t g = 1u + (c >> 5), bl = c & 31u, site0 = ahead;
        const uint32_t i = i0 + lane, j = j0 + c, Ta = count[0][lane];
        if (c + THREADS / 32u < kMixCols) ahead = first_site(j + THREADS / 32u);
        const bool active = i < j && j < n && Ta < count[g][bl];
        if (!__any_sync(0xffffffffu, active)) continue;
        uint32_t l = 0, h = 0;
        pairs_of(std::integral_constant<int, 1>(), g, bl, j, 0u, site0, &Ta, &active, &l, &h);
        if (active) {
            s_lo[lane][c] = l;
            s_hi[lane][c] = h;
        }
    }
    __syncthreads();
    // the tile's bounds, row by row in output order
    for (uint32_t t = threadIdx.x; t < kMixRows * kMixCols; t += THREADS) {
        const uint32_t r = t / kMixCols, c = t % kMixCols;
        const uint32_t i = i0 + r, j = j0 + c;
        if (i < j && j < n) {
            const size_t p = static_cast<size_t>(i) * (2ull * n - i - 1ull) / 2ull + (j - i - 1u);
            __stcs(&lo[p], s_lo[r][c]);
            __stcs(&hi[p], s_hi[r][c]);
        }
    }
}

}  // namespace

size_t mrca_scratch_bytes(const ga_run *run, uint32_t n)
{
    const uint32_t S = run->cfg.surface_sites;
    if (run->cfg.mode != GA_SYNC) {
        MixedLayout l;
        return carve_mixed(nullptr, S, run->cfg.differentia_bits, n, l);
    }
    return sync_scratch_bytes(S, run->cfg.differentia_bits, n);
}

namespace {

cudaError_t launch_mrca_mixed(ga_run *run, const uint32_t *d_ids, uint32_t n, uint32_t *d_lo,
                              uint32_t *d_hi, void *scratch)
{
    const uint32_t S = run->cfg.surface_sites, b = run->cfg.differentia_bits;
    MixedLayout l;
    carve_mixed(scratch, S, b, n, l);
    const uint32_t *pop = reinterpret_cast<const uint32_t *>(run->pop[run->cur]);
    const uint32_t rw = run->record_bytes / 4u, words = surface_words(S, b);
    const uint32_t per_block = 256u / S;
    mixed_table_kernel<<<(n + per_block - 1u) / per_block, 256, 0, run->stream>>>(
        pop, rw, run->n_agents, d_ids, n, run->cfg.curation, run->log2_sites, words, l.cnt, l.held,
        l.surf, l.ranks, l.order, run->d_status);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    run->launches += 1;
    const dim3 grid((n + kMixCols - 1u) / kMixCols, (n + kMixRows - 1u) / kMixRows);
    const bool few = grid.x * grid.y / 2u < 2u * 152u;
    const auto kernel = few ? (b == 1u ? mixed_pair_kernel<1024, true> : mixed_pair_kernel<1024, false>)
                            : (b == 1u ? mixed_pair_kernel<256, true> : mixed_pair_kernel<256, false>);
    e = launch_dependent(kernel, grid, few ? 1024u : 256u, run->stream, n, S, words, b, margin(b),
                         static_cast<const uint32_t *>(l.cnt), static_cast<const uint32_t *>(l.held),
                         static_cast<const uint32_t *>(l.surf), static_cast<const uint32_t *>(l.ranks),
                         static_cast<const uint8_t *>(l.order), d_lo, d_hi, run->d_status);
    if (e == cudaSuccess) run->launches += 1;
    return e;
}

}  // namespace

cudaError_t launch_mrca(ga_run *run, const uint32_t *d_ids, uint32_t n, uint32_t *d_lo,
                        uint32_t *d_hi, void *scratch)
{
    if (run->cfg.mode != GA_SYNC) return launch_mrca_mixed(run, d_ids, n, d_lo, d_hi, scratch);
    const uint32_t S = run->cfg.surface_sites, b = run->cfg.differentia_bits;
    const uint32_t T = static_cast<uint32_t>(run->generation);
    const cudaError_t e =
        launch_sync_mrca(run->pop[run->cur], run->record_bytes, run->n_agents, d_ids, n, scratch, run->cfg.curation,
                         run->log2_sites, S, b, T, d_lo, d_hi, run->d_status, run->stream);
    if (e == cudaSuccess) run->launches += 2;
    return e;
}

}  // namespace ga

// ---------------------------------------------------------------------------------------
// ga_mrca_bounds_noalloc: the same MRCA kernels with their scratch held in a fixed
// device array instead of memory allocated per call, for callers that cannot allocate
// device memory (see include/ga.h).
//
// The array is a file-scope __device__ variable, so every GPU that loads this library holds
// its own copy until the process exits.  In host code the name g_mrca_fixed_scratch is only
// a host-side stand-in for the symbol, never a device address; each call looks the address
// up with cudaGetSymbolAddress, with the caller's device current, and passes it to the
// kernels (a lookup per call stays right after a device reset reloads the module, which a
// cached address would not).  Every call on a device reuses the same array: the status word
// is cleared at the start of each call, the table and strings are fully rewritten before
// they are read.
// ---------------------------------------------------------------------------------------
namespace ga {
namespace {

constexpr uint32_t kFixedMaxSample = 4096;    // largest n accepted
constexpr uint32_t kFixedMaxSites = 256;      // S * b <= 256 bits
constexpr size_t kFixedStatusBytes = 256;     // device status word, padded
// status, then the scratch of a call with n = 4096 and S = 256: 256 + 2,304 + 4,096 x 32 bytes
constexpr size_t kFixedScratchBytes = kFixedStatusBytes + kTableBytes + static_cast<size_t>(kFixedMaxSample) * 32u;

static __device__ __align__(256) unsigned char g_mrca_fixed_scratch[kFixedScratchBytes];

}  // namespace
}  // namespace ga

extern "C" int ga_mrca_bounds_noalloc(const void *d_records, uint32_t record_bytes,
                                      uint32_t n_agents, uint32_t curation,
                                      uint32_t surface_sites, uint32_t differentia_bits,
                                      uint32_t generation, const uint32_t *d_agent_ids,
                                      uint32_t n, uint32_t *d_lo, uint32_t *d_hi, void *stream)
{
    using namespace ga;
    const uint32_t S = surface_sites, b = differentia_bits;
    if (!d_records || !d_agent_ids || !d_lo || !d_hi) return GA_EINVAL;
    if (n < 2 || n > kFixedMaxSample) return GA_EINVAL;
    if (curation > GA_HYBRID) return GA_EINVAL;
    if (S == 0u || (S & (S - 1u)) != 0u || S < (curation == GA_HYBRID ? 8u : 4u)) return GA_EINVAL;
    if (!(b == 1u || b == 2u || b == 4u || b == 8u) || S * b > kFixedMaxSites) return GA_EINVAL;
    const uint32_t words = (S * b + 31u) / 32u;
    if (record_bytes != (8u + 4u * words + 15u) / 16u * 16u || n_agents == 0u) return GA_EINVAL;
    if (reinterpret_cast<uintptr_t>(d_records) % 16u != 0u) return GA_EINVAL;
    // an error left pending by earlier, unrelated work on this thread is not this call's
    cudaGetLastError();
    void *base = nullptr;
    if (cudaGetSymbolAddress(&base, g_mrca_fixed_scratch) != cudaSuccess || base == nullptr) {
        cudaGetLastError();
        return GA_ECUDA;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int *status = static_cast<int *>(base);
    uint32_t log2_sites = 0;
    while ((1u << log2_sites) < S) ++log2_sites;

    if (cudaMemsetAsync(status, 0, sizeof(int), st) != cudaSuccess) return GA_ECUDA;
    if (launch_sync_mrca(d_records, record_bytes, n_agents, d_agent_ids, n,
                         static_cast<uint8_t *>(base) + kFixedStatusBytes, curation, log2_sites, S, b, generation, d_lo, d_hi, status, st) != cudaSuccess)
        return GA_ECUDA;
    int device_status = GA_OK;
    if (cudaMemcpyAsync(&device_status, status, sizeof(int), cudaMemcpyDeviceToHost, st) !=
            cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return GA_ECUDA;
    return device_status;
}

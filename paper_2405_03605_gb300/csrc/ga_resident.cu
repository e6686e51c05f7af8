// ga_resident.cu -- resident stepping: a run whose population fits in the SMs' shared memory
// stays there for a whole chunk of generations, in one cooperative launch, and its islands
// trade migrants through mailboxes in global memory (L2) instead of through launch boundaries.
// The paper's processors keep their populations in place and exchange only migrants with their
// neighbours (Sec. 2); this is that arrangement on the GPU.  A launch per generation cannot
// follow it there: it takes at least 2.4 us, even as a dependent one, and 4.3 for a run of 320,000
// agents, whose arithmetic needs 2.
//
// Scope: synchronous runs whose counters all equal the generation, any record size, islands of
// 8 to 64 agents.  Results are bit-identical to the streamed kernels: the same draws, landing
// slots, tournaments, mutations and deposits.
//
// Mapping: each warp, a block of its own, holds a few consecutive islands (units of Shape<N>::P)
// in shared memory for the whole launch and works through them one unit at a time.  The
// migration bookkeeping is done for all the warp's islands at once, one (island, direction)
// pair per lane.  On a migration generation g the warp
//   1. pushes: lane (I, d) writes the member that the neighbour in direction d draws into that
//      neighbour's mailbox for direction d ^ 1 and this migration's parity;
//   2. draws what needs no arrival: the next migration's emigrants and landing slots (they
//      depend on no state) and its first islands' births;
//   3. polls: lane (I, d) reads I's mailbox for direction d until it holds generation g;
//   4. lands the arrivals in its islands' records (shared memory) and reproduces.
//
// Mailboxes: a 16-byte record is its own ready flag (its counter is g); wider records travel as
// three 16-byte chunks of three words and the generation, their counter being g (32-byte records:
// the third chunk one word and the generation three times).  Each chunk is one 128-bit relaxed
// store and load at GPU scope, so it is seen whole or not at all.  They are double-buffered by migration parity: a sender can only overwrite a chunk after it has received
// the receiver's next push, which the receiver makes after reading that chunk.  Every island
// pushes before it polls and the cooperative launch keeps every warp resident, so each poll is
// answered once the neighbour reaches the same generation.  Runs without mailboxes in their
// workspace (wider records, more than 8,192 islands) keep them in the destination buffer,
// each island's in the place of its own records: those are written when the launch ends, by
// the warp that has read the island's last arrival.
//
// Waits are bounded: a poll gives up after the run's wait limit (wall clock, %globaltimer) and
// kMinPolls reads, records GA_ETIMEOUT in the status word and sets the launch's abort word; every poll also
// watches the abort word, so once one warp gives up every warp leaves at its next migration
// generation.  The population is then undefined; the status is returned by the next ga_sync.
//
// What bounds it: small runs the two L2 trips of a migration (32x32 torus of 32-agent islands:
// 1.10 us per generation), larger ones issue (9,991 islands of 32: 2.50 us per generation; 7.2 us
// with one ordinary launch each, 4.3 with dependent ones).  One warp per block: what depends on the
// block alone stays in uniform registers (250 generations of 9,991 islands of 16-byte and 5,893 of
// 48-byte records: 665 and 562 us, four warps per block 707 and 612).
#include "ga_device.cuh"
#include "ga_internal.h"
#include "ga_island.cuh"

namespace ga {

RunParams run_params(const ga_run *run, const void *src, void *dst, uint32_t g0, uint32_t n_gens,
                     bool migrate);

namespace {

// Units per warp: as few as keep an SM's warps to a limit, more where they don't fit at once.  An SM
// has four schedulers, so a generation lengthens where a sixth warp falls to one of them: with one
// unit to a warp the limit is 20.  Us per generation with one unit to a warp and with two, on
// either side of it (2,916 to 3,025 and 3,080 islands of 32): float model 2.08 / 2.20 and 2.34 / 2.20,
// every 4 generations 1.23 / 1.49 and 1.46 / 1.49; trait model every 4 0.70 / 0.73 and 0.81 / 0.73.
// (A limit of 18, which takes two from 2,737 on, made the float model slower there than with a warp
// to every island before: 1.55 against 1.41 every 4.)  But
//   - float model, and islands of 16, with tournaments of run-time size and several generations to
//     a migration: a unit's work is long, so one to a warp up to 28 warps: 3,422 islands of 32 every 4
//     1.51 / 1.63, every 16 1.38 / 1.42;
//   - 16-byte trait records in islands of 32 or 64, tournaments of 5, a migration in one or two
//     generations: so short that from 16 warps on two to a warp are faster, as the bookkeeping of
//     one fills few of a warp's lanes: 2,401 islands of 32 1.40 / 1.43, 2,601 1.50 / 1.45, 3,025 1.55 /
//     1.50; 2,652 of 64 2.02 / 1.95.
// With more units to a warp, 18: 14,042 islands of 32 five or six to a warp (18.5 and 15.4 warps) 3.19
// and 2.95, float model 5.83 and 5.52.
uint32_t units_per_warp(const ga_run *run, uint32_t n_units, uint32_t sms)
{
    const bool five = run->cfg.tournament_size == 5u, fit = run->cfg.model == GA_MODEL_FITNESS;
    const uint32_t N = run->cfg.island_size, k = run->per_neighbor ? run->every_k : 0xFFFFFFFFu;
    uint32_t single = 20u;
    if (!five && k > 1u && (fit || N == 16u)) single = 28u;
    else if (five && k <= 2u && !fit && N >= 32u && run->record_bytes == 16u) single = 16u;
    if (n_units <= single * sms) return 1u;
    const uint32_t units = (n_units + 18u * sms - 1u) / (18u * sms);
    return units < 2u ? 2u : units;
}

// Reads that a wait makes at least before it gives up (3 to 5 ms).  The clock goes on while the GPU runs
// another process; without them a launch that was set aside for longer than the limit would give up
// though its neighbours are about to answer.
constexpr uint32_t kMinPolls = 4096;

struct ResidentArgs {
    RunParams r;
    RoundKeys rk;
    uint4 *mail;             // mailboxes: island i's from mail + i * mail_stride
    uint32_t mail_stride;    // [parity][direction][chunk] of an island, in 16-byte chunks
    uint32_t *abort_word;    // 0; set to 1 by a warp that gave up waiting
    unsigned long long wait_ns;
    uint32_t every_k, per_neighbor;
    uint32_t drop_island;    // fault injection: this island's pushes are dropped (~0u: none)
    uint32_t units;          // units of Shape<N>::P islands per warp
};

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// 128-bit relaxed accesses at GPU scope, each one memory operation: the reader sees all of a
// 16-byte chunk or none of it.  The reader has to use all four words: of a load with unused words
// only the others are loaded, and no longer in one access (32-byte records whose third chunk
// carried two unused words arrived with that chunk's new generation and its old first word some
// three times in 100,000 migrants).
__device__ __forceinline__ uint4 load128(const uint4 *p)
{
    unsigned long long lo, hi;
    asm volatile("{\n\t.reg .b128 v;\n\t"
                 "ld.relaxed.gpu.global.b128 v, [%2];\n\t"
                 "mov.b128 {%0, %1}, v;\n\t}"
                 : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
    return make_uint4(static_cast<uint32_t>(lo), static_cast<uint32_t>(lo >> 32),
                      static_cast<uint32_t>(hi), static_cast<uint32_t>(hi >> 32));
}

__device__ __forceinline__ void store128(uint4 *p, uint4 v)
{
    const unsigned long long lo = static_cast<unsigned long long>(v.x) | (static_cast<unsigned long long>(v.y) << 32);
    const unsigned long long hi = static_cast<unsigned long long>(v.z) | (static_cast<unsigned long long>(v.w) << 32);
    asm volatile("{\n\t.reg .b128 v;\n\t"
                 "mov.b128 v, {%0, %1};\n\t"
                 "st.relaxed.gpu.global.b128 [%2], v;\n\t}"
                 :: "l"(lo), "l"(hi), "l"(p) : "memory");
}

__device__ __forceinline__ uint32_t load_relaxed(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Deposit masks of the launch's generation `it` ((0, 0) past the table in a device-check build).  The
// resident kernel starts when the set-up kernel that wrote them has ended, so they are constant.
__device__ __forceinline__ uint2 const_mask_at(const RunParams &p, uint32_t it)
{
    return in_bounds(it < p.gen_sites_left, p.status) ? __ldg(&p.gen_masks[it]) : make_uint2(0u, 0u);
}

// Next migration generation at or after g (~0u: none before `end`).
__device__ __forceinline__ uint32_t next_migration(uint32_t g, uint32_t end, uint32_t k, uint32_t on)
{
    if (!on) return ~0u;
    const uint32_t r = g % k;
    const uint64_t m = static_cast<uint64_t>(g) + (r ? k - r : 0u);
    return m < end ? static_cast<uint32_t>(m) : ~0u;
}

template <int SW>
struct Record {
    static constexpr int LW = 2 + SW;
    static constexpr int Q = (LW + 3) / 4;       // 128-bit words of a record
    static constexpr int C = Q == 1 ? 1 : 3;     // 128-bit chunks of a mailbox
};

// Shared memory of one warp, in bytes: its records, then by (island, direction) the neighbour,
// the landing slots of two migrations and the emigrant.
template <int N, int SW>
__host__ __device__ constexpr uint32_t warp_bytes(uint32_t islands)
{
    return islands * (N * Record<SW>::Q * 16u + 4u * (4u + 2u + 1u) + 4u);
}

// Resident warps per SM asked of the compiler, for the registers that leaves (20: 96, 28: 72, 32: 64).
// Fewer registers let the warps of runs on other streams fit beside this one's, and few of them hold a
// single run back: 16-byte records in islands of 32 take 74 to 78 unasked and 62 to 64 here without a
// spill.  65,536 agents, us per generation for one run and for four at once: 1.48 and 6.2 with 20, 1.40
// and 4.0 with 32 (before islands shared warps 1.61 and 4.0); float model 1.98 and 8.3, 1.88 and 5.8.  20
// where the cap costs a single run more than 5% for some size: float runs in islands of 64, and of 16
// with several generations to a migration, and tournaments of 5 in islands of 64 with several; wider
// records, which were not slower beside one another.
template <int N, int SW, int TS, int MODEL, bool IV>
constexpr int resident_warps()
{
    if (SW != 2) return 20;
    if (N == 64) return MODEL == 0 && (!IV || TS == 0) ? 28 : 20;
    if (N == 32) return MODEL == 1 && IV ? 28 : 32;
    if (N == 16) return !IV ? 32 : MODEL == 0 ? 28 : 20;
    return 28;
}

// N, SW, TS, MODEL: island size, surface words, tournament size (0: read from the run) and genome
// model, as in step_block; IV: migrations more than a generation apart.
template <int N, int SW, int TS, int MODEL, bool IV, int WARPS = resident_warps<N, SW, TS, MODEL, IV>()>
__global__ void __launch_bounds__(32, WARPS) resident_kernel(const ResidentArgs a)
{
    constexpr int A = Shape<N>::A, P = Shape<N>::P, SEG = Shape<N>::SEG;
    constexpr int LW = Record<SW>::LW, Q = Record<SW>::Q, C = Record<SW>::C;
    extern __shared__ uint4 s_all[];
    const RunParams &p = a.r;
    const uint32_t lane = threadIdx.x;  // one warp per block
    const uint32_t seg_lane = lane % SEG;
    const uint32_t per_warp = a.units * P;
    const uint32_t first = blockIdx.x * per_warp;
    const uint32_t count = min(per_warp, p.n_islands - first);
    const uint32_t pairs = count * 4u;  // (island, direction) pairs of the warp
    const uint32_t end = p.g0 + p.n_gens;

    uint4 *recs = s_all;
    uint32_t *s_nb = reinterpret_cast<uint32_t *>(recs + per_warp * (N * Q));
    uint8_t *s_slot = reinterpret_cast<uint8_t *>(s_nb + per_warp * 4u);  // [2][per_warp * 4]
    uint8_t *s_e = s_slot + per_warp * 8u;

    for (uint32_t i = lane; i < count * (N * Q); i += 32u)
        cp_async16(&recs[i], &p.src[static_cast<size_t>(first) * (N * Q) + i]);
    cp_async_commit();
    for (uint32_t idx = lane; idx < pairs; idx += 32u) {
        const uint32_t isl = first + (idx >> 2), d = idx & 3u;
        const uint32_t y = div_cols(isl, p.cols_m, p.cols_l), x = isl - y * p.cols;
        const uint32_t yn = d == 0u ? (y == 0u ? p.rows - 1u : y - 1u)
                          : d == 1u ? (y + 1u == p.rows ? 0u : y + 1u) : y;
        const uint32_t xn = d == 2u ? (x + 1u == p.cols ? 0u : x + 1u)
                          : d == 3u ? (x == 0u ? p.cols - 1u : x - 1u) : x;
        const uint32_t nb = yn * p.cols + xn;
        s_nb[idx] = in_bounds(nb < p.n_islands, p.status) ? nb : 0u;
    }
    __syncwarp();

    // The draws of migration generation gm, two per (island, direction) pair and one per lane at
    // a time: items [0, pairs) draw the member that the neighbour takes from this island (word 3,
    // bits 8..15, of the neighbour's own draw for the slot facing it), items [pairs, 2 pairs) the
    // landing slot of the arrival (the partial Fisher-Yates draw over [0, N) in direction order,
    // among the island's four lanes).
    auto prepare = [&](uint32_t gm, uint32_t par) {
        for (uint32_t base = 0; base < 2u * pairs; base += 32u) {
            const uint32_t item = base + lane;
            const bool own = item >= pairs;
            const uint32_t idx = own ? item - pairs : item;
            const bool ok = item < 2u * pairs;
            const uint32_t d = idx & 3u;
            const uint32_t isl = own ? first + (idx >> 2) : s_nb[idx];
            const uint32_t u = philox_rk(gm, isl, (own ? d : d ^ 1u) | (kBirth << 16), p.run_id, a.rk).w;
            const uint32_t r = d + (((u >> 16) * static_cast<uint32_t>(N - d)) >> 16);
            uint32_t rr[4];
#pragma unroll
            for (int dd = 0; dd < 4; ++dd) rr[dd] = __shfl_sync(0xffffffffu, r, dd, 4);
            uint32_t v[4], slot = 0;
#pragma unroll
            for (int dd = 0; dd < 4; ++dd) {
                uint32_t vd = dd, vr = rr[dd];
#pragma unroll
                for (int e = 0; e < dd; ++e) {
                    if (rr[e] == static_cast<uint32_t>(dd)) vd = v[e];
                    if (rr[e] == rr[dd]) vr = v[e];
                }
                if (static_cast<uint32_t>(dd) == d) slot = vr;
                v[dd] = vd;
            }
            if (ok) {
                if (own) s_slot[par * (per_warp * 4u) + idx] = static_cast<uint8_t>(slot);
                else s_e[idx] = static_cast<uint8_t>((((u >> 8) & 0xFFu) * N) >> 8);
            }
        }
    };
    // mailbox of island i for direction d, migration parity 0 (parity 1: 4 C chunks further)
    auto box_of = [&](uint32_t i, uint32_t d) { return a.mail + static_cast<size_t>(i) * a.mail_stride + d * C; };
    // this lane's first pair: its own mailbox and the neighbour's that it fills
    uint4 *const box_in = box_of(first + (lane < pairs ? lane >> 2 : 0u), lane & 3u);
    uint4 *const box_out = box_of(lane < pairs ? s_nb[lane] : first, (lane & 3u) ^ 1u);

    uint32_t gm = next_migration(p.g0, end, a.every_k, a.per_neighbor);
    uint32_t par = 0;
    if (gm != ~0u) prepare(gm, par);
    cp_async_wait<0>();
    __syncwarp();
    bool aborted = false;
    for (uint32_t it = 0, len = 0; it < p.n_gens; it += len) {
        const uint32_t g = p.g0 + it;
        uint2 dm = make_uint2(0u, 0u);
        int site = -1;
        if constexpr (SW == 2) dm = const_mask_at(p, it);
        else site = gen_site_at(p, it);
        const SlotDraws<N> sd = slot_draws<N>(p, a.rk, g, seg_lane);
        uint4 w[A];
        if (g == gm) {
            __syncwarp();  // the islands' records, written by their own lanes, are pushed by others
            for (uint32_t idx = lane; idx < pairs; idx += 32u) {
                const uint4 *r = recs + ((idx >> 2) * N + s_e[idx]) * Q;
                uint4 *box = (idx == lane ? box_out : box_of(s_nb[idx], (idx & 3u) ^ 1u)) + par * (4u * C);
                if (first + (idx >> 2) != a.drop_island) {
                    if constexpr (C == 1) {
                        store128(box, r[0]);
                    } else {
                        const uint4 r0 = r[0], r1 = r[1];
                        uint4 r2 = make_uint4(0u, 0u, 0u, 0u);
                        if constexpr (Q == 3) r2 = r[2];
                        store128(box, make_uint4(r0.x, r0.z, r0.w, g));
                        store128(box + 1, make_uint4(r1.x, r1.y, r1.z, g));
                        store128(box + 2, Q == 3 ? make_uint4(r1.w, r2.x, r2.y, g) : make_uint4(r1.w, g, g, g));
                    }
                }
            }
            const uint64_t after = static_cast<uint64_t>(g) + a.every_k;
            const uint32_t gm_next = after < end ? static_cast<uint32_t>(after) : ~0u;
            bool gave_up = false;
            for (uint32_t base = 0; base < pairs; base += 32u) {
                const uint32_t idx = base + lane;
                const bool act = idx < pairs;
                const uint4 *box = (base == 0u ? box_in : box_of(first + (act ? idx >> 2 : 0u), idx & 3u)) +
                                   par * (4u * C);
                uint4 in[C];
                auto read = [&]() {
#pragma unroll
                    for (int c = 0; c < C; ++c) in[c] = load128(box + c);
                };
                auto arrived = [&]() {
                    if constexpr (C == 1) return in[0].y == g;
                    else return in[0].w == g && in[1].w == g && in[2].w == g && (Q == 3 || (in[2].y == g && in[2].z == g));
                };
                // while the pushes and the first reads travel: the next migration's draws and the
                // first islands' birth draws.  An arrival is read right after the pushes, and a
                // second time in between where the warp holds one unit and has nothing else to
                // do (32x32 torus, 1,000 generations: 1,230 us, 1,255 with one early read,
                // 1,292 with one read after the draws); wider records, three chunks each, are
                // read once after the draws (256 sites, 5,893 islands: 651 us, 689 before them).
                if (C == 1 && act) read();
                if (base == 0u && gm_next != ~0u) prepare(gm_next, par ^ 1u);
                uint4 again = make_uint4(0u, 0u, 0u, 0u);
                if (C == 1 && act && a.units == 1u) again = load128(box);
                if (C != 1 && act) read();
                if (base == 0u) island_draws<N>(w, sd, a.rk, first + lane / SEG);
                if (C == 1 && a.units == 1u && !arrived()) in[0] = again;
                if (act && !arrived()) {
                    const unsigned long long t0 = global_ns();
                    for (uint32_t polls = 0;; ++polls) {
                        read();
                        const uint32_t ab = load_relaxed(a.abort_word);
                        if (arrived()) break;
                        if (ab != 0u) {
                            gave_up = true;
                            break;
                        }
                        if (global_ns() - t0 > a.wait_ns && polls >= kMinPolls) {
                            atomicCAS(p.status, 0, GA_ETIMEOUT);
                            atomicExch(a.abort_word, 1u);
                            gave_up = true;
                            break;
                        }
                        if (polls >= 8u) __nanosleep(64);
                    }
                }
                if (__any_sync(0xffffffffu, gave_up)) {
                    aborted = true;
                    break;
                }
                __syncwarp();  // every push has read its record
                if (act) {
                    const uint32_t slot = s_slot[par * (per_warp * 4u) + idx];
                    uint4 *r = recs + ((idx >> 2) * N + slot) * Q;
                    if (in_bounds(slot < static_cast<uint32_t>(N), p.status)) {
                        if constexpr (C == 1) {
                            r[0] = in[0];
                        } else {
                            r[0] = make_uint4(in[0].x, g, in[0].y, in[0].z);
                            r[1] = make_uint4(in[1].x, in[1].y, in[1].z, in[2].x);
                            if constexpr (Q == 3) r[2] = make_uint4(in[2].y, in[2].z, 0u, 0u);
                        }
                    }
                }
            }
            if (aborted) break;
            __syncwarp();
            par ^= 1u;
            gm = gm_next;
        }
        else island_draws<N>(w, sd, a.rk, first + lane / SEG);
        // IV (16-byte records, migrations more than a generation apart): the generations up to the
        // next migration in registers (16,384 agents, one migration in 16: 0.31 us per generation,
        // 0.42 with the records stored and loaded in each)
        len = IV ? (gm != ~0u ? gm : end) - g : 1u;
        uint4 *own = recs + lane * Q;
        for (uint32_t u = 0; u < count; u += P, own += 32u * A * Q) {
            const uint32_t li = u + lane / SEG;
            unsigned mask = 0xffffffffu;
            if constexpr (P > 1) {
                mask = __ballot_sync(0xffffffffu, li < count);
                if (li >= count) continue;  // lanes of a missing last island
            }
            const uint32_t island = first + li;
            if (u != 0u) island_draws<N>(w, sd, a.rk, island);
            uint32_t rec[A][LW];
#pragma unroll
            for (int ag = 0; ag < A; ++ag)
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const uint4 v = own[32u * ag * Q + q];
                    const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (4 * q + k < LW) rec[ag][4 * q + k] = w4[k];
                }
            // wider records take the deposit in shared memory, below
            if constexpr (SW == 2) {
                reproduce<N, SW, TS, MODEL, 0, 1>(rec, w, p, a.rk, island, seg_lane, mask, g, 0, dm);
                if constexpr (IV) {
                    for (uint32_t j = 1; j < len; ++j) {
                        const uint2 dj = const_mask_at(p, it + j);
                        birth_draws<N>(w, p, a.rk, g + j, island, seg_lane);
                        reproduce<N, SW, TS, MODEL, 0, 1>(rec, w, p, a.rk, island, seg_lane, mask, g + j, 0, dj);
                    }
                }
            } else {
                reproduce<N, SW, TS, MODEL, 0, 0>(rec, w, p, a.rk, island, seg_lane, mask, g, -1);
            }
#pragma unroll
            for (int ag = 0; ag < A; ++ag)
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    uint32_t w4[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) w4[k] = 4 * q + k < LW ? rec[ag][4 * q + k] : 0u;
                    own[32u * ag * Q + q] = make_uint4(w4[0], w4[1], w4[2], w4[3]);
                }
            if constexpr (SW > 2) {
                const uint32_t pos = static_cast<uint32_t>(site) * p.bits;
                if (site >= 0 && in_bounds(pos + p.bits <= 32u * SW, p.status)) {
                    const uint32_t m = p.dif_mask << (pos & 31u);
#pragma unroll
                    for (int ag = 0; ag < A; ++ag) {
                        uint32_t *word = reinterpret_cast<uint32_t *>(own + 32u * ag * Q) + 2u + (pos >> 5);
                        *word = (*word & ~m) | ((w[ag].w << (pos & 31u)) & m);
                    }
                }
            }
        }
    }
    __syncwarp();
    if (!aborted)
        for (uint32_t i = lane; i < count * (N * Q); i += 32u)
            p.dst[static_cast<size_t>(first) * (N * Q) + i] = recs[i];
}

using ResidentKernel = void (*)(ResidentArgs);

struct ResidentPick {
    ResidentKernel k = nullptr;
    uint32_t islands_per_unit = 1;
    uint32_t bytes_per_island = 0;  // shared memory
    uint32_t boxes = 0;             // 16-byte chunks of an island's mailboxes, both parities
};

template <int N, int SW>
ResidentPick picked(ResidentKernel k)
{
    // the mailboxes fit in the place of the island's own records
    static_assert(8 * Record<SW>::C <= N * Record<SW>::Q, "mailboxes larger than the island");
    ResidentPick m;
    m.k = k;
    m.islands_per_unit = Shape<N>::P;
    m.bytes_per_island = warp_bytes<N, SW>(1);
    m.boxes = 8u * Record<SW>::C;
    return m;
}

// Tournament size 5 (the paper's) is compiled in; other sizes are read from the run.  dense: 21 to 28
// warps per SM with one unit each (float model, islands of 16, every 4 generations: 110,000 agents
// 1.67 against 1.72 us per generation with the 96-register kernel, 131,072, where that one takes two
// units to a warp, 1.96 against 2.12; every 16 1.84 against 1.90).
template <int N, int SW, int MODEL = 0>
ResidentPick pick_ts(uint32_t tsize, bool intervals, bool dense = false)
{
    if constexpr (SW == 2) {
        if constexpr (N == 16 && MODEL == 1)
            if (intervals && dense && tsize != 5u) return picked<N, SW>(resident_kernel<N, SW, 0, MODEL, true, 28>);
        if (intervals)
            return picked<N, SW>(tsize == 5u ? resident_kernel<N, SW, 5, MODEL, true>
                                             : resident_kernel<N, SW, 0, MODEL, true>);
    }
    return picked<N, SW>(tsize == 5u ? resident_kernel<N, SW, 5, MODEL, false>
                                     : resident_kernel<N, SW, 0, MODEL, false>);
}

// The float-fitness model: 16-byte records, islands of 16 to 64 agents.  32-byte records: not
// for islands of 8, whose mailboxes would not fit in the place of their records.
template <int N>
ResidentPick pick_n(uint32_t surface_words, uint32_t model, uint32_t tsize, bool intervals, bool dense = false)
{
    if (model == GA_MODEL_FITNESS) {
        if constexpr (N >= 16)
            if (surface_words <= 2u) return pick_ts<N, 2, 1>(tsize, intervals, dense);
        return ResidentPick();
    }
    if (surface_words <= 2u) return pick_ts<N, 2>(tsize, intervals);
    if (surface_words <= 6u) {
        if constexpr (N >= 16) return pick_ts<N, 6>(tsize, intervals);
        return ResidentPick();
    }
    return pick_ts<N, 8>(tsize, intervals);
}

ResidentPick pick(const ga_run *run, uint32_t sms)
{
    const uint32_t sw = run->surface_words, model = run->cfg.model, ts = run->cfg.tournament_size;
    const bool iv = run->per_neighbor == 0u || run->every_k > 1u;
    switch (run->cfg.island_size) {
    case 8: return pick_n<8>(sw, model, ts, iv);
    case 16: return pick_n<16>(sw, model, ts, iv, run->n_islands > 40u * sms && run->n_islands <= 56u * sms);
    case 32: return pick_n<32>(sw, model, ts, iv);
    case 64: return pick_n<64>(sw, model, ts, iv);
    default: return ResidentPick();
    }
}

// Before a launch: the curation sites (and deposit masks) of its generations, every mailbox
// empty (all ones) and the abort word clear.
__global__ void resident_init_kernel(uint4 *__restrict__ mail, uint32_t n_islands, uint32_t stride,
                                     uint32_t boxes, uint32_t *__restrict__ abort_word, uint32_t policy,
                                     uint32_t log2_sites, uint32_t sites, uint32_t t0, uint32_t count,
                                     int32_t *__restrict__ out, uint32_t bits, uint2 *__restrict__ masks)
{
    wait_previous_grid();
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x, all = gridDim.x * blockDim.x;
    if (t == 0u) *abort_word = 0u;
    for (uint32_t i = t; i < count; i += all)
        store_curation_site(policy, log2_sites, sites, t0 + i, bits, &out[i], masks ? &masks[i] : nullptr);
    const uint32_t total = n_islands * boxes;
    for (uint32_t i = t; i < total; i += all)
        mail[static_cast<size_t>(i / boxes) * stride + i % boxes] = make_uint4(~0u, ~0u, ~0u, ~0u);
}

}  // namespace

size_t resident_state_bytes(uint32_t n_islands, uint32_t record_bytes)
{
    if (record_bytes != 16u || n_islands > kResidentMaxIslands) return 0;
    // 256 bytes that nothing uses (callers may have sized workspaces by them), then two parities of four
    // 16-byte mailboxes per island
    return 256u + static_cast<size_t>(n_islands) * 4u * 2u * 16u;
}

bool resident_eligible(const ga_run *run)
{
    if (!run->resident_state || run->cfg.mode != GA_SYNC || !run->counters_uniform) return false;
    const uint32_t N = run->cfg.island_size;
    if (N < 8u || N > 64u) return false;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    const bool narrow = run->cfg.tournament_size == 5u && run->cfg.model == GA_MODEL_TRAIT;
    const uint32_t per_sm = N == 32u ? 40u : N == 64u ? (narrow ? 36u : 32u) : kResidentMaxIslands;
    return run->n_islands <= static_cast<uint64_t>(sms) * per_sm;
}

// A streamed launch covers a migration interval of k generations, so resident launches save
// fewer launches as k grows, while the streamed kernels keep three times the warps on an SM.  The
// most agents, in thousands, up to which they are faster; rows: islands of 8, 16, 32, 64; columns:
// 16-byte trait records, the float model, 32-byte, 48-byte records.  Streamed / resident, us per
// generation (the slower of tournaments of 5 and 3) on either side of some lines:
//   k = 1   16-byte: 16: 350 4.1 / 3.2, 400 4.1 / 4.5; 32: 1,000 7.1 / 6.5, 1,100 7.1 / 7.3; 64: 1,100 8.5 / 8.1
//           float: 32: 650 8.9 / 8.5, 750 9.0 / 10.1;  32-byte: 16: 700 8.94 / 8.93, 1,000 12.0 / 31
//           48-byte: 16: 650 10.2 / 8.8, 700 10.7 / 28 (too few warps fit); 64: 700 10.4 / 7.5
//   k = 2   48-byte: 16: 600 5.85 / 5.77, 700 6.5 / 22; 32: 600 5.45 / 4.37;  32-byte: 64: 450 3.9 / 3.9;
//           float: 64: 900 14.1 / 11.3, 1,100 14.1 / 16.9
//   k = 4   32-byte: 16: 65 1.00, 98 0.91 of the streamed rate; 32: 98 1.02, 131 0.92; 64: 114 1.05, 131 0.95
//   k = 6   48-byte: 32: 150 1.02, 175 0.93; 64: 114 0.97 to 1.06, 131 0.89 to 0.98;  k = 8: 32: 65 0.99, 81 0.96
struct ResidentLines {
    uint32_t every;  // up to this migration interval
    uint16_t most[4][4];
};
constexpr ResidentLines kResidentLines[] = {
    {1u, {{150, 0, 0, 150}, {380, 375, 700, 650}, {1000, 650, 1100, 700}, {1400, 1000, 1000, 700}}},
    {2u, {{99, 0, 0, 99}, {300, 225, 300, 600}, {500, 500, 550, 600}, {1400, 950, 450, 600}}},
    {4u, {{66, 0, 0, 66}, {200, 200, 66, 150}, {400, 400, 99, 200}, {600, 600, 115, 150}}},
    {6u, {{66, 0, 0, 66}, {200, 200, 0, 50}, {400, 400, 50, 150}, {600, 600, 66, 115}}},
    {8u, {{66, 0, 0, 0}, {200, 200, 0, 0}, {400, 400, 0, 66}, {600, 600, 0, 33}}},
    {~0u, {{0, 0, 0, 0}, {200, 200, 0, 0}, {400, 400, 0, 0}, {400, 400, 0, 0}}},
};

bool resident_pays(const ga_run *run)
{
    const uint32_t N = run->cfg.island_size, k = run->per_neighbor ? run->every_k : ~0u;
    if (N < 8u || N > 64u) return false;
    const ResidentLines *row = kResidentLines;
    while (k > row->every) ++row;
    const uint32_t kind = run->cfg.model == GA_MODEL_FITNESS ? 1u : run->record_bytes == 16u ? 0u : run->record_bytes / 16u;
    const uint32_t size = N == 8u ? 0u : N == 16u ? 1u : N == 32u ? 2u : 3u;
    return run->n_agents <= row->most[size][kind] * 1000u;
}

bool resident_plan(const ga_run *run, ResidentPlan &plan)
{
    if (run->cfg.mode != GA_SYNC || !run->counters_uniform) return false;
    int dev = 0, sms = 0, smem = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    plan.sms = static_cast<uint32_t>(sms);
    const ResidentPick m = pick(run, plan.sms);
    if (!m.k) return false;
    if (cudaFuncSetAttribute(reinterpret_cast<const void *>(m.k),
                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (static_cast<uint64_t>(run->n_islands) * m.bytes_per_island > static_cast<uint64_t>(sms) * smem) return false;
    const uint32_t n_units = (run->n_islands + m.islands_per_unit - 1u) / m.islands_per_unit;
    for (uint32_t units = units_per_warp(run, n_units, plan.sms);; ++units) {
        const size_t bytes = static_cast<size_t>(units) * m.islands_per_unit * m.bytes_per_island;
        if (bytes > static_cast<size_t>(smem)) return false;
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, m.k, 32, bytes) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        const uint32_t blocks = (n_units + units - 1u) / units;
        if (blocks <= plan.sms * static_cast<uint32_t>(per_sm)) {
            plan.units = units;
            plan.blocks = blocks;
            plan.shared_bytes = bytes;
            return true;
        }
    }
}

cudaError_t launch_resident(ga_run *run, const ResidentPlan &plan, const void *src, void *dst, uint32_t g0,
                            uint32_t n_gens, cudaStream_t stream)
{
    const ResidentPick m = pick(run, plan.sms);
    if (!m.k) return cudaErrorInvalidValue;
    ResidentArgs a;
    a.r = run_params(run, src, dst, g0, n_gens, false);
    a.rk = round_keys(Key{static_cast<uint32_t>(run->cfg.seed), static_cast<uint32_t>(run->cfg.seed >> 32)});
    if (run->resident_state) {
        a.mail = reinterpret_cast<uint4 *>(static_cast<uint8_t *>(run->resident_state) + 256);
        a.mail_stride = m.boxes;
    } else {
        a.mail = static_cast<uint4 *>(dst);
        a.mail_stride = run->cfg.island_size * run->record_bytes / 16u;
    }
    a.abort_word = run->d_abort;
    a.wait_ns = static_cast<unsigned long long>(run->resident_wait_us) * 1000ull;
    a.every_k = run->every_k;
    a.per_neighbor = run->per_neighbor;
    a.drop_island = run->drop_island;
    a.units = plan.units;
    const uint32_t entries = run->n_islands * m.boxes > n_gens ? run->n_islands * m.boxes : n_gens;
    const uint32_t blocks = (entries + 255u) / 256u;
    cudaError_t e = launch_dependent(
        resident_init_kernel, blocks < 1216u ? blocks : 1216u, 256, stream, a.mail, run->n_islands,
        a.mail_stride, m.boxes, a.abort_word, run->cfg.curation, run->log2_sites, run->cfg.surface_sites, g0,
        n_gens, run->d_sites, run->cfg.differentia_bits, run->surface_words <= 2u ? run->d_masks : nullptr);
    if (e != cudaSuccess) return e;
    run->launches += 1;
    void *args[] = {&a};
    e = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(m.k), dim3(plan.blocks), dim3(32),
                                    args, plan.shared_bytes, stream);
    if (e == cudaSuccess) run->launches += 1;
    else cudaGetLastError();  // returned here, not left pending for a later call
    return e;
}

}  // namespace ga

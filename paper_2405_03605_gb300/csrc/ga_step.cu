// ga_step.cu -- founder initialisation, the single-run island-step kernel (the block body
// lives in ga_island.cuh) and the curation-site kernels.
#include "ga_device.cuh"
#include "ga_internal.h"
#include "ga_island.cuh"

namespace ga {

constexpr int kUnitsThreads = 256;

// Warps per block of the one-unit kernel.  Four: the warps of a block wait at its one barrier for
// the warp that does the bookkeeping, and smaller blocks leave more of the others at work (4.2M
// agents, a migration per generation, us a generation with 4 and 8 warps: 48-byte records,
// islands of 8 69.6 and 74.5, of 32 63.9 and 67.4, of 128 66.7 and 71.5; 32-byte records, islands
// of 32 46.6 and 49.3; 16-byte records, islands of 128 27.4 and 30.9).  Two is slower for most
// (islands of 32, 4 generations to a launch: 26.6 against 23.7).  Eight for 16-byte records in
// islands of 4 and 8, whose bookkeeping takes every lane of four warps or two (65,536 to 1M agents
// 1 to 3% faster than with four).
template <int N, int SW>
constexpr int step_warps() { return N <= 8 && SW <= 2 ? 8 : 4; }

// Blocks per SM asked of the compiler: 12 (40 registers) for 48-byte records with equal counters
// in islands of 16 and 32, which take 44 to 46 unasked: 61.7 against 63.9 us a generation for 4.2M
// agents in islands of 32, 15.5 against 15.9 for 1M.  7 (64 to 68 registers) for 16-byte records with equal
// counters in islands of 128, which take 80 unasked: 500,000 agents 4.4 against 5.2 us with a migration
// every generation, 2.14 against 2.18 every 16.
template <int N, int SW, int CF>
constexpr int step_min_blocks()
{
    return CF != 0 ? 1 : SW == 8 && (N == 16 || N == 32) ? 12 : SW == 2 && N == 128 ? 7 : 1;
}

// Single run: per-run values and round keys are kernel parameters (constant bank).
struct StepArgs {
    RunParams r;
    RoundKeys rk;
};

template <int N, int SW, int TS, int MODEL = 0, int CF = 1>
__global__ void __launch_bounds__((32 * step_warps<N, SW>()), (step_min_blocks<N, SW, CF>()))
    island_step_kernel(const StepArgs a)
{
    wait_previous_grid();
    step_block<N, SW, TS, step_warps<N, SW>(), MODEL, CF>(a.r, a.rk, blockIdx.x);
}

// Multi-unit kernel (step_units in ga_island.cuh) for 16-byte records whose counters all
// equal the generation, islands of 16, 32 or 64 agents, any tournament size, both genome
// models; TS = 0 reads the tournament size from the run; ONE: launches of one generation.
// Resident blocks per SM asked of the compiler: 8 (32 registers) below 64 agents; the two
// agents per lane of 64-agent islands need 40 registers (6 blocks).  The float model's queue needs
// 64: 4 (50 generations of 16.8M agents: 7,433 us; 7,638 with 5 blocks, 7,865 with 3; 6,900 since
// launches of one generation are compiled apart).
template <int N, bool QUEUE>
constexpr int units_min_blocks() { return QUEUE ? 4 : N >= 64 ? 6 : 8; }

template <int N, int TS, int MODEL, bool ONE, bool QUEUE = MODEL == 1>
__global__ void __launch_bounds__(kUnitsThreads, (units_min_blocks<N, QUEUE>())) island_units_kernel(const StepArgs a)
{
    wait_previous_grid();
    step_units<N, TS, units_per_block<N>(), MODEL, true, ONE, QUEUE>(a.r, a.rk, blockIdx.x);
}

// Every record becomes the founder: trait 0, counter 0, surface word w = word 0 of
// Philox((0, 0, w | FOUNDER << 16, run_id)); surface bits past S*b are zero.
__global__ void founder_kernel(uint4 *__restrict__ dst, uint32_t n_agents, uint32_t q_per_rec,
                               uint32_t surface_words, uint32_t top_bits, Key key,
                               uint32_t run_id)
{
    __shared__ uint32_t words[12];
    wait_previous_grid();
    if (threadIdx.x < 12) {
        uint32_t val = 0u;
        const uint32_t k = threadIdx.x;
        if (k >= 2 && k - 2 < surface_words) {
            val = philox(0u, 0u, (k - 2) | (kFounder << 16), run_id, key).x;
            if (k - 2 == surface_words - 1 && top_bits) val &= (1u << top_bits) - 1u;
        }
        words[k] = val;
    }
    __syncthreads();
    const size_t total = static_cast<size_t>(n_agents) * q_per_rec;
    for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < total;
         i += static_cast<size_t>(gridDim.x) * blockDim.x) {
        const uint32_t q = static_cast<uint32_t>(i % q_per_rec);
        dst[i] = make_uint4(words[4 * q], words[4 * q + 1], words[4 * q + 2], words[4 * q + 3]);
    }
}

__global__ void counter_check_kernel(const uint32_t *__restrict__ pop, uint32_t record_words,
                                     uint32_t n_agents, uint32_t generation, int *__restrict__ flag)
{
    for (size_t a = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; a < n_agents;
         a += static_cast<size_t>(gridDim.x) * blockDim.x)
        if (pop[a * record_words + 1u] != generation) *flag = 1;  // every writer stores 1
}

__global__ void curation_sites_kernel(uint32_t policy, uint32_t log2_sites, uint32_t sites,
                                      uint32_t t0, uint32_t count, int32_t *__restrict__ out,
                                      uint32_t bits, uint2 *__restrict__ masks)
{
    wait_previous_grid();
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += gridDim.x * blockDim.x)
        store_curation_site(policy, log2_sites, sites, t0 + i, bits, &out[i], masks ? &masks[i] : nullptr);
}

namespace {

using StepKernel = void (*)(StepArgs);

// The template's surface-word count fills the record: 16-byte records carry 2 surface words,
// 32-byte records 6 and 48-byte records 8 (words past the run's own S*b bits are zero).
// Tournament size 5 (the paper's, Sec. 3) has its own instantiation; other sizes use the
// kernel that reads the size from its arguments.
template <int N, int SW>
StepKernel pick_ts(uint32_t tsize)
{
    return tsize == 5 ? island_step_kernel<N, SW, 5> : island_step_kernel<N, SW, 0>;
}

template <int N>
StepKernel pick_sw(uint32_t surface_words, uint32_t tsize)
{
    if (surface_words <= 2) return pick_ts<N, 2>(tsize);
    if (surface_words <= 6) return pick_ts<N, 6>(tsize);
    if (surface_words <= 8) return pick_ts<N, 8>(tsize);
    return nullptr;
}

// The float-fitness model (16-byte records: fitness, counter, 64-bit surface -- the paper's
// 128-bit genome of Sec. 3) has kernels for islands of 16, 32 and 64.
template <int N>
StepKernel pick_fitness(uint32_t surface_words, uint32_t tsize)
{
    if (surface_words > 2) return nullptr;
    return tsize == 5 ? island_step_kernel<N, 2, 5, 1> : island_step_kernel<N, 2, 0, 1>;
}

// Generations to a launch from which on the float model's kernel without the queue is faster: the queue
// shortens the first generation alone, and the registers it takes halve the warps on an SM in the
// later ones.  With the queue and without, 2.5M agents, us per generation:
//   tournaments of 5   16 agents: 6 23.07 / 23.14, 8 22.75 / 22.42, none 22.02 / 20.74;  32: 8 24.62 / 24.78,
//                      16 24.57 / 24.09, none 24.47 / 23.43;  64: 16 30.36 / 30.65, none 30.22 / 30.21
//   of 3               16: 4 24.29 / 24.67, 6 23.83 / 23.68, none 22.74 / 21.44;  32: 2 27.69 / 28.45,
//                      4 26.58 / 25.88, none 25.46 / 23.43;  64: 16 31.88 / 31.24 (5M agents 54.8 / 57.5), none
//                      31.78 / 30.72 (54.5 / 55.4; 500,000 10.6 / 10.1)
template <int N, int TS>
constexpr uint32_t plain_from()
{
    if (TS == 5) return N == 16 ? 8u : N == 32 ? 16u : kMaxGensPerLaunch + 1u;
    return N == 16 ? 6u : N == 32 ? 4u : 32u;
}

// Launches of one generation have a kernel of their own (see step_units).
template <int N, int TS, int MODEL>
StepKernel units_of(uint32_t n_gens)
{
    if (n_gens == 1u) return island_units_kernel<N, TS, MODEL, true>;
    if constexpr (MODEL == 1 && plain_from<N, TS>() <= kMaxGensPerLaunch)
        if (n_gens >= plain_from<N, TS>()) return island_units_kernel<N, TS, MODEL, false, false>;
    return island_units_kernel<N, TS, MODEL, false>;
}

template <int N>
StepKernel pick_units(uint32_t tsize, bool fitness, uint32_t n_gens)
{
    if (fitness) return tsize == 5 ? units_of<N, 5, 1>(n_gens) : units_of<N, 0, 1>(n_gens);
    return tsize == 5 ? units_of<N, 5, 0>(n_gens) : units_of<N, 0, 0>(n_gens);
}

// Kernels without the closed-form curation path, for launches whose counters all equal the
// generation: 16-byte trait records of the island sizes that island_units_kernel does not take, and
// 32- and 48-byte trait records of islands of 16 to 128.
template <int N, int SW>
StepKernel uniform_ts(uint32_t tsize)
{
    return tsize == 5u ? island_step_kernel<N, SW, 5, 0, 0> : island_step_kernel<N, SW, 0, 0, 0>;
}

template <int N>
StepKernel uniform_wide(uint32_t surface_words, uint32_t tsize)
{
    return surface_words <= 6u ? uniform_ts<N, 6>(tsize) : uniform_ts<N, 8>(tsize);
}

StepKernel pick_uniform(uint32_t island_size, uint32_t surface_words, uint32_t tsize, uint32_t model)
{
    if (model != GA_MODEL_TRAIT) return nullptr;
    if (surface_words > 2u) {
        switch (island_size) {
        case 16: return uniform_wide<16>(surface_words, tsize);
        case 32: return uniform_wide<32>(surface_words, tsize);
        case 64: return uniform_wide<64>(surface_words, tsize);
        case 128: return uniform_wide<128>(surface_words, tsize);
        default: return nullptr;
        }
    }
    switch (island_size) {
    case 4: return uniform_ts<4, 2>(tsize);
    case 8: return uniform_ts<8, 2>(tsize);
    case 128: return uniform_ts<128, 2>(tsize);
    default: return nullptr;
    }
}

StepKernel pick_kernel(uint32_t island_size, uint32_t surface_words, uint32_t tsize,
                       uint32_t model)
{
    if (model == GA_MODEL_FITNESS) {
        switch (island_size) {
        case 16: return pick_fitness<16>(surface_words, tsize);
        case 32: return pick_fitness<32>(surface_words, tsize);
        case 64: return pick_fitness<64>(surface_words, tsize);
        default: return nullptr;
        }
    }
    if (model != GA_MODEL_TRAIT) return nullptr;
    switch (island_size) {
    case 4: return pick_sw<4>(surface_words, tsize);
    case 8: return pick_sw<8>(surface_words, tsize);
    case 16: return pick_sw<16>(surface_words, tsize);
    case 32: return pick_sw<32>(surface_words, tsize);
    case 64: return pick_sw<64>(surface_words, tsize);
    case 128: return pick_sw<128>(surface_words, tsize);
    default: return nullptr;
    }
}

// SM count of the current device, read once (a function-local static: initialised once even
// when handles are used from several threads).
uint32_t sm_count()
{
    static const uint32_t sms = [] {
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return n > 0 ? static_cast<uint32_t>(n) : 1u;
    }();
    return sms;
}

}  // namespace

RunParams run_params(const ga_run *run, const void *src, void *dst, uint32_t g0, uint32_t n_gens,
                     bool migrate)
{
    RunParams r;
    r.src = static_cast<const uint4 *>(src);
    r.dst = static_cast<uint4 *>(dst);
    r.rows = run->cfg.rows;
    r.cols = run->cfg.cols;
    r.n_islands = run->n_islands;
    division_magic(run->cfg.cols, r.cols_m, r.cols_l);
    r.tsize = run->cfg.tournament_size;
    r.theta_ben = run->theta_ben;
    r.theta_del = run->theta_del;
    r.policy = run->cfg.curation;
    r.log2_sites = run->log2_sites;
    r.sites = run->cfg.surface_sites;
    r.bits = run->cfg.differentia_bits;
    r.run_id = run->cfg.run_id;
    r.g0 = g0;
    r.n_gens = n_gens;
    r.migrate = migrate ? 1u : 0u;
    r.gen_sites = run->d_sites + (g0 - run->sites_base);
    r.effect_scale = static_cast<float>(run->cfg.effect_scale);
    r.gen_sites_left = kSiteTableCap - static_cast<uint32_t>(g0 - run->sites_base);
    r.status = run->d_status;
    r.gen_masks = run->d_masks + (g0 - run->sites_base);
    const uint32_t b = run->cfg.differentia_bits;
    r.dif_mask = (1u << b) - 1u;
    r.dif_rep = b == 1u ? 0xFFFFFFFFu : b == 2u ? 0x55555555u : b == 4u ? 0x11111111u : 0x01010101u;
    return r;
}

bool step_supported(uint32_t island_size, uint32_t surface_words, uint32_t model)
{
    return pick_kernel(island_size, surface_words, 1, model) != nullptr;
}

cudaError_t launch_founder(ga_run *run, void *dst)
{
    const uint32_t q = run->record_bytes / 16;
    const uint32_t top = (run->cfg.surface_sites * run->cfg.differentia_bits) % 32u;
    const Key key{static_cast<uint32_t>(run->cfg.seed), static_cast<uint32_t>(run->cfg.seed >> 32)};
    const size_t total = static_cast<size_t>(run->n_agents) * q;
    size_t blocks = (total + 255) / 256;
    const size_t cap = static_cast<size_t>(sm_count()) * 8;
    if (blocks > cap) blocks = cap;
    if (blocks == 0) blocks = 1;
    run->launches += 1;
    return launch_dependent(founder_kernel, static_cast<unsigned>(blocks), 256, run->stream,
                            static_cast<uint4 *>(dst), run->n_agents, q, run->surface_words, top, key,
                            run->cfg.run_id);
}

cudaError_t launch_counter_check(ga_run *run, uint32_t generation, int *d_flag)
{
    size_t blocks = (static_cast<size_t>(run->n_agents) + 255) / 256;
    const size_t cap = static_cast<size_t>(sm_count()) * 8;
    if (blocks > cap) blocks = cap;
    if (blocks == 0) blocks = 1;
    counter_check_kernel<<<static_cast<unsigned>(blocks), 256, 0, run->stream>>>(
        static_cast<const uint32_t *>(static_cast<const void *>(run->pop[run->cur])),
        run->record_bytes / 4u, run->n_agents, generation, d_flag);
    run->launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_island_step(ga_run *run, const void *src, void *dst, uint32_t g0,
                               uint32_t n_gens, bool migrate, cudaStream_t stream)
{
    const bool uniform = run->cfg.mode == GA_SYNC && run->counters_uniform;
    if (run->cfg.mode == GA_SYNC && run->counters_uniform && run->surface_words <= 2) {
        const uint32_t N = run->cfg.island_size, ts = run->cfg.tournament_size;
        const bool fit = run->cfg.model == GA_MODEL_FITNESS;
        StepKernel ku = nullptr;
        uint32_t islands_per_block = 0;
        switch (N) {
        case 16:
            ku = pick_units<16>(ts, fit, n_gens);
            islands_per_block = units_per_block<16>() * 16;
            break;
        case 32:
            ku = pick_units<32>(ts, fit, n_gens);
            islands_per_block = units_per_block<32>() * 8;
            break;
        case 64:
            ku = pick_units<64>(ts, fit, n_gens);
            islands_per_block = units_per_block<64>() * 8;
            break;
        default: break;
        }
        if (ku) {
            StepArgs a;
            a.r = run_params(run, src, dst, g0, n_gens, migrate);
            a.rk = round_keys(Key{static_cast<uint32_t>(run->cfg.seed),
                                  static_cast<uint32_t>(run->cfg.seed >> 32)});
            const uint32_t blocks = (run->n_islands + islands_per_block - 1) / islands_per_block;
            run->launches += 1;
            return launch_dependent(ku, blocks, kUnitsThreads, stream, a);
        }
    }
    StepKernel k =
        uniform ? pick_uniform(run->cfg.island_size, run->surface_words, run->cfg.tournament_size, run->cfg.model)
                : nullptr;
    if (!k)
        k = pick_kernel(run->cfg.island_size, run->surface_words, run->cfg.tournament_size,
                        run->cfg.model);
    if (!k) return cudaErrorInvalidValue;
    StepArgs a;
    a.r = run_params(run, src, dst, g0, n_gens, migrate);
    a.rk = round_keys(Key{static_cast<uint32_t>(run->cfg.seed),
                          static_cast<uint32_t>(run->cfg.seed >> 32)});
    const uint32_t N = run->cfg.island_size;
    const uint32_t warps = N <= 8u && run->surface_words <= 2u ? step_warps<8, 2>() : step_warps<32, 2>();
    const uint32_t islands_per_block = warps * (N >= 32 ? 1u : 32u / N);
    const uint32_t blocks = (run->n_islands + islands_per_block - 1) / islands_per_block;
    run->launches += 1;
    return launch_dependent(k, blocks, 32u * warps, stream, a);
}

cudaError_t launch_site_table(ga_run *run, uint32_t g0, uint32_t count, cudaStream_t stream)
{
    const bool masks = run->surface_words <= 2u;
    const cudaError_t e = launch_curation_sites(
        run->cfg.curation, run->cfg.surface_sites, g0, count, run->d_sites, stream,
        run->cfg.differentia_bits, masks ? run->d_masks : nullptr);
    run->launches += 1;
    return e;
}

cudaError_t launch_curation_sites(uint32_t policy, uint32_t sites, uint32_t t0, uint32_t count,
                                  int32_t *d_sites, cudaStream_t stream, uint32_t bits,
                                  uint2 *d_masks)
{
    if (count == 0) return cudaSuccess;
    uint32_t s = 0;
    while ((1u << s) < sites) ++s;
    uint32_t blocks = (count + 255u) / 256u;
    if (blocks > 8192u) blocks = 8192u;
    return launch_dependent(curation_sites_kernel, blocks, 256, stream, policy, s, sites, t0, count, d_sites,
                            bits, d_masks);
}

}  // namespace ga

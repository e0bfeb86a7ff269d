// Host side of the C ABI: argument checks, per-device context, launch configuration.
#include "nuna_internal.h"
#include "nuna_debug.h"
#include "nuna_kernels.cuh"

#include <cuda.h>

#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <tuple>
#include <type_traits>
#include <utility>
#include <vector>

namespace nuna {

std::atomic<unsigned long long> g_launches{0};
static std::mutex g_ctx_mutex;
static std::atomic<Context*> g_ctx[kMaxDevices];              // written under g_ctx_mutex

static int static_status_read_and_clear(const Context* c, unsigned* out);     // the allocation-free entry point's status word (end of file)
constexpr unsigned kMinFlagTileVec = 16;                    // smallest two-shot tile (vectors): 256 bytes of shard per flag
constexpr size_t kTaggedMaxShard = (size_t)8 << 20;         // largest message, in bytes per rank, that the tagged two-shot takes
constexpr unsigned kStaticTileVec = 128;                    // tile of the allocation-free entry point: 2 KiB of shard per flag

static int env_int(const char* name, int fallback)
{
    const char* s = getenv(name);
    return (s && *s) ? atoi(s) : fallback;
}

constexpr size_t align_up(size_t n, size_t to) { return (n + to - 1) / to * to; }

// Sets device memory that a kernel on any stream may use next, to zero or to what `host` holds: cudaMemset, and cudaMemcpy from
// pageable memory, return before they are done, and only the legacy stream and those that wait for it come after them.  On a
// stream of the context's own it waits for nobody else's work.
static bool set_now(const Context* c, void* p, const void* host, size_t bytes)
{
    const cudaError_t e = host ? cudaMemcpyAsync(p, host, bytes, cudaMemcpyHostToDevice, c->setup) : cudaMemsetAsync(p, 0, bytes, c->setup);
    return cudaStreamSynchronize(c->setup) == cudaSuccess && e == cudaSuccess;
}

int init_barrier_words(Context* c)
{
    return set_now(c, c->bw, nullptr, sizeof(BarrierWords)) ? NUNA_OK : NUNA_ERR_CUDA;
}

// After a latched timeout the barrier's arrival counter is in an undefined state: zero it and clear the
// status, but keep both epochs moving forward -- the ready flags of earlier launches must never match a
// later launch's epoch.  The device is idle (the caller synchronised).
static int rewind_barrier_words(const Context* c, BarrierWords* dev, const BarrierWords& seen)
{
    BarrierWords h = {};
    h.epoch = seen.epoch + 1u;
    h.ticket = ((seen.ticket >> 32) + 1ull) << 32;
    return set_now(c, dev, &h, sizeof h) ? NUNA_OK : NUNA_ERR_CUDA;
}

// Returns the current device's context, creating it on first use (allocates: not capturable).
int get_context(Context** out)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return NUNA_ERR_CUDA;
    if ((*out = g_ctx[dev].load(std::memory_order_acquire)) != nullptr) return NUNA_OK;
    std::lock_guard<std::mutex> lock(g_ctx_mutex);
    if (!g_ctx[dev].load(std::memory_order_relaxed)) {
        Context* c = new Context();
        c->device = dev;
        cudaDeviceProp prop;
        if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) { delete c; return NUNA_ERR_CUDA; }
        c->num_sms = prop.multiProcessorCount;
        c->l2_bytes = (size_t)prop.l2CacheSize;
        if (cudaStreamCreateWithFlags(&c->setup, cudaStreamNonBlocking) != cudaSuccess) { delete c; return NUNA_ERR_CUDA; }
        if (cudaMalloc(&c->bw, sizeof(BarrierWords)) != cudaSuccess || init_barrier_words(c) != NUNA_OK) {
            if (c->bw) cudaFree(c->bw);
            cudaStreamDestroy(c->setup);
            delete c;
            return NUNA_ERR_CUDA;
        }
        c->opt.timeout_ns = (unsigned long long)env_int("NUNA_TIMEOUT_MS", 1000) * 1000000ull;
        c->opt.blocks = env_int("NUNA_BLOCKS", 0);
        c->opt.unroll = env_int("NUNA_UNROLL", 0);
        c->opt.auto_min_bytes = (size_t)env_int("NUNA_AUTO_MIN_BYTES", 0);
        c->opt.coloc = env_int("NUNA_COLOC", 0);
        c->opt.domains = env_int("NUNA_DOMAINS", 0);
        c->opt.stage_vecs = env_int("NUNA_STAGE_VECS", 0);
        c->opt.twoshot_vecs = env_int("NUNA_TWOSHOT_VECS", 0);
        c->opt.keep_shard = env_int("NUNA_KEEP_SHARD", 0);
        c->opt.ag_bulk_vecs = env_int("NUNA_AG_BULK_VECS", 0);
        c->opt.regs_vecs = env_int("NUNA_REGS_VECS", 0);
        c->opt.prefetch = env_int("NUNA_PREFETCH", 0);
        g_ctx[dev].store(c, std::memory_order_release);
    }
    *out = g_ctx[dev].load(std::memory_order_relaxed);
    return NUNA_OK;
}

// Grows the two-shot scratch: shard intermediate, one ready flag per smallest tile of it, and behind them, where larger ones are
// needed, the slots of the tagged form.  The caller holds c->mutex.  An outgrown allocation is never freed before nuna_shutdown: a
// CUDA graph captured earlier (a chain, or a user's capture of a two-shot call) still carries its address as a kernel argument.
// The slots take twice their shard's bytes, so they double, whatever the shard grows by: what has been outgrown of them is never
// more than what is in use, and most growths leave them where they are.
int ensure_scratch(Context* c, size_t bytes)
{
    if (bytes <= c->scratch_bytes && c->scratch) return NUNA_OK;
    const size_t want = (std::max<size_t>(bytes, 4096) + 4095) & ~(size_t)4095;
    const size_t nflags = want / (kMinFlagTileVec * 16) + 1;         // one ready flag per smallest tile
    const size_t slots_at = align_up(want + nflags * sizeof(unsigned), 256);
    size_t slots_shard = 64 << 10;
    while (slots_shard < std::min(want, kTaggedMaxShard)) slots_shard *= 2;
    const bool more_slots = slots_shard > c->slots_shard;
    const size_t total = slots_at + (more_slots ? tagged_bytes(slots_shard) : 0);
    void* p = nullptr;
    if (cudaMalloc(&p, total) != cudaSuccess) return NUNA_ERR_CUDA;
    // flags and tags start at zero; epochs start at one, so a fresh one never reads as "ready"
    if (!set_now(c, static_cast<char*>(p) + want, nullptr, total - want)) {
        cudaFree(p);
        return NUNA_ERR_CUDA;
    }
    if (c->scratch) c->retired_scratch.push_back(c->scratch);
    c->scratch = p;
    c->flags = reinterpret_cast<unsigned*>(static_cast<char*>(p) + want);
    c->scratch_bytes = want;
    if (more_slots) {
        c->slots = static_cast<char*>(p) + slots_at;
        c->slots_shard = slots_shard;
    }
    return NUNA_OK;
}

// ---- argument validation -------------------------------------------------------------------

size_t elem_size(int dtype) { return dtype == NUNA_F32 ? 4 : 2; }
static size_t elems_per_vec(int dtype) { return 16 / elem_size(dtype); }

// Whether a destination range overlaps a source range or another destination range.  One pass over the ranges in the
// order of their addresses; buffers usually come nearly in that order, so sorting them costs little (16 ranks: 376 pairs
// to compare otherwise, 0.2 us of the 2 us that a small call takes).
static bool aliased(const void* const* src, size_t src_bytes, void* const* dst, size_t dst_bytes, int nranks)
{
    struct Range { uintptr_t from; bool is_dst; } v[2 * NUNA_MAX_RANKS];
    int n = 0;
    const auto add = [&](const void* at, bool is_dst) {
        int i = n++;
        for (; i > 0 && v[i - 1].from > (uintptr_t)at; --i) v[i] = v[i - 1];
        v[i] = {(uintptr_t)at, is_dst};
    };
    for (int r = 0; r < nranks; ++r) {
        if (src_bytes) add(src[r], false);
        if (dst_bytes) add(dst[r], true);
    }
    uintptr_t src_end = 0, dst_end = 0;                    // the furthest end of the ranges before the current one
    for (int i = 0; i < n; ++i) {
        if (v[i].from < dst_end || (v[i].is_dst && v[i].from < src_end)) return true;
        uintptr_t& end = v[i].is_dst ? dst_end : src_end;
        end = std::max(end, v[i].from + (v[i].is_dst ? dst_bytes : src_bytes));
    }
    return false;
}

int check_args(const void* const* src, void* const* dst, int nranks, size_t src_elems, size_t dst_elems,
               int dtype, unsigned flags, bool device_ptrs)
{
    if (nranks > NUNA_MAX_RANKS) return NUNA_ERR_TOO_MANY_RANKS;
    if (nranks < 1) return NUNA_ERR_INVALID_ARG;
    if (dtype != NUNA_BF16 && dtype != NUNA_F16 && dtype != NUNA_F32) return NUNA_ERR_UNSUPPORTED_DTYPE;
    if ((flags & ~(NUNA_PLACE_MASK | NUNA_TWOSHOT_PUT | NUNA_HINT_RESIDENT | NUNA_LAUNCH_PDL | NUNA_PLACE_SM_LISTS |
                   NUNA_PLACE_CLUSTER | NUNA_PLACE_STAGED | NUNA_TWOSHOT_SYNC | NUNA_CHAIN_PERSISTENT | NUNA_CHAIN_GRAPH |
                   NUNA_TWOSHOT_SYS_SCOPE | NUNA_PLACE_REGS)) != 0u ||
        (flags & NUNA_PLACE_MASK) == 3u)
        return NUNA_ERR_INVALID_ARG;
    if (src_elems > ((size_t)1 << 40) || dst_elems > ((size_t)1 << 40)) return NUNA_ERR_TOO_LARGE;
    if (src_elems == 0 && dst_elems == 0) return NUNA_OK;
    if (!src || !dst) return NUNA_ERR_INVALID_ARG;
    for (int r = 0; r < nranks; ++r) {
        if (!src[r] || !dst[r]) return NUNA_ERR_INVALID_ARG;
        if (device_ptrs && (((uintptr_t)src[r] | (uintptr_t)dst[r]) & 15u)) return NUNA_ERR_ALIGNMENT;
    }
    return aliased(src, src_elems * elem_size(dtype), dst, dst_elems * elem_size(dtype), nranks) ? NUNA_ERR_ALIAS : NUNA_OK;
}

// Bits that only nuna_chain_create understands.
static bool has_chain_bits(unsigned flags) { return (flags & (NUNA_CHAIN_PERSISTENT | NUNA_CHAIN_GRAPH)) != 0u; }

static RankPtrs make_ptrs(const void* const* src, void* const* dst, int nranks)
{
    RankPtrs p;
    memset(&p, 0, sizeof p);
    for (int r = 0; r < nranks; ++r) {
        p.src[r] = reinterpret_cast<const uint4*>(src[r]);
        p.dst[r] = reinterpret_cast<uint4*>(dst[r]);
    }
    return p;
}

// ---- launch configuration --------------------------------------------------------------------

// Vectors per thread per item.  One: with one work item per block and N independent 16-byte loads in
// flight per thread, more vectors per thread only mean fewer blocks (measured at 2 and 4 ranks: 64 KiB
// per rank 1.43 us with one vector, 1.64 us with four; no difference at 16 MiB).  NUNA_OPT_UNROLL
// overrides it for experiments.
static int pick_unroll(const Options& o, int nranks)
{
    int u = 1;
    if (o.unroll == 1 || o.unroll == 2 || o.unroll == 4) u = o.unroll;
    while (u > 1 && u * nranks > 16) u >>= 1;
    return u;
}

// Resident blocks per SM of a kernel, looked up once per device (racing first calls compute the same value).  The kernel is
// a template argument, so that the slot it is kept in belongs to that one instantiation: instantiations of one template
// share their pointer's type but not their registers.
template <auto kKernel>
static int resident_blocks(const Context* c)
{
    static std::atomic<int> cache[kMaxDevices];
    int n = cache[c->device].load(std::memory_order_relaxed);
    if (n == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kKernel, kThreads, 0) != cudaSuccess || n < 1) n = 1;
        cache[c->device].store(n, std::memory_order_relaxed);
    }
    return n;
}

// Grid size: `waves` x (SMs x resident blocks per SM), never more than the work items.  Streaming
// kernels (two-shot put, reduce-scatter, allgather) run one item per block (waves = 0: no cap): leaving
// the balancing to the hardware block scheduler measured 0.99 of the copy peak at 64 MiB per rank
// against 0.90 for a persistent grid-stride loop.  The one-shot wants its N readers of a tile close in
// time so that re-reads hit L2: four waves measured best (0.70 of peak at 64 MiB against 0.63 for one
// wave and 0.62 for an uncapped grid).
static unsigned pick_grid(const Context* c, const Options& o, size_t nitems, int blocks_per_sm, int waves = 1)
{
    size_t cap = waves > 0 ? (size_t)c->num_sms * (size_t)blocks_per_sm * (size_t)waves : ((size_t)1 << 22);
    if (o.blocks > 0) cap = (size_t)o.blocks;
    return (unsigned)std::max<size_t>(1, std::min(nitems, cap));
}

constexpr unsigned kLaunchPlain = 0u, kLaunchCooperative = 1u, kLaunchPdl = 2u;

// Programmatic dependent launch pays off while a kernel is short enough for its launch latency to
// matter.  For the one-shot it was measured to cost a few percent from about 16 MiB of sources (its
// multi-wave grid competes with the successor's early blocks), so it is dropped there; the streaming
// kernels (two-shot put, reduce-scatter, allgather) keep it at every size (4 MiB per rank: 12.6 -> 12.0 us).
static unsigned launch_mode(unsigned flags, size_t total_src_bytes = 0)
{
    return ((flags & NUNA_LAUNCH_PDL) && total_src_bytes <= ((size_t)16 << 20)) ? kLaunchPdl : kLaunchPlain;
}

// The flags a collective runs with.  Every collective kernel waits for its predecessor before it touches the buffers
// (pdl_wait), so it may be launched with or without the programmatic attribute with the same result, and a call that
// goes into a stream directly gets it without asking.  A run of plain launches that the host issues faster than the
// device drains costs a fixed 2.05 us step per kernel on B200: short kernels came out at 4.10 us each whatever their
// work, longer ones rounded up to the next multiple of 2.05 us (a kernel of 3.8 us as a graph node took 6.15, one of
// 16.0 took 18.4).  Behind a programmatic launch there is no such step, the host call is 0.4 us cheaper, and the
// prefetch ahead of the wait pays as it does with the flag (8 x 4 MiB flag two-shot: 15.6 -> 14.2 us).  While a stream
// is captured the caller's choice stands: the graph has the edges it asked for.  (The legacy default stream cannot be
// captured, and must not be asked about while another stream is.)
static unsigned effective_flags(unsigned flags, void* stream)
{
    if (flags & NUNA_LAUNCH_PDL) return flags;
    const cudaStream_t s = (cudaStream_t)stream;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (s != nullptr && s != cudaStreamLegacy && (cudaStreamIsCapturing(s, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone))
        return flags;
    return flags | NUNA_LAUNCH_PDL;
}

static thread_local unsigned t_cluster_dim = 0;           // > 0: next launch() uses clusters of this many blocks
static thread_local unsigned t_block = 0;                 // > 0: next launch() uses blocks of this many threads
static thread_local unsigned t_dyn_smem = 0;              // next launch() requests this much dynamic shared memory

template <typename... Args, typename... Act>
static int launch(void (*kernel)(Args...), unsigned grid, cudaStream_t stream, unsigned mode, Act&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(t_block > 0 ? t_block : (unsigned)kThreads, 1, 1);
    t_block = 0;
    cfg.dynamicSmemBytes = t_dyn_smem;
    t_dyn_smem = 0;
    cfg.stream = stream;
    cudaLaunchAttribute attr[3];
    int nattr = 0;
    if (t_cluster_dim > 0) {
        attr[nattr].id = cudaLaunchAttributeClusterDimension;
        attr[nattr].val.clusterDim.x = t_cluster_dim;
        attr[nattr].val.clusterDim.y = 1;
        attr[nattr].val.clusterDim.z = 1;
        ++nattr;
        t_cluster_dim = 0;
    }
    if (mode & kLaunchCooperative) {
        attr[nattr].id = cudaLaunchAttributeCooperative;
        attr[nattr].val.cooperative = 1;
        ++nattr;
    } else if (mode & kLaunchPdl) {
        attr[nattr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[nattr].val.programmaticStreamSerializationAllowed = 1;
        ++nattr;
    }
    cfg.attrs = attr;
    cfg.numAttrs = nattr;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<Args>(args)...);
    if (e != cudaSuccess) {
        fprintf(stderr, "nuna: kernel launch failed: %s\n", cudaGetErrorString(e));
        return NUNA_ERR_CUDA;
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return NUNA_OK;
}

template <typename... Args>
constexpr size_t param_bytes()
{
    size_t n = 0;
    ((n = align_up(n, alignof(Args)) + sizeof(Args)), ...);
    return n;
}

// launch() for a kernel whose last argument is a ParamPad, which it supplies.
template <typename... Args, typename... Act>
static int launch_padded(void (*kernel)(Args...), unsigned grid, cudaStream_t stream, unsigned mode, Act&&... args)
{
    static_assert(param_bytes<std::remove_const_t<Args>...>() % 64 == 32, "see ParamPad");
    using Pad = std::tuple_element_t<sizeof...(Args) - 1, std::tuple<std::remove_const_t<Args>...>>;
    return launch(kernel, grid, stream, mode, std::forward<Act>(args)..., Pad{});
}

// Compile-time dispatch over the rank count N and the unroll factor U (N * U <= 16 vectors in flight).
template <int V> using IC = std::integral_constant<int, V>;

template <int N, int U, typename F>
static int dispatch_dt(int dtype, F&& f)
{
    switch (dtype) {
        case NUNA_BF16: return f(IC<N>{}, IC<U>{}, IC<kBf16>{});
        case NUNA_F16: return f(IC<N>{}, IC<U>{}, IC<kF16>{});
        case NUNA_F32: return f(IC<N>{}, IC<U>{}, IC<kF32>{});
        default: return NUNA_ERR_UNSUPPORTED_DTYPE;
    }
}

template <int N, typename F>
static int dispatch_u(int u, int dtype, F&& f)
{
    if constexpr (N * 4 <= 16) { if (u == 4) return dispatch_dt<N, 4>(dtype, f); }
    if constexpr (N * 2 <= 16) { if (u >= 2) return dispatch_dt<N, 2>(dtype, f); }
    return dispatch_dt<N, 1>(dtype, f);
}

template <typename F>
static int dispatch(int nranks, int u, int dtype, F&& f)
{
    switch (nranks) {
        case 1: return dispatch_u<1>(u, dtype, f);   case 2: return dispatch_u<2>(u, dtype, f);
        case 3: return dispatch_u<3>(u, dtype, f);   case 4: return dispatch_u<4>(u, dtype, f);
        case 5: return dispatch_u<5>(u, dtype, f);   case 6: return dispatch_u<6>(u, dtype, f);
        case 7: return dispatch_u<7>(u, dtype, f);   case 8: return dispatch_u<8>(u, dtype, f);
        case 9: return dispatch_u<9>(u, dtype, f);   case 10: return dispatch_u<10>(u, dtype, f);
        case 11: return dispatch_u<11>(u, dtype, f); case 12: return dispatch_u<12>(u, dtype, f);
        case 13: return dispatch_u<13>(u, dtype, f); case 14: return dispatch_u<14>(u, dtype, f);
        case 15: return dispatch_u<15>(u, dtype, f); case 16: return dispatch_u<16>(u, dtype, f);
        default: return NUNA_ERR_TOO_MANY_RANKS;
    }
}
#define NUNA_NUD(n_, u_, d_) constexpr int N = decltype(n_)::value; constexpr int U = decltype(u_)::value; \
    constexpr int DT = decltype(d_)::value; (void)U; (void)DT

static size_t ceil_div(size_t a, size_t b) { return (a + b - 1) / b; }

// ---- collectives ---------------------------------------------------------------------------------

// NUNA_PLACE_AUTO picks, per size, the one-shot kernel that was measured fastest on B200, never one that is
// slower than the round-robin baseline.  Measured at 2, 3, 4, 8 and 16 ranks, 8 KiB ... 4 MiB per rank
// (us per graph node, 8 ranks; round-robin | group through L1 | group through registers):
//   dependent launch, cold:      8 KiB 1.60 | 1.16 | 1.26   64 KiB 1.78 | 1.90 | 1.41   512 KiB 3.38 | 3.65 | 2.09   4 MiB 15.6 | 17.2 | 11.8
//   dependent launch, resident:  8 KiB 1.18 | 1.16 | 1.05   64 KiB 1.21 | 1.19 | 1.09   512 KiB 2.99 | 2.48 | 1.64   4 MiB 15.1 | 17.1 | 10.5
//   plain launch, resident:      8 KiB 1.58 | 1.55 | 1.53   64 KiB 1.62 | 1.59 | 1.58   512 KiB 3.41 | 2.88 | 2.15   4 MiB 15.1 | 17.1 | 11.2
//   plain launch, cold:          8 KiB 2.02 | 1.56 | 2.00   64 KiB 2.16 | 2.46 | 2.27   512 KiB 3.78 | 4.24 | 3.29   4 MiB 15.5 | 17.2 | 12.5
// The group that shares its tile through registers wins at every size behind a dependent launch and on
// L2-resident sources; launched plainly on cold sources it wins from 1 MiB of sources in total (2 MiB below 8
// ranks) and the round-robin kernel is kept below that.  The other co-located forms (through L1, through shared
// memory) stay opt-in.
enum class OneShotKernel { RoundRobin, Group, Staged, Regs };

static OneShotKernel auto_kernel(const Context* c, const Options& o, int nranks, size_t bytes, unsigned flags)
{
    (void)c;
    if (nranks < 2) return OneShotKernel::RoundRobin;
    if (bytes < o.auto_min_bytes) return OneShotKernel::RoundRobin;
    if (flags & (NUNA_LAUNCH_PDL | NUNA_HINT_RESIDENT)) return OneShotKernel::Regs;
    const size_t total = bytes * (size_t)nranks;
    const size_t from = nranks >= 8 ? ((size_t)1 << 20) : ((size_t)2 << 20);
    return total >= from ? OneShotKernel::Regs : OneShotKernel::RoundRobin;
}


// ---- per-SM work lists for the one-shot (Algorithm 1 applied to its regular workload) ----------------
//
// Thread blocks = work items (tile, d); item (t, d) touches the N source chunks of tile t and the
// destination chunk (d, t).  Domains and the order of SMs inside a domain come from the probe
// (nearest = lowest mean hit latency).  `domains` = 0 uses what the probe found (one, or the two dies);
// a larger count splits every probed domain into equal latency quantiles (the paper's sweep over the
// number of routing domains, Section 6.5), 1 forces a single domain.  The per-SM budget R_max is
// ceil(groups per domain / SMs of the smallest domain) whole groups, so a small workload fills only the
// nearest SMs, one group each, and a large one spreads evenly.  Up to kGenericPlanTiles tiles the lists
// are produced by the general planner (nuna_plan_placement); beyond that by the closed form it reduces to
// for this workload (tile t -> domain t mod D, SMs of the domain filled in preference order), which the
// host tests check against the general planner.
constexpr size_t kGenericPlanTiles = 1024;

void plan_oneshot_lists(const nuna_topology_t* topo, int num_sms, int nranks, size_t ntiles, size_t tile_bytes,
                        bool generic, int domains, std::vector<std::vector<unsigned>>& lists)
{
    lists.assign((size_t)num_sms, {});
    const bool split = topo && topo->verdict == NUNA_TOPO_NONUNIFORM && topo->num_domains == 2 && domains != 1;
    const int base_domains = split ? 2 : 1;
    std::vector<int> dom(num_sms, 0), rank(num_sms, 0), order(num_sms);
    for (int s = 0; s < num_sms; ++s) {
        order[s] = s;
        if (split && s < NUNA_MAX_SMS) dom[s] = topo->sm_domain[s];
    }
    if (topo && topo->sms_reported > 0)
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
            const float la = a < NUNA_MAX_SMS ? topo->sm_lat_hit[a] : 0.f, lb = b < NUNA_MAX_SMS ? topo->sm_lat_hit[b] : 0.f;
            return la < lb;
        });
    for (int i = 0; i < num_sms; ++i) rank[order[i]] = i;
    // more domains than the probe found: cut each probed domain into `sub` latency quantiles
    int D = base_domains;
    if (domains > base_domains) {
        const int sub = std::max(1, std::min(domains / base_domains, num_sms / base_domains));
        std::vector<int> size(base_domains, 0), seen(base_domains, 0);
        for (int s = 0; s < num_sms; ++s) size[dom[s]]++;
        std::vector<int> fine(num_sms, 0);
        for (int i = 0; i < num_sms; ++i) {                          // in preference order
            const int s = order[i], b = dom[s];
            const int q = std::min(sub - 1, (int)((long long)seen[b]++ * sub / std::max(1, size[b])));
            fine[s] = b * sub + q;
        }
        dom = fine;
        D = base_domains * sub;
    }
    std::vector<int> dsize(D, 0);
    for (int s = 0; s < num_sms; ++s) dsize[dom[s]]++;
    const int smallest = std::max(1, *std::min_element(dsize.begin(), dsize.end()));
    const size_t per_domain = ceil_div(ntiles, (size_t)D);
    const size_t budget = std::max<size_t>(1, ceil_div(per_domain, (size_t)smallest));        // groups per SM
    if (generic) {
        const int N = nranks;
        std::vector<int> tb_gpu(ntiles * N, 0), begin(ntiles * N + 1, 0), chunks;
        chunks.reserve(ntiles * N * (N + 1));
        for (size_t t = 0; t < ntiles; ++t)
            for (int d = 0; d < N; ++d) {
                for (int r = 0; r < N; ++r) chunks.push_back((int)(r * ntiles + t));
                chunks.push_back((int)((N + d) * ntiles + t));
                begin[t * N + d + 1] = (int)chunks.size();
            }
        std::vector<long long> cbytes(2 * (size_t)N * ntiles, (long long)tile_bytes);
        std::vector<int> stack(num_sms, 0), m_compute(ntiles * N, -1);
        nuna_plan_input_t in = {};
        in.num_tbs = (int)(ntiles * N); in.tb_gpu = tb_gpu.data(); in.tb_chunk_begin = begin.data(); in.tb_chunks = chunks.data();
        in.num_chunks = (int)cbytes.size(); in.chunk_bytes = cbytes.data();
        in.num_cus = num_sms; in.cu_domain = dom.data(); in.cu_rank = rank.data();
        in.num_stacks = 1; in.cu_stack = stack.data();
        in.r_max_cu = (long long)(budget * (size_t)N * (size_t)(N + 1) * tile_bytes);
        in.r_max_stack = (long long)1 << 60;
        in.nar_max = D;
        if (nuna_plan_placement(&in, m_compute.data(), nullptr, nullptr, nullptr) == NUNA_OK) {
            for (size_t t = 0; t < ntiles; ++t) lists[(size_t)m_compute[t * N]].push_back((unsigned)t);
            return;
        }
        lists.assign((size_t)num_sms, {});
    }
    // closed form
    std::vector<std::vector<int>> dom_sms(D);
    for (int i = 0; i < num_sms; ++i) dom_sms[dom[order[i]]].push_back(order[i]);
    std::vector<size_t> used(D, 0);
    for (size_t t = 0; t < ntiles; ++t) {
        const int d = (int)(t % (size_t)D);
        size_t slot = used[d]++ / budget;
        if (slot >= dom_sms[d].size()) slot = dom_sms[d].size() - 1;      // cannot happen with the budget above
        lists[(size_t)dom_sms[d][slot]].push_back((unsigned)t);
    }
}

// Looks up (or builds and uploads) the work lists of a shape.  The plan is returned BY VALUE: its device
// tables stay allocated until nuna_shutdown even when a later probe retires the plan, so a copy taken
// under the lock stays usable after the lock is dropped.
static int get_sm_plan(Context* c, int nranks, size_t nvec, int coloc, int domains, cudaStream_t stream, SmPlan* out)
{
    std::lock_guard<std::mutex> lock(c->mutex);
    const auto key = std::make_tuple(nranks, nvec, coloc, domains);
    auto it = c->sm_plans.find(key);
    if (it == c->sm_plans.end()) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(stream, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone)
            return NUNA_ERR_CAPTURING;                 // building a plan allocates: make one plain call first
        const size_t lanes = (size_t)(kThreads / coloc);
        const size_t ntiles = ceil_div(nvec, lanes);
        std::vector<std::vector<unsigned>> lists;
        plan_oneshot_lists(c->have_topology ? &c->topology : nullptr, c->num_sms, nranks, ntiles, lanes * 16,
                           ntiles <= kGenericPlanTiles, domains, lists);
        std::vector<unsigned> off((size_t)c->num_sms + 1, 0), tiles;
        tiles.reserve(ntiles);
        for (int s = 0; s < c->num_sms; ++s) {
            tiles.insert(tiles.end(), lists[s].begin(), lists[s].end());
            off[s + 1] = (unsigned)tiles.size();
        }
        SmPlan pl;
        pl.total = (unsigned)tiles.size();
        const size_t words = off.size() + std::max<size_t>(tiles.size(), 1) + 2 * (size_t)c->num_sms + 2;
        unsigned* d = nullptr;
        if (cudaMalloc(&d, words * sizeof(unsigned)) != cudaSuccess) return NUNA_ERR_CUDA;
        std::vector<unsigned> host(words, 0u);
        std::copy(off.begin(), off.end(), host.begin());
        std::copy(tiles.begin(), tiles.end(), host.begin() + off.size());
        const size_t cur0 = off.size() + std::max<size_t>(tiles.size(), 1);
        pl.nonempty = 0;
        for (int s = 0; s < c->num_sms; ++s) pl.nonempty += !lists[s].empty();
        if (!set_now(c, d, host.data(), words * sizeof(unsigned))) {
            cudaFree(d);
            return NUNA_ERR_CUDA;
        }
        pl.base = d;
        pl.off = d;
        pl.tiles = d + off.size();
        pl.cursor = d + cur0;
        pl.present = d + cur0 + c->num_sms;
        pl.ctl = d + cur0 + 2 * (size_t)c->num_sms;
        it = c->sm_plans.emplace(key, pl).first;
    }
    *out = it->second;
    return NUNA_OK;
}

static int coloc_for(const Options& o, int nranks)
{
    int coloc = o.coloc > 0 ? o.coloc : 8;
    while (coloc > 1 && coloc / 2 >= nranks) coloc >>= 1;
    return coloc >= 8 ? 8 : coloc >= 4 ? 4 : 2;
}

// Everything a later launch of this shape would have to allocate (called before stream capture).
int prepare_oneshot(Context* c, int nranks, int dtype, size_t count, unsigned flags)
{
    if ((flags & NUNA_PLACE_MASK) == NUNA_PLACE_AWARE && (flags & NUNA_PLACE_SM_LISTS)) {
        const Options o = snapshot(c);
        SmPlan pl;
        return get_sm_plan(c, nranks, count / elems_per_vec(dtype), coloc_for(o, nranks), o.domains, (cudaStream_t)0, &pl);
    }
    return NUNA_OK;
}

template <int N, int C, int DT>
static int launch_sm_lists(Context* c, const Options& o, const RankPtrs& p, size_t count, unsigned mode, cudaStream_t stream)
{
    constexpr auto k = k_oneshot_sm<N, C, DT, false>;
    SmPlan pl;
    const int st = get_sm_plan(c, N, count / Elem<DT>::kElems, C, o.domains, stream, &pl);
    if (st != NUNA_OK) return st;
    SmLists sl;
    sl.off = pl.off; sl.tiles = pl.tiles; sl.cursor = pl.cursor; sl.present = pl.present; sl.ctl = pl.ctl;
    sl.nonempty = pl.nonempty; sl.num_sms = c->num_sms;
    const size_t cap = (size_t)c->num_sms * (size_t)resident_blocks<k>(c);
    const unsigned grid = (unsigned)std::min(cap, std::max<size_t>((size_t)c->num_sms, (size_t)pl.total));
    const unsigned blocks_per_sm = (unsigned)std::max<size_t>(1, grid / (size_t)c->num_sms);
    return launch(k, grid, stream, mode, p, count, sl, blocks_per_sm, (unsigned*)nullptr);
}

template <int N, int DT>
static int launch_cluster(const Options& o, const RankPtrs& p, size_t count, unsigned mode, cudaStream_t stream)
{
    auto k = k_oneshot_cluster<N, DT>;
    const size_t nvec = count / Elem<DT>::kElems;
    const size_t ntiles = std::max<size_t>(1, ceil_div(nvec, (size_t)kThreads));
    size_t clusters = std::min<size_t>(ntiles, (size_t)1 << 20);
    if (o.blocks > 0) clusters = std::max<size_t>(1, std::min<size_t>(clusters, (size_t)o.blocks / N));
    t_cluster_dim = N;
    return launch(k, (unsigned)(clusters * N), stream, mode, p, count, ntiles);
}

template <int N, int C, int DT>
static int launch_group(Context* c, const Options& o, const RankPtrs& p, size_t count, unsigned mode, cudaStream_t stream)
{
    constexpr auto k = k_oneshot_group<N, C, DT>;
    const size_t nvec = count / Elem<DT>::kElems;
    const size_t ntiles = ceil_div(nvec, (size_t)(kThreads / C));
    const size_t nitems = std::max<size_t>(ntiles * ((N + C - 1) / C), (count % Elem<DT>::kElems) ? (size_t)N : 0);
    const unsigned grid = pick_grid(c, o, nitems, resident_blocks<k>(c));
    return launch(k, grid, stream, mode, p, count, ntiles);
}

// How the kernels that hold a tile in registers and store it to several destinations (k_oneshot_regs, k_twoshot_put)
// are launched: vectors per source per tile, threads per block, and how many blocks prefetch ahead of the wait.
struct TileShape {
    unsigned tv, threads, prefetch_blocks;
};

// The same for L2-resident sources.  Measured at 2, 3, 4, 6, 8, 12 and 16 ranks, 8 KiB ... 8 MiB per rank, tiles of 8 ... 256
// vectors in blocks of 32 ... 256 threads, dependent graph nodes, one-shot (the put form chooses the same within 1 %); us:
// * Small messages want few, narrow blocks: up to u = 32 half the SMs up to 4 ranks (2 x 64 KiB 0.960 with 32 vectors, 0.934 with
//   64) and all of them beyond, in 128 threads (8 x 16 KiB 1.05 -> 1.00).
// * Up to u = 128 a block per SM.  Few ranks have that much less to do per vector that two blocks of 64 vectors per SM are ahead
//   (2 x 96 KiB 0.960 -> 0.936, 6 x 128 KiB 1.103 -> 1.057 against 64 vectors in 64 threads).  Every SM gets a tile: 8 ranks x
//   128 KiB take 147 tiles of 56 vectors, 1.11, where 128 tiles of 64 took 1.15.
// * Between, four full-width blocks per SM as for cold sources; up to 4 ranks three blocks of 128 threads up to u = 256
//   (2 x 512 KiB 1.17 -> 1.08).
// * Larger messages are dealt evenly, in blocks as wide as their tiles: tiles of up to 128 vectors, whose number is a whole
//   multiple of the SMs (8 x 1 MiB 2.54 -> 2.32, 8 x 1.5 MiB 3.18 -> 2.95 against 128 vectors throughout); of up to 256 for few
//   ranks and the longest messages (2 x 4 MiB 3.06 with 128 vectors, 2.16 with 256; 6 x 4 MiB 6.67, 6.49).
// * What sources and destinations of one call take of L2 leaves no room for a second set beyond half of it: the hint cannot be
//   true of a chain then, and half-full blocks keep more DRAM requests in flight (8 x 4 MiB 10.3 -> 9.9).
static TileShape hot_shape(const Context* c, int nranks, size_t units, size_t total, size_t per_sm)
{
    const size_t sms = (size_t)c->num_sms;
    const bool few = nranks <= 4;
    const auto deal = [&](size_t blocks, size_t least) {
        return (unsigned)std::min<size_t>(kThreads, std::max(least, ceil_div(ceil_div(units, blocks), (size_t)8) * 8));
    };
    const auto tight = [](unsigned tv) { return TileShape{tv, (tv + 31u) / 32u * 32u, 0u}; };
    const auto even = [&](size_t most) { return tight(deal(sms * ceil_div(units, sms * most), 8)); };
    const TileShape four = {deal(sms * per_sm, 56), (unsigned)kThreads, 0u};
    if (2 * total > c->l2_bytes / 2) return {128u, (unsigned)kThreads, 0u};
    if (units <= sms * 32) return {deal(few ? sms / 2 : sms, 16), 128u, 0u};
    if (units <= sms * 128) {
        if (nranks <= 6) return {64u, 128u, 0u};
        const TileShape t = tight(deal(sms, 8));
        return {t.tv, nranks <= 8 ? std::max(t.threads, units <= sms * 64 ? 128u : 0u) : t.threads, 0u};
    }
    if (few) return units <= sms * 256 ? TileShape{deal(sms * 3, 8), 128u, 0u} : units <= sms * 384 ? four : even(256);
    if (units <= sms * (nranks <= 8 ? 384 : 448)) return four;
    return nranks <= 8 && units > sms * 1000 ? even(256) : even(128);
}

// One tile per block.  Measured at 2, 4, 8 and 16 ranks, 16 KiB ... 64 MiB per rank, tiles of 16 ... 256 vectors in blocks
// of 32 ... 256 threads, as dependent graph nodes (us at 8 ranks; u = vectors per source and SM; `ksplit` blocks share a
// tile, each with a part of the destinations):
// * u <= 56: one block per SM, tiles of 8 ... 56 vectors (8 KiB: 1.08 resident against 1.38 with eight full blocks).
// * up to 6 MiB of sources: four blocks per SM, as many as stay resident, tiles of 56 ... 256 vectors (512 KiB cold: 2.1
//   against 2.8 with full tiles; 16 ranks x 256 KiB, three blocks per SM: 3.46 with 586 blocks, 2.42 with 294).
// * 6 to 16 MiB of sources, cold: eight blocks per SM, i.e. two waves, tiles from 112 vectors: the second wave's loads run
//   beside the first one's stores (2 MiB 6.16 -> 5.4, 1.5 MiB 4.79 -> 4.2; 4 ranks x 4 MiB 5.87 -> 5.4; 4 ranks x 2 MB,
//   three sets in turn: 3.6 with one full wave of 216 vectors, 2.6 with 112).
// * 16 to 64 MiB, cold: tiles of 192 vectors (256 up to 4 ranks) in blocks of just so many threads, and only the first wave
//   prefetches: later blocks would ask L2 for what they load at once (4 MiB 11.4 -> 11.0, 6 MiB 16.9 -> 16.1, 8 MiB
//   21.5 -> 21.1; 4 ranks x 8 MiB 11.5 -> 10.9).
// * beyond, cold: no prefetch, half the destinations per block; half-full blocks from 5 to 8 ranks (64 MiB 159.3 -> 157.6).
// * L2-resident sources: hot_shape, below.  (Cold, narrow blocks are slower up to 8 MiB of sources: more of them start
//   on an SM while the predecessor still drains, unevenly -- 512 KiB 2.07 with 256 threads, 2.6 with 64.)
// `resident` = full-width blocks of the kernel an SM holds.
static TileShape tile_shape(const Context* c, const Options& o, int nranks, size_t nvec, int ksplit, int resident, unsigned flags,
                            bool may_prefetch)
{
    const size_t sms = (size_t)c->num_sms, units = nvec * (size_t)ksplit, total = nvec * 16 * (size_t)nranks;
    const size_t per_sm = (size_t)std::max(1, std::min(4, resident));
    const bool hot = (flags & NUNA_HINT_RESIDENT) != 0u;
    const auto tile_for = [&](size_t blocks) { return ceil_div(ceil_div(units, blocks), (size_t)8) * 8; };
    const auto clamp = [](size_t v, size_t lo) { return (unsigned)std::min<size_t>(kThreads, std::max(lo, v)); };
    const unsigned everyone = may_prefetch && !hot && o.prefetch != 1 ? ~0u : 0u, first_wave = everyone ? (unsigned)(sms * 4) : 0u;
    if (o.regs_vecs > 0) return {(unsigned)std::min(kThreads, std::max(8, o.regs_vecs / 8 * 8)), (unsigned)kThreads, everyone};
    if (o.blocks > 0 && (size_t)o.blocks < sms * per_sm)             // a capped grid: as few tiles as blocks, then full tiles
        return {clamp(tile_for((size_t)o.blocks), 8), (unsigned)kThreads, everyone};
    if (hot) return hot_shape(c, nranks, units, total, per_sm);
    if (units <= sms * 56) return {clamp(tile_for(sms), 8), (unsigned)kThreads, everyone};
    const unsigned four = clamp(tile_for(sms * per_sm), 56);
    if (total < ((size_t)6 << 20)) return {four, (unsigned)kThreads, everyone};
    if (total <= ((size_t)16 << 20))
        return {std::min(four, clamp(tile_for(sms * 2 * per_sm), 112)), (unsigned)kThreads, total <= ((size_t)8 << 20) ? everyone : first_wave};
    if (total <= ((size_t)64 << 20)) {
        const unsigned tv = nranks <= 4 || nranks > 8 ? 256u : 192u;
        return {tv, tv, first_wave};
    }
    return {nranks <= 4 || nranks > 8 ? 256u : 128u, (unsigned)kThreads, 0u};
}

// Whether a kernel runs its form without the tile loop, which wants a block per item (us per node, looping | once):
// * cold, up to 4 ranks, at every size (2 x 64 KiB 0.999 | 0.947, 4 x 512 KiB 1.845 | 1.787, 3 x 4 MiB 4.39 | 4.32); beyond, the
//   loop is ahead (8 x 64 KiB 1.358 | 1.398, 16 x 256 KiB 2.38 | 3.61: every block pays for the longer text of more ranks).
// * L2-resident, where the text is shorter, but for the four full-width blocks per SM of hot_shape, where the loop is 1 ... 2 % ahead
//   (8 x 384 KiB 1.505 | 1.55), and beyond 8 ranks from u = 448 (12 x 2 MiB 6.59 | 6.82).
static bool runs_once(const Context* c, int nranks, size_t units, const TileShape& t, unsigned flags)
{
    if (!(flags & NUNA_HINT_RESIDENT)) return nranks <= 4;
    const bool large = units > (size_t)c->num_sms * 448;
    return large ? nranks <= 8 : t.threads < (unsigned)kThreads;
}

template <int N, int C, int DT>
static int launch_regs(Context* c, const Options& o, const RankPtrs& p, size_t count, unsigned flags, unsigned mode, cudaStream_t stream)
{
    constexpr int kSplit = (N + C - 1) / C;
    constexpr auto looping = k_oneshot_regs<N, C, DT, false, false>;
    const bool hot = (flags & NUNA_HINT_RESIDENT) != 0u;
    const size_t nvec = count / Elem<DT>::kElems;
    const TileShape t = tile_shape(c, o, N, nvec, kSplit, resident_blocks<looping>(c), flags, mode == kLaunchPdl);
    const size_t ntiles = ceil_div(nvec, (size_t)t.tv);
    const size_t nitems = std::max<size_t>(ntiles * kSplit, (count % Elem<DT>::kElems) ? (size_t)N : 0);
    const unsigned grid = pick_grid(c, o, std::max<size_t>(nitems, 1), 0, 0);
    const bool once = grid >= nitems && runs_once(c, N, nvec * kSplit, t, flags);
    const auto go = [&](auto kernel) { return launch_padded(kernel, grid, stream, mode, p, count, ntiles, t.tv, hot ? 0 : 1, t.prefetch_blocks); };
    t_block = t.threads;
    if constexpr (kSplit == 1) { if (hot && once) return go(k_oneshot_regs<N, C, DT, true, true>); }
    // 8 ranks x 512 KiB 1.745 -> 1.705 us; below 8 ranks it is up to 2 % slower than the general form
    if constexpr (kSplit == 1 && N >= 8) { if (hot) return go(k_oneshot_regs<N, C, DT, false, true>); }
    if constexpr (N <= 4) { if (!hot && once) return go(k_oneshot_regs<N, C, DT, true, false>); }
    return go(looping);
}

// Staged group kernel: one tile per block.  Tile size (vectors per source): large enough that a tile's
// N slices amortise the copy set-up, small enough that a mid-sized message still gives every SM several
// blocks; 32 KiB of shared memory per block at most.
template <int N, int DT>
static int launch_stage(Context* c, const Options& o, const RankPtrs& p, size_t count, unsigned flags, unsigned mode,
                        cudaStream_t stream)
{
    auto k = k_oneshot_stage<N, DT>;
    constexpr unsigned kLanes = kThreads / pow2_at_least(N);
    const size_t nvec = count / Elem<DT>::kElems;
    // measured at 8 ranks (cold): 4 KiB tiles up to 512 KiB per rank, 8 KiB to 4 MiB, 16 KiB to 16 MiB, 32 KiB beyond
    const size_t bytes = count * (size_t)Elem<DT>::kBytes;
    unsigned tile_bytes = bytes <= ((size_t)512 << 10) ? 4096u : bytes <= ((size_t)4 << 20) ? 8192u
                        : bytes <= ((size_t)16 << 20) ? 16384u : 32768u;
    unsigned tv = tile_bytes / 16u / (unsigned)pow2_at_least(N);
    if (o.stage_vecs > 0) tv = (unsigned)o.stage_vecs;
    tv = std::max(kLanes, std::min(tv, 2048u / N)) / kLanes * kLanes;     // a multiple of the row width, <= 32 KiB per tile
    const size_t ntiles = ceil_div(nvec, (size_t)tv);
    const size_t grid = std::max<size_t>(ntiles, (count % Elem<DT>::kElems) ? 1 : 0);
    t_dyn_smem = (unsigned)N * tv * 16u;
    return launch(k, (unsigned)std::max<size_t>(1, grid), stream, mode, p, count, tv,
                  (flags & NUNA_HINT_RESIDENT) ? 0 : 1, &c->bw->status, o.timeout_ns);
}

int launch_oneshot(Context* c, const RankPtrs& p, int nranks, int dtype, size_t count, unsigned flags, cudaStream_t stream)
{
    const Options o = snapshot(c);
    const size_t bytes = count * elem_size(dtype);                   // per rank
    const size_t epv = elems_per_vec(dtype);
    const unsigned mode = launch_mode(flags, bytes * (size_t)nranks);
    const size_t nvec = count / epv;
    const unsigned place = flags & NUNA_PLACE_MASK;
    OneShotKernel which = OneShotKernel::RoundRobin;
    if (place == NUNA_PLACE_AWARE)
        which = (flags & NUNA_PLACE_REGS) ? OneShotKernel::Regs : (flags & NUNA_PLACE_STAGED) ? OneShotKernel::Staged : OneShotKernel::Group;
    else if (place == NUNA_PLACE_AUTO) which = auto_kernel(c, o, nranks, bytes, flags);
    if (which == OneShotKernel::Regs) {
        const unsigned m = launch_mode(flags);
        // destinations per thread: all of them, so that a tile crosses the L2 -> SM fabric once (beyond 8 ranks the
        // sixteen-destination form: 9 ranks x 512 KiB 2.25 us against 2.71 in two passes of eight, 16 ranks x 1 MiB
        // 6.39 against 7.35); half of them for cold messages beyond 64 MiB of sources, where two blocks per tile keep more
        // DRAM loads in flight (8 ranks x 16 MiB: 41.0 us with four, 41.4 with eight; x 64 MiB 157.6 against 160.2)
        const int all = nranks > 8 ? 16 : std::min(8, pow2_at_least(nranks));
        const bool large_cold = !(flags & NUNA_HINT_RESIDENT) && bytes * (size_t)nranks > ((size_t)64 << 20);
        int coloc = o.coloc > 0 ? o.coloc : (large_cold ? std::min(8, std::max(2, pow2_at_least(nranks) / 2)) : all);
        while (coloc > 2 && coloc / 2 >= nranks) coloc >>= 1;
        return dispatch(nranks, 1, dtype, [&](auto n_, auto, auto d_) -> int {
            constexpr int N = decltype(n_)::value, DT = decltype(d_)::value;
            if constexpr (N > 8) { if (coloc >= 16) return launch_regs<N, 16, DT>(c, o, p, count, flags, m, stream); }
            if (coloc >= 8) return launch_regs<N, 8, DT>(c, o, p, count, flags, m, stream);
            if (coloc >= 4) return launch_regs<N, 4, DT>(c, o, p, count, flags, m, stream);
            return launch_regs<N, 2, DT>(c, o, p, count, flags, m, stream);
        });
    }
    if (which == OneShotKernel::Staged) {
        return dispatch(nranks, 1, dtype, [&](auto n_, auto, auto d_) -> int {
            constexpr int N = decltype(n_)::value, DT = decltype(d_)::value;
            return launch_stage<N, DT>(c, o, p, count, flags, launch_mode(flags), stream);
        });
    }
    if (which == OneShotKernel::Group) {
        // co-location factor: C destinations of a tile share a block (C <= N rounded up to a power of two)
        const int coloc = coloc_for(o, nranks);
        if (place == NUNA_PLACE_AWARE && (flags & NUNA_PLACE_CLUSTER) && nranks >= 2 && nranks <= 8) {
            return dispatch(nranks, 1, dtype, [&](auto n_, auto, auto d_) -> int {
                constexpr int N = decltype(n_)::value, DT = decltype(d_)::value;
                if constexpr (N >= 2 && N <= 8) return launch_cluster<N, DT>(o, p, count, mode, stream);
                else return NUNA_ERR_INVALID_ARG;
            });
        }
        if (place == NUNA_PLACE_AWARE && (flags & NUNA_PLACE_SM_LISTS)) {
            return dispatch(nranks, 1, dtype, [&](auto n_, auto, auto d_) -> int {
                constexpr int N = decltype(n_)::value, DT = decltype(d_)::value;
                if (coloc >= 8) return launch_sm_lists<N, 8, DT>(c, o, p, count, mode, stream);
                if (coloc >= 4) return launch_sm_lists<N, 4, DT>(c, o, p, count, mode, stream);
                return launch_sm_lists<N, 2, DT>(c, o, p, count, mode, stream);
            });
        }
        return dispatch(nranks, 1, dtype, [&](auto n_, auto, auto d_) -> int {
            constexpr int N = decltype(n_)::value, DT = decltype(d_)::value;
            if (coloc >= 8) return launch_group<N, 8, DT>(c, o, p, count, mode, stream);
            if (coloc >= 4) return launch_group<N, 4, DT>(c, o, p, count, mode, stream);
            return launch_group<N, 2, DT>(c, o, p, count, mode, stream);
        });
    }
    return dispatch(nranks, pick_unroll(o, nranks), dtype, [&](auto n_, auto u_, auto d_) -> int {
        NUNA_NUD(n_, u_, d_);
        constexpr auto k = k_oneshot_rr<N, U, DT>;
        const size_t ntiles = ceil_div(nvec, (size_t)kThreads * U);
        const size_t nitems = std::max<size_t>(ntiles * N, (count % epv) ? (size_t)N : 0);
        // one resident wave while the message is small enough for latency to matter, four beyond
        const unsigned grid = pick_grid(c, o, nitems, resident_blocks<k>(c), bytes >= ((size_t)8 << 20) ? 4 : 1);
        return launch_padded(k, grid, stream, mode, p, count, ntiles);
    });
}

// Launches the flag-synchronised two-shot on explicit scratch / flag / control storage (the context's, or
// the fixed arrays of the allocation-free entry point): one block per work item, tiles + lead blocks.
// tv = 0 picks the tile size by message size.  min_tv is the smallest tile the flag array was sized for.
int launch_twoshot_flags(int num_sms, int blocks_override, const RankPtrs& p, int nranks, int dtype, size_t count,
                         unsigned tv, unsigned min_tv, uint4* scratch, unsigned* tile_flags, BarrierWords* bw,
                         unsigned long long timeout_ns, bool pdl, unsigned debug_bits, cudaStream_t stream)
{
    const size_t bytes = count * elem_size(dtype);
    const size_t nvec = count / elems_per_vec(dtype);
    const bool in_place = (debug_bits & 64u) != 0u;
    // The register-thrifty instantiation, six blocks per SM instead of four: once a message is bandwidth-bound.  In place it is
    // ahead later, with a lead of eight blocks per SM instead of six, and in tiles of 32 KiB instead of 24, 16 of 2 ranks in both (us, four |
    // six: 2 x 16 MiB 13.6 | 14.0, 32 MiB 24.5 | 23.4, 64 MiB 44.0 | 42.9; 3 x 23 MiB 24.6 | 25.7; 4 x 16 MiB 23.5 | 24.2, 64 MiB 88.1 | 84.5;
    // 8 x 16 MiB 42.7 | 44.5).
    const size_t all_src = bytes * (size_t)nranks;
    const bool many_resident = !in_place ? all_src >= ((size_t)64 << 20) : all_src > (nranks <= 2 ? (size_t)32 << 20 : (size_t)160 << 20);
    bool mid_sized = false;
    if (tv == 0) {
        // (Below takes_tags' limit these are the tiles of calls that ask for the flags' scope or cap the blocks, and of the hooks.)
        // Tile bytes across all N sources, from a sweep at 8 ranks (16 ... 256 vectors per tile at every size):
        // small tiles while the message is small (more blocks, less latency per tile), 32 KiB once there are
        // plenty.  At 8 MiB of sources 16 KiB tiles make 1024 blocks for 592 resident ones and the second
        // wave's consumers wait (10.3 us against 7.6 us with 12 KiB tiles), hence the step back there.  From 10 ranks
        // fewer blocks are resident, and larger tiles are ahead from 4 to 14 MiB (16 ranks x 320 KiB 6.3 us with 24 KiB
        // tiles, 8.3 with 12; x 512 KiB 6.9 against 8.7; 12 x 400 KiB 6.1 against 7.9; 9 x 700 KiB 7.1 against 6.6).
        // Between 16 and 64 MiB of sources 24 KiB tiles with a lead of five blocks per SM are ahead (3 MiB per rank 11.6
        // against 12.3 us, 4 MiB 14.2 against 15.1, 6 MiB 19.1 against 21.3, 7 MiB 21.6 against 24.2; at 8 MiB 27.2
        // against 24.8, hence the upper limit; a lead of four is 2 % faster at 4 MiB and 10 ... 30 % slower elsewhere).
        const size_t src_bytes = bytes * (size_t)nranks;
        mid_sized = nranks <= 8 && src_bytes > ((size_t)16 << 20) && src_bytes < ((size_t)64 << 20);   // 16 ranks: no gain
        const bool many = nranks >= 10;
        const unsigned tile_src = src_bytes <= ((size_t)512 << 10) ? 4096u : src_bytes <= ((size_t)1 << 20) ? 8192u
                                : src_bytes <= ((size_t)4 << 20) ? 12288u
                                : src_bytes <= ((size_t)8 << 20) ? (many ? 24576u : 12288u)
                                : src_bytes <= ((size_t)14 << 20) ? (many ? 32768u : 16384u)
                                : src_bytes <= ((size_t)16 << 20) ? 16384u : mid_sized ? 24576u : 32768u;
        tv = (!in_place ? tile_src : nranks <= 2 ? 16384u : many_resident ? 32768u : 24576u) / 16u / (unsigned)nranks;
    }
    tv = std::max(min_tv, std::min(tv, 2048u / (unsigned)nranks));
    tv = std::max(1u, tv / 8u * 8u);
    if (tv < min_tv) tv = min_tv;
    const size_t ntiles = std::max<size_t>(1, ceil_div(nvec, (size_t)tv));
    unsigned lead_max = (unsigned)num_sms * (mid_sized ? 5u : 8u);
    if (in_place) lead_max = (unsigned)num_sms * (many_resident ? 8u : 6u);
    if (blocks_override > 0) lead_max = (unsigned)std::max(1, blocks_override);
    const size_t lead = std::min<size_t>(ntiles, lead_max);
    const unsigned grid = (unsigned)(ntiles + lead);
    return dispatch(nranks, 1, dtype, [&](auto n_, auto, auto d_) -> int {
        constexpr int N = decltype(n_)::value, DT = decltype(d_)::value;
        t_dyn_smem = (unsigned)N * tv * 16u;
        const unsigned mode = pdl ? kLaunchPdl : kLaunchPlain;
        const auto go = [&](auto kernel) {
            return launch_padded(kernel, grid, stream, mode, p, scratch, tile_flags, count, tv, lead_max, bw, timeout_ns, debug_bits);
        };
        if constexpr (N <= 8) { if (in_place) return go(many_resident ? k_twoshot_flags<N, DT, 6, true> : k_twoshot_flags<N, DT, 4, true>); }
        return go(many_resident ? k_twoshot_flags<N, DT, 6, false> : k_twoshot_flags<N, DT, 4, false>);
    });
}

// How the tagged two-shot is launched, always in full-width blocks: narrow ones start on an SM while the predecessor still
// drains, unevenly (8 x 64 KiB 1.8 us in 256 threads, 2.5 in 64).  Measured at 2, 4, 8 and 16 ranks, 16 KiB ... 16 MiB per rank, cold, tiles
// of 16 ... 256 vectors, leads of 1 ... 1184 tiles, dependent graph nodes (us):
// * Up to four tiles per SM each block gathers the tile before its own (lead 1: 8 x 512 KiB 2.9, 3.6 with a lead of three tiles per
//   SM): tiles of 56 ... 128 vectors, from 96 up to 8 ranks (8 x 512 KiB 2.95 with 56, 2.89; 16 x 256 KiB 2.88 with 56, 3.00), fewer
//   and larger ones up to 4 ranks (2 x 1 MiB 2.75 with 96 vectors, 2.53 with 192).  Up to 11 ranks registers hold four blocks per SM
//   and all of them are resident together; from 12 they hold three, and the last quarter starts as the first leave (16 x 1 MiB 7.4).
// * Beyond, a lead of three tiles per SM, so that what a block gathers was reduced a wave earlier (8 x 4 MiB 11.5; five 11.6,
//   one 11.7, eight 11.9), and tiles of 128 vectors (192 12.1), 192 up to 4 ranks (2 x 8 MiB 8.84; 128 9.2, 256 8.97).
struct TaggedShape {
    unsigned tv, lead;
};

static TaggedShape tagged_shape(const Context* c, int nranks, size_t nvec)
{
    const size_t sms = (size_t)c->num_sms;
    const auto deal = [&](size_t blocks, size_t least, size_t most) {
        return (unsigned)std::min(most, std::max(least, ceil_div(ceil_div(nvec, blocks), (size_t)8) * 8));
    };
    if (nvec <= sms * 32) return {nranks <= 4 ? 96u : 32u, 1u};
    if (nranks <= 4) return nvec <= sms * 4 * 192 ? TaggedShape{deal(sms * 2, 96, 192), 1u} : TaggedShape{192u, (unsigned)sms * 3};
    const size_t least = nranks <= 8 && nvec > sms * 96 ? 96 : 56;
    return nvec <= sms * 4 * 128 ? TaggedShape{deal(sms * 4, least, 128), 1u} : TaggedShape{128u, (unsigned)sms * 3};
}

// Whether a two-shot call runs the tagged form.  us per node, flags | tagged: 2 ranks x 64 KiB 3.19 | 1.96, 4 MiB 9.9 | 6.1,
// 8 MiB 9.4 | 9.8; 4 x 512 KiB 6.4 | 2.6, 4 MiB 8.8 | 7.9; 8 x 8 KiB 3.3 | 2.0, 512 KiB 5.0 | 2.9, 4 MiB 14.2 | 12.2, 8 MiB 24.7 | 22.7,
// 16 MiB 44.6 | 45.9; 16 x 64 KiB 5.6 | 2.6, 1 MiB 10.1 | 7.5, 4 MiB 25.6 | 22.7.  The fewer the ranks, the more the shard's doubled
// bytes are beside theirs.  On sources that are in L2 there is less to hide them behind (flags, scratch or in place | tagged, with the
// hint: 3 x 5 MiB 7.51 | 7.51, 6 MiB 8.50 | 8.79, 4 x 5 MiB 9.09 | 8.88, 6 MiB 10.22 | 10.56; 8 x 8 MiB 25.5 | 23.5).  Captured plainly the order is
// that of cold sources (3 x 6 MiB 11.6 | 10.5, 4 x 6 MiB 13.3 | 12.0, 8 x 8 MiB 26.6 | 24.6, 16 x 8 MiB 46.5 | 45.1; 3 x 6 MiB from L2 9.2 | 9.7).
// What asks about the flags (their scope, their tile, the shard's lines) gets the form that has them.
static bool takes_tags(const Options& o, int nranks, size_t bytes, unsigned flags)
{
    const bool five = nranks <= 2 || (nranks <= 4 && (flags & NUNA_HINT_RESIDENT));
    return bytes <= (five ? kTaggedMaxShard / 8 * 5 : nranks <= 4 ? kTaggedMaxShard / 4 * 3 : kTaggedMaxShard) && !(flags & NUNA_TWOSHOT_SYS_SCOPE) && !o.keep_shard &&
           o.twoshot_vecs <= 0 && o.blocks <= 0;
}

// Whether the flag two-shot, the allgather and the alltoall ask L2 for their blocks' first tiles ahead of the
// dependent-launch wait: cold device-memory sources, and a message small enough that the predecessor's drain is a visible
// share of it.  us with | without, by MiB of sources: flag two-shot, 8 ranks, 2 4.8 | 5.2, 8 10.1 | 11.7, 32 14.5 | 15.9, 128
// 44.0 | 45.4; 2 ranks 32 15.2 | 16.5, but 128 53.6 | 52.3; allgather, 16 ranks, 4 10.9 | 12.5, 4 ranks 32 26.8 | 28.0, 128
// 103.3 | 104.3; alltoall, 8 ranks, 4 2.2 | 2.8, 32 10.3 | 11.5, 128 40.9 | 41.8.  Beyond 8 ranks 8 MiB (16 ranks, flag two-shot, 7.3 | 8.2)
// is as far as it has been measured to pay.
static bool prefetch_pays(const Options& o, unsigned flags, int nranks, size_t bytes)
{
    if (!(flags & NUNA_LAUNCH_PDL) || (flags & NUNA_HINT_RESIDENT) || o.prefetch == 1) return false;
    return bytes * (size_t)nranks <= (nranks <= 8 ? (size_t)128 << 20 : (size_t)8 << 20);
}

// The put form: one tile per block by default; `max_blocks` > 0 makes it a grid-stride loop over that many blocks.
int launch_twoshot_put(Context* c, const RankPtrs& p, int nranks, int dtype, size_t count, unsigned flags, cudaStream_t stream,
                       unsigned max_blocks)
{
    const Options o = snapshot(c);
    const unsigned mode = launch_mode(flags);
    const size_t nvec = count / elems_per_vec(dtype);
    return dispatch(nranks, pick_unroll(o, nranks), dtype, [&](auto n_, auto u_, auto d_) -> int {
        NUNA_NUD(n_, u_, d_);
        constexpr auto looping = k_twoshot_put<N, U, DT, false>;
        // host-memory sources (max_blocks > 0) are read through the link, not through L2: no prefetch, full tiles
        const TileShape t = max_blocks > 0 ? TileShape{(unsigned)kThreads, (unsigned)kThreads, 0u}
                                           : tile_shape(c, o, nranks, nvec, 1, resident_blocks<looping>(c), flags, mode == kLaunchPdl);
        const size_t ntiles = ceil_div(nvec, (size_t)t.tv * U);
        unsigned grid = pick_grid(c, o, std::max<size_t>(ntiles, 1), 0, 0);
        if (max_blocks > 0 && o.blocks <= 0) grid = std::min(grid, max_blocks);
        const auto go = [&](auto kernel) {
            return launch_padded(kernel, grid, stream, mode, p, count, ntiles, t.tv, (flags & NUNA_HINT_RESIDENT) ? 0 : 1, t.prefetch_blocks);
        };
        t_block = t.threads;
        if constexpr (U == 1) { if (grid >= ntiles && runs_once(c, N, nvec, t, flags)) return go(k_twoshot_put<N, U, DT, true>); }
        return go(looping);
    });
}

// Whether the flag two-shot uses the owners' destinations as its shard.  us, scratch | in place, dependent launches: 2 ranks x 8 MiB
// 9.4 | 8.4, 64 MiB 53.2 | 42.7; 3 x 23 MiB 27.8 | 25.3; 4 x 16 MiB 26.5 | 23.5, 64 MiB 92 | 84.5; 6 x 12 MB 26.5 | 25.1; 8 x 9 MiB 27.7 |
// 26.1, 16 MiB 44.0 | 42.7, but 22 MiB 61.5 | 63.7, 6 x 24 MB 49.9 | 50.9; 12 x 10 MB 43.0 | 44.3; 16 x 12 MB 63.4 | 63.8.  Launched
// plainly, without a prefetch: 2 x 16 MiB 17.5 | 19.5, 3 x 64 MiB 71.8 | 67.4, 4 x 16 MiB 28.0 | 26.9, 8 x 16 MiB 46.8 | 48.2.
// With the resident hint there is no prefetch either: 2 x 9 MiB 9.5 | 9.2, 10 MiB 10.5 | 10.5, 12 MiB 11.9 | 14.4, 16 MiB 16.5 | 18.5, but 18 MiB 18.2 | 16.8, 64 MiB 52.3 | 47.6; 3 x
// 23 MiB 29.2 | 27.7; 5 x 9 MiB 20.7 | 19.7, 25 MiB 49.0 | 47.0; 6 x 9 MiB 23.7 | 22.4, 20 MiB 43.8 | 43.8; 7 x 12 MiB 32.7 | 33.7, 18 MiB 45.3 |
// 47.8; 8 x 9 MiB 28.2 | 28.9, 16 MiB 45.5 | 47.6.
static bool shard_in_place(const Options& o, int nranks, size_t bytes, unsigned flags)
{
    const size_t total = bytes * (size_t)nranks;
    const bool hint = (flags & NUNA_HINT_RESIDENT) != 0u;
    const bool pays = !(flags & NUNA_LAUNCH_PDL) ? nranks == 3 || nranks == 4
                    : nranks > 4                 ? nranks <= (hint ? 6 : 8) && total <= ((size_t)128 << 20)
                                                 : !hint || nranks != 2 || total <= ((size_t)20 << 20) || total > ((size_t)32 << 20);
    return pays && !(flags & NUNA_TWOSHOT_SYS_SCOPE) && !o.keep_shard && o.twoshot_vecs <= 0 && o.blocks <= 0;
}

// The form whose shard words carry their own flags: a block per tile and `lead` more that only gather.
static int launch_twoshot_tagged(const Context* c, const Options& o, const RankPtrs& p, int nranks, int dtype, size_t count, uint4* slots,
                                 unsigned long long timeout_ns, unsigned flags, unsigned debug_bits, cudaStream_t stream)
{
    const unsigned mode = launch_mode(flags);
    const size_t nvec = count / elems_per_vec(dtype), bytes = count * elem_size(dtype);
    const TaggedShape t = tagged_shape(c, nranks, nvec);
    const size_t ntiles = std::max<size_t>(1, ceil_div(nvec, (size_t)t.tv));
    const unsigned grid = (unsigned)(ntiles + std::min<size_t>(ntiles, t.lead));
    const unsigned bits = debug_bits | (prefetch_pays(o, flags, nranks, bytes) ? 16u : 0u);
    return dispatch(nranks, 1, dtype, [&](auto n_, auto, auto d_) -> int {
        constexpr int N = decltype(n_)::value, DT = decltype(d_)::value;
        return launch_padded(k_twoshot_tagged<N, DT>, grid, stream, mode, p, slots, count, t.tv, t.lead, c->bw, timeout_ns, bits);
    });
}

int launch_twoshot(Context* c, const RankPtrs& p, int nranks, int dtype, size_t count, unsigned flags, cudaStream_t stream)
{
    if (flags & NUNA_TWOSHOT_PUT) return launch_twoshot_put(c, p, nranks, dtype, count, flags, stream, 0u);
    uint4 *scratch, *slots;
    unsigned* tile_flags;
    Options o;
    {
        std::lock_guard<std::mutex> lock(c->mutex);
        o = c->opt;
        scratch = reinterpret_cast<uint4*>(c->scratch);
        slots = reinterpret_cast<uint4*>(c->slots);
        tile_flags = c->flags;
    }
    if (takes_tags(o, nranks, count * elem_size(dtype), flags))
        return launch_twoshot_tagged(c, o, p, nranks, dtype, count, slots, o.timeout_ns, flags, 0u, stream);
    return launch_twoshot_flags(c->num_sms, o.blocks, p, nranks, dtype, count, (unsigned)std::max(0, o.twoshot_vecs), kMinFlagTileVec,
                                scratch, tile_flags, c->bw, o.timeout_ns, (flags & NUNA_LAUNCH_PDL) != 0,
                                (o.keep_shard ? 4u : 0u) | ((flags & NUNA_TWOSHOT_SYS_SCOPE) ? 8u : 0u) |
                                    (prefetch_pays(o, flags, nranks, count * elem_size(dtype)) ? 16u : 0u) |
                                    (shard_in_place(o, nranks, count * elem_size(dtype), flags) ? 64u : 0u), stream);
}

// `asked`: the caller gave NUNA_LAUNCH_PDL itself.
int launch_reduce_scatter(Context* c, const RankPtrs& p, int nranks, int dtype, size_t shard, unsigned flags, bool asked,
                          cudaStream_t stream)
{
    const Options o = snapshot(c);
    const size_t epv = elems_per_vec(dtype);
    const unsigned mode = launch_mode(flags);
    if (shard % epv) {
        const size_t tiles = std::max<size_t>(1, ceil_div(shard / epv, (size_t)kRaggedTile));
        return dispatch(nranks, 1, dtype, [&](auto n_, auto u_, auto d_) -> int {
            NUNA_NUD(n_, u_, d_);
            constexpr auto k = k_reduce_scatter_ragged<N, DT>;
            return launch_padded(k, pick_grid(c, o, (tiles + 1) * N, resident_blocks<k>(c), 0), stream, mode, p, shard, tiles);
        });
    }
    const size_t shard_vec = shard / epv, total = shard * elem_size(dtype) * (size_t)nranks * (size_t)nranks;
    const int unroll = pick_unroll(o, nranks);
    // The form that works ahead.  A caller who asks for dependent launches, and does not say that the sources are in L2, gets it from
    // 32 full tiles (64 up to 4 ranks), below which the early successor's blocks get in the way, to 128 MiB of sources, 256 beyond 8
    // ranks.  us, ordinary | ahead, in a run of such calls on cold sources, by bytes per source: 8 ranks 64 KiB 1.16 | 1.32, 128 KiB
    // 1.73 | 1.34, 512 KiB 2.20 | 1.86, 4 MiB 6.38 | 5.51, 16 MiB 21.7 | 20.5, 32 MiB 43.2 | 43.7; 2 x 128 KiB 1.21 | 1.16, 512 KiB 1.70 | 1.27;
    // 4 x 4 MiB 4.49 | 3.66; 16 x 1 MiB 4.01 | 4.05, 4 MiB 10.9 | 9.3, 16 MiB 39.7 | 39.0.
    // Nothing is known of what stands before any other call.  If its sources are in L2 all the same (8 x 512 KiB 1.37 | 1.40, 1 MiB
    // 1.71 | 1.93, 2 MiB 2.38 | 2.54, but 4 MiB 5.44 | 4.50, 8 MiB 10.7 | 9.4), or a kernel that does not release early comes before it
    // (with that kernel's time, one that writes the sources, and one that writes elsewhere: 8 x 1 MiB 6.98 | 7.29, 9.99 | 10.65, 4 MiB
    // 16.41 | 16.74, 14.38 | 14.70, 8 MiB 28.24 | 28.57, 20.32 | 20.14; 4 x 4 MiB 10.54 | 10.74, 11.50 | 11.97, 8 MiB 17.06 | 17.22, 14.94 | 15.06;
    // 16 x 2 MiB 16.24 | 16.93, 13.86 | 14.56, 3 MiB 22.13 | 22.39, 16.50 | 16.61), it costs at most 2.3 % from 32 MiB of sources, 48 beyond 8
    // ranks, and up to 15 % below.
    // Beyond 4 ranks blocks of 192 threads, 128 from 9 ranks, once full-width ones do not fit beside each other: they leave, and make
    // room for the successor's, more evenly (8 x 4 MiB 5.49 | 5.31, 16 x 2 MiB 5.67 | 5.04, 4 MiB 9.62 | 9.31); from 9 ranks full-width
    // ones are ahead again beyond 64 MiB of sources (12 x 8 MiB 13.87 | 14.68, 16 x 8 MiB 18.65 | 19.02, 16 MiB 37.99 | 39.56).
    const size_t full = ceil_div(shard_vec, (size_t)kThreads) * (size_t)nranks, sms = (size_t)c->num_sms;
    const bool ahead = asked ? full >= (nranks <= 4 ? 64 : 32) : total >= (nranks <= 8 ? (size_t)32 << 20 : (size_t)48 << 20);
    if (ahead && mode == kLaunchPdl && !(flags & NUNA_HINT_RESIDENT) && o.prefetch != 1 && o.blocks <= 0 && unroll == 1 &&
        total <= (nranks <= 8 ? (size_t)128 << 20 : (size_t)256 << 20)) {
        const bool wide = nranks <= 4 || full <= sms * 4 || (nranks > 8 && total > ((size_t)64 << 20));
        const unsigned threads = wide ? (unsigned)kThreads : nranks <= 8 ? 192u : 128u;
        const unsigned tiles = (unsigned)ceil_div(shard_vec, (size_t)threads);
        return dispatch(nranks, 1, dtype, [&](auto n_, auto, auto d_) -> int {
            constexpr int N = decltype(n_)::value, DT = decltype(d_)::value;
            t_block = threads;
            return launch_padded(k_reduce_scatter_ahead<N, DT>, tiles * N, stream, mode, p, shard_vec, tiles, (unsigned)sms * 4u);
        });
    }
    return dispatch(nranks, unroll, dtype, [&](auto n_, auto u_, auto d_) -> int {
        NUNA_NUD(n_, u_, d_);
        constexpr auto k = k_reduce_scatter<N, U, DT>;
        const size_t tiles = ceil_div(shard_vec, (size_t)kThreads * U);
        const unsigned grid = pick_grid(c, o, tiles * N, resident_blocks<k>(c), 0);
        return launch_padded(k, grid, stream, mode, p, shard_vec, tiles);
    });
}

// Allgather and alltoall copy bits: they work on 16-byte vectors, shifted to the destination's alignment when a shard is
// no whole number of them; what is left at the ends goes in 16-bit units (every element type is a multiple of that).
int launch_allgather(Context* c, const RankPtrs& p, int nranks, size_t shard_bytes, unsigned flags, cudaStream_t stream)
{
    const Options o = snapshot(c);
    const unsigned mode = launch_mode(flags);
    const size_t shard_vec = shard_bytes / 16;
    // small tiles: about four blocks per SM, 16 ... 256 vectors each
    const size_t per = ceil_div(ceil_div(shard_vec * (size_t)nranks, (size_t)c->num_sms * 4), (size_t)8) * 8;
    const unsigned small_tv = (unsigned)std::min<size_t>(kThreads, std::max<size_t>(16, per));
    const bool prefetch = prefetch_pays(o, flags, nranks, shard_vec * 16);
    if (shard_bytes % 16) {
        const unsigned tv = std::min(kRaggedGather, small_tv);
        const size_t tiles = std::max<size_t>(1, ceil_div(shard_vec + 7, (size_t)tv));          // the first may be short by 7 vectors
        return launch(k_allgather_ragged, pick_grid(c, o, tiles * nranks, 0, 0), stream, mode, p, nranks, shard_bytes, tiles, tv,
                      prefetch ? 1 : 0);
    }
    const size_t out_total = shard_bytes * (size_t)nranks * (size_t)nranks;
    if (o.ag_bulk_vecs == 0 && out_total <= ((size_t)128 << 20)) {
        // register form with small tiles
        const size_t tiles = ceil_div(shard_vec + (shard_vec % 8 ? 7 : 0), (size_t)small_tv);   // the first tile of a shard may be short
        const unsigned grid = (unsigned)(tiles * nranks);
        if (o.blocks <= 0 || (size_t)o.blocks >= grid) {           // one tile per block: a capped grid takes the looping form below
            // Blocks of no more threads than the tile once tiles are large: more of them fit beside each other.  Full-width |
            // narrow, cold, us: 8 ranks, tiles of 104 vectors 2.15 | 2.18, 112 2.25 | 2.16, 192 3.28 | 2.99; 16 ranks 96 3.01 | 2.93,
            // 144 4.37 | 3.90; 12 ranks 112 2.78 | 2.80, 144 3.49 | 3.25.  With fewer ranks to store to, the line lies further up:
            // 4 ranks 112 1.91 | 1.93, 128 1.96 | 2.08, 160 2.08 | 2.09, 192 2.28 | 2.25; 6 ranks 128 2.20 | 2.34, 160 2.61 | 2.66, 192 3.18 | 2.69.  Two
            // and three ranks and smaller tiles are up to 30 % faster in full-width blocks.
            if (nranks >= 4 && small_tv >= (nranks >= 8 ? 112u : 176u)) t_block = (small_tv + 31u) / 32u * 32u;
            return launch_padded(shard_vec % 8 ? k_allgather_small<true> : k_allgather_small<false>, grid, stream, mode, p, nranks, shard_vec,
                                 small_tv, prefetch ? 1 : 0);
        }
    }
    if (o.ag_bulk_vecs != 1) {
        // Default: the bulk-copy form, one block per (rank, tile); the copy engine moves the tile in once and
        // out N times.  Measured against the register form below: 16 x 64 KiB 4.11 vs 4.99 us, 16 x 8 KiB 2.02
        // vs 3.68 us, 8 x 8 MiB 97.4 vs 102.2 us.  Small tiles (1 KiB) while there are few of them, 2 KiB beyond.
        const size_t out_bytes = shard_bytes * (size_t)nranks * (size_t)nranks;
        unsigned tv = o.ag_bulk_vecs >= 8 ? (unsigned)o.ag_bulk_vecs : (out_bytes <= ((size_t)64 << 20) ? 64u : 128u);
        tv = std::min(2048u, tv) / 8u * 8u;
        const size_t tiles = ceil_div(shard_vec, (size_t)tv);
        if (tiles * (size_t)nranks <= ((size_t)1 << 24)) {
            t_dyn_smem = tv * 16u;
            return launch_padded(k_allgather_bulk, (unsigned)(tiles * nranks), stream, mode, p, nranks, shard_vec, tiles, tv, &c->bw->status,
                          o.timeout_ns, prefetch ? 1 : 0);
        }
    }
    // One block per (rank, tile) storing to all N destinations.  Splitting a tile's destinations over
    // several blocks (dsplit > 1) was measured slower at every size tried (16 x 64 KiB: 4.4 us with 1,
    // 5.4 us with 8): the stores, not the block count, are the limit.
    constexpr int U = 2;
    const int dsplit = 1;
    constexpr auto k = k_allgather<U>;
    const size_t tiles = ceil_div(shard_vec, (size_t)kThreads * U);
    const unsigned grid = pick_grid(c, o, tiles * nranks * dsplit, resident_blocks<k>(c), 0);
    return launch(k, grid, stream, mode, p, nranks, shard_vec, tiles, dsplit);
}

int launch_alltoall(Context* c, const RankPtrs& p, int nranks, size_t block_bytes, unsigned flags, cudaStream_t stream)
{
    const Options o = snapshot(c);
    const unsigned mode = launch_mode(flags);
    if (block_bytes % 16) {
        // four vectors per thread from 16 MiB of sources (8 x 8 x 1 MB blocks 23.6 against 22.9 us, 8 x 8 x 18 KB 1.6 against 1.9)
        const bool wide = block_bytes * (size_t)nranks * (size_t)nranks >= ((size_t)16 << 20);
        const size_t tiles = std::max<size_t>(1, ceil_div(block_bytes / 16 + 7, (size_t)kRaggedRow * (wide ? 4 : 2)));
        return launch_padded(wide ? k_alltoall_ragged<4> : k_alltoall_ragged<2>, pick_grid(c, o, tiles * nranks * nranks, 0, 0), stream, mode, p,
                      nranks, block_bytes, tiles);
    }
    const size_t block_vec = block_bytes / 16;
    if (o.ag_bulk_vecs != 1) {
        // bulk-copy form (default), as for the allgather; 8 KiB tiles (8 x 8 blocks of 64 KiB: 2.84 us against
        // 3.02 us for the register form and 3.11 us with 2 KiB tiles)
        const unsigned tv = o.ag_bulk_vecs >= 8 ? std::min(2048u, (unsigned)o.ag_bulk_vecs) / 8u * 8u : 512u;
        const size_t tiles = ceil_div(block_vec, (size_t)tv);
        const size_t grid = tiles * (size_t)nranks * (size_t)nranks;
        if (grid <= ((size_t)1 << 24)) {
            t_dyn_smem = tv * 16u;
            return launch_padded(k_alltoall_bulk, (unsigned)grid, stream, mode, p, nranks, block_vec, tiles, tv, &c->bw->status, o.timeout_ns,
                          prefetch_pays(o, flags, nranks, block_vec * 16 * (size_t)nranks) ? 1 : 0);
        }
    }
    constexpr int U = 2;
    constexpr auto k = k_alltoall<U>;
    const size_t tiles = ceil_div(block_vec, (size_t)kThreads * U);
    const unsigned grid = pick_grid(c, o, tiles * nranks * nranks, resident_blocks<k>(c), 0);
    return launch(k, grid, stream, mode, p, nranks, block_vec, tiles);
}

// ---- single-kernel chain ---------------------------------------------------------------------------------

// One cluster runs the whole chain.  Measured on B200 (160 nodes, 8 ranks): 1.45 us per node at 16 KiB per rank
// against 1.08 us for the graph with dependent launch, 2.5 against 1.15 us at 128 KiB, 12 against 2.4 us at
// 1 MiB: a node still costs two dependent memory round trips (loads; then the stores the cluster barrier has to
// see performed) plus the barrier on sixteen SMs, which is no less than a launch hidden behind its predecessor.
// So the library never picks it by itself (limit 0); NUNA_CHAIN_PERSISTENT runs it on request.
constexpr size_t kChainPersistentMaxBytes = 0;                      // per rank

bool chain_persistent_supported(const Context* c, int nsets, int nranks, int dtype, size_t count)
{
    (void)c;
    return nsets >= 1 && nsets <= kMaxChainSets && nranks >= 1 && count * elem_size(dtype) <= ((size_t)4 << 20);
}

bool chain_persistent_pays_off(int dtype, size_t count) { return count * elem_size(dtype) <= kChainPersistentMaxBytes; }

int launch_chain_persistent(Context* c, const ChainSets& sets, int nsets, int nnodes, int nranks, int dtype, size_t count,
                            cudaStream_t stream)
{
    (void)c;
    // two destinations per thread while that still gives every thread of the cluster an item, all of them beyond
    const bool wide = (count / elems_per_vec(dtype)) * (size_t)((nranks + 1) / 2) > (size_t)16 * kThreads;
    return dispatch(nranks, 1, dtype, [&](auto n_, auto, auto d_) -> int {
        constexpr int N = decltype(n_)::value, DT = decltype(d_)::value;
        constexpr int kAll = pow2_at_least(N) > 8 ? 8 : (pow2_at_least(N) < 2 ? 2 : pow2_at_least(N));
        auto k = wide ? k_chain_persistent<N, kAll, DT> : k_chain_persistent<N, 2, DT>;
        // sixteen blocks per cluster need the non-portable opt-in; fall back to the portable eight
        static std::atomic<int> cluster_size[kMaxDevices];
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = 0;
        int cs = cluster_size[dev].load(std::memory_order_relaxed);
        if (cs == 0) {
            cs = 8;
            if (cudaFuncSetAttribute(k_chain_persistent<N, kAll, DT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                cudaFuncSetAttribute(k_chain_persistent<N, 2, DT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
                cudaLaunchConfig_t cfg = {};
                cfg.gridDim = dim3(16, 1, 1);
                cfg.blockDim = dim3(kThreads, 1, 1);
                cudaLaunchAttribute at;
                at.id = cudaLaunchAttributeClusterDimension;
                at.val.clusterDim.x = 16; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
                cfg.attrs = &at;
                cfg.numAttrs = 1;
                int nclusters = 0;
                if (cudaOccupancyMaxActiveClusters(&nclusters, k, &cfg) == cudaSuccess && nclusters >= 1) cs = 16;
            }
            cudaGetLastError();
            cluster_size[dev].store(cs, std::memory_order_relaxed);
        }
        t_cluster_dim = (unsigned)cs;
        return launch(k, (unsigned)cs, stream, kLaunchPlain, sets, nsets, nnodes, count);
    });
}

}  // namespace nuna

using namespace nuna;

// The device address of `bytes` bytes of page-locked host memory, or null unless all of them are page-locked and the
// device sees them in one piece.  The first byte does not speak for the rest: a program may have registered a part of
// its buffer, or registered it in parts, so the ranges are followed to the end (one step for any single allocation).
static void* mapped_host(const void* host, size_t bytes)
{
    typedef CUresult (*Attributes)(unsigned, CUpointer_attribute*, void**, CUdeviceptr);
    static const Attributes attributes = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult found;
        const bool ok = cudaGetDriverEntryPoint("cuPointerGetAttributes", &fn, cudaEnableDefault, &found) == cudaSuccess &&
                        found == cudaDriverEntryPointSuccess;
        return ok ? reinterpret_cast<Attributes>(fn) : nullptr;
    }();
    if (!attributes) return nullptr;
    uintptr_t first = 0;
    for (size_t done = 0; done < bytes;) {
        // one driver call for all of them: 16 buffers cost 1 us more with a call per attribute
        unsigned type = 0, managed = 0;
        CUdeviceptr at = 0, start = 0;
        size_t size = 0;
        CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                      CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
        void* to[] = {&type, &managed, &at, &start, &size};
        if (attributes(5, what, to, (CUdeviceptr)(uintptr_t)host + done) != CUDA_SUCCESS || type != CU_MEMORYTYPE_HOST || managed || !at ||
            (done && at != first + done) || start > at || start + size <= at)
            return nullptr;
        if (!done) first = at;
        done += start + size - at;
    }
    return reinterpret_cast<void*>(first);
}

// The allreduce forms behind their argument checks; `flags` are the ones to run with.
static int run_oneshot(const void* const* src, void* const* dst, int nranks, size_t count, int dtype, unsigned flags, void* stream)
{
    Context* c = nullptr;
    const int st = get_context(&c);
    if (st != NUNA_OK) return st;
    return launch_oneshot(c, make_ptrs(src, dst, nranks), nranks, dtype, count, flags, (cudaStream_t)stream);
}

static int run_twoshot(const void* const* src, void* const* dst, int nranks, size_t count, int dtype, unsigned flags, void* stream)
{
    Context* c = nullptr;
    int st = get_context(&c);
    if (st != NUNA_OK) return st;
    if (!(flags & NUNA_TWOSHOT_PUT)) {
        std::lock_guard<std::mutex> lock(c->mutex);
        const size_t need = (count * elem_size(dtype) + 15) & ~(size_t)15;
        if (need > c->scratch_bytes || !c->scratch) {
            cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
            if (cudaStreamIsCapturing((cudaStream_t)stream, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone)
                return NUNA_ERR_CAPTURING;             // growing the scratch allocates: call nuna_init first
            if ((st = ensure_scratch(c, need)) != NUNA_OK) return st;
        }
    }
    return launch_twoshot(c, make_ptrs(src, dst, nranks), nranks, dtype, count, flags, (cudaStream_t)stream);
}

extern "C" {

int nuna_init(size_t scratch_bytes)
{
    Context* c = nullptr;
    int st = get_context(&c);
    if (st != NUNA_OK) return st;
    std::lock_guard<std::mutex> lock(c->mutex);
    return ensure_scratch(c, scratch_bytes);
}

int nuna_set_option(int option, long long value)
{
    if (value < 0) return NUNA_ERR_INVALID_ARG;
    Context* c = nullptr;
    int st = get_context(&c);
    if (st != NUNA_OK) return st;
    std::lock_guard<std::mutex> lock(c->mutex);
    switch (option) {
        case NUNA_OPT_BLOCKS: c->opt.blocks = (int)std::min<long long>(value, 1 << 22); break;
        case NUNA_OPT_UNROLL: c->opt.unroll = (int)value; break;
        case NUNA_OPT_COLOC: c->opt.coloc = (int)value; break;
        case NUNA_OPT_AUTO_MIN_BYTES: c->opt.auto_min_bytes = (size_t)value; break;
        case NUNA_OPT_TIMEOUT_MS: c->opt.timeout_ns = (unsigned long long)(value ? value : 1000) * 1000000ull; break;
        case NUNA_OPT_DOMAINS: c->opt.domains = (int)std::min<long long>(value, NUNA_MAX_SMS); break;
        case NUNA_OPT_STAGE_VECS: c->opt.stage_vecs = (int)std::min<long long>(value, 4096); break;
        case NUNA_OPT_TWOSHOT_VECS: c->opt.twoshot_vecs = (int)std::min<long long>(value, 4096); break;
        case NUNA_OPT_AG_BULK_VECS: c->opt.ag_bulk_vecs = (int)std::min<long long>(value, 2048); break;
        case NUNA_OPT_REGS_VECS: c->opt.regs_vecs = (int)std::min<long long>(value, kThreads); break;
        case NUNA_OPT_PREFETCH: c->opt.prefetch = (int)std::min<long long>(value, 1); break;
        default: return NUNA_ERR_INVALID_ARG;
    }
    return NUNA_OK;
}

int nuna_allreduce_oneshot(const void* const* src, void* const* dst, int nranks, size_t count, int dtype,
                           unsigned flags, void* stream)
{
    if (has_chain_bits(flags)) return NUNA_ERR_INVALID_ARG;
    int st = check_args(src, dst, nranks, count, count, dtype, flags & ~NUNA_TWOSHOT_PUT, true);
    if (st != NUNA_OK || count == 0) return st;
    if (flags & NUNA_TWOSHOT_PUT) return NUNA_ERR_INVALID_ARG;
    return run_oneshot(src, dst, nranks, count, dtype, effective_flags(flags, stream), stream);
}

int nuna_allreduce_twoshot(const void* const* src, void* const* dst, int nranks, size_t count, int dtype,
                           unsigned flags, void* stream)
{
    if (has_chain_bits(flags)) return NUNA_ERR_INVALID_ARG;
    int st = check_args(src, dst, nranks, count, count, dtype, flags, true);
    if (st != NUNA_OK || count == 0) return st;
    return run_twoshot(src, dst, nranks, count, dtype, effective_flags(flags, stream), stream);
}

int nuna_allreduce(const void* const* src, void* const* dst, int nranks, size_t count, int dtype, unsigned flags,
                   void* stream)
{
    if (has_chain_bits(flags)) return NUNA_ERR_INVALID_ARG;
    const int st = check_args(src, dst, nranks, count, count, dtype, flags, true);
    if (st != NUNA_OK || count == 0) return st;
    // Measured on B200 at 2, 3, 4, 6, 8 and 16 ranks, 8 KiB ... 64 MiB per rank, cold and L2-resident (us per graph node).
    // Without NUNA_PLACE_AUTO the one-shot is the round-robin kernel, whose re-reads cost more the more ranks there are.
    // Behind a dependent launch the put form is ahead of it (8 ranks x 8 KiB 1.14 against 1.29, x 1 MiB 3.14 against 4.92)
    // but for the smallest messages of few ranks (2 x 8 KiB 0.92 against 0.86; L2-resident 2 x 256 KiB 1.04 against 1.01);
    // launched plainly, where nothing is prefetched, the one-shot's many blocks pay up to 1 MiB per rank at 2 ranks (2.24
    // against 2.16), 512 KiB at 4, 64 KiB at 8 and 8 KiB at 16.
    // With NUNA_PLACE_AUTO the one-shot is the register-sharing kernel, equal to the put form within 2 % at every size and
    // ahead of it beyond 64 MiB of sources, where two blocks share a tile (8 x 64 MiB 157 against 160); beyond 8 ranks and
    // 16 MiB the put form is ahead (16 x 2 MiB 11.55 against 11.95).
    flags = effective_flags(flags, stream);
    const size_t bytes = count * elem_size(dtype);
    const bool autop = (flags & NUNA_PLACE_MASK) == NUNA_PLACE_AUTO, pdl = (flags & NUNA_LAUNCH_PDL) != 0u;
    const bool sync_form = (flags & NUNA_TWOSHOT_SYNC) && !(flags & NUNA_TWOSHOT_PUT);
    const unsigned base = flags & ~(NUNA_TWOSHOT_SYNC | NUNA_TWOSHOT_PUT | (sync_form ? 0u : NUNA_TWOSHOT_SYS_SCOPE));
    size_t limit;                                              // the largest message, in bytes per rank, for the one-shot
    if (sync_form) {
        // asked for explicitly; the one-shot takes what is too small for two dependent phases
        limit = nranks <= 2 ? ((size_t)1 << 20) : nranks <= 4 ? ((size_t)512 << 10) : nranks <= 8 ? ((size_t)128 << 10) : ((size_t)64 << 10);
        if (autop) limit = std::max(limit, (pdl ? (size_t)8 << 20 : nranks <= 8 ? (size_t)2 << 20 : (size_t)512 << 10) / (size_t)std::max(1, nranks));
        limit *= 8;
    } else if (autop) {
        limit = nranks <= 8 ? ~(size_t)0 : ((size_t)16 << 20) / (size_t)nranks;
    } else if (pdl) {
        limit = nranks > 4 ? 0 : (flags & NUNA_HINT_RESIDENT) ? ((size_t)256 << 10) : ((size_t)16 << 10);
    } else {
        limit = nranks <= 2 ? ((size_t)1 << 20) : nranks <= 4 ? ((size_t)512 << 10) : nranks <= 8 ? ((size_t)64 << 10) : ((size_t)8 << 10);
    }
    if (nranks <= 1 || bytes <= limit) return run_oneshot(src, dst, nranks, count, dtype, base, stream);
    return run_twoshot(src, dst, nranks, count, dtype, sync_form ? base : (base | NUNA_TWOSHOT_PUT), stream);
}

int nuna_reduce_scatter(const void* const* src, void* const* dst, int nranks, size_t shard_count, int dtype,
                        unsigned flags, void* stream)
{
    if (has_chain_bits(flags)) return NUNA_ERR_INVALID_ARG;
    if (nranks >= 1 && nranks <= NUNA_MAX_RANKS && shard_count > ((size_t)1 << 40) / (size_t)nranks)
        return NUNA_ERR_TOO_LARGE;
    int st = check_args(src, dst, nranks, shard_count * (size_t)(nranks > 0 ? nranks : 0), shard_count, dtype,
                        flags & ~NUNA_TWOSHOT_PUT, true);
    if (st != NUNA_OK || shard_count == 0) return st;
    if (flags & NUNA_TWOSHOT_PUT) return NUNA_ERR_INVALID_ARG;
    Context* c = nullptr;
    if ((st = get_context(&c)) != NUNA_OK) return st;
    return launch_reduce_scatter(c, make_ptrs(src, dst, nranks), nranks, dtype, shard_count, effective_flags(flags, stream),
                                 (flags & NUNA_LAUNCH_PDL) != 0u, (cudaStream_t)stream);
}

int nuna_allgather(const void* const* src, void* const* dst, int nranks, size_t shard_count, int dtype,
                   unsigned flags, void* stream)
{
    if (has_chain_bits(flags)) return NUNA_ERR_INVALID_ARG;
    if (nranks >= 1 && nranks <= NUNA_MAX_RANKS && shard_count > ((size_t)1 << 40) / (size_t)nranks)
        return NUNA_ERR_TOO_LARGE;
    int st = check_args(src, dst, nranks, shard_count, shard_count * (size_t)(nranks > 0 ? nranks : 0), dtype,
                        flags & ~NUNA_TWOSHOT_PUT, true);
    if (st != NUNA_OK || shard_count == 0) return st;
    if (flags & NUNA_TWOSHOT_PUT) return NUNA_ERR_INVALID_ARG;
    Context* c = nullptr;
    if ((st = get_context(&c)) != NUNA_OK) return st;
    return launch_allgather(c, make_ptrs(src, dst, nranks), nranks, shard_count * elem_size(dtype), effective_flags(flags, stream), (cudaStream_t)stream);
}

int nuna_alltoall(const void* const* src, void* const* dst, int nranks, size_t block_count, int dtype,
                  unsigned flags, void* stream)
{
    if (has_chain_bits(flags)) return NUNA_ERR_INVALID_ARG;
    if (nranks >= 1 && nranks <= NUNA_MAX_RANKS && block_count > ((size_t)1 << 40) / (size_t)nranks)
        return NUNA_ERR_TOO_LARGE;
    const size_t per_rank = block_count * (size_t)(nranks > 0 ? nranks : 0);
    int st = check_args(src, dst, nranks, per_rank, per_rank, dtype, flags & ~NUNA_TWOSHOT_PUT, true);
    if (st != NUNA_OK || block_count == 0) return st;
    if (flags & NUNA_TWOSHOT_PUT) return NUNA_ERR_INVALID_ARG;
    Context* c = nullptr;
    if ((st = get_context(&c)) != NUNA_OK) return st;
    return launch_alltoall(c, make_ptrs(src, dst, nranks), nranks, block_count * elem_size(dtype), effective_flags(flags, stream), (cudaStream_t)stream);
}

int nuna_allreduce_host(const void* const* src, void* const* dst, int nranks, size_t count, int dtype,
                        unsigned flags, int two_shot)
{
    if (has_chain_bits(flags)) return NUNA_ERR_INVALID_ARG;
    int st = check_args(src, dst, nranks, count, count, dtype, flags, false);
    if (st != NUNA_OK || count == 0) return st;
    if (!two_shot && (flags & NUNA_TWOSHOT_PUT)) return NUNA_ERR_INVALID_ARG;
    Context* c = nullptr;
    if ((st = get_context(&c)) != NUNA_OK) return st;
    std::lock_guard<std::mutex> lock(c->host_mutex);       // staging buffers and the private stream: one call at a time
    const size_t bytes = count * elem_size(dtype);
    if (!c->stream && cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking) != cudaSuccess) return NUNA_ERR_CUDA;

    // Page-locked host buffers are visible to the device: the put form of the two-shot reads every source
    // byte once and writes every destination byte once, so it can run directly on them -- one kernel, reads
    // and writes crossing the host link in both directions at once, no staging copies.  (Bringing the sources
    // in by copy engine in 1-16 pipelined chunks while the kernel stores straight into the host destinations
    // was measured slower at every size -- 8 x 512 KiB: 214-690 us against 174 us -- because each of the
    // 8 x chunks asynchronous copies costs about 4 us of host time to enqueue.)  The one-shot without a placement of its
    // own gives the same bits, so it goes the same way (8 x 12 KB: 77 us with staging copies, 17 in place).
    if (two_shot ? (flags & NUNA_TWOSHOT_PUT) != 0u : (flags & NUNA_PLACE_MASK) != NUNA_PLACE_AWARE) {
        const void* msrc[NUNA_MAX_RANKS];
        void* mdst[NUNA_MAX_RANKS];
        bool mapped = true;
        for (int r = 0; r < nranks && mapped; ++r) {
            msrc[r] = mapped_host(src[r], bytes);
            mdst[r] = mapped_host(dst[r], bytes);
            mapped = msrc[r] && mdst[r] && (((uintptr_t)msrc[r] | (uintptr_t)mdst[r]) & 15u) == 0;
        }
        if (mapped) {
            // Few blocks: reads of host memory issued by many SMs at once get less out of the link than the same reads from
            // a few (8 x 512 KiB: 166 us with one block per tile).  The fewer, though, the longer the first call on buffers
            // that were just page-locked, when every translation of theirs is still missing.  us on the first call | later, 12,
            // 20 and 24 blocks: 8 x 512 KiB 167 153 148 | 124.2 123.7 124.9, 4 x 1 MiB 172 157 160 | 124.6 124.4 124.4, 2 x 512 KiB
            // 64 59 58 | 42.7 41.7 41.7, 2 x 2 MiB 191 187 187 | 126.7 122.0 122.3.  Twelve suffice for the first call, and are
            // ahead later, beyond 8 ranks (16 x 256 KiB 154 149 153 | 127 134 138) and for little data of many ranks (8 x 128 KiB
            // 64 64 62 | 44.0 45.5 47.0, 8 x 64 KiB 47 46 46 | 31.7 33.1 33.1; 2 x 64 KiB 25 24 24 | 19.5 18.8 18.7).
            // What is left: either direction of the link alone takes 86 us of device time for 4 MiB.
            const bool twelve = nranks > 8 || (nranks > 4 && bytes * (size_t)nranks <= ((size_t)1 << 20));
            st = launch_twoshot_put(c, make_ptrs(msrc, mdst, nranks), nranks, dtype, count, flags & ~NUNA_LAUNCH_PDL, c->stream,
                                    twelve ? 12u : 20u);
            if (st != NUNA_OK) return st;
            return cudaStreamSynchronize(c->stream) == cudaSuccess ? NUNA_OK : NUNA_ERR_CUDA;
        }
    }

    const size_t slot = (bytes + 255) & ~(size_t)255;
    const size_t need = slot * 2 * (size_t)nranks;
    if (need > c->staging_bytes) {
        if (c->staging) cudaFree(c->staging);
        c->staging = nullptr;
        c->staging_bytes = 0;
        if (cudaMalloc(&c->staging, need) != cudaSuccess) return NUNA_ERR_CUDA;
        c->staging_bytes = need;
    }
    if (two_shot && !(flags & NUNA_TWOSHOT_PUT)) {
        std::lock_guard<std::mutex> inner(c->mutex);
        if ((st = ensure_scratch(c, slot)) != NUNA_OK) return st;
    }
    const void* dsrc[NUNA_MAX_RANKS];
    void* ddst[NUNA_MAX_RANKS];
    char* base = static_cast<char*>(c->staging);
    for (int r = 0; r < nranks; ++r) {
        dsrc[r] = base + slot * (size_t)r;
        ddst[r] = base + slot * (size_t)(nranks + r);
        if (cudaMemcpyAsync(const_cast<void*>(dsrc[r]), src[r], bytes, cudaMemcpyHostToDevice, c->stream) != cudaSuccess)
            return NUNA_ERR_CUDA;
    }
    const RankPtrs p = make_ptrs(dsrc, ddst, nranks);
    st = two_shot ? launch_twoshot(c, p, nranks, dtype, count, flags, c->stream)
                  : launch_oneshot(c, p, nranks, dtype, count, flags, c->stream);
    if (st != NUNA_OK) return st;
    for (int d = 0; d < nranks; ++d)
        if (cudaMemcpyAsync(dst[d], ddst[d], bytes, cudaMemcpyDeviceToHost, c->stream) != cudaSuccess)
            return NUNA_ERR_CUDA;
    return cudaStreamSynchronize(c->stream) == cudaSuccess ? NUNA_OK : NUNA_ERR_CUDA;
}

int nuna_device_status(int* out)
{
    if (!out) return NUNA_ERR_INVALID_ARG;
    Context* c = nullptr;
    int st = get_context(&c);
    if (st != NUNA_OK) return st;
    if (cudaDeviceSynchronize() != cudaSuccess) return NUNA_ERR_CUDA;
    BarrierWords h;
    if (cudaMemcpy(&h, c->bw, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return NUNA_ERR_CUDA;
    unsigned worst = h.status;
    if (h.status != 0 && (st = rewind_barrier_words(c, c->bw, h)) != NUNA_OK) return st;
    // the allocation-free entry point keeps its own words in the library's fixed arrays
    unsigned static_status = 0;
    if ((st = static_status_read_and_clear(c, &static_status)) != NUNA_OK) return st;
    *out = (int)std::max(worst, static_status);
    return NUNA_OK;
}

int nuna_launch_floor(unsigned blocks, unsigned flags, void* stream)
{
    if (blocks == 0 || blocks > (1u << 20) || (flags & ~NUNA_LAUNCH_PDL)) return NUNA_ERR_INVALID_ARG;
    return launch(k_empty, blocks, (cudaStream_t)stream, launch_mode(flags), 0);
}

// See nuna_debug.h.
int nuna_debug_launch_floor(unsigned blocks, unsigned flags, int trigger_first, void* stream)
{
    if (blocks == 0 || blocks > (1u << 20) || (flags & ~NUNA_LAUNCH_PDL)) return NUNA_ERR_INVALID_ARG;
    if (trigger_first) return launch(k_empty_trigger_first, blocks, (cudaStream_t)stream, launch_mode(flags), 0);
    return launch(k_empty, blocks, (cudaStream_t)stream, launch_mode(flags), 0);
}

unsigned long long nuna_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

const char* nuna_status_string(int status)
{
    switch (status) {
        case NUNA_OK: return "ok";
        case NUNA_ERR_INVALID_ARG: return "invalid argument";
        case NUNA_ERR_UNSUPPORTED_DTYPE: return "unsupported dtype";
        case NUNA_ERR_ALIGNMENT: return "pointer not 16-byte aligned";
        case NUNA_ERR_ALIAS: return "destination overlaps a source or another destination";
        case NUNA_ERR_CUDA: return "CUDA runtime error";
        case NUNA_ERR_TIMEOUT: return "flag barrier timed out";
        case NUNA_ERR_CAPTURING: return "operation would allocate or synchronise during stream capture";
        case NUNA_ERR_TOO_MANY_RANKS: return "more than NUNA_MAX_RANKS ranks";
        case NUNA_ERR_TOO_LARGE: return "size beyond the supported maximum";
        default: return "unknown status";
    }
}

int nuna_shutdown(void)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return NUNA_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_ctx_mutex);
    // out of the table first: a call that comes while this one waits for the device finds none, and waits for the lock
    Context* c = g_ctx[dev].exchange(nullptr, std::memory_order_acq_rel);
    if (!c) return NUNA_OK;
    cudaDeviceSynchronize();
    if (c->bw) cudaFree(c->bw);
    if (c->scratch) cudaFree(c->scratch);
    for (void* d : c->retired_scratch) cudaFree(d);
    if (c->staging) cudaFree(c->staging);
    if (c->stream) cudaStreamDestroy(c->stream);
    cudaStreamDestroy(c->setup);
    for (auto& kv : c->sm_plans) cudaFree(kv.second.base);
    for (unsigned* d : c->retired_plans) cudaFree(d);
    delete c;
    return NUNA_OK;
}

// See nuna_debug.h.
int nuna_debug_host_mapped(const void* host, size_t bytes) { return host && bytes && mapped_host(host, bytes) ? 1 : 0; }

/* Test hook: the per-SM work lists planned for a one-shot of `ntiles` tiles under `topo` (NULL = no probe),
 * by the general planner (generic != 0) or the closed form.  off: [num_sms + 1], tiles: [ntiles].          */
int nuna_debug_plan_oneshot(const nuna_topology_t* topo, int num_sms, int nranks, size_t ntiles, size_t tile_bytes,
                            int generic, int domains, unsigned* off, unsigned* tiles)
{
    if (num_sms < 1 || nranks < 1 || nranks > NUNA_MAX_RANKS || !off || !tiles || domains < 0) return NUNA_ERR_INVALID_ARG;
    std::vector<std::vector<unsigned>> lists;
    plan_oneshot_lists(topo, num_sms, nranks, ntiles, tile_bytes, generic != 0, domains, lists);
    size_t n = 0;
    off[0] = 0;
    for (int s = 0; s < num_sms; ++s) {
        for (unsigned t : lists[s]) tiles[n++] = t;
        off[s + 1] = (unsigned)n;
    }
    return n == ntiles ? NUNA_OK : NUNA_ERR_INVALID_ARG;
}

/* Test hook (not part of the public header): every block of a `grid`-block launch arrives at a flag
 * barrier that expects `expected` arrivals and waits at most timeout_ms.  Writes how many blocks
 * passed.  With expected > grid nothing ever completes the barrier, the waits run out, and the
 * status word latches NUNA_ERR_TIMEOUT -- without trapping or hanging the device.                    */
int nuna_debug_barrier_selftest(unsigned grid, unsigned expected, unsigned timeout_ms, unsigned* passed)
{
    Context* c = nullptr;
    int st = get_context(&c);
    if (st != NUNA_OK) return st;
    if (!passed || grid == 0 || grid > (unsigned)c->num_sms || expected == 0) return NUNA_ERR_INVALID_ARG;
    unsigned* d = nullptr;
    if (cudaMalloc(&d, sizeof(unsigned)) != cudaSuccess) return NUNA_ERR_CUDA;
    cudaMemset(d, 0, sizeof(unsigned));
    st = launch(k_barrier_selftest, grid, (cudaStream_t)0, kLaunchCooperative, c->bw, expected,
                (unsigned long long)timeout_ms * 1000000ull, d);
    if (st == NUNA_OK && cudaDeviceSynchronize() != cudaSuccess) st = NUNA_ERR_CUDA;
    if (st == NUNA_OK && cudaMemcpy(passed, d, sizeof(unsigned), cudaMemcpyDeviceToHost) != cudaSuccess) st = NUNA_ERR_CUDA;
    cudaFree(d);
    return st;
}

/* Measurement hook: one launch of the one-shot allreduce (8 ranks, bf16, whole vectors) under a placement --
 * 0 round-robin, 1 co-located groups, 2 per-SM work lists -- with the latency of every work item's first load
 * sampled per warp into hist[NUNA_DEBUG_LAT_BINS] (bins of NUNA_DEBUG_LAT_STEP cycles, added to what hist
 * already holds).  Destinations receive the ordinary result.  Synchronises the device.                   */
int nuna_debug_access_latency(const void* const* src, void* const* dst, size_t count, int placement, unsigned* hist)
{
    constexpr int N = 8;
    int st = check_args(src, dst, N, count, count, NUNA_BF16, 0u, true);
    if (st != NUNA_OK) return st;
    if (!hist || count == 0 || count % 8 != 0 || placement < 0 || placement > 2) return NUNA_ERR_INVALID_ARG;
    Context* c = nullptr;
    if ((st = get_context(&c)) != NUNA_OK) return st;
    const Options o = snapshot(c);
    const RankPtrs p = make_ptrs(src, dst, N);
    const size_t nvec = count / 8;
    unsigned* d_hist = nullptr;
    if (cudaMalloc(&d_hist, kLatBins * sizeof(unsigned)) != cudaSuccess) return NUNA_ERR_CUDA;
    cudaMemset(d_hist, 0, kLatBins * sizeof(unsigned));
    if (placement == 0) {
        constexpr auto k = k_latency_rr<N, kBf16>;
        const size_t ntiles = ceil_div(nvec, (size_t)kThreads);
        st = launch(k, pick_grid(c, o, ntiles * N, resident_blocks<k>(c)), (cudaStream_t)0, kLaunchPlain, p, count, ntiles, d_hist);
    } else if (placement == 1) {
        constexpr auto k = k_latency_group<N, 8, kBf16>;
        const size_t ntiles = ceil_div(nvec, (size_t)(kThreads / 8));
        st = launch(k, pick_grid(c, o, ntiles, resident_blocks<k>(c)), (cudaStream_t)0, kLaunchPlain, p, count, ntiles, d_hist);
    } else {
        constexpr auto k = k_oneshot_sm<N, 8, kBf16, true>;
        SmPlan pl;
        st = get_sm_plan(c, N, nvec, 8, o.domains, (cudaStream_t)0, &pl);
        if (st == NUNA_OK) {
            SmLists sl;
            sl.off = pl.off; sl.tiles = pl.tiles; sl.cursor = pl.cursor; sl.present = pl.present; sl.ctl = pl.ctl;
            sl.nonempty = pl.nonempty; sl.num_sms = c->num_sms;
            const size_t cap = (size_t)c->num_sms * (size_t)resident_blocks<k>(c);
            const unsigned grid = (unsigned)std::min(cap, std::max<size_t>((size_t)c->num_sms, (size_t)pl.total));
            st = launch(k, grid, (cudaStream_t)0, kLaunchPlain, p, count, sl,
                        (unsigned)std::max<size_t>(1, grid / (size_t)c->num_sms), d_hist);
        }
    }
    if (st == NUNA_OK && cudaDeviceSynchronize() != cudaSuccess) st = NUNA_ERR_CUDA;
    unsigned h[kLatBins];
    if (st == NUNA_OK && cudaMemcpy(h, d_hist, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) st = NUNA_ERR_CUDA;
    if (st == NUNA_OK)
        for (int b = 0; b < kLatBins; ++b) hist[b] += h[b];
    cudaFree(d_hist);
    return st;
}

// See nuna_debug.h.  The same tile size, grid and form of the kernel as launch_regs<8, 8, bf16>.
int nuna_debug_oneshot_regs_traced(const void* const* src, void* const* dst, size_t count, unsigned flags, unsigned slot,
                                   unsigned long long* trace, unsigned* grid_blocks, void* stream)
{
    constexpr int N = 8;
    int st = check_args(src, dst, N, count, count, NUNA_BF16, flags & (NUNA_LAUNCH_PDL | NUNA_HINT_RESIDENT), true);
    if (st != NUNA_OK) return st;
    if (!trace || count == 0 || (flags & ~(NUNA_LAUNCH_PDL | NUNA_HINT_RESIDENT)) != 0u) return NUNA_ERR_INVALID_ARG;
    Context* c = nullptr;
    if ((st = get_context(&c)) != NUNA_OK) return st;
    const Options o = snapshot(c);
    constexpr auto looping = k_oneshot_regs<N, 8, kBf16, false, false>;
    const bool hot = (flags & NUNA_HINT_RESIDENT) != 0u;
    const size_t nvec = count / 8;
    const unsigned mode = launch_mode(flags);
    const TileShape t = tile_shape(c, o, N, nvec, 1, resident_blocks<looping>(c), flags, mode == kLaunchPdl);
    const size_t ntiles = ceil_div(nvec, (size_t)t.tv);
    const size_t nitems = std::max<size_t>(ntiles, (count % 8) ? (size_t)N : 0);
    const unsigned grid = pick_grid(c, o, std::max<size_t>(nitems, 1), 0, 0);
    if (grid_blocks) *grid_blocks = grid;
    t_block = t.threads;
    const bool once = hot && grid >= nitems && runs_once(c, N, nvec, t, flags);
    const auto k = once ? k_oneshot_regs_timed<N, 8, kBf16, true, true> : hot ? k_oneshot_regs_timed<N, 8, kBf16, false, true>
                                                                             : k_oneshot_regs_timed<N, 8, kBf16, false, false>;
    return launch(k, grid, (cudaStream_t)stream, mode, make_ptrs(src, dst, N), count, ntiles, t.tv, hot ? 0 : 1,
                  t.prefetch_blocks, trace, slot, (unsigned)NUNA_DEBUG_TRACE_BLOCKS);
}

/* Test hook: a flag-synchronised two-shot whose consumers wait for a flag value that nobody publishes
 * (debug_bits = 1): every consumer wait runs out after timeout_ms, the kernel returns, destinations stay
 * unwritten and the status word latches NUNA_ERR_TIMEOUT; nothing traps or hangs.  debug_bits = 0 is the
 * ordinary kernel with an explicit timeout.                                                            */
int nuna_debug_twoshot(const void* const* src, void* const* dst, int nranks, size_t count, int dtype,
                       unsigned timeout_ms, unsigned debug_bits)
{
    int st = check_args(src, dst, nranks, count, count, dtype, 0u, true);
    if (st != NUNA_OK || count == 0) return st;
    const bool tagged = (debug_bits & 32u) != 0u;
    if ((debug_bits & ~37u) != 0u || (tagged && count * elem_size(dtype) > kTaggedMaxShard)) return NUNA_ERR_INVALID_ARG;
    Context* c = nullptr;
    if ((st = get_context(&c)) != NUNA_OK) return st;
    uint4 *scratch, *slots;
    unsigned* tile_flags;
    {
        std::lock_guard<std::mutex> lock(c->mutex);
        if ((st = ensure_scratch(c, (count * elem_size(dtype) + 15) & ~(size_t)15)) != NUNA_OK) return st;
        scratch = reinterpret_cast<uint4*>(c->scratch);
        slots = reinterpret_cast<uint4*>(c->slots);
        tile_flags = c->flags;
    }
    if (tagged)
        return launch_twoshot_tagged(c, snapshot(c), make_ptrs(src, dst, nranks), nranks, dtype, count, slots,
                                     (unsigned long long)timeout_ms * 1000000ull, 0u, debug_bits & 1u, (cudaStream_t)0);
    return launch_twoshot_flags(c->num_sms, 0, make_ptrs(src, dst, nranks), nranks, dtype, count, 0u, kMinFlagTileVec, scratch,
                                tile_flags, c->bw, (unsigned long long)timeout_ms * 1000000ull, false, debug_bits,
                                (cudaStream_t)0);
}

}  // extern "C"

// ---- two-shot allreduce for callers that cannot allocate ------------------------------------------
//
// Everything the flag-barrier two-shot needs beyond its inputs and outputs -- the shard
// intermediate and the barrier words -- lives in the two file-scope device arrays below, which
// every GPU that loads this library carries from module load to process exit (4 MiB + 384 bytes).
// In host code the names `g_static_shard` and `g_static_barrier` are only stand-ins for the
// symbols, not device addresses; the addresses a kernel can use come from cudaGetSymbolAddress,
// looked up once per device, with that device current, on the entry point's first call there.
namespace nuna {

static __device__ __align__(256) unsigned char g_static_shard[NUNA_STATIC_MAX_COUNT * 2];
static __device__ __align__(256) unsigned int g_static_flags[NUNA_STATIC_MAX_COUNT * 2 / (kStaticTileVec * 16) + 1];   // one per tile
static __device__ __align__(256) BarrierWords g_static_barrier;

struct StaticSetup {
    bool ready = false;
    uint4* shard = nullptr;              // device address of g_static_shard on this device
    unsigned* flags = nullptr;           // device address of g_static_flags
    BarrierWords* barrier = nullptr;     // device address of g_static_barrier
    int num_sms = 0;
};
static StaticSetup g_static_setup[kMaxDevices];
static std::mutex g_static_mutex;

// Once per device: resolve the symbols.  No allocation, and nothing is written: epoch, ticket and ready flags are zero from the
// moment the module is loaded (device variables without an initialiser), before any stream can use them.  A memset here would
// return before it is done, and would come after nobody but the legacy stream: on another one it could take back tickets that
// the call's blocks have drawn.  The shard needs no clearing (every element is written before it is read).
static int static_setup(StaticSetup** out)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return NUNA_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    StaticSetup& s = g_static_setup[dev];
    if (!s.ready) {
        void* shard = nullptr;
        void* flags = nullptr;
        void* barrier = nullptr;
        if (cudaGetSymbolAddress(&shard, g_static_shard) != cudaSuccess || !shard) return NUNA_ERR_CUDA;
        if (cudaGetSymbolAddress(&flags, g_static_flags) != cudaSuccess || !flags) return NUNA_ERR_CUDA;
        if (cudaGetSymbolAddress(&barrier, g_static_barrier) != cudaSuccess || !barrier) return NUNA_ERR_CUDA;
        if (cudaDeviceGetAttribute(&s.num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || s.num_sms < 1)
            return NUNA_ERR_CUDA;
        s.shard = static_cast<uint4*>(shard);
        s.flags = static_cast<unsigned*>(flags);
        s.barrier = static_cast<BarrierWords*>(barrier);
        s.ready = true;
    }
    *out = &s;
    return NUNA_OK;
}

// For nuna_device_status: the status latched by the allocation-free entry point on the current device
// (0 if that entry point was never used here).  A latched timeout leaves cursor and departure counter in
// an undefined state, so the control words are zeroed again; the device is idle (the caller synchronised).
static int static_status_read_and_clear(const Context* c, unsigned* out)
{
    *out = 0;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return NUNA_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    StaticSetup& s = g_static_setup[dev];
    if (!s.ready) return NUNA_OK;
    BarrierWords h;
    if (cudaMemcpy(&h, s.barrier, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return NUNA_ERR_CUDA;
    *out = h.status;
    return h.status != 0 ? rewind_barrier_words(c, s.barrier, h) : NUNA_OK;
}

}  // namespace nuna

extern "C" int nuna_allreduce_twoshot_static(const void* const* src, void* const* dst, int nranks, size_t count,
                                             int dtype, void* stream)
{
    int st = check_args(src, dst, nranks, count, count, dtype, 0u, true);
    if (st != NUNA_OK || count == 0) return st;
    if (count * elem_size(dtype) > (size_t)NUNA_STATIC_MAX_COUNT * 2) {
        fprintf(stderr, "nuna_allreduce_twoshot_static: %zu bytes per rank exceed the fixed scratch array "
                        "(NUNA_STATIC_MAX_COUNT = %d 16-bit elements, %d bytes); use nuna_allreduce_twoshot for larger "
                        "messages\n", count * elem_size(dtype), (int)NUNA_STATIC_MAX_COUNT, (int)NUNA_STATIC_MAX_COUNT * 2);
        return NUNA_ERR_TOO_LARGE;
    }
    StaticSetup* s = nullptr;
    if ((st = static_setup(&s)) != NUNA_OK) return st;
    // tiles of 4 KiB per source (the fixed flag array has one word per 4 KiB of the shard), fewer vectors for many ranks
    return launch_twoshot_flags(s->num_sms, 0, make_ptrs(src, dst, nranks), nranks, dtype, count, kStaticTileVec, kStaticTileVec,
                                s->shard, s->flags, s->barrier, 1000000000ull, (effective_flags(0u, stream) & NUNA_LAUNCH_PDL) != 0u, 0u,
                                (cudaStream_t)stream);
}

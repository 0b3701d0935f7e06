// Launching the step kernels: the per-frame kernels of gk_game.cuh, the launch
// shape, and the choice between them and the multi-frame (gk_rollout.cu) and
// work-list (gk_worklist.cu) kernels, which compile apart.
#include <atomic>
#include <map>
#include <mutex>
#include <tuple>

#include "gk_game.cuh"

namespace gk {

// the other translation units' kernels and column tables
StepKernel rollout_kernel(int lw, bool uniform, bool spawn);
int fill_rollout_columns();
WorklistKernel worklist_kernel(bool multi, bool spawn);
int fill_worklist_columns();
int launch_team(const KArgs& a, int sms, void* stream);
int fill_team_columns();

__global__ void k_copy(const uint4* __restrict__ src, uint4* __restrict__ dst, size_t n) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (; i < n; i += stride) __stcs(dst + i, __ldcs(src + i));
}

// The step kernel of a launch: lw lanes per game (8 only in multi-frame
// launches of the plain generator).  The spawn options have kernels of their
// own, since the generator with them sets the registers of a kernel that
// only calls it (compiled into the plain ones: 324 -> 359 us for 64 frames of
// 1,024 games, 240 -> 251 us per frame of the mixed batch's work list).
StepKernel step_kernel(int lw, bool multi, bool uniform, bool spawn) {
    if (multi) return rollout_kernel(lw, uniform, spawn);
    if (spawn) {
        if (lw == 32) return k_generals<false, true, 32, false>;
        return uniform ? k_generals<false, true, 16, true> : k_generals<false, true, 16, false>;
    }
    if (lw == 32) return uniform ? k_generals<false, false, 32, true> : k_generals<false, false, 32, false>;
    return uniform ? k_generals<false, false, 16, true> : k_generals<false, false, 16, false>;
}

bool has_spawn_options(const KArgs& a) { return a.spawn_dmax > 0 || a.spawn_bfs || a.castle_radius > 0; }

// Every step-kernel instantiation may take up to the per-CTA maximum of
// dynamic shared memory on the current device: set once per device, so no
// launch shape needs its own opt-in (the limit gates launches only).
int allow_max_smem() {
    static SmemLimit limit;
    static const void* fns[15];
    static std::once_flag once;
    std::call_once(once, [] {
        int n = 0;
        for (int uniform = 0; uniform < 2; ++uniform) {
            for (int lw : {32, 16}) fns[n++] = (const void*)step_kernel(lw, false, uniform, false);
            for (int lw : {32, 16, 8}) fns[n++] = (const void*)step_kernel(lw, true, uniform, false);
        }
        for (int multi = 0; multi < 2; ++multi)
            for (int lw : {32, 16}) fns[n++] = (const void*)step_kernel(lw, multi, false, true);
        fns[n++] = (const void*)step_kernel(16, false, true, true);
    });
    return limit.raise(fns, 15, 227 * 1024);
}

uint32_t bucket_geom(int npad_max, int nw_stride, int pmax) {
    return pack_geom(npad_max, nw_stride, pmax);
}

int worklist_shape(bool multi, int* cta_smem, int* ctas) {
    // three CTAs of 8 warps per SM (the register budget's limit); each takes an
    // equal share of the SM's shared memory less the per-CTA reservation
    // (the same shape with spawn options: their kernel has the same budget)
    const void* f = (const void*)worklist_kernel(multi, false);
    int dev = 0, sms = 0, smem_sm = 0, reserved = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return (int)e;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    const int want = 3;
    int bytes = ((smem_sm / want - reserved - 64) / 16) * 16;  // 64: the kernel's static item slot
    if (bytes > 227 * 1024) bytes = 227 * 1024;
    // the kernel's own static slot counts against the per-CTA limit too
    if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)) != cudaSuccess)
        return (int)e;
    if ((e = cudaFuncSetAttribute((const void*)worklist_kernel(multi, true), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  bytes)) != cudaSuccess)
        return (int)e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, 256, (size_t)bytes)) != cudaSuccess)
        return (int)e;
    if (per_sm < 1) return (int)cudaErrorInvalidConfiguration;
    *cta_smem = bytes;
    *ctas = per_sm * sms;
    return 0;
}

int launch_worklist(const KArgs& a, const WArgs& w, int cta_smem, int ctas, void* stream) {
    const cudaStream_t st = (cudaStream_t)stream;  // the counters arrive zeroed (see k_worklist)
    const bool multi = a.frames > 1 || a.action_log;
    const int grid = ctas < w.n_items ? ctas : w.n_items;
    if (grid <= 0) return 0;
    return launch_chained(worklist_kernel(multi, has_spawn_options(a)), dim3(grid), dim3(256), cta_smem, st, a, w);
}

int warp_smem_bytes(int npad_max, int pmax, int* nw_stride) {
    int nw = (npad_max + 31) / 32;
    nw = (nw + 1) & ~1;  // even: the regions stay 8-byte aligned
    if (nw_stride) *nw_stride = nw;
    const int bytes = 4 * npad_max + 4 * (nw * (pmax + 3) + vis_region_words(nw, pmax)) +
                      count_region_bytes(npad_max, pmax) + 4 * 24;
    return (bytes + 15) & ~15;  // the next group's board is copied 16 bytes at a time
}

int max_resident_ctas(int warps_per_cta, int smem_bytes, int* out) {
    cudaError_t e = (cudaError_t)allow_max_smem();
    if (e != cudaSuccess) return (int)e;
    int per_sm = 0, dev = 0, sms = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_generals<false, false, 32, false>, 32 * warps_per_cta,
                                                           smem_bytes)) != cudaSuccess)
        return (int)e;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    *out = per_sm * sms;
    return 0;
}

int init_tables() {
    static std::mutex mu;
    static bool ready[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return (int)e;
    std::lock_guard<std::mutex> lk(mu);
    if (dev >= 0 && dev < 64 && ready[dev]) return 0;
    for (int (*fill)() : {fill_columns, fill_rollout_columns, fill_worklist_columns, fill_team_columns}) {
        const int f = fill();
        if (f != 0) return f;
    }
    if (dev >= 0 && dev < 64) ready[dev] = true;
    return 0;
}

// Resident CTAs of kernel f per SM for a launch shape, from the occupancy
// calculator; cached per (kernel, threads, bytes) for the process.
int ctas_per_sm(const void* f, int threads, int smem) {
    static std::mutex mu;
    static std::map<std::tuple<const void*, int, int, int>, int> cache;
    int dev = 0;
    cudaGetDevice(&dev);
    const auto key = std::make_tuple(f, threads, smem, dev);
    {
        std::lock_guard<std::mutex> lk(mu);
        auto it = cache.find(key);
        if (it != cache.end()) return it->second;
    }
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f, threads, (size_t)smem) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    std::lock_guard<std::mutex> lk(mu);
    cache[key] = n;
    return n;
}

// Launch shape of one step launch: warps per CTA.  `fixed` > 0 is the
// caller's choice (gen_set_launch, the autotuner); otherwise the count among
// 8, 4, 2, 1 whose CTAs keep the most warps resident per SM (ties: more warps
// per CTA).  Either way, launches too small to give every SM a CTA take
// fewer warps per CTA.
int pick_warps(const void* f, int fixed, int games_per_warp, int warp_smem, int n_items, int sms) {
    int w = fixed;
    if (w <= 0) {
        int best = 0;
        w = 1;
        for (int cand : {8, 4, 2, 1}) {
            const int smem = cand * games_per_warp * warp_smem;
            if (smem > 227 * 1024) continue;
            const int warps = ctas_per_sm(f, 32 * cand, smem) * cand;
            if (warps > best) {
                best = warps;
                w = cand;
            }
        }
    }
    while (w > 1 && (n_items + games_per_warp * w - 1) / (games_per_warp * w) < sms) w >>= 1;
    return w;
}

int launch_groups(const KArgs& a, int lw, bool multi, bool spawn, int fixed_warps, int max_ctas, int sms,
                  cudaStream_t st) {
    const StepKernel f = step_kernel(lw, multi, a.uniform != 0, spawn);
    const int per_warp = 32 / lw;
    const int warps = pick_warps((const void*)f, fixed_warps, per_warp, a.warp_smem, a.n_items, sms);
    const int games_per_cta = per_warp * warps;
    const int smem = a.warp_smem * games_per_cta;
    int blocks = (a.n_items + games_per_cta - 1) / games_per_cta;
    // multi-frame launches: a grid of many waves, groups stride over any items beyond it
    if (multi && max_ctas > 0 && blocks > 64 * max_ctas) blocks = 64 * max_ctas;
    return launch_chained(f, dim3(blocks), dim3(32 * warps), smem, st, a);
}

int sm_count() {
    static std::atomic<int> count{0};
    int sms = count.load(std::memory_order_relaxed);
    if (sms == 0) {
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        sms = n > 0 ? n : 1;
        count.store(sms, std::memory_order_relaxed);
    }
    return sms;
}

// A CTA per game (gk_team.cu) while the batch is small.  Of one size class, up
// to 9 games per SM, where three warps per game still run all at once: 32
// frames of 24x24 1v1 games, against a warp per game, 85 / 122 / 162 us for
// 64 / 1,024 / 1,400 games against 127 / 142 / 184, but 188 against 185 for
// 1,536.
constexpr int kTeamGames = 9;
// Of several classes, against one launch per class on forked streams (up to
// four classes; 1v1 games of 15..30 a side, per frame: 1,024 games 8.4
// against 21.1 us, 6,144 23.9 against 29.4, 8,192 31.0 against 32.2, 12,288
// 46.9 against 39.4) or against the work list (mixed games of 20..40 a side:
// 512 games 12.9 against 21.4 us, 4,096 37.7 against 43.0, 6,144 51.7 against
// 46.8).
constexpr int kTeamGamesFewClasses = 40, kTeamGamesManyClasses = 27;
bool team_batch(const KArgs& a, int per_sm, int sms) {
    return a.op == OP_STEP && a.do_outputs && a.lane_groups == 0 && a.n_items <= per_sm * sms;
}
int launch_small(const KArgs& a, int classes, void* stream, bool* taken) {
    const int sms = sm_count();
    *taken = team_batch(a, classes > 4 ? kTeamGamesManyClasses : kTeamGamesFewClasses, sms);
    return *taken ? launch_team(a, sms, stream) : 0;
}

int launch_step(const KArgs& a, int warps_per_cta, int max_ctas, void* stream) {
    if (a.n_items <= 0) return 0;

    const bool multi = a.frames > 1 || a.action_log;
    const cudaStream_t st = (cudaStream_t)stream;
    {
        const int e = allow_max_smem();
        if (e != 0) return e;
    }
    const int sms = sm_count();
    if (team_batch(a, kTeamGames, sms)) return launch_team(a, sms, stream);
    // several games per warp for small two-player boards, once the batch is
    // large enough: below it a warp per game is faster (measured on 24x24 1v1: 1,024 games per frame 98 against 87 M
    // frames/s, resident 194 against 122 M; pairs win from 2,048 games per
    // frame and 4,096 resident)
    const bool large = a.n_items >= (multi ? 24 : 12) * sms;
    const bool small = a.pmax <= kPairMaxPlayers && (a.lane_groups == 2 || (a.lane_groups == 0 && large));
    const int wcap = warps_per_cta > 0 ? warps_per_cta : 1;  // the fixed shape must fit too
    int per_warp = 1;
    const bool spawn = has_spawn_options(a);
    // four per warp from 32 games per SM on (16 frames of 24x24 1v1 games:
    // 4,096 games 137 us with four, 127 us with two; 6,144 166 and 172; 8,192
    // 199 and 238)
    if (small && multi && !spawn && a.npad_max <= kQuadMaxCells && a.n_items >= 32 * sms && 4 * wcap * a.warp_smem <= 227 * 1024)
        per_warp = 4;
    else if (small && a.npad_max <= kPairMaxCells && 2 * wcap * a.warp_smem <= 227 * 1024)
        per_warp = 2;
    return launch_groups(a, 32 / per_warp, multi, spawn, warps_per_cta, max_ctas, sms, st);
}

int launch_copy(const void* src, void* dst, size_t n16, int blocks, void* stream) {
    k_copy<<<blocks, 256, 0, (cudaStream_t)stream>>>(reinterpret_cast<const uint4*>(src),
                                                      reinterpret_cast<uint4*>(dst), n16);
    return (int)cudaGetLastError();
}

}  // namespace gk

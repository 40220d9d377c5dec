// ci_gen.cuh -- the generation kernel template and its launch-shape
// dispatch, instantiated per strategy source in ci_gen_<source>.cu so the
// instantiations compile in parallel.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <mutex>

#include "ci_device.cuh"
#include "ci_tune.h"

namespace ci {

// One warp per group of 32 lanes.  Blocks of consecutive groups are handed to
// the SMs in order as they fall free: the SMs do not run at the same speed (two
// dies, one memory each), so a fixed share per SM ends with the slowest, and
// stores in address order reach 7.6 TB/s where the same stores from a
// persistent grid reached 6.5 (1 GiB, nothing else in the kernel).  Measured
// against a persistent grid when it was brought in: 2^20 x 1024 consumed 610
// instead of 690 us, 2^20 x 256 written 175 instead of 199 us.  W warps per
// block; a state of one wave takes smaller blocks as far as the SMs' 32 blocks
// each hold it, since idle warps of larger ones leave schedulers unused (2^17 x
// 1024 digested: 82 us, 92 with one or two of a block's four warps at work;
// 50001 x 1001 XORshift 53, 57 then).
// The squaring sources (kHeavy) nearly fill a scheduler with each warp: one-warp
// blocks up to two warps per scheduler (10^4 x 1024 of Algorithm 5 as printed:
// 94 us, 139 spread), beyond them a wave is spread over all resident blocks so
// that every SM gets its share (2^16 x 1024: 261 us, 270 in one-warp blocks).
constexpr uint64_t kNeverSpread = 1ull << 32;
struct GenGrid {
    unsigned grid, warps;  // blocks; warps per block
    uint32_t in_order;     // the same if blocks hold consecutive groups, else 0: warp w of block b takes w * grid + b
};
// `spread_from`: one-wave states of more groups per SM are spread.
inline GenGrid gen_grid(uint64_t groups, int W, uint64_t resident_blocks, uint64_t spread_from) {
    const uint64_t sms = (uint64_t)sm_count();
    unsigned warps = (unsigned)W;
    if (groups <= resident_blocks * W) {
        if (groups > spread_from * sms)
            return {(unsigned)(groups < resident_blocks ? groups : resident_blocks), warps, 0u};
        const uint64_t w = (groups + 32 * sms - 1) / (32 * sms);
        if (w < (uint64_t)W) warps = (unsigned)w;
    }
    return {(unsigned)((groups + warps - 1) / warps), warps, warps};
}
__device__ __forceinline__ uint64_t warp_group(uint32_t in_order) {
    const uint64_t w = threadIdx.x >> 5;
    return in_order ? (uint64_t)blockIdx.x * in_order + w : w * gridDim.x + blockIdx.x;
}
template <class Kernel>
int resident_blocks_per_sm(Kernel kern, int threads, size_t smem) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, smem) != cudaSuccess || n <= 0) n = 1;
    return n;
}

// Written sinks stage a 32 x KT tile per warp in dynamic shared memory.
template <class Src, int SINK, class TC>
constexpr int kTileVecs = SINK >= dev::SINK_QC ? 0 : SINK == dev::SINK_SCALAR ? dev::kScalarTile<Src> : TC::KT * 8;
template <class Src, int SINK, int W, class TC>
__global__ void __launch_bounds__(W * 32) k_generate(DevState st, uint64_t n, uint32_t in_order, uint32_t *out,
                                                     uint64_t *counts) {
    extern __shared__ uint4 dyn_tiles[];
    const int w = threadIdx.x >> 5;
    uint4 *tile = dyn_tiles + w * kTileVecs<Src, SINK, TC>;
    const uint64_t g = warp_group(in_order);
    if (g < st.P / 32) dev::warp_task<Src, SINK, TC>(st, g, n, out, n, 0, counts, tile);
}

// Written sink through TMA bulk tensor stores (xor sources, store policy 2).
template <class Src, int W>
__global__ void __launch_bounds__(W * 32) k_generate_tma(DevState st, uint64_t n, uint32_t in_order,
                                                         const __grid_constant__ CUtensorMap map) {
    extern __shared__ uint4 tma_tiles[];
    // the 128-byte swizzle needs 1024-byte aligned tiles: round the base up
    // (the launch allocates 1 KB of slack)
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(tma_tiles);
    uint4 *base = reinterpret_cast<uint4 *>(reinterpret_cast<char *>(tma_tiles) + ((1024u - (sbase & 1023u)) & 1023u));
    const int w = threadIdx.x >> 5;
    uint4 *tiles = base + w * 256 * dev::kTmaTiles;
    const uint64_t g = warp_group(in_order);
    if (g < st.P / 32) dev::warp_task_tma<Src>(st, g, n, &map, tiles);
}

// Short rows as one bulk store per warp group (xor sources): one warp per
// block, as many blocks per SM as their 128 n bytes of staging allow.
template <class Src>
__global__ void __launch_bounds__(32) k_generate_span(DevState st, uint32_t n, uint32_t *out) {
    extern __shared__ __align__(128) uint32_t span_stage[];
    dev::warp_task_span<Src>(st, blockIdx.x, n, out, span_stage);
}

// Which written rows leave as spans: out 16-byte aligned, and rows that are
// not whole 32-byte sectors (the others' TMA tiles write whole sectors) up to
// the length where too few warps fit an SM beside their staging, or shorter
// than a TMA tile.  400 MB in rows of n, span against the next best form: n =
// 36 83 us / 95 TMA, 100 70 / 117, 249 84 / 92 line-staged, 260 95 / 117 TMA,
// 290 96 / 95 line-staged, 333 113 / 90; n = 200 81 / 69 TMA, 144 80 / 69.
constexpr uint64_t kSpanMax = 280;
inline bool span_rows(uint64_t n, const uint32_t *out) {
    return n <= kSpanMax && (n % 8 != 0 || n < 32) && (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
}

template <class Src>
static cudaError_t launch_gen_span(const DevState &st, uint64_t n, uint32_t *out, cudaStream_t stream) {
    auto kern = k_generate_span<Src>;
    static_assert(128 * kSpanMax <= 48 * 1024, "staging within the default shared-memory limit");
    static std::once_flag once;  // a hint: as many warps per SM as the shared memory holds
    std::call_once(once, [&] { cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100); });
    kern<<<(unsigned)(st.P / 32), 32, 128 * n, stream>>>(st, (uint32_t)n, out);
    return cudaGetLastError();
}

// Lets `kern` use `smem` bytes of dynamic shared memory on the current device,
// once per device (`done`: a bit per device ordinal, the kernel's own).
template <class Kernel>
static void allow_smem(Kernel kern, size_t smem, std::atomic<uint64_t> &done) {
    if (smem <= 48 * 1024) return;
    int dev = 0;
    const bool known = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64;
    if (known && (done.load(std::memory_order_relaxed) >> dev & 1u)) return;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (known) done.fetch_or(1ull << dev, std::memory_order_relaxed);
}

// Tensor map over out[rows][cols] (uint32, row stride cols words) with a
// 32 x 32 box and the 128-byte swizzle; false when TMA cannot be used (then
// the caller takes the 16-byte-store path).
bool make_out_tensor_map(CUtensorMap *map, uint32_t *out, uint64_t rows, uint64_t cols);

template <class Src, int W>
static cudaError_t launch_gen_tma(const DevState &st, uint64_t n, uint32_t *out, cudaStream_t stream, bool *used) {
    *used = false;
    CUtensorMap map;
    if (!make_out_tensor_map(&map, out, st.S, n)) return cudaSuccess;
    auto kern = k_generate_tma<Src, W>;
    // + slack for the 1024-byte alignment of the base
    auto smem = [](unsigned warps) { return (size_t)warps * dev::kTmaTiles * 4096 + 1024; };
    static std::atomic<uint64_t> smem_set{0};
    allow_smem(kern, smem(W), smem_set);
    static const int per_sm = resident_blocks_per_sm(kern, W * 32, smem(W));
    const GenGrid gg = gen_grid(st.P / 32, W, (uint64_t)sm_count() * per_sm, kNeverSpread);
    *used = true;
    kern<<<gg.grid, gg.warps * 32, smem(gg.warps), stream>>>(st, n, gg.in_order, map);
    return cudaGetLastError();
}

template <class Src, int SINK, int W, class TC>
static cudaError_t launch_gen_t(const DevState &st, uint64_t n, uint32_t *out, uint64_t *counts,
                                cudaStream_t stream) {
    auto kern = k_generate<Src, SINK, W, TC>;
    constexpr size_t tile = kTileVecs<Src, SINK, TC> * sizeof(uint4);
    static std::atomic<uint64_t> smem_set{0};
    allow_smem(kern, W * tile, smem_set);
    static const int per_sm = resident_blocks_per_sm(kern, W * 32, W * tile);
    // short written calls of the squaring sources are over before one-warp blocks
    // pay (30000 x 12 BBS: 13.7 us, 12.7 spread)
    const uint64_t spread_from = !Src::kHeavy ? kNeverSpread : SINK <= dev::SINK_SCALAR && n < 32 ? 0 : 8;
    const GenGrid gg = gen_grid(st.P / 32, W, (uint64_t)sm_count() * per_sm, spread_from);
    kern<<<gg.grid, gg.warps * 32, gg.warps * tile, stream>>>(st, n, gg.in_order, out, counts);
    return cudaGetLastError();
}

// Small calls of short rows leave by 16-byte stores although the policy is TMA:
// they are as fast, and the tensor map costs the host 0.3 us (1000 x 64: 7.6
// us against 7.9; 32768 x 128 8.3 against 7.8, 1000 x 200 10.3 against 7.6).
inline bool tma_rows(uint64_t S, uint64_t n) { return n > 128 || S * n >= 1ull << 21; }

template <class Src, int SINK, int W>
static cudaError_t gen_tile(const TuneChoice &c, const DevState &st, uint64_t n, uint32_t *out, uint64_t *counts,
                            cudaStream_t stream) {
    if constexpr (SINK <= dev::SINK_SCALAR && !Src::kHeavy)
        if (span_rows(n, out)) return launch_gen_span<Src>(st, n, out, stream);
    if constexpr (SINK == dev::SINK_V4 && !Src::kHeavy) {
        if (c.cache_policy == 2 && tma_rows(st.S, n)) {
            bool used = false;
            const cudaError_t e = launch_gen_tma<Src, W>(st, n, out, stream, &used);
            if (used || e != cudaSuccess) return e;
            return launch_gen_t<Src, SINK, W, dev::TileCfg<32, 0>>(st, n, out, counts, stream);
        }
        if (c.tile_depth == 64)
            return c.cache_policy ? launch_gen_t<Src, SINK, W, dev::TileCfg<64, 1>>(st, n, out, counts, stream)
                                  : launch_gen_t<Src, SINK, W, dev::TileCfg<64, 0>>(st, n, out, counts, stream);
        return c.cache_policy ? launch_gen_t<Src, SINK, W, dev::TileCfg<32, 1>>(st, n, out, counts, stream)
                              : launch_gen_t<Src, SINK, W, dev::TileCfg<32, 0>>(st, n, out, counts, stream);
    } else if constexpr (SINK == dev::SINK_V4) {
        return c.cache_policy ? launch_gen_t<Src, SINK, W, dev::TileCfg<32, 1>>(st, n, out, counts, stream)
                              : launch_gen_t<Src, SINK, W, dev::TileCfg<32, 0>>(st, n, out, counts, stream);
    } else {
        return launch_gen_t<Src, SINK, W, dev::TileDefault>(st, n, out, counts, stream);
    }
}

template <class Src, int SINK>
static cudaError_t gen_warps(const TuneChoice &c, const DevState &st, uint64_t n, uint32_t *out, uint64_t *counts,
                             cudaStream_t stream) {
    switch (c.warps_per_block) {
        case 4:
            return gen_tile<Src, SINK, 4>(c, st, n, out, counts, stream);
        case 16:
            return gen_tile<Src, SINK, 16>(c, st, n, out, counts, stream);
        default:
            return gen_tile<Src, SINK, 8>(c, st, n, out, counts, stream);
    }
}

template <class Src>
static cudaError_t gen_source(int sink, const TuneChoice &c, const DevState &st, uint64_t n, uint32_t *out,
                              uint64_t *counts, cudaStream_t stream) {
    switch (sink) {
        case dev::SINK_V4:
            return gen_warps<Src, dev::SINK_V4>(c, st, n, out, counts, stream);
        case dev::SINK_SCALAR:
            return gen_warps<Src, dev::SINK_SCALAR>(c, st, n, out, counts, stream);
        case dev::SINK_QC:
            return gen_warps<Src, dev::SINK_QC>(c, st, n, out, counts, stream);
        default:
            return gen_warps<Src, dev::SINK_DIGEST>(c, st, n, out, counts, stream);
    }
}

}  // namespace ci

// spread.cuh -- launch shapes of the persistent kernels.  Like
// launchers_common.cuh it is included inside an anonymous namespace, after R
// (the spin precision) is defined.
#pragma once

// Blocks of a persistent launch: resident blocks per SM x SMs (device 0 of
// the process is assumed representative; computed once per kernel).
template <typename K>
uint32_t resident_blocks(K kernel, int threads = kBlock) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0);
    if (per_sm < 1) per_sm = 1;
    return uint32_t(sms) * uint32_t(per_sm);
}

// Launch shape of `warps` warps of work for a kernel that keeps cap blocks of
// `threads` threads resident.  A launch that fills the GPU takes them all.  A
// smaller FP64 launch takes blocks of one or two warps, which the hardware
// deals out over all SMs: an FP64 warp instruction holds the SM's FP64 pipe
// for many cycles, and in blocks of 256 threads the 64 warps of a 16^3 colour
// pass sat on 8 SMs with that pipe 70% busy (25 us a pass, 55 us a sweep; 34
// us a sweep spread out).  Two warps a block above 8 warps per SM keep the SM
// below its block limit.  FP32 launches stay in full blocks: spread out, a
// 12^3 lattice swept 6% slower, a 90 x 75 x 61 one 3% slower and a 64^3 one no
// faster (they wait on memory latency and on the launch, not on a pipe).
struct Spread {
    uint32_t blocks;
    int threads;
};

uint32_t sm_count() {
    static const uint32_t sms = [] {
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return uint32_t(n > 0 ? n : 1);
    }();
    return sms;
}

Spread spread_warps(uint32_t warps, uint32_t cap, int threads = kBlock) {
    const uint32_t sms = sm_count();
    const uint32_t wpb = uint32_t(threads / 32);
    if (warps == 0) warps = 1;
    if (warps >= cap * wpb) return Spread{cap, threads};
    if (!kIsF64<R>) return Spread{(warps + wpb - 1) / wpb, threads};
    if (warps <= 8 * sms) return Spread{warps, 32};
    return Spread{(warps + 1) / 2, 64};
}

// Consecutive tiles a warp of a grid-stride kernel takes per step (an instance
// each): `most` (2, 4 or 8), or 2 or 1 when the launch would otherwise leave
// resident warps without work (a lone 64^3 lattice has 2048 pair tiles for
// 2432 warps, and 4 a step kept only 512 of them busy; a 16^3 one walked its
// 32 tiles on 8 warps).  Constrained sweeps alone, half of them measured, 4
// tiles a step against this rule: 16^3 36.8 -> 24.6 us, 64^3 43.5 -> 33.9 us,
// 256^3 unchanged; 16^3 in FP64, spread over the SMs as well, 275 -> 55.9 us.
int tiles_per_step(uint32_t ntiles, uint32_t warps, int most) {
    const uint32_t even = ntiles / warps;
    if (even >= uint32_t(most)) return most;
    return even >= 2 ? 2 : 1;
}

// Launch with programmatic serialisation (chain): the kernel's blocks may start
// while the previous launch drains; it waits for it (griddepcontrol.wait) before
// it touches any memory.
template <typename... K, typename... A>
cudaError_t launch_chained_if(bool chain, void (*kernel)(K...), uint32_t blocks, int threads, cudaStream_t s, A... a) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(uint32_t(threads));
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = chain ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, a...);
}

// Whether a pass that leaves room on the GPU is chained.  FP64: only where it
// and the next fit the SMs side by side; blocks dealt out while the SMs are busy
// pile up on some, and with them FP64 work (32^3: 39 -> 66 us a sweep).
bool chain_small(const Spread& sp, uint32_t cap) {
    return kIsF64<R> ? 2 * sp.blocks <= sm_count() : sp.blocks < cap;
}

template <typename... K, typename... A>
cudaError_t launch_chained(void (*kernel)(K...), uint32_t blocks, int threads, cudaStream_t s, A... a) {
    return launch_chained_if(true, kernel, blocks, threads, s, a...);
}

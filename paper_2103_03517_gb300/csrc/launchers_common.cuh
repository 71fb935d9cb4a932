// launchers_common.cuh -- host launchers shared by both precisions.  It is
// included inside `namespace mcgb { namespace { ... } }` of kernels_f32.cu
// and kernels_f64.cu, after each has defined R (the spin precision), V
// (sites per thread of a site tile), MINB (resident blocks per SM of the
// general colour pass) and kFieldChunk (tiles per grid-stride step of the
// neighbour-field kernel).
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

Spread spread_warps(uint32_t warps, uint32_t cap, int threads = kBlock) {
    static const uint32_t sms = [] {
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return uint32_t(n > 0 ? n : 1);
    }();
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

template <int MEASURE>
void colour_pass_t(const GroupArgs& g, uint32_t ntiles, const R* cone, int colour, cudaStream_t s) {
    static const uint32_t cap = resident_blocks(colour_pass_kernel<R, V, MINB, MEASURE>);
    const Spread sp = spread_warps(ntiles, cap);
    colour_pass_kernel<R, V, MINB, MEASURE><<<sp.blocks, sp.threads, 0, s>>>(g, ntiles, cone, colour);
}

// measure: 0 none, 1 magnetisation and energies, 2 also torques
void colour_pass(const GroupArgs& g, uint32_t ntiles, const void* cone, int colour, int measure, cudaStream_t s) {
    const R* c = static_cast<const R*>(cone);
    if (measure >= 2) colour_pass_t<2>(g, ntiles, c, colour, s);
    else if (measure == 1) colour_pass_t<1>(g, ntiles, c, colour, s);
    else colour_pass_t<0>(g, ntiles, c, colour, s);
}

void sweep_end(const GroupArgs& g, cudaStream_t s) {
    sweep_end_kernel<R><<<(g.n + kBlock - 1) / kBlock, kBlock, 0, s>>>(g);
}

template <int C>
void pair_field_t(const GroupArgs& g, uint32_t ntiles, int colour, uint32_t cap, cudaStream_t s) {
    const Spread sp = spread_warps((ntiles + C - 1) / C, cap);
    pair_field_kernel<R, V, C><<<sp.blocks, sp.threads, 0, s>>>(g, ntiles, colour);
}

// launch shapes: at most {default, 8, 2} tiles per grid-stride step
void pair_field(const GroupArgs& g, uint32_t ntiles, int colour, int shape, cudaStream_t s) {
    static const uint32_t cap = resident_blocks(pair_field_kernel<R, V, kFieldChunk>);
    const int c = tiles_per_step(ntiles, cap * (kBlock / 32), shape == 1 ? 8 : shape == 2 ? 2 : kFieldChunk);
    if (c == 8) pair_field_t<8>(g, ntiles, colour, cap, s);
    else if (c == 4) pair_field_t<4>(g, ntiles, colour, cap, s);
    else if (c == 2) pair_field_t<2>(g, ntiles, colour, cap, s);
    else pair_field_t<1>(g, ntiles, colour, cap, s);
}

void ml_reset(const GroupArgs& g, cudaStream_t s) {
    ml_reset_kernel<R><<<(g.n + kBlock - 1) / kBlock, kBlock, 0, s>>>(g);
}

void mlong(const GroupArgs& g, uint32_t ntiles, cudaStream_t s) {
    static const uint32_t cap = resident_blocks(mlong_kernel<R, V>);
    const Spread sp = spread_warps(ntiles, cap);
    mlong_kernel<R, V><<<sp.blocks, sp.threads, 0, s>>>(g, ntiles);
}

void measure(const GroupArgs& g, uint32_t ntiles, cudaStream_t s) {
    static const uint32_t cap = resident_blocks(measure_kernel<R, V>);
    const Spread sp = spread_warps(ntiles, cap);
    measure_kernel<R, V><<<sp.blocks, sp.threads, 0, s>>>(g, ntiles);
}

// Entry bound of the crystal kernels: the smallest instance that holds nb.
template <template <int> class F, typename... A>
void by_entries(int nb, A... a) {
    if (nb <= 8) F<8>::run(a...);
    else if (nb <= 12) F<12>::run(a...);
    else if (nb <= 14) F<14>::run(a...);
    else if (nb <= 18) F<18>::run(a...);
    else F<kXtalMaxNb>::run(a...);
}

template <int NB>
struct XtalPass {
    static void run(LatDev* L, uint32_t ntiles, const void* cone, int sub, int colour, int finalize, cudaStream_t s) {
        static const uint32_t cap = resident_blocks(xtal_pass_kernel<R, NB>);
        const Spread sp = spread_warps(ntiles, cap);
        xtal_pass_kernel<R, NB><<<sp.blocks, sp.threads, 0, s>>>(L, ntiles, static_cast<const R*>(cone), sub, colour,
                                                                 finalize);
    }
};

template <int NB>
struct XtalSample {
    template <int LEVEL>
    static void go(LatDev* L, uint32_t ntiles, uint32_t tiles_per_subset, cudaStream_t s) {
        static const uint32_t cap = resident_blocks(xtal_sample_kernel<R, NB, LEVEL>);
        const Spread sp = spread_warps(ntiles, cap);
        xtal_sample_kernel<R, NB, LEVEL><<<sp.blocks, sp.threads, 0, s>>>(L, ntiles, tiles_per_subset);
    }
    // level 2: with the torque sums
    static void run(LatDev* L, uint32_t ntiles, uint32_t tiles_per_subset, int level, cudaStream_t s) {
        if (level >= 2) go<2>(L, ntiles, tiles_per_subset, s);
        else go<1>(L, ntiles, tiles_per_subset, s);
    }
};

template <int NB>
struct XtalField {
    static void run(LatDev* L, uint32_t ntiles, int sub, int colour, cudaStream_t s) {
        static const uint32_t cap = resident_blocks(xtal_field_kernel<R, NB>);
        const Spread sp = spread_warps(ntiles, cap);
        xtal_field_kernel<R, NB><<<sp.blocks, sp.threads, 0, s>>>(L, ntiles, sub, colour);
    }
};

void xtal_field_launch(LatDev* L, uint32_t ntiles, int sub, int colour, int nb, cudaStream_t s) {
    by_entries<XtalField>(nb, L, ntiles, sub, colour, s);
}

void xtal_pass(LatDev* L, uint32_t ntiles, const void* cone, int sub, int colour, int finalize, int nb,
               cudaStream_t s) {
    by_entries<XtalPass>(nb, L, ntiles, cone, sub, colour, finalize, s);
}

void xtal_sample(LatDev* L, uint32_t ntiles, uint32_t tiles_per_subset, int nb, int level, cudaStream_t s) {
    by_entries<XtalSample>(nb, L, ntiles, tiles_per_subset, level, s);
}

void grain_sample(LatDev* L, uint32_t ntiles, int n_grains, cudaStream_t s) {
    static const uint32_t cap = resident_blocks(grain_sum_kernel<R, V>);
    const Spread sp = spread_warps(ntiles, cap);
    grain_sum_kernel<R, V><<<sp.blocks, sp.threads, 0, s>>>(L, ntiles);
    grain_finish_kernel<R><<<(n_grains + kBlock) / kBlock, kBlock, 0, s>>>(L);
}

void profile(LatDev* d, uint32_t Lh, uint32_t rows, cudaStream_t s) {
    const uint32_t threads = Lh * ((rows + 31) / 32);
    profile_kernel<R><<<(threads + kBlock - 1) / kBlock, kBlock, 0, s>>>(d);
}

// launchers_common.cuh -- host launchers shared by both precisions.  It is
// included inside `namespace mcgb { namespace { ... } }` of kernels_f32.cu
// and kernels_f64.cu, after each has defined R (the spin precision), V
// (sites per thread of a site tile), MINB (resident blocks per SM of the
// general colour pass) and kFieldChunk (tiles per grid-stride step of the
// neighbour-field kernel).
#pragma once

#include "spread.cuh"

// Lattices up to which a launch that forms samples, a block per lattice, is chained
// as it is: blocks dealt out while the SMs are busy pile up on some, and with
// them their FP64 chains.  Above it, sweep_close takes blocks of kCloseThreads
// threads, all but one warp idle, of which an SM holds four, and sample_close is
// not chained.  A measured sweep by itself, us, one warp chained / one warp not
// chained / spread blocks chained: 40 x 24^3 40 / 29.5 / 26.6, 8 x 32^3 18.5 /
// 20.0 / -, 32 lattices of 16^3 ... 128^3 211 / 209 / 206.
constexpr int kChainedSamples = 16;

// The end of a sweep after its black pass (sweep_close_kernel).
cudaError_t sweep_close(const GroupArgs& g, bool measure, bool now, cudaStream_t s) {
    const int threads = measure && now && g.n > kChainedSamples ? kCloseThreads : 32;
    return launch_chained(sweep_close_kernel<R>, uint32_t(g.n), threads, s, g, measure ? (now ? 2 : 1) : 0);
}

template <int MEASURE>
void colour_pass_t(const GroupArgs& g, uint32_t ntiles, const R* cone, int colour, bool now, cudaStream_t s) {
    static const uint32_t cap = resident_blocks(colour_pass_kernel<R, V, MINB, MEASURE>);
    const Spread sp = spread_warps(ntiles, cap);
    const bool full = sp.threads == kBlock;  // FP64: the launch fills the SMs (64^3: 133 -> 127 us a sweep)
    launch_chained_if(!kIsF64<R> || full || chain_small(sp, cap), colour_pass_kernel<R, V, MINB, MEASURE>, sp.blocks, sp.threads, s, g, ntiles, cone, colour);
    if (colour == 1) sweep_close(g, MEASURE > 0, now, s);
}

// measure: 0 none, 1 magnetisation and energies, 2 also torques
void colour_pass(const GroupArgs& g, uint32_t ntiles, const void* cone, int colour, int measure, bool now,
                 cudaStream_t s) {
    const R* c = static_cast<const R*>(cone);
    if (measure >= 2) colour_pass_t<2>(g, ntiles, c, colour, now, s);
    else if (measure == 1) colour_pass_t<1>(g, ntiles, c, colour, now, s);
    else colour_pass_t<0>(g, ntiles, c, colour, now, s);
}

void sample_close(const GroupArgs& g, cudaStream_t s) {
    launch_chained_if(g.n <= kChainedSamples, sample_close_kernel<R>, uint32_t(g.n), 32 * kSampleRecords, s, g);
}

void sweep_end(const GroupArgs& g, cudaStream_t s) {
    launch_chained(sweep_end_kernel<R>, uint32_t(g.n + kBlock - 1) / kBlock, kBlock, s, g);
}

// The constrained sweeps' launches are chained where they do not fill the GPU
// (8^3 ... 32^3 alone 10% faster a sweep); a full one's blocks, started early,
// only take room from the launch that they wait for (80 x 64^3 1.2% slower).
template <int C>
void pair_field_t(const GroupArgs& g, uint32_t ntiles, int colour, uint32_t cap, cudaStream_t s) {
    const Spread sp = spread_warps((ntiles + C - 1) / C, cap);
    launch_chained_if(chain_small(sp, cap), pair_field_kernel<R, V, C>, sp.blocks, sp.threads, s, g, ntiles, colour);
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

void init_spins(const LatParams& p, int wall, const double v[3], cudaStream_t s) {
    static const uint32_t cap = resident_blocks(init_spins_kernel<R>);
    const uint32_t want = (p.stride + kBlock - 1) / kBlock;
    init_spins_kernel<R><<<want < cap ? want : cap, kBlock, 0, s>>>(p, wall, V3<R>{R(v[0]), R(v[1]), R(v[2])});
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

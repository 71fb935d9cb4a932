// kernels_f32.cu -- float instances of the libmc kernels and their launchers.
// FP32 spins and energies (fast intrinsics: rsqrtf, __expf, __fdividef);
// FP64 for the sample, torque and M_L bookkeeping.
#ifndef MC_MINB_F32
#define MC_MINB_F32 3
#endif
#ifndef MC_MINB_PAIR_F32
#define MC_MINB_PAIR_F32 3
#endif
#ifndef MC_PAIR_CHUNK
#define MC_PAIR_CHUNK 4
#endif
#ifndef MC_PAIR_CHUNK_LEAD
#define MC_PAIR_CHUNK_LEAD 4
#endif
#include <algorithm>

#include "kernels.h"
#include "pass_impl.cuh"
#include "row_pass.cuh"
#include "wave_pass.cuh"
#include "resident_pass.cuh"

namespace mcgb {
namespace {

using R = float;
constexpr int MINB = MC_MINB_F32;  // minimum resident blocks per SM of the colour pass
// The same for the row kernel with faces (GEN 1): three blocks without a sample,
// two with one, whose sums would spill 160 to 380 bytes a thread at 80 registers.
constexpr int MINB_FACES = 3, MINB_FACES_M = 2;
// With film tables (GEN 2) two blocks: at three an unmeasured pass spills too,
// and most sizes lose.  Unmeasured us a sweep, two / three blocks / three with the
// warps in turn and a tile's tables read one tile ahead: 128 x 128 x 8 9.5 /
// 11.7 / 12.2, 256 x 256 x 8 13.6 / 17.6 / 18.1, 512 x 512 x 8 32.7 / 35.5 /
// 36.6, 500 x 500 x 20 66.8 / 74.6 / 79.9, 1024 x 1024 x 15 224 / 237 / 234
// (measured 256 / 263 / 280); 768 x 768 x 24 208 / 201 / 201 (236 / 233 / 249).
constexpr int MINB_FILM = 2;
constexpr int MINB_PAIR = MC_MINB_PAIR_F32;  // the same for the pair pass
constexpr int MINB_PAIR_LEAD = 2;            // the same for the pair pass in site order
constexpr int kPairChunk = MC_PAIR_CHUNK;    // consecutive pair tiles per grid-stride step
constexpr int kPairChunkLead = MC_PAIR_CHUNK_LEAD;  // the same in site order
constexpr int kFieldChunk = 4;               // the same for the neighbour-field kernel
constexpr int V = kSitesPerThreadF32;

#include "launchers_common.cuh"

template <int B, int MEASURE, int GEN, int LAW, int TURNS = 0>
cudaError_t row_pass_t(const GroupArgs& g, uint32_t ntiles, const R* cone, int colour, bool now, cudaStream_t s) {
    static const uint32_t cap = resident_blocks(row_pass_kernel<B, MEASURE, GEN, 1, LAW, TURNS>);
    const Spread sp = spread_warps(ntiles, cap);
    const cudaError_t e =
        launch_chained(row_pass_kernel<B, MEASURE, GEN, 1, LAW, TURNS>, sp.blocks, sp.threads, s, g, ntiles, cone, colour);
    if (e != cudaSuccess || colour != 1) return e;  // the sweep's end
    return sweep_close(g, MEASURE > 0, now, s);
}

// launch shape 0: the default blocks per SM of the instance (B0 of a pass
// without a sample, B0M of one with it); 1: the other candidate (B1, B1M)
template <int GEN, int B0, int B0M, int B1, int B1M, int LAW, int TURNS>
cudaError_t row_pass_s(const GroupArgs& g, uint32_t ntiles, const R* c, int colour, int measure, int shape,
                       bool now, cudaStream_t s) {
    if constexpr (!TURNS) {
        if (shape == 1) {
            if (measure >= 2) return row_pass_t<B1M, 2, GEN, LAW>(g, ntiles, c, colour, now, s);
            if (measure == 1) return row_pass_t<B1M, 1, GEN, LAW>(g, ntiles, c, colour, now, s);
            return row_pass_t<B1, 0, GEN, LAW>(g, ntiles, c, colour, now, s);
        }
    }
    if (measure >= 2) return row_pass_t<B0M, 2, GEN, LAW, TURNS>(g, ntiles, c, colour, now, s);
    if (measure == 1) return row_pass_t<B0M, 1, GEN, LAW, TURNS>(g, ntiles, c, colour, now, s);
    return row_pass_t<B0, 0, GEN, LAW, TURNS>(g, ntiles, c, colour, now, s);
}

template <int LAW>
cudaError_t row_pass_l(const GroupArgs& g, uint32_t ntiles, const R* c, int colour, int measure, int gen, int shape,
                       bool turns, bool now, cudaStream_t s) {
    const bool t = turns && shape == 0;
    if (gen == 2)
        return row_pass_s<2, MINB_FILM, MINB_FILM, MINB_FILM + 1, MINB_FILM, LAW, 0>(g, ntiles, c, colour, measure, shape, now, s);
    if (gen == 1) {
        if (t) return row_pass_s<1, MINB_FACES, MINB_FACES_M, 2, 2, LAW, 1>(g, ntiles, c, colour, measure, shape, now, s);
        return row_pass_s<1, MINB_FACES, MINB_FACES_M, 2, 2, LAW, 0>(g, ntiles, c, colour, measure, shape, now, s);
    }
    if (t) return row_pass_s<0, MINB, MINB, MINB - 1, MINB - 1, LAW, 1>(g, ntiles, c, colour, measure, shape, now, s);
    return row_pass_s<0, MINB, MINB, MINB - 1, MINB - 1, LAW, 0>(g, ntiles, c, colour, measure, shape, now, s);
}

cudaError_t row_pass(const GroupArgs& g, uint32_t ntiles, const void* cone, int colour, int measure, int law, int gen,
                     int shape, bool turns, bool now, cudaStream_t s) {
    const R* c = static_cast<const R*>(cone);
    if (law) return row_pass_l<1>(g, ntiles, c, colour, measure, gen, shape, turns, now, s);
    return row_pass_l<0>(g, ntiles, c, colour, measure, gen, shape, turns, now, s);
}

template <int C>
void row_field_t(const GroupArgs& g, uint32_t ntiles, int colour, uint32_t cap, cudaStream_t s) {
    const Spread sp = spread_warps((ntiles + C - 1) / C, cap);
    launch_chained_if(chain_small(sp, cap), row_field_kernel<C>, sp.blocks, sp.threads, s, g, ntiles, colour);
}

// launch shapes as for pair_field
void row_field(const GroupArgs& g, uint32_t ntiles, int colour, int shape, cudaStream_t s) {
    static const uint32_t cap = resident_blocks(row_field_kernel<kFieldChunk>);
    const int c = tiles_per_step(ntiles, cap * (kBlock / 32), shape == 1 ? 8 : shape == 2 ? 2 : kFieldChunk);
    if (c == 8) row_field_t<8>(g, ntiles, colour, cap, s);
    else if (c == 4) row_field_t<4>(g, ntiles, colour, cap, s);
    else if (c == 2) row_field_t<2>(g, ntiles, colour, cap, s);
    else row_field_t<1>(g, ntiles, colour, cap, s);
}

// the all-periodic instance samples red sites first and stores their field
// (the next constrained sweep's red field); the other keeps black
template <int GEN>
void row_sample_g(const GroupArgs& g, uint32_t ntiles, cudaStream_t s) {
    constexpr int B = GEN == 2 ? MINB_FILM : (GEN == 1 ? MINB_FACES_M : MINB);
    static const uint32_t cap = resident_blocks(row_pass_kernel<B, 2, GEN, 0>);
    const Spread sp = spread_warps(ntiles, cap);
    launch_chained_if(chain_small(sp, cap), row_pass_kernel<B, 2, GEN, 0>, sp.blocks, sp.threads, s, g, ntiles,
                      static_cast<const R*>(nullptr), GEN ? 1 : 0);
}

void row_sample(const GroupArgs& g, uint32_t ntiles, int gen, cudaStream_t s) {
    if (gen == 2) row_sample_g<2>(g, ntiles, s);
    else if (gen == 1) row_sample_g<1>(g, ntiles, s);
    else row_sample_g<0>(g, ntiles, s);
}

template <bool LEADER, int C, int B = LEADER ? MINB_PAIR_LEAD : MINB_PAIR, int NT = kBlock>
void pair_pass_t(const GroupArgs& g, uint32_t ntiles, const void* cone, int colour, int sub, cudaStream_t s) {
    static const uint32_t cap = resident_blocks(pair_pass_kernel<R, B, C, LEADER, NT>, NT);
    const Spread sp = spread_warps((ntiles + C - 1) / C, cap, NT);
    launch_chained_if(chain_small(sp, cap), pair_pass_kernel<R, B, C, LEADER, NT>, sp.blocks, sp.threads, s, g, ntiles,
                      static_cast<const R*>(cone), colour, sub);
}

// Consecutive pair tiles a warp takes per step: the fewest of 1, 2 and `most` with
// which about one step a warp does the launch.  Fewer leave a warp a second step
// when others have none, more leave warps without work; constrained sweeps of
// periodic lattices alone, us a sweep at 1 / 2 / 4 tiles: 64^3 (0.8 tiles a
// warp) 25.1 / 27.8 / 35.3, 128 x 128 x 32 (1.7) 40.3 / 30.5 / 38.2, 88^3 (2.2)
// 63.6 / 55.3 / 58.3, 128 x 96 x 64 (2.5) 65.5 / 54.2 / 52.7, 96^3 (2.8) 72.9 /
// 59.1 / 53.1, 256 x 64 x 64 (3.4) 75.9 / 57.4 / 45.5.
int pair_tiles_per_step(uint32_t ntiles, uint32_t warps, int most) {
    if (ntiles <= warps) return 1;
    return 5 * ntiles <= 11 * warps ? 2 : most;
}

// launch shapes: at most {default, 8, 2} tiles per grid-stride step, and the
// default step with more resident warps per SM: pair order one more block
// of 256 threads (fewer registers, some spilled), site order blocks of 128
// threads, five per SM (20 warps at up to 102 registers, against 16 warps
// in two blocks of 256)
template <bool LEADER>
void pair_pass_s(const GroupArgs& g, uint32_t ntiles, const void* cone, int colour, int shape, int sub,
                 cudaStream_t s) {
    constexpr int C0 = LEADER ? kPairChunkLead : kPairChunk;
    constexpr int B0 = LEADER ? MINB_PAIR_LEAD : MINB_PAIR;
    static const uint32_t cap = resident_blocks(pair_pass_kernel<R, B0, C0, LEADER>);
    const int c = pair_tiles_per_step(ntiles, cap * (kBlock / 32), shape == 1 ? 8 : shape == 2 ? 2 : C0);
    if (c == 1) pair_pass_t<LEADER, 1>(g, ntiles, cone, colour, sub, s);
    else if (c == 2) pair_pass_t<LEADER, 2>(g, ntiles, cone, colour, sub, s);
    else if (c == 8) pair_pass_t<LEADER, 8>(g, ntiles, cone, colour, sub, s);
    else if (shape == 3) {
        if constexpr (LEADER) pair_pass_t<LEADER, C0, 5, 128>(g, ntiles, cone, colour, sub, s);
        else pair_pass_t<LEADER, C0, B0 + 1>(g, ntiles, cone, colour, sub, s);
    } else pair_pass_t<LEADER, C0>(g, ntiles, cone, colour, sub, s);
}

void pair_pass(const GroupArgs& g, uint32_t ntiles, const void* cone, int colour, int leader, int shape, int sub,
               cudaStream_t s) {
    if (leader) pair_pass_s<true>(g, ntiles, cone, colour, shape, sub, s);
    else pair_pass_s<false>(g, ntiles, cone, colour, shape, sub, s);
}

// The wavefront kernel takes more than the default 48 KB of dynamic shared
// memory (opt_in_smem).
template <int MEASURE>
bool wave_opt_in() {
    return opt_in_smem(wave_sweep_kernel<MEASURE>, int(kWaveSmemBytes)) == cudaSuccess;
}

template <int MEASURE>
cudaError_t wave_sweep_t(const WaveArgs& a, uint32_t nblocks, const R* cone, int dir, cudaStream_t s) {
    if (!wave_opt_in<MEASURE>()) return cudaErrorInvalidConfiguration;
    // programmatic serialisation, as for the row passes
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nblocks);
    cfg.blockDim = dim3(kWaveThreads);
    cfg.dynamicSmemBytes = kWaveSmemBytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, wave_sweep_kernel<MEASURE>, a, cone, dir);
}

cudaError_t wave_sweep(const WaveArgs& a, uint32_t nblocks, const void* cone, int dir, int measure, cudaStream_t s) {
    const R* c = static_cast<const R*>(cone);
    if (measure >= 2) return wave_sweep_t<2>(a, nblocks, c, dir, s);
    if (measure == 1) return wave_sweep_t<1>(a, nblocks, c, dir, s);
    return wave_sweep_t<0>(a, nblocks, c, dir, s);
}

uint32_t wave_blocks() {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (wave_opt_in<0>())
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, wave_sweep_kernel<0>, kWaveThreads, kWaveSmemBytes);
    if (per_sm < 1) per_sm = 1;
    return uint32_t(sms) * uint32_t(per_sm);
}

// Resident sweeps: shape 0 = blocks of 512 threads (16 warps, up to 128
// registers), 1 = 640 threads (20 warps, up to 96 registers; 768 threads
// would spill at 80); one block per SM, opted in to the shared memory of the
// largest brick.
template <int NT, int MEASURE>
bool resident_opt_in() {
    return opt_in_smem(resident_sweep_kernel<NT, MEASURE>) == cudaSuccess;
}

template <int NT, int MEASURE>
cudaError_t resident_t(const ResidentPlan& r, const ResidentArgs& a, const R* cone, cudaStream_t s) {
    if (!resident_opt_in<NT, MEASURE>()) return cudaErrorInvalidConfiguration;
    // cooperative: the launch fails rather than run with a block not resident,
    // since the blocks wait for one another at the grid barriers
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(uint32_t(a.nyc * a.nzc));
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = a.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, resident_sweep_kernel<NT, MEASURE>, a,
                              *reinterpret_cast<const CUtensorMap*>(r.map_y),
                              *reinterpret_cast<const CUtensorMap*>(r.map_z), cone);
}

template <int NT>
cudaError_t resident_m(const ResidentPlan& r, const ResidentArgs& a, const R* cone, int measure, cudaStream_t s) {
    if (measure >= 2) return resident_t<NT, 2>(r, a, cone, s);
    if (measure == 1) return resident_t<NT, 1>(r, a, cone, s);
    return resident_t<NT, 0>(r, a, cone, s);
}

// n sweeps in launches of at most kResMaxSweeps, each after its control
// words are zeroed
cudaError_t resident_sweeps(const ResidentPlan& r, const void* cone, int n, int measure, int shape, cudaStream_t s) {
    const R* c = static_cast<const R*>(cone);
    for (int done = 0; done < n;) {
        ResidentArgs a = r.args;
        a.n_sweeps = std::min(n - done, measure ? kBrickMaxMeasured : kResMaxSweeps);
        // the records lie behind the control words (create_lattice): one memset
        const size_t clear = measure ? size_t(reinterpret_cast<char*>(a.record + size_t(a.n_sweeps) * kRecordWords) -
                                              reinterpret_cast<char*>(a.ctl))
                                     : sizeof(ResCtl);
        cudaError_t e = cudaMemsetAsync(a.ctl, 0, clear, s);
        if (e == cudaSuccess)
            e = shape == 1 ? resident_m<640>(r, a, c, measure, s) : resident_m<512>(r, a, c, measure, s);
        if (e == cudaSuccess && measure) {
            e = brick_close(a, static_cast<const ResidentArgs*>(nullptr), 1, a.n_sweeps, s);
        }
        if (e != cudaSuccess) return e;
        done += a.n_sweeps;
    }
    return cudaSuccess;
}

// cuTensorMapEncodeTiled, taken from the driver at run time (the library
// links the CUDA runtime only).
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled() {
    static const EncodeTiledFn fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<EncodeTiledFn>(f);
    }();
    return fn;
}

// The bricks of a resident lattice of Ly x Lz rows on the current device:
// the split (nyc, nzc) with the fewest rows in the largest brick, then the
// fewest halo rows, then the fewest blocks, among those with one block per
// SM at most whose brick fits a block's shared memory (both launch shapes
// must keep a block resident).  Then the tensor maps of the halo faces: the
// spins as a 64 x Ly x Lz x 6 array of floats (x, y, z, 3 colour + component;
// strides 256 B, 256 Ly B, 4 stride B).  False if no split fits or a map
// cannot be made.
bool resident_plan(const LatParams& p, ResidentPlan* r) {
    const int Ly = p.Ly, Lz = p.Lz;
    ResidentArgs* out = &r->args;
    int dev = 0, sms = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const long long cap = (long long)optin - (long long)kResStaticSmem;
    long long best[3] = {0, 0, 0};
    bool found = false;
    for (int nyc = 1; nyc <= Ly && nyc <= sms; ++nyc)
        for (int nzc = 1; nzc <= Lz && nyc * nzc <= sms && nyc * nzc <= kResMaxBlocks; ++nzc) {
            const int by = (Ly + nyc - 1) / nyc, bz = (Lz + nzc - 1) / nzc;
            if (by > 255 || bz > 255) continue;
            const uint32_t smem = resident_smem_bytes(by, bz, nyc, nzc);
            if ((long long)smem > cap) continue;
            const long long key[3] = {(long long)by * bz, (long long)resident_halo_rows(by, bz, nyc, nzc),
                                      (long long)nyc * nzc};
            if (!found || std::lexicographical_compare(key, key + 3, best, best + 3)) {
                found = true;
                std::copy(key, key + 3, best);
                *out = ResidentArgs{};
                out->nyc = nyc;
                out->nzc = nzc;
                out->by = by;
                out->bz = bz;
                out->smem = smem;
            }
        }
    if (!found) return false;
    int per_sm = 0;
    if (!resident_opt_in<512, 0>() || !resident_opt_in<640, 0>()) return false;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, resident_sweep_kernel<640, 0>, 640, out->smem);
    if (per_sm < 1) return false;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, resident_sweep_kernel<512, 0>, 512, out->smem);
    if (per_sm < 1) return false;
    const EncodeTiledFn enc = encode_tiled();
    if (!enc) return false;
    const cuuint64_t dim[4] = {cuuint64_t(kResLh), cuuint64_t(Ly), cuuint64_t(Lz), 6};
    const cuuint64_t strides[3] = {cuuint64_t(kResLh) * 4, cuuint64_t(kResLh) * 4 * cuuint64_t(Ly),
                                   cuuint64_t(p.stride) * 4};
    const cuuint32_t box_y[4] = {cuuint32_t(kResLh), 1, cuuint32_t(out->bz), 3};
    const cuuint32_t box_z[4] = {cuuint32_t(kResLh), cuuint32_t(out->by), 1, 3};
    const cuuint32_t unit[4] = {1, 1, 1, 1};
    for (int k = 0; k < 2; ++k) {
        const CUresult e = enc(reinterpret_cast<CUtensorMap*>(k == 0 ? r->map_y : r->map_z),
                               CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, p.spins, dim, strides, k == 0 ? box_y : box_z,
                               unit, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                               CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (e != CUDA_SUCCESS) return false;
    }
    return true;
}

void slab_export(LatDev* L, cudaStream_t s) { slab_export_kernel<<<1, 32, 0, s>>>(L); }

void slab_close(LatDev* L, int measure, cudaStream_t s) { slab_close_kernel<<<1, 32, 0, s>>>(L, measure); }

cudaError_t slab_halo(float* const (*dst)[2], const float* const (*src)[2], const uint32_t* stride,
                      const uint32_t (*src_stride)[2], uint32_t plane, int n, cudaStream_t s) {
    if (n < 1 || n > kMaxSlabs) return cudaErrorInvalidValue;
    SlabHaloArgs a{};
    for (int i = 0; i < n; ++i) {
        for (int k = 0; k < 2; ++k) {
            a.dst[i][k] = dst[i][k];
            a.src[i][k] = src[i][k];
            a.src_stride[i][k] = src_stride[i][k];
        }
        a.stride[i] = stride[i];
    }
    a.plane = plane;
    a.n = n;
    const uint32_t bx = (plane + 255) / 256;
    slab_halo_kernel<<<dim3(bx < 64 ? bx : 64, 2, uint32_t(n)), 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t slab_close_all(LatDev* const* lats, int n, int measure, cudaStream_t s) {
    if (n < 1 || n > kMaxSlabs) return cudaErrorInvalidValue;
    SlabDevs d{};
    for (int i = 0; i < n; ++i) d.lat[i] = lats[i];
    d.n = n;
    slab_close_all_kernel<<<1, 32 * (n < 32 ? n : 32), 0, s>>>(d, measure);
    return cudaGetLastError();
}

}  // namespace

const KernelSet& kernels_f32() {
    static const KernelSet k{colour_pass, row_pass,    pair_pass,   sweep_end,         pair_field,
                             ml_reset,    mlong,       measure,     row_sample,        grain_sample,
                             profile,     init_spins,  sample_close, row_field, "f32",
                             wave_sweep,  wave_blocks, slab_export,       slab_close,   slab_halo,
                             slab_close_all, resident_sweeps, resident_plan};
    return k;
}

}  // namespace mcgb

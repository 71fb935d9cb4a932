// kernels.h -- host-side launchers of the libmc kernels, one set per
// precision (kernels_f64.cu, kernels_f32.cu).
#pragma once
#include <cuda_runtime.h>

#include <vector>

#include "mc_internal.h"

namespace mcgb {

// Launch shapes the autotuner chooses among: an index into each kernel's
// candidate list (0 = the default, measured best on the batched workloads).
//   row:   FP32 row kernel, minimum resident blocks per SM (registers per
//          thread): {3, 2} (boundaries: 2 in passes with a sample), with film
//          tables {2, 3} (2 in passes with a sample);
//          for a resident lattice, threads per block {512, 640};
//   pair:  pair pass, consecutive tiles per grid-stride step {4, 8, 2}, and
//          4 with one more resident block per SM;
//   field: neighbour-field kernel, the same {4, 8, 2}.
constexpr int kRowShapes = 2, kPairShapes = 4, kFieldShapes = 3;
struct LaunchShape {
    int row = 0, pair = 0, field = 0;
};

// A resident lattice's launch: its arguments and two TMA descriptors
// (CUtensorMap, 128 bytes each) of its spins seen as a 64 x Ly x Lz x 6
// array (x, y, z, colour and component), with the boxes of a y face (64 x 1
// x bz x 3) and of a z face (64 x by x 1 x 3) of a brick.
struct alignas(128) ResidentPlan {
    unsigned char map_y[128];
    unsigned char map_z[128];
    ResidentArgs args;
};

// Launchers of a bcc, fcc or hcp lattice (one lattice a launch), a set per
// precision.
struct XtalKernels {
    // pass over sub-set (sub, colour) of ntiles 32-site tiles (finalize != 0
    // closes the sweep)
    cudaError_t (*pass)(const XtalArgs& a, uint32_t ntiles, const void* cone, int sub, int colour, int finalize,
                        cudaStream_t s);
    // the sample over the 2 nsub sub-sets (ntiles = 2 nsub tiles_per_subset),
    // which closes the sweep (level 2: with the torques)
    cudaError_t (*sample)(const XtalArgs& a, uint32_t ntiles, uint32_t tiles_per_subset, int level, cudaStream_t s);
    // constrained sweeps: the neighbour field of sub-set (sub, colour) into
    // LatParams::pfield
    void (*field)(const XtalArgs& a, uint32_t ntiles, int sub, int colour, cudaStream_t s);
};
const XtalKernels& xtal_f64();
const XtalKernels& xtal_f32();

struct KernelSet {
    // Table A1 colour pass over the lattices of g (ntiles = warp tiles of the
    // launch; the launcher sizes a persistent grid from the occupancy).
    // measure: 0 none, 1 magnetisation and energies, 2 also torques.
    // now: see row_pass.
    void (*colour_pass)(const GroupArgs& g, uint32_t ntiles, const void* cone, int colour, int measure, bool now,
                        cudaStream_t s);
    // FP32 colour pass over lattices in the row layout (adjacent site pairs
    // per lane; law = 0) or outside it with rows of even Lh (law = 1: the
    // general kernel's arithmetic); gen = 0: all axes periodic, no film tables;
    // gen = 1: any boundaries; gen = 2: film tables, any boundaries; turns: the
    // warps of a block share its tiles in turn (LaunchSet::turns).  Null in the FP64 set.  After a
    // black pass (colour 1) it also launches the close of the lattices' sweeps
    // (sweep_close_kernel); of measured ones the samples are formed there (now) or
    // by sample_close.  Returns the status of the
    // launches (made with programmatic serialisation).
    cudaError_t (*row_pass)(const GroupArgs& g, uint32_t ntiles, const void* cone, int colour, int measure, int law,
                            int gen, int shape, bool turns, bool now, cudaStream_t s);
    // Table A2 pair pass over sub-set (sub, colour) (sub = 0 for simple cubic
    // lattices); leader != 0 takes the pairs in site order
    // (LatParams::pair_leader).
    void (*pair_pass)(const GroupArgs& g, uint32_t ntiles, const void* cone, int colour, int leader, int shape,
                      int sub, cudaStream_t s);
    // End of an unmeasured constrained sweep of every lattice of g.
    void (*sweep_end)(const GroupArgs& g, cudaStream_t s);
    // Neighbour field of every site of the given colour into LatParams::pfield
    // (site tiles), before that colour's pair pass.
    void (*pair_field)(const GroupArgs& g, uint32_t ntiles, int colour, int shape, cudaStream_t s);
    // Zero M_L and its carried change of every lattice of g (before mlong).
    void (*ml_reset)(const GroupArgs& g, cudaStream_t s);
    // Exact M_L of every lattice of g (site tiles).
    void (*mlong)(const GroupArgs& g, uint32_t ntiles, cudaStream_t s);
    // Standalone sample + end of sweep (site tiles).
    void (*measure)(const GroupArgs& g, uint32_t ntiles, cudaStream_t s);
    // The same over lattices in the row layout (gen as in row_pass, law 0); with gen
    // = 0 it also stores the red sites' field for the next constrained sweep
    // (LatParams::pfield).  Null in the FP64 set.
    void (*row_sample)(const GroupArgs& g, uint32_t ntiles, int gen, cudaStream_t s);
    // One grain sample of a film lattice (ntiles site tiles, n_grains grains).
    void (*grain_sample)(LatDev* L, uint32_t ntiles, int n_grains, cudaStream_t s);
    // Slice sums for the profile of one lattice.
    void (*profile)(LatDev* d, uint32_t Lh, uint32_t rows, cudaStream_t s);
    // The spins of a new lattice p (host copy): all along v, or a wall along x.
    void (*init_spins)(const LatParams& p, int wall, const double v[3], cudaStream_t s);
    // The samples of the measured launched sweeps since the last call (at most
    // kSampleRecords), of every lattice of g.
    void (*sample_close)(const GroupArgs& g, cudaStream_t s);
    // pair_field over all-periodic lattices in the row layout.  Null in the FP64
    // set.
    void (*row_field)(const GroupArgs& g, uint32_t ntiles, int colour, int shape, cudaStream_t s);
    const char* name;
    // FP32 wavefront sweep (red and black pass in one launch) of the
    // lattices of a, nblocks blocks; dir = 0 reads spins and writes
    // spins_alt, dir = 1 the reverse; measure as for colour_pass.  Null in
    // the FP64 set.  Returns the status of the launch.
    cudaError_t (*wave_sweep)(const WaveArgs& a, uint32_t nblocks, const void* cone, int dir, int measure,
                              cudaStream_t s);
    // Blocks of the wavefront kernel resident on the current device at once
    // (the work-unit plan is made for this many).  Null in the FP64 set.
    uint32_t (*wave_blocks)();
    // Slabs of a lattice split along z (FP32 row layout; null in the FP64
    // set): export slab L's counts to LatParams::slab_counts, close L's
    // sweep from its (summed) counts.
    void (*slab_export)(LatDev* L, cudaStream_t s);
    void (*slab_close)(LatDev* L, int measure, cudaStream_t s);
    // Slabs on one device: the halo planes of one colour of n slabs, each
    // from its neighbours (dst / src: [slab][lower, upper] plane bases,
    // strides per slab), and export, sum and close of n slabs in one launch.
    cudaError_t (*slab_halo)(float* const (*dst)[2], const float* const (*src)[2], const uint32_t* stride,
                             const uint32_t (*src_stride)[2], uint32_t plane, int n, cudaStream_t s);
    cudaError_t (*slab_close_all)(LatDev* const* lats, int n, int measure, cudaStream_t s);
    // Resident sweeps (resident_pass.cuh) of the lattice of a plan: n sweeps
    // in cooperative launches of at most kResMaxSweeps, measure as for
    // colour_pass, shape 0 or 1 (blocks of 512 or 640 threads).  Null in the
    // FP64 set.  Returns the status of the launches.
    cudaError_t (*resident_sweeps)(const ResidentPlan& r, const void* cone, int n, int measure, int shape,
                                   cudaStream_t s);
    // The brick split of FP32 lattice p (host copy: dims, stride, spins) on
    // the current device and the tensor maps of its halo faces: fills
    // everything but args.lat and args.ctl; false when its rows do not fit
    // the SMs' shared memory.  Null in the FP64 set.
    bool (*resident_plan)(const LatParams& p, ResidentPlan* out);
};

// Launch tables of a set of lattices: site tiles and pair tiles of every
// lattice (lattice l owns tiles [start[l], start[l+1])), and for the colour
// passes the split by colour-pass kernel (LatParams::colour_kernel).
struct LaunchSet {
    GroupArgs all, pairs, pairs_lead;
    uint32_t nt_all = 0, nt_pairs = 0, nt_pairs_lead = 0;  // pair tiles: pair order, site order
    // colour passes: lattices and tiles of each colour-pass kernel
    GroupArgs col[kColourKinds];
    uint32_t nt_col[kColourKinds] = {};
    bool turns[kColourKinds] = {};  // every lattice of the list is large with long rows (long_rows)
    // wavefront lattices (LatParams::wave): their work-unit plan (nb_wave
    // blocks; 0 = none), and the row-kernel list without them, which runs
    // beside a wavefront launch (col keeps them, for sweeps that run
    // as two row passes)
    WaveArgs wave = {};
    uint32_t nb_wave = 0;
    GroupArgs row_rest;
    uint32_t nt_row_rest = 0;
    // resident lattices (LatParams::rctl) whose unconstrained sweeps run as
    // resident launches, one lattice after another: a lattice alone, or every
    // lattice of a group made only of large resident lattices; n_res launch
    // plans, owned by the lattices (none: n_res = 0)
    ResidentPlan* const* res = nullptr;
    int n_res = 0;
    // a lattice alone whose unconstrained sweeps run as brick launches, else
    // null; its Lh
    BrickArgs* brick = nullptr;
    uint32_t brick_lh = 0;
    // a group whose unconstrained sweeps run as brick launches of all its
    // lattices side by side, else null
    struct BrickSet* brick_set = nullptr;
    int sample_level = 2;  // sample of a measured colour pass: 1 or 2 (torques)
    // a bcc / fcc / hcp lattice alone (xtal.lat, else null) and its sub-lattices
    XtalArgs xtal = {};
    int nsub = 1;
    LaunchShape shape;  // autotuned launch shapes
};

// Brick sweeps (brick_pass.cuh; FP32 simple cubic lattices without film
// tables): the split of lattice p (host copy) over the current device's SMs,
// everything of out but its pointers and key; false when its rows do not fit
// their shared memory.  Then n sweeps of a plan in one cooperative launch (at
// most kResMaxSweeps, or kBrickMaxMeasured measured), measure as for colour_pass;
// *ran: the launch was accepted (if not, nothing of it ran).
bool brick_plan(const LatParams& p, BrickArgs* out);
// The splits of several lattices swept side by side, each with blocks of its
// own (splits only: out[i] keeps its pointers and key): the estimated us of a
// sweep of the slowest, or 0 when they do not fit the SMs together.
double brick_group_plan(const std::vector<const LatParams*>& lats, std::vector<BrickArgs>* out);
cudaError_t brick_sweeps(const BrickArgs& b, uint32_t Lh, const void* cone, int n, int measure, bool* ran,
                         cudaStream_t s);
// The same for lattices of one kernel instance (law, no faces, parity of Lh):
// their plans and first blocks in device memory, blocks and shared memory of
// the launch.
struct BrickClass {
    BrickArgs* args = nullptr;
    uint32_t* first = nullptr;
    int n = 0, law = 0, odd = 0;
    uint32_t blocks = 0, smem = 0;
    int refuse = 0;  // the most of its lattices' (BrickArgs::refuse)
};
cudaError_t brick_group_sweeps(const BrickClass& c, const void* cone, int n, int measure, bool* ran, cudaStream_t s);

const KernelSet& kernels_f64();
const KernelSet& kernels_f32();

}  // namespace mcgb

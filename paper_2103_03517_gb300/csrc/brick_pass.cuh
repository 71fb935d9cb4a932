// brick_pass.cuh -- FP32 sweeps of Table A1 over one simple cubic lattice of
// any shape and boundaries held in the SMs' shared memory for a whole run of
// sweeps (films excepted), for the lattices that resident_pass.cuh does not
// take: rows of any length, open, pinned and anti-periodic faces, rows that
// do not have the row layout.
//
// What bounds it.  A small lattice swept by launches spends its time between
// passes: a 64^3 pass has 2.2 us of issue time over all SMs at the row
// kernel's instruction count and took 6 us as a launch in a graph (measured
// ones 10), most of it the launch, the first loads' latency and the drained
// end.  Here a run of sweeps is one cooperative launch; what is left per pass
// is the exchange between neighbouring blocks.  That exchange is one trip
// through L2: a block stores the spins on its faces as 16-byte packets that end
// in a tag, and the neighbour polls the packets it needs, with no fence,
// flag or copy between (a 16-byte access of scope .gpu is single-copy atomic,
// so a packet whose tag is the awaited one carries that pass's spin).
//
// The lattice's rows (y, z) are shared out over the blocks as bricks ny x nz
// (rows of even Lh), or as runs of consecutive rows that start on an even row
// (odd Lh, where two neighbouring colour indices that share a Philox call may
// lie in two rows).  A block keeps both colours of its rows, [colour][row][3]
// [Lh], and a table with one entry per row: its place, its four neighbour
// rows (in the block, or the packets of another block's row) and its faces.
// A warp moves 32 pairs of neighbouring colour indices at a time, rows on
// faces first.  Arithmetic, order and draws are those of the kernel that the
// lattice's single passes take (LAW 0: the row kernels, pair_math.cuh; LAW 1:
// the general kernel), so a chain is the same bit for bit whichever runs it.
//
// Packets.  The packet of a site is rewritten two passes after it was read:
// by then its writer has read the reader's own packet of the pass between,
// which the reader stored after its read.  Tags hold the pass and an epoch that
// every launch counts up, so that no packet of an earlier launch, and none of
// zeroed memory, can match (brick_tag0; before the epochs repeat the packets are
// cleared, since a lattice swept alone, in a group, or in memory that several
// sizes share does not write the same packets in every launch).
//
// Cone angle.  Every block adds its accepted count of a sweep and its arrival
// to one word (running totals, one word per parity of the sweep: a block adds
// to a word again only after every block has read it), and a service warp of
// each block polls the word and hands the next cone angle to its block's
// workers, which meanwhile have loaded and drawn their first tile of the next
// sweep.  (A slot per block that all blocks poll, in place of the word, costs
// 1 us a sweep more at 144 blocks: 144 x 144 polls meet in few L2 lines.)
//
// Measured sweeps.  The blocks add their sample sums into the sweep's own
// record, and a launch after the run turns the records into moments and ring
// entries, one warp per sweep (brick_close_kernel).  Closing each sweep as it
// ended kept the service warp of block 0 busy for 4 us with FP64 divisions and
// round trips, which every block then waited for: 6.1 us a measured sweep of
// 32^3 against 3.1 us unmeasured.
//
// Every wait is bounded (a count of polls that takes about one second): the block
// then raises the abort flag, its workers leave together at the next barrier (a
// reduction of their fail flags) without writing their rows back, and the lattice's
// error is set.  Its spins are undefined then: until the barrier a lane whose wait
// ran out still publishes what it computed, and a block that has finished its last
// pass writes back.
#pragma once
#include "resident_pass.cuh"

namespace mcgb {

constexpr int kBrickWarps = 19;                  // workers of a block (20 warps, five a scheduler: 96 registers,
                                                 // what 17 warps would get too)
constexpr int kBrickThreads = 32 * (kBrickWarps + 1);  // and the service warp

// One row of a block.  own: offset of its first float; nb: the neighbour rows
// -y, +y, -z, +z: offset in the block, or ~(first packet); row: its index
// y + Ly z in the lattice; flags: bit 0 parity of y + z, bit 1 a face row,
// bit 2 pinned, bits 8 + 2 d: 1 - the factor of neighbour d (1, 0 or -1).
struct alignas(16) BrickRow {
    int own, nb[4];
    uint32_t row, flags, pad;
};
static_assert(sizeof(BrickRow) == 32, "a row's entry is two 16-byte loads");

__host__ __device__ inline uint32_t brick_smem_bytes(uint32_t rows, uint32_t Lh) {
    return ((2u * rows * 3u * Lh * 4u + 15u) & ~15u) + rows * uint32_t(sizeof(BrickRow));
}

__device__ __forceinline__ uint4 ld_packet(const float4* p) {
    unsigned long long lo, hi;
    asm volatile("{\n\t.reg .b128 q;\n\tld.relaxed.gpu.global.b128 q, [%2];\n\tmov.b128 {%0, %1}, q;\n\t}"
                 : "=l"(lo), "=l"(hi)
                 : "l"(p)
                 : "memory");
    return make_uint4(uint32_t(lo), uint32_t(lo >> 32), uint32_t(hi), uint32_t(hi >> 32));
}

__device__ __forceinline__ void st_packet(float4* p, float x, float y, float z, uint32_t tag) {
    const unsigned long long lo = (unsigned long long)__float_as_uint(x) | ((unsigned long long)__float_as_uint(y) << 32);
    const unsigned long long hi = (unsigned long long)__float_as_uint(z) | ((unsigned long long)tag << 32);
    asm volatile("{\n\t.reg .b128 q;\n\tmov.b128 q, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], q;\n\t}" ::"l"(p),
                 "l"(lo), "l"(hi)
                 : "memory");
}

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* a) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.u64 %0, [%1];" : "=l"(v) : "l"(a) : "memory");
    return v;
}

// Barrier of the workers that also tells each whether any of them failed.
__device__ __forceinline__ bool workers_failed(bool mine) {
    uint32_t any;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
        "barrier.cta.red.or.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(any)
        : "r"(uint32_t(mine)), "n"(32 * kBrickWarps)
        : "memory");
    return any != 0;
}

// Polls of one L2 access each that take about a second.
constexpr uint32_t kBrickPolls = 1u << 20;

__device__ __forceinline__ float brick_factor(uint32_t flags, int d) {
    return 1.0f - float((flags >> (8 + 2 * d)) & 3u);
}

// Factor of a bond across an x face with boundary mode bc.
__device__ __forceinline__ float x_face_factor(int bc) { return bc == 0 ? 1.0f : (bc == 3 ? -1.0f : 0.0f); }

// The spins of a lane's pair (k even) in its four neighbour rows.  Rows of the
// block come from shared memory; the packets of other blocks' rows are all
// requested before the first is looked at, and asked for again until all carry
// the awaited tag.  A pair is two packets, (x0, x1, y0, tag) and (z0, z1, y1,
// tag), so that two of its three components are packed operands as they come.
// False if the wait runs out (the abort flag is then raised) or another block
// gave up.
__device__ __forceinline__ bool brick_neighbours(const float* oth, const float4* pk, const BrickRow& e, uint32_t k,
                                                 uint32_t Lh, uint32_t tag, int* abort, P3 n[4]) {
    for (uint32_t i = 0;; ++i) {
        uint32_t bad = 0;
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            if (e.nb[d] < 0) {
                const uint4 u = ld_packet(pk + uint32_t(~e.nb[d]) + k), v = ld_packet(pk + uint32_t(~e.nb[d]) + k + 1);
                n[d] = P3{make_float2(__uint_as_float(u.x), __uint_as_float(u.y)),
                          make_float2(__uint_as_float(u.z), __uint_as_float(v.z)),
                          make_float2(__uint_as_float(v.x), __uint_as_float(v.y))};
                bad |= (u.w ^ tag) | (v.w ^ tag);
            } else {
                const float* r = oth + e.nb[d] + k;
                n[d] = P3{*reinterpret_cast<const float2*>(r), *reinterpret_cast<const float2*>(r + Lh),
                          *reinterpret_cast<const float2*>(r + 2 * Lh)};
            }
        }
        if (bad == 0) return true;
        if (*reinterpret_cast<volatile int*>(abort)) return false;
        if (i == kBrickPolls) {
            atomicExch(abort, 1);
            return false;
        }
    }
}

__device__ __forceinline__ void st_pair_packets(float4* p, const P3& v, uint32_t tag) {
    st_packet(p, v.x.x, v.x.y, v.y.x, tag);
    st_packet(p + 1, v.z.x, v.z.y, v.y.y, tag);
}

// The same for one site (rows of odd Lh): a packet is (x, y, z, tag).
__device__ __forceinline__ bool brick_neighbours(const float* oth, const float4* pk, const BrickRow& e, uint32_t k,
                                                 uint32_t Lh, uint32_t tag, int* abort, V3<float> n[4]) {
    for (uint32_t i = 0;; ++i) {
        uint32_t bad = 0;
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            if (e.nb[d] < 0) {
                const uint4 u = ld_packet(pk + uint32_t(~e.nb[d]) + k);
                n[d] = V3<float>{__uint_as_float(u.x), __uint_as_float(u.y), __uint_as_float(u.z)};
                bad |= u.w ^ tag;
            } else {
                const float* r = oth + e.nb[d] + k;
                n[d] = V3<float>{r[0], r[Lh], r[2 * Lh]};
            }
        }
        if (bad == 0) return true;
        if (*reinterpret_cast<volatile int*>(abort)) return false;
        if (i == kBrickPolls) {
            atomicExch(abort, 1);
            return false;
        }
    }
}

// The block's nr rows, both colours, from the lattice (LOAD) or back into it, by
// WARPS warps.  SIX: a unit is 32 sites of a row, or short rows that make up at
// most 32; a lane moves the six floats of its site index, those of two units (LOAD)
// before it waits for the first.  Otherwise a component of a row at a time, each
// waited for and each with its address formed anew: a block of 192 rows of 32 took
// 14 us to load and 7.5 to store that way, and 3 sweeps of 8 x 64^3 107 us a call
// (75 by launches); all SIX, and the row table made in one pass, 78.
template <bool LOAD, bool SIX, int WARPS>
__device__ __forceinline__ void brick_rows(float* bsm, float* s, const BrickRow* tab, uint32_t nr, uint32_t Lh,
                                           uint32_t half, uint32_t stride, int warp, int lane) {
    if constexpr (!SIX) {
        for (int c = 0; c < 2; ++c)
            for (uint32_t i = uint32_t(warp); i < 3u * nr; i += uint32_t(WARPS)) {
                const BrickRow& e = tab[i / 3u];
                const uint32_t comp = i % 3u;
                float* g = s + size_t(3 * c + int(comp)) * stride + size_t(e.row) * Lh;
                float* b = bsm + size_t(c) * half + e.own + comp * Lh;
                const float* src = LOAD ? g : b;
                float* dst = LOAD ? b : g;
                for (uint32_t k = uint32_t(lane); k < Lh; k += 32) dst[k] = src[k];
            }
        return;
    }
    constexpr int U = LOAD ? 2 : 1;
    const uint32_t segs = (Lh + 31u) / 32u;
    const uint32_t lg = Lh > 16u ? 5u : 32u - uint32_t(__clz(int(Lh - 1u)));  // lanes of a row: 1 << lg
    const uint32_t per = 32u >> lg, units = (nr + per - 1u) / per * segs;
    for (uint32_t u0 = uint32_t(warp); u0 < units; u0 += uint32_t(U * WARPS)) {
        float v[U][6];
        float* g[U];
        float* b[U];
        bool has[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const uint32_t u = u0 + uint32_t(j * WARPS);
            const uint32_t r0 = segs == 1u ? u : u / segs;
            const uint32_t i = r0 * per + (uint32_t(lane) >> lg);
            const uint32_t k = 32u * (u - r0 * segs) + (uint32_t(lane) & ((1u << lg) - 1u));
            has[j] = u < units && i < nr && k < Lh;
            if (has[j]) {
                g[j] = s + size_t(tab[i].row) * Lh + k;
                b[j] = bsm + tab[i].own + k;
                if (LOAD)
#pragma unroll
                    for (int c = 0; c < 6; ++c) v[j][c] = g[j][size_t(c) * stride];
            }
        }
#pragma unroll
        for (int j = 0; j < U; ++j)
            if (has[j])
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    float* const at = b[j] + (c >= 3 ? half : 0u) + uint32_t(c % 3) * Lh;
                    if (LOAD) *at = v[j][c];
                    else g[j][size_t(c) * stride] = *at;
                }
    }
}

// Which form of row table, load and store an instance has.  They differ by a few us
// a call, but the compiler gives the sweeps of an instance other registers with
// each, and those differ by up to 7% a sweep; this is the shortest call whose sweeps
// are no slower than with the plainest.  us a sweep, all of the short form / as
// here: 60^3 open 4.28 / 3.97, 40 x 160 x 136 9.90 / 9.72 (without torques 11.43
// / 10.79), 96^3 without torques 10.86 / 10.26, 128 x 100 x 80 open without
// torques 12.23 / 11.76, 138^3 38.1 / 37.1.
template <int LAW, int FACES, int ODD, int MEASURE, int GROUP>
struct BrickForm {
    static constexpr bool plain = LAW == 0 && FACES && MEASURE == 1;
    static constexpr bool table_once = LAW == 0 || GROUP;
    static constexpr bool load_six = !ODD && !plain;
    static constexpr bool store_six = !ODD && !plain && (LAW == 0 || FACES || GROUP);
};

// LAW 0: packed pairs (row kernels), 1: the general kernel's scalar law;
// FACES: any boundaries (0: all periodic); ODD: rows of odd Lh (LAW 1);
// MEASURE as in the row kernel; GROUP: the lattices of grp, each with blocks of
// its own that know nothing of the others, instead of `one` (plan and keys then come
// from memory: these instances spill 22 to 72 bytes a thread at 96 registers, the
// others at most 24).
template <int LAW, int FACES, int ODD, int MEASURE, int GROUP>
__global__ void __launch_bounds__(kBrickThreads, 1)
    brick_sweep_kernel(const __grid_constant__ BrickArgs one, const __grid_constant__ BrickGroup grp,
                       const float* __restrict__ cone) {
    constexpr int NS = MEASURE >= 2 ? kNumSums : kSumTux;  // sums sampled
    constexpr int NW = kBrickWarps;
    using Form = BrickForm<LAW, FACES, ODD, MEASURE, GROUP>;
    extern __shared__ __align__(16) float bsm[];
    __shared__ uint64_t tbar;                  // the cone angle of a sweep is known
    __shared__ unsigned cta_acc, wdone;        // accepted moves, warps done with the sweep
    __shared__ long long cta_sums[kNumSums];   // fixed-point sample sums
    __shared__ float s_cone;                   // 1 - cos of the cone angle
    __shared__ int s_fail;
    int lat = 0;
    if (GROUP)
        for (int hi = grp.n - 1; lat < hi;) {  // the last lattice whose first block is not above this one
            const int mid = (lat + hi + 1) >> 1;
            if (__ldg(&grp.first[mid]) <= blockIdx.x) lat = mid;
            else hi = mid - 1;
        }
    const BrickArgs& a = GROUP ? grp.args[lat] : one;
    const uint32_t key0 = a.key0, key1 = a.key1;  // launch constants of a lattice alone, and with them the round keys
    const FastDiv div_half = a.div_half;
    const int n_sweeps = GROUP ? grp.n_sweeps : a.n_sweeps;
    LatDev* const L = a.lat;
    const LatParams& p = L->p;
    BrickCtl* const ctl = a.ctl;
    const int tid = int(threadIdx.x), lane = tid & 31, warp = tid >> 5;
    const uint32_t Lh = uint32_t(p.Lh), Ly = uint32_t(p.Ly), Lz = uint32_t(p.Lz), stride = p.stride;
    const uint32_t G = a.nyc * a.nzc, blk = blockIdx.x - (GROUP ? __ldg(&grp.first[lat]) : 0u);
    float* const s = static_cast<float*>(p.spins);
    // this block's rows: a brick, or a run of rows
    uint32_t y0 = 0, ny = 1, z0 = 0, nr, r0 = 0;
    if (ODD) {
        const uint32_t pairs = (Ly * Lz + 1) / 2;  // row pairs, shared out evenly
        r0 = 2u * uint32_t(uint64_t(pairs) * blk / G);
        nr = min(2u * uint32_t(uint64_t(pairs) * (blk + 1) / G), Ly * Lz) - r0;
    } else {
        const uint32_t bi = blk % a.nyc, bj = blk / a.nyc;
        y0 = bi * Ly / a.nyc;
        ny = (bi + 1) * Ly / a.nyc - y0;
        z0 = bj * Lz / a.nzc;
        nr = ny * ((bj + 1) * Lz / a.nzc - z0);
    }
    const uint32_t rowf = 3u * Lh, half = a.rows * rowf;  // floats of a row, of a colour
    BrickRow* const tab = reinterpret_cast<BrickRow*>(reinterpret_cast<char*>(bsm) + ((2u * half * 4u + 15u) & ~15u));
    if (tid == 0) {
        mbar_init(&tbar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        cta_acc = 0;
        wdone = 0;
        s_fail = 0;
    }
    if (tid < kNumSums) cta_sums[tid] = 0;
    // the row table, by warp 0: face rows from its front, the others from its end
    // in one pass, or behind them in two (ODD: in order, one pass)
    if (warp == 0) {
        constexpr int phases = ODD || Form::table_once ? 1 : 2;
        uint32_t front = 0, end = nr;
        for (int phase = 0; phase < phases; ++phase)
            for (uint32_t i0 = 0; i0 < nr; i0 += 32) {
                const uint32_t i = i0 + uint32_t(lane);
                BrickRow e{};
                bool mine = false, last = false;
                if (i < nr) {
                    const uint32_t f = ODD ? r0 + i : y0 + i % ny + Ly * (z0 + i / ny);
                    const uint32_t y = f % Ly, z = f / Ly;
                    e.own = int(i * rowf);
                    e.row = f;
                    bool face = false;
#pragma unroll
                    for (int d = 0; d < 4; ++d) {
                        const bool isz = d >= 2, plus = d & 1;
                        const uint32_t n = isz ? Lz : Ly, w = isz ? z : y;
                        const bool cross = plus ? w + 1 == n : w == 0;
                        const uint32_t w2 = cross ? (plus ? 0 : n - 1) : (plus ? w + 1 : w - 1);
                        const int bc = isz ? p.bc[2] : p.bc[1];
                        const bool absent = cross && (bc == 1 || bc == 2);
                        const uint32_t yn = isz ? y : w2, zn = isz ? w2 : z, fn = yn + Ly * zn;
                        uint32_t j = 0;  // its place in the block
                        bool in;
                        if (ODD) {
                            in = fn >= r0 && fn < r0 + nr;
                            j = fn - r0;
                        } else {
                            in = yn >= y0 && yn < y0 + ny && zn >= z0 && (zn - z0) * ny < nr;
                            j = (yn - y0) + ny * (zn - z0);
                        }
                        if (absent) {
                            e.nb[d] = e.own;  // read and multiplied by zero
                            e.flags |= 1u << (8 + 2 * d);
                        } else {
                            e.nb[d] = in ? int(j * rowf) : ~int(fn * Lh);
                            face = face || !in;
                            if (cross && bc == 3) e.flags |= 2u << (8 + 2 * d);
                        }
                    }
                    e.flags |= ((y + z) & 1u) | (face ? 2u : 0u);
                    if ((p.bc[1] == 2 && (y == 0 || y + 1 == Ly)) || (p.bc[2] == 2 && (z == 0 || z + 1 == Lz))) e.flags |= 4u;
                    mine = ODD || Form::table_once || face == (phase == 0);
                    last = !ODD && Form::table_once && !face;
                }
                const uint32_t below = (1u << lane) - 1u;
                const uint32_t f = __ballot_sync(0xffffffffu, mine && !last);
                if (mine && !last) tab[front + uint32_t(__popc(f & below))] = e;
                front += uint32_t(__popc(f));
                if (!ODD && Form::table_once) {
                    const uint32_t o = __ballot_sync(0xffffffffu, last);
                    if (last) tab[end - 1u - uint32_t(__popc(o & below))] = e;
                    end -= uint32_t(__popc(o));
                }
            }
    }
    __syncthreads();
    brick_rows<true, Form::load_six, NW + 1>(bsm, s, tab, nr, Lh, half, stride, warp, lane);
    int theta = L->st.theta;
    const uint32_t sweep0 = L->st.sweep;
    const uint32_t epoch = *reinterpret_cast<volatile uint32_t*>(&ctl->epoch), T0 = brick_tag0(epoch);
    const Par<float> par = load_par<float>(p);
    const bool adapt = MEASURE == 0 || p.adapt_in_measure;
    __syncthreads();
    // ------------------------------------------------------ the service warp
    if (warp == NW) {
        LatState& st = L->st;
        bool ok = true;
        long long acc = 0;
        unsigned long long even = 0, odd = 0;  // totals of the sweeps of either parity so far
        for (int sw = 0; sw < n_sweeps && ok; ++sw) {
            if (sw + 1 == n_sweeps && blk != 0) break;
            // every block's count of this sweep
            const uint32_t want = G * uint32_t(sw / 2 + 1) + uint32_t(a.inject);
            unsigned long long v = 0;
            if (lane == 0) {
                uint32_t i = 0;
                while (uint32_t((v = ld_relaxed_u64(&ctl->count[sw & 1])) >> 40) != want) {
                    if (*reinterpret_cast<volatile int*>(&s_fail) || *reinterpret_cast<volatile int*>(&ctl->abort) ||
                        ++i == kBrickPolls) {
                        ok = false;
                        break;
                    }
                }
            }
            ok = __shfl_sync(0xffffffffu, int(ok), 0) != 0;
            v = __shfl_sync(0xffffffffu, v, 0) & ((1ull << 40) - 1ull);
            acc = (long long)(v - (sw & 1 ? odd : even));
            if (sw & 1) odd = v;
            else even = v;
            if (adapt) theta = cone_rule(theta, acc, p.n_mov);
            if (lane == 0) {
                if (ok) s_cone = cone[theta];
                else *reinterpret_cast<volatile int*>(&s_fail) = 1;
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tbar)) : "memory");
            }
            __syncwarp();
            if (MEASURE > 0 && ok && blk == 0 && lane < 2)
                a.record[size_t(sw) * kRecordWords + kRecTheta + lane] = lane == 0 ? (long long)theta : acc;
        }
        if (ok && blk == 0) {  // the run's end
            if (lane == 0) {
                st.last_acc = acc;
                st.theta = theta;
                st.ml_hi += st.dml_hi;
                st.ml_lo += st.dml_lo;
                st.dml_hi = 0;
                st.dml_lo = 0;
                st.sweep = sweep0 + uint32_t(n_sweeps);
            }
        }
        if (!ok && lane == 0) {
            *reinterpret_cast<volatile int*>(&s_fail) = 1;
            atomicExch(&ctl->abort, 1);
            atomicCAS(&st.error, 0, -4);  // MC_ERR_TIMEOUT
        }
        if (blk == 0 && lane == 0) *reinterpret_cast<volatile uint32_t*>(&ctl->epoch) = epoch + 1u;
        return;
    }
    // ----------------------------------------------------------- the workers
    // the black spins of the face rows at the start, for the first red pass
    float4* const pk = static_cast<float4*>(a.packets);
    for (uint32_t i = uint32_t(warp); i < nr; i += NW) {
        const BrickRow& e = tab[i];
        if (!(e.flags & 2u)) continue;
        const float* r = bsm + half + e.own;
        float4* d = pk + stride + size_t(e.row) * Lh;
        if (ODD) {
            for (uint32_t k = uint32_t(lane); k < Lh; k += 32) st_packet(d + k, r[k], r[Lh + k], r[2 * Lh + k], T0);
        } else {
            for (uint32_t k = 2u * uint32_t(lane); k < Lh; k += 64)
                st_pair_packets(d + k, P3{make_float2(r[k], r[k + 1]), make_float2(r[Lh + k], r[Lh + k + 1]),
                                          make_float2(r[2 * Lh + k], r[2 * Lh + k + 1])}, T0);
        }
    }
    const uint32_t sites = nr * Lh;                   // colour indices of the block
    const uint32_t np = ODD ? (sites + 1u) / 2u : sites / 2u;
    const uint32_t ntiles = (np + 31u) / 32u;
    float cval = cone[theta];
    bool failed = false;
    bool alive = true;
    for (int sw = 0; sw < n_sweeps && alive; ++sw) {
        const uint32_t sweep = sweep0 + uint32_t(sw);
        unsigned nacc = 0;
        for (int c = 0; c < 2 && alive; ++c) {
            const uint32_t tag_in = T0 + 2u * uint32_t(sw) + uint32_t(c), tag_out = tag_in + 1u;
            float* const own = bsm + (c ? half : 0u);
            const float* const oth = bsm + (c ? 0u : half);
            const float4* const pin = pk + size_t(c ^ 1) * stride;
            float4* const pout = pk + size_t(c) * stride;
            bool first = c == 0 && sw > 0;
            int lf[NS];  // this lane's fixed-point parts of the sample, kPartTiles tiles at a time
#pragma unroll
            for (int i = 0; i < NS; ++i) lf[i] = 0;
            uint32_t nparts = 0;
            long long fix = 0;
            for (uint32_t tile = uint32_t(warp); tile < ntiles; tile += NW) {
                const uint32_t P = tile * 32u + uint32_t(lane);
                const bool valid = P < np;
                const uint32_t Pc = valid ? P : np - 1u;
                P3 S, h, O;
                bool mov[2];
                uint32_t site0, k;
                BrickRow e, e1;  // ODD: of the two sites
                uint32_t k1 = 0;
                bool two = true;
                if constexpr (!ODD) {
                    const uint32_t i = fast_div(Pc, div_half);
                    k = 2u * (Pc - i * (Lh >> 1));
                    e = tab[i];
                    const uint32_t xoff = (e.flags + uint32_t(c)) & 1u;
                    const float* o = own + e.own + k;
                    const float* x = oth + e.own;
                    S = P3{*reinterpret_cast<const float2*>(o), *reinterpret_cast<const float2*>(o + Lh),
                           *reinterpret_cast<const float2*>(o + 2 * Lh)};
                    O = P3{*reinterpret_cast<const float2*>(x + k), *reinterpret_cast<const float2*>(x + Lh + k),
                           *reinterpret_cast<const float2*>(x + 2 * Lh + k)};
                    // the fourth x neighbour of the pair: k + 2 or k - 1 in the row
                    const uint32_t ke = xoff ? (k + 2u == Lh ? 0u : k + 2u) : (k == 0 ? Lh - 1u : k - 1u);
                    const V3<float> E{x[ke], x[Lh + ke], x[2 * Lh + ke]};
                    P3 n[4];
                    if (!brick_neighbours(oth, pin, e, k, Lh, tag_in, &ctl->abort, n)) failed = true;
                    const uint32_t x0 = xoff + 2u * k;
                    site0 = x0 + 2u * Lh * e.row;
                    mov[0] = mov[1] = true;
                    if constexpr (FACES == 0) {
                        const P3 b{make_float2(xoff ? O.x.y : E.x, xoff ? E.x : O.x.x),
                                   make_float2(xoff ? O.y.y : E.y, xoff ? E.y : O.y.x),
                                   make_float2(xoff ? O.z.y : E.z, xoff ? E.z : O.z.x)};
                        h = P3{p2add(O.x, b.x), p2add(O.y, b.y), p2add(O.z, b.z)};
#pragma unroll
                        for (int d = 0; d < 4; ++d) h = P3{p2add(h.x, n[d].x), p2add(h.y, n[d].y), p2add(h.z, n[d].z)};
                    } else {
                        const P3 xm{make_float2(xoff ? O.x.x : E.x, xoff ? O.x.y : O.x.x),
                                    make_float2(xoff ? O.y.x : E.y, xoff ? O.y.y : O.y.x),
                                    make_float2(xoff ? O.z.x : E.z, xoff ? O.z.y : O.z.x)};
                        const P3 xp{make_float2(xoff ? O.x.y : O.x.x, xoff ? E.x : O.x.y),
                                    make_float2(xoff ? O.y.y : O.y.x, xoff ? E.y : O.y.y),
                                    make_float2(xoff ? O.z.y : O.z.x, xoff ? E.z : O.z.y)};
                        const float fb = x_face_factor(p.bc[0]);
                        const float2 Fm = make_float2(x0 == 0 ? fb : 1.0f, 1.0f);
                        const float2 Fp = make_float2(1.0f, x0 + 3u == 2u * Lh ? fb : 1.0f);
                        h = P3{p2fma(Fp, xp.x, p2mul(Fm, xm.x)), p2fma(Fp, xp.y, p2mul(Fm, xm.y)),
                               p2fma(Fp, xp.z, p2mul(Fm, xm.z))};
#pragma unroll
                        for (int d = 0; d < 4; ++d) {
                            const float2 F = p2(brick_factor(e.flags, d));
                            h = P3{p2fma(F, n[d].x, h.x), p2fma(F, n[d].y, h.y), p2fma(F, n[d].z, h.z)};
                        }
                        mov[0] = !(e.flags & 4u) && !(p.bc[0] == 2 && x0 == 0);
                        mov[1] = !(e.flags & 4u) && !(p.bc[0] == 2 && x0 + 3u == 2u * Lh);
                    }
                } else {
                    V3<float> Sv[2], hv[2], Ov[2];
                    const uint32_t q = 2u * Pc;
                    two = q + 1u < sites;
                    site0 = 0;
                    k = 0;
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        const uint32_t qv = v && !two ? q : q + uint32_t(v);
                        const uint32_t i = fast_div(qv, p.div_lh), kv = qv - i * Lh;
                        const BrickRow ev = tab[i];
                        const uint32_t xoff = (ev.flags + uint32_t(c)) & 1u;
                        const float* o = own + ev.own + kv;
                        const float* x = oth + ev.own;
                        Sv[v] = V3<float>{o[0], o[Lh], o[2 * Lh]};
                        Ov[v] = V3<float>{x[kv], x[Lh + kv], x[2 * Lh + kv]};
                        const uint32_t ke = xoff ? (kv + 1u == Lh ? 0u : kv + 1u) : (kv == 0 ? Lh - 1u : kv - 1u);
                        const V3<float> E{x[ke], x[Lh + ke], x[2 * Lh + ke]};
                        V3<float> nv[4];
                        if (!brick_neighbours(oth, pin, ev, kv, Lh, tag_in, &ctl->abort, nv)) failed = true;
                        const uint32_t xs = xoff + 2u * kv;
                        // -x, +x in order; the row's wrap crosses a face of the x axis
                        const float fb = FACES ? x_face_factor(p.bc[0]) : 1.0f;
                        const float fm = xs == 0 ? fb : 1.0f, fp = xs + 1u == 2u * Lh ? fb : 1.0f;
                        const V3<float> m = xoff ? Ov[v] : E, pl = xoff ? E : Ov[v];
                        V3<float> t{__fmaf_rn(fp, pl.x, __fmul_rn(fm, m.x)), __fmaf_rn(fp, pl.y, __fmul_rn(fm, m.y)),
                                    __fmaf_rn(fp, pl.z, __fmul_rn(fm, m.z))};
#pragma unroll
                        for (int d = 0; d < 4; ++d) {
                            const float F = FACES ? brick_factor(ev.flags, d) : 1.0f;
                            t.x = __fmaf_rn(F, nv[d].x, t.x);
                            t.y = __fmaf_rn(F, nv[d].y, t.y);
                            t.z = __fmaf_rn(F, nv[d].z, t.z);
                        }
                        hv[v] = t;
                        mov[v] = true;
                        if (FACES) mov[v] = !(ev.flags & 4u) && !(p.bc[0] == 2 && (xs == 0 || xs + 1u == 2u * Lh));
                        if (v == 0) {
                            site0 = xs + 2u * Lh * ev.row;
                            e = ev;
                            k = kv;
                        } else {
                            e1 = ev;
                            k1 = kv;
                            mov[v] = mov[v] && two;
                        }
                    }
                    S = pack(Sv);
                    h = pack(hv);
                    O = pack(Ov);
                }
                const uint4 w = philox(make_uint4(site0, sweep, tag_of(c, kPurposeMove), 0u), key0, key1);
                if (first) {  // the cone angle, now that everything else is at hand
                    first = false;
                    if (!mbar_wait(&tbar, uint32_t(sw - 1) & 1u) || *reinterpret_cast<volatile int*>(&s_fail)) failed = true;
                    cval = *reinterpret_cast<volatile float*>(&s_cone);
                }
                P3 Sf;
                unsigned n = 0;
                V3<float> Sv[2], hv[2], Sn[2];
                if constexpr (LAW == 0) {
                    n = pair_move(par, cval, w, S, h, mov, nullptr, Sf);
                } else {
                    unpack(S, Sv);
                    unpack(h, hv);
                    const V3<float> ax[2] = {V3<float>{par.e[0], par.e[1], par.e[2]},
                                             V3<float>{par.e[0], par.e[1], par.e[2]}};
                    n = scalar_move(par, cval, w, Sv, hv, ax, mov, Sn);
                    Sf = pack(Sn);
                }
                if (valid) {
                    nacc += n;
                    if constexpr (!ODD) {
                        if (n) {
                            float* o = own + e.own + k;
                            *reinterpret_cast<float2*>(o) = Sf.x;
                            *reinterpret_cast<float2*>(o + Lh) = Sf.y;
                            *reinterpret_cast<float2*>(o + 2 * Lh) = Sf.z;
                        }
                        if (e.flags & 2u) {
                            st_pair_packets(pout + size_t(e.row) * Lh + k, Sf, tag_out);
                        }
                    } else {
                        float* o = own + e.own + k;
                        o[0] = Sf.x.x;
                        o[Lh] = Sf.y.x;
                        o[2 * Lh] = Sf.z.x;
                        if (e.flags & 2u) st_packet(pout + size_t(e.row) * Lh + k, Sf.x.x, Sf.y.x, Sf.z.x, tag_out);
                        if (two) {
                            o = own + e1.own + k1;
                            o[0] = Sf.x.y;
                            o[Lh] = Sf.y.y;
                            o[2 * Lh] = Sf.z.y;
                            if (e1.flags & 2u)
                                st_packet(pout + size_t(e1.row) * Lh + k1, Sf.x.y, Sf.y.y, Sf.z.y, tag_out);
                        }
                    }
                    if constexpr (MEASURE > 0) {
                        if (c == 1) {
                            if constexpr (LAW == 0) {
                                const P3 ea{p2(par.e[0]), p2(par.e[1]), p2(par.e[2])};
                                pair_tile_parts<MEASURE, NS>(par, Sf, h, ea, O, ea, lf);
                            } else {
                                const V3<float> ax[2] = {V3<float>{par.e[0], par.e[1], par.e[2]},
                                                         V3<float>{par.e[0], par.e[1], par.e[2]}};
                                V3<float> Ov[2];
                                unpack(O, Ov);
                                scalar_tile_parts<MEASURE, NS>(par, Sn, hv, ax, Ov, ax, two ? 2 : 1, lf);
                            }
                        }
                    }
                }
                if constexpr (MEASURE > 0) {
                    if (c == 1 && ++nparts == uint32_t(kPartTiles)) {
                        fix += pair_parts_flush<NS>(lf, lane);
                        nparts = 0;
                    }
                }
            }
            if (c == 1) {  // the block's count (and sums) of the sweep, by the last warp done
                if constexpr (MEASURE > 0) {
                    if (nparts) fix += pair_parts_flush<NS>(lf, lane);
                    if (lane < NS && fix)
                        atomicAdd(reinterpret_cast<unsigned long long*>(&cta_sums[lane]), static_cast<unsigned long long>(fix));
                }
                const unsigned wacc = __reduce_add_sync(0xffffffffu, nacc);
                unsigned mine = 0;
                __syncwarp();
                if (lane == 0) {
                    if (wacc) atomicAdd(&cta_acc, wacc);
                    __threadfence_block();
                    mine = atomicAdd(&wdone, 1u) == unsigned(NW - 1);
                    if (mine) {
                        __threadfence_block();
                        const unsigned v = *reinterpret_cast<volatile unsigned*>(&cta_acc);
                        cta_acc = 0;
                        wdone = 0;
                        atomicAdd(&ctl->count[sw & 1], (1ull << 40) | v);
                    }
                }
                if constexpr (MEASURE > 0) {
                    if (__shfl_sync(0xffffffffu, mine, 0)) {
                        __threadfence_block();
                        if (lane < NS) {
                            const long long v = *reinterpret_cast<volatile long long*>(&cta_sums[lane]);
                            cta_sums[lane] = 0;
                            if (v)
                                atomicAdd(reinterpret_cast<unsigned long long*>(&a.record[size_t(sw) * kRecordWords + lane]),
                                          static_cast<unsigned long long>(v));
                        }
                    }
                }
            }
            if (workers_failed(failed)) alive = false;  // the pass is complete in the block
        }
    }
    if (!alive) {
        if (tid == 0) {
            *reinterpret_cast<volatile int*>(&s_fail) = 1;
            atomicExch(&ctl->abort, 1);
            atomicCAS(&L->st.error, 0, -4);  // MC_ERR_TIMEOUT
        }
        return;
    }
    // the rows back into the lattice
    brick_rows<false, Form::store_six, NW>(bsm, s, tab, nr, Lh, half, stride, warp, lane);
}

// Before a launch (of one lattice, or of many, by blockIdx.y): the control words
// (not the epoch) and the records of n measured sweeps zeroed, and before a
// launch whose epoch brick_clears all packets of the memory as well.
template <int THREADS>
__global__ void __launch_bounds__(THREADS) brick_prep_kernel(const __grid_constant__ BrickArgs one, const BrickArgs* many,
                                                             int n) {
    const BrickArgs& a = many ? many[blockIdx.y] : one;
    const uint32_t i = blockIdx.x * uint32_t(THREADS) + threadIdx.x;
    if (i < uint32_t(n * kRecordWords)) a.record[i] = 0;
    if (i == 0) {
        a.ctl->abort = 0;
        a.ctl->closed = 0;
        a.ctl->count[0] = a.ctl->count[1] = 0;
    }
    if (brick_clears(a.ctl->epoch)) {
        float4* const p = static_cast<float4*>(a.packets);
        for (uint32_t k = i; k < a.n_packets; k += gridDim.x * uint32_t(THREADS)) p[k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
}

}  // namespace mcgb

// xtal_pass.cuh -- colour passes, neighbour field and sample of the bcc, fcc
// and hcp lattices (Sec. 2: bcc as 2 interleaved simple cubic sub-lattices, fcc
// as 4, hcp as 4 simple tetragonal ones, each split red/black by cell parity
// and visited in turn).  Spins of sub-lattice s and colour c are the simple
// cubic colour arrays of that sub-lattice: component a at spins[((2 s + c) 3 +
// a) stride + q], q = (x >> 1) + Lh (y + Ly z) for cell (x, y, z).  One lattice
// per launch, one lane per site, persistent warps.
//
// The neighbours of a site depend on its sub-lattice alone, so each sub-lattice
// has its own instance with the entries as compile-time constants: an entry is
// then one three-term sum (of the cell's three x, y and z terms, taken once per
// site with their wraps) and three loads off a launch constant.  Walking a table
// in shared memory instead, with the wraps and the address formed per entry,
// cost 726 warp instructions per 32 sites of an fcc sub-set (25 us a pass of
// 96^3 cells, 41% issued per cycle); here 342 and 14.5 us.  What bounds it now is
// latency, of a site's loads and of its draw and move behind them: 38% issued per
// cycle at 16 warps per SM.
#pragma once
#include "kernels.h"
#include "pair_math.cuh"
#include "pass_impl.cuh"

namespace mcgb {

// ------------------------------------------------------------- neighbour entries
// An entry (t, d) of sub-lattice s: the site of sub-lattice t in the cell at
// offset d in {-1, 0, 1}^3.  Types 1 bcc, 2 fcc, 3 hcp.  Positions in units of
// 1/2 (bcc, fcc) or 1/6 (hcp) of the cell; hcp in the orthohexagonal cell (a,
// sqrt(3) a, sqrt(8/3) a), so that the squared distances below are integers.
struct XtalEnt {
    int t = 0, dx = 0, dy = 0, dz = 0;
    bool nn = true;   // nearest (coupling J) or next-nearest (J2)
    bool fwd = true;  // one of each entry and its reverse (sub-lattice t -> s, offset -d)
};

__host__ __device__ constexpr int xtal_nsub(int type) { return type == 1 ? 2 : 4; }

__host__ __device__ constexpr int xtal_basis(int type, int s, int a) {
    if (type == 1) return s;                        // (0,0,0), (1,1,1)
    if (type == 2) return s == 0 ? 0 : s == 1 ? (a < 2) : s == 2 ? (a != 1) : (a > 0);
    if (s == 0) return 0;                           // hcp: (0,0,0), (3,3,0), (3,1,3), (0,4,3)
    return a == 0 ? (s < 3 ? 3 : 0) : a == 1 ? (s == 1 ? 3 : s == 2 ? 1 : 4) : (s == 1 ? 0 : 3);
}

// 1 nearest, 2 next-nearest, 0 neither
__host__ __device__ constexpr int xtal_shell(int type, int s, int t, int dx, int dy, int dz) {
    const int u = type == 3 ? 6 : 2;
    const int x = xtal_basis(type, t, 0) - xtal_basis(type, s, 0) + u * dx;
    const int y = xtal_basis(type, t, 1) - xtal_basis(type, s, 1) + u * dy;
    const int z = xtal_basis(type, t, 2) - xtal_basis(type, s, 2) + u * dz;
    if (type == 3) return 3 * x * x + 9 * y * y + 8 * z * z == 108 ? 1 : 0;
    const int r2 = x * x + y * y + z * z;
    return r2 == (type == 1 ? 3 : 2) ? 1 : (r2 == 4 ? 2 : 0);
}

// Entry i of sub-lattice s, in the order in which the field is summed: by t,
// then d_z, d_y, d_x from -1 to 1 (J2: next-nearest entries among them).
__host__ __device__ constexpr XtalEnt xtal_entry(int type, bool j2, int s, int i) {
    int n = 0;
    for (int t = 0; t < xtal_nsub(type); ++t)
        for (int dz = -1; dz <= 1; ++dz)
            for (int dy = -1; dy <= 1; ++dy)
                for (int dx = -1; dx <= 1; ++dx) {
                    const int shell = xtal_shell(type, s, t, dx, dy, dz);
                    if (shell == 0 || (shell == 2 && !j2)) continue;
                    if (n++ == i) {
                        XtalEnt e;
                        e.t = t;
                        e.dx = dx;
                        e.dy = dy;
                        e.dz = dz;
                        e.nn = shell == 1;
                        e.fwd = t > s || (t == s && (dz > 0 || (dz == 0 && (dy > 0 || (dy == 0 && dx > 0)))));
                        return e;
                    }
                }
    return XtalEnt{};
}

__host__ __device__ constexpr int xtal_entries(int type, bool j2) {
    return type == 1 ? (j2 ? 14 : 8) : type == 2 ? (j2 ? 18 : 12) : 12;
}

// ------------------------------------------------------------------- geometry
// Colour index q's cell and the x, y and z terms of its neighbours' colour
// indices (offsets -1, 0, 1, wrapped): the colour index of the cell at offset d
// is kx[dx + 1] + ry[dy + 1] + rz[dz + 1] in the colour (c + dx + dy + dz) & 1.
struct XCell {
    uint32_t x, y, z;
    uint32_t kx[3], ry[3], rz[3];
};

__device__ __forceinline__ XCell xtal_cell(const LatParams& p, int colour, uint32_t q) {
    const uint32_t Lh = uint32_t(p.Lh), Ly = uint32_t(p.Ly), Lz = uint32_t(p.Lz), plane = Lh * Ly;
    const uint32_t row = fast_div(q, p.div_lh);
    const uint32_t k = q - row * Lh;
    const uint32_t z = fast_div(row, p.div_ly);
    const uint32_t y = row - z * Ly;
    const uint32_t xoff = (y + z + uint32_t(colour)) & 1u;
    XCell c;
    c.x = 2u * k + xoff;
    c.y = y;
    c.z = z;
    c.kx[0] = xoff ? k : (k == 0 ? Lh - 1u : k - 1u);
    c.kx[1] = k;
    c.kx[2] = xoff ? (k + 1u == Lh ? 0u : k + 1u) : k;
    c.ry[0] = Lh * (y == 0 ? Ly - 1u : y - 1u);
    c.ry[1] = Lh * y;
    c.ry[2] = Lh * (y + 1u == Ly ? 0u : y + 1u);
    c.rz[0] = plane * (z == 0 ? Lz - 1u : z - 1u);
    c.rz[1] = plane * z;
    c.rz[2] = plane * (z + 1u == Lz ? 0u : z + 1u);
    return c;
}

template <typename R, int TYPE, int J2, int SUB, bool HALF, int I = 0>
__device__ __forceinline__ void xtal_load(const XtalArgs& a, const XCell& c, int colour, V3<R>* nb) {
    constexpr XtalEnt e = xtal_entry(TYPE, J2 != 0, SUB, I);
    if constexpr (!HALF || e.fwd) {
        const uint32_t q = c.kx[e.dx + 1] + c.ry[e.dy + 1] + c.rz[e.dz + 1];
        const R* b = static_cast<const R*>(a.spins) +
                     size_t(2 * e.t + ((colour + e.dx + e.dy + e.dz + 4) & 1)) * 3 * a.stride;
        nb[I] = V3<R>{b[q], b[a.stride + q], b[2 * size_t(a.stride) + q]};
    }
    if constexpr (I + 1 < xtal_entries(TYPE, J2 != 0)) xtal_load<R, TYPE, J2, SUB, HALF, I + 1>(a, c, colour, nb);
}

template <typename R, int TYPE, int J2, int SUB, bool HALF, int I = 0>
__device__ __forceinline__ void xtal_add(const XtalArgs& a, const V3<R>* nb, V3<R>& h) {
    constexpr XtalEnt e = xtal_entry(TYPE, J2 != 0, SUB, I);
    if constexpr (!HALF || e.fwd) {
        R J;
        if constexpr (kIsF64<R>) J = e.nn ? a.J : a.J2;
        else J = e.nn ? a.fJ : a.fJ2;
        h.x = h.x + J * nb[I].x;
        h.y = h.y + J * nb[I].y;
        h.z = h.z + J * nb[I].z;
    }
    if constexpr (I + 1 < xtal_entries(TYPE, J2 != 0)) xtal_add<R, TYPE, J2, SUB, HALF, I + 1>(a, nb, h);
}

// h = sum over the neighbours of a site of sub-lattice SUB, colour `colour`, in
// cell c, of J S_j.  HALF: the forward entries only (every bond once over the
// lattice).  Every neighbour is loaded before the first is added: taken entry by
// entry, in the registers the compiler then chose, few of the 3 x 8 to 18 loads
// were in flight and a site waited for L2 several times over.
template <typename R, int TYPE, int J2, int SUB, bool HALF = false>
__device__ __forceinline__ V3<R> xtal_field(const XtalArgs& a, const XCell& c, int colour) {
    V3<R> nb[xtal_entries(TYPE, J2 != 0)];
    xtal_load<R, TYPE, J2, SUB, HALF>(a, c, colour, nb);
    V3<R> h{R(0), R(0), R(0)};
    xtal_add<R, TYPE, J2, SUB, HALF>(a, nb, h);
    return h;
}

// Blocks per SM that the kernels are compiled for: two in FP32, so that the loads
// of a whole site fit the registers (80 to 128).  Blocks of 10 + 10 sweeps at two
// / three / four: fcc 96^3 2310 / 2439, 64^3 1145 / 1341 / 1431, with J2 96^3 2650
// / - / 2846 us, hcp 96^3 2297 / 2449, bcc 128^3 with J2 2493 / 2604, 64^3 774 / 777
// / 800; without a bound (40 to 66 registers) fcc 96^3 2706.
template <typename R>
constexpr int kXtalMinb = kIsF64<R> ? 1 : 2;

// ------------------------------------------------------------------- kernels
// Pass over sub-set (SUB, colour); finalize != 0 closes the sweep (the last
// sub-set of an unmeasured sweep).  Launched with programmatic serialisation:
// its blocks start while the previous pass drains and wait for it here.
template <typename R, int TYPE, int J2, int SUB>
__global__ void __launch_bounds__(kBlock, kXtalMinb<R>) xtal_pass_kernel(const __grid_constant__ XtalArgs a, uint32_t ntiles,
                                                           const R* __restrict__ cone, int colour, int finalize) {
    asm volatile("griddepcontrol.launch_dependents;");
    const LatParams& p = a.lat->p;
    LatState& st = a.lat->st;
    const WarpChunk wc = warp_chunk(ntiles);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (wc.begin >= wc.end) return;
    const int lane = wc.lane;
    const Par<R> par = load_par<R>(p);
    const R c = cone[st.theta];
    const uint32_t sweep = st.sweep;
    const uint32_t tag = tag_of(colour, kPurposeMove);
    R* own = static_cast<R*>(a.spins) + size_t(2 * SUB + colour) * 3 * a.stride;
    const V3<R> e_ax{par.e[0], par.e[1], par.e[2]};
    unsigned nacc = 0;
    for (uint32_t tile = wc.begin; tile < wc.end; ++tile) {
        const uint32_t q = tile * 32u + uint32_t(lane);
        if (q >= p.Nc) continue;
        const XCell cell = xtal_cell(p, colour, q);
        const uint32_t site = uint32_t(SUB) + uint32_t(xtal_nsub(TYPE)) *
                                                  (cell.x + uint32_t(p.Lx) * (cell.y + uint32_t(p.Ly) * cell.z));
        const V3<R> S{own[q], own[a.stride + q], own[2 * size_t(a.stride) + q]};
        const V3<R> h = xtal_field<R, TYPE, J2, SUB>(a, cell, colour);
        V3<R> Sn;
        R P;
        if (!cone_trial(S, c, site, sweep, tag, p.key0, p.key1, Sn, P)) continue;
        if (metropolis(delta_e(par, S, Sn, h, e_ax), par, P)) {
            own[q] = Sn.x;
            own[a.stride + q] = Sn.y;
            own[2 * size_t(a.stride) + q] = Sn.z;
            ++nacc;
        }
    }
    publish(st, lane, nacc, false, 0, colour, wc.end - wc.begin, ntiles, finalize != 0,
            [&] { finalize_sweep(p, st, 0, false, lane); });
}

// Constrained sweeps (Table A2) of a crystal: the neighbour field of every
// site of sub-set (SUB, colour) into LatParams::pfield as (h_x, h_y, h_z, 0),
// summed from the spins (which the pair passes keep in step; the sub-set's own
// spins are not among its neighbours).
template <typename R, int TYPE, int J2, int SUB>
__global__ void __launch_bounds__(kBlock, kXtalMinb<R>) xtal_field_kernel(const __grid_constant__ XtalArgs a, uint32_t ntiles, int colour) {
    const LatParams& p = a.lat->p;
    const WarpChunk wc = warp_chunk(ntiles);
    Spin4<R>* fld = static_cast<Spin4<R>*>(p.pfield);
    for (uint32_t tile = wc.begin; tile < wc.end; ++tile) {
        const uint32_t q = tile * 32u + uint32_t(wc.lane);
        if (q >= p.Nc) continue;
        const V3<R> h = xtal_field<R, TYPE, J2, SUB>(a, xtal_cell(p, colour, q), colour);
        fld[q] = Spin4<R>{h.x, h.y, h.z, R(0)};
    }
}

// S.h of the exchange sum, with its FP32 rounding order in so many words: left
// to the compiler it would change from instance to instance and with it the
// energies of small lattices (by up to 5e-9)
template <typename R>
__device__ __forceinline__ R xtal_dot(V3<R> S, V3<R> h) {
    if constexpr (kIsF64<R>) return S.x * h.x + S.y * h.y + S.z * h.z;
    else return __fmaf_rn(S.z, h.z, __fmaf_rn(S.x, h.x, __fmul_rn(S.y, h.y)));
}

// Sample of the current state: M, the exchange sum over every bond once (sum_i
// S_i . h_i over the forward entries), the uniaxial, cubic and torque sums;
// tiles of 32 sites over the 2 nsub sub-sets; closes the sweep.  FP64: the warp
// sums of a tile are reduced in a fixed butterfly order and rounded to fixed
// point on lane i (int64).  FP32: a lane adds its sites of 16 tiles in fixed
// point before the warp adds the lanes, exact integers either way (a warp sum per
// tile instead: bcc 48^3 591 against 551 us a block of 10 + 10 sweeps, fcc 32^3 748
// against 704, 96^3 the same); of fewer tiles where |S . h|, whose couplings are
// inside the sum, could take 16 of them out of an int32, and for couplings that take
// one site out of it the exchange sum is formed in 64 bits.  LEVEL 2: with the
// torques.
template <typename R, int TYPE, int J2, int LEVEL>
__global__ void __launch_bounds__(kBlock, kXtalMinb<R>) xtal_sample_kernel(const __grid_constant__ XtalArgs a, uint32_t ntiles,
                                                             uint32_t tiles_per_subset) {
    constexpr int NS = LEVEL >= 2 ? kNumSums : kSumTux;  // sums sampled
    asm volatile("griddepcontrol.launch_dependents;");
    const LatParams& p = a.lat->p;
    const WarpChunk wc = warp_chunk(ntiles);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (wc.begin >= wc.end) return;
    const int lane = wc.lane;
    const Par<R> par = load_par<R>(p);
    const V3<R> e_ax{par.e[0], par.e[1], par.e[2]};
    long long fix = 0;
    int lf[NS] = {}, nparts = 0;
    // tiles whose parts fit an int32 at scale 2^22: |S . h| is at most `most` (up to
    // the rounding of a unit spin)
    const float most = 1.01f * (float(TYPE == 1 ? 8 : 12) * fabsf(a.fJ) + (J2 ? 6.0f * fabsf(a.fJ2) : 0.0f));
    const int parts = most < 512.0f / kPartTiles ? kPartTiles : most < 512.0f ? int(512.0f / most) : 0;
    for (uint32_t tile = wc.begin; tile < wc.end; ++tile) {
        const uint32_t set = tile / tiles_per_subset;  // 2 sub + colour
        const int sub = int(set >> 1), colour = int(set & 1u);
        const uint32_t q = (tile - set * tiles_per_subset) * 32u + uint32_t(lane);
        Sums<R> sums;
        for (int i = 0; i < kNumSums; ++i) sums.v[i] = R(0);
        if (q < p.Nc) {
            const XCell cell = xtal_cell(p, colour, q);
            const R* own = static_cast<const R*>(a.spins) + size_t(set) * 3 * a.stride;
            const V3<R> S{own[q], own[a.stride + q], own[2 * size_t(a.stride) + q]};
            V3<R> h;
            if (sub == 0) h = xtal_field<R, TYPE, J2, 0, true>(a, cell, colour);
            else if (sub == 1) h = xtal_field<R, TYPE, J2, 1, true>(a, cell, colour);
            else if constexpr (xtal_nsub(TYPE) == 4) {
                if (sub == 2) h = xtal_field<R, TYPE, J2, 2, true>(a, cell, colour);
                else h = xtal_field<R, TYPE, J2, 3, true>(a, cell, colour);
            }
            add_site<R, LEVEL>(sums, S, e_ax);
            sums.v[kSumEx] = xtal_dot(S, h);
        }
        if constexpr (kIsF64<R>) {
            fix += __double2ll_rn(warp_sums_f64<NS>(sums.v, lane) * kFixScale);
        } else {
            if (parts == 0) {
                long long ex = __float2ll_rn(sums.v[kSumEx] * float(kFixScaleF32));
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) ex += __shfl_xor_sync(0xffffffffu, ex, o);
                if (lane == kSumEx) fix += ex;
                sums.v[kSumEx] = 0.0f;
            }
#pragma unroll
            for (int i = 0; i < NS; ++i) lf[i] += __float2int_rn(sums.v[i] * float(kFixScaleF32));
            if (++nparts >= max(parts, 1)) {
                fix += pair_parts_flush<NS>(lf, lane);
                nparts = 0;
            }
        }
    }
    if constexpr (!kIsF64<R>) {
        if (nparts) fix += pair_parts_flush<NS>(lf, lane);
    }
    publish(a.lat->st, lane, 0, true, fix, 3, wc.end - wc.begin, ntiles, true,
            [&] { finalize_sweep(p, a.lat->st, 1, LEVEL >= 2, lane); });
}

}  // namespace mcgb

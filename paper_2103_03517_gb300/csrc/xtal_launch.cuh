// xtal_launch.cuh -- launchers of the crystal kernels (xtal_pass.cuh), one
// instance per lattice type, next-nearest exchange and sub-lattice.  Included
// inside an anonymous namespace after R is defined.
#pragma once
#include "spread.cuh"

template <typename... K, typename... A>
cudaError_t xtal_launch(void (*kernel)(K...), uint32_t ntiles, uint32_t cap, cudaStream_t s, A... a) {
    const Spread sp = spread_warps(ntiles, cap);
    return launch_chained_if(!kIsF64<R> || chain_small(sp, cap), kernel, sp.blocks, sp.threads, s, a...);
}

template <int TYPE, int J2>
struct Xtal {
    template <int SUB>
    static cudaError_t pass1(const XtalArgs& a, uint32_t nt, const R* cone, int colour, int finalize, cudaStream_t s) {
        static const uint32_t cap = resident_blocks(xtal_pass_kernel<R, TYPE, J2, SUB>);
        return xtal_launch(xtal_pass_kernel<R, TYPE, J2, SUB>, nt, cap, s, a, nt, cone, colour, finalize);
    }
    static cudaError_t pass(const XtalArgs& a, uint32_t nt, const R* cone, int sub, int colour, int finalize,
                            cudaStream_t s) {
        if (sub == 0) return pass1<0>(a, nt, cone, colour, finalize, s);
        if (sub == 1) return pass1<1>(a, nt, cone, colour, finalize, s);
        if constexpr (xtal_nsub(TYPE) == 4) {
            if (sub == 2) return pass1<2>(a, nt, cone, colour, finalize, s);
            return pass1<3>(a, nt, cone, colour, finalize, s);
        }
        return cudaErrorInvalidValue;
    }
    template <int SUB>
    static void field1(const XtalArgs& a, uint32_t nt, int colour, cudaStream_t s) {
        static const uint32_t cap = resident_blocks(xtal_field_kernel<R, TYPE, J2, SUB>);
        const Spread sp = spread_warps(nt, cap);
        xtal_field_kernel<R, TYPE, J2, SUB><<<sp.blocks, sp.threads, 0, s>>>(a, nt, colour);
    }
    static void field(const XtalArgs& a, uint32_t nt, int sub, int colour, cudaStream_t s) {
        if (sub == 0) field1<0>(a, nt, colour, s);
        else if (sub == 1) field1<1>(a, nt, colour, s);
        else if constexpr (xtal_nsub(TYPE) == 4) {
            if (sub == 2) field1<2>(a, nt, colour, s);
            else field1<3>(a, nt, colour, s);
        }
    }
    template <int LEVEL>
    static cudaError_t sample1(const XtalArgs& a, uint32_t nt, uint32_t per, cudaStream_t s) {
        static const uint32_t cap = resident_blocks(xtal_sample_kernel<R, TYPE, J2, LEVEL>);
        return xtal_launch(xtal_sample_kernel<R, TYPE, J2, LEVEL>, nt, cap, s, a, nt, per);
    }
    static cudaError_t sample(const XtalArgs& a, uint32_t nt, uint32_t per, int level, cudaStream_t s) {
        return level >= 2 ? sample1<2>(a, nt, per, s) : sample1<1>(a, nt, per, s);
    }
};

// f(Xtal<type, j2>) of lattice a
template <typename F>
auto by_type(const XtalArgs& a, F&& f) {
    if (a.type == 1) return a.j2 ? f(Xtal<1, 1>{}) : f(Xtal<1, 0>{});
    if (a.type == 2) return a.j2 ? f(Xtal<2, 1>{}) : f(Xtal<2, 0>{});
    return f(Xtal<3, 0>{});
}

cudaError_t pass(const XtalArgs& a, uint32_t nt, const void* cone, int sub, int colour, int finalize, cudaStream_t s) {
    return by_type(a, [&](auto x) { return x.pass(a, nt, static_cast<const R*>(cone), sub, colour, finalize, s); });
}

void field(const XtalArgs& a, uint32_t nt, int sub, int colour, cudaStream_t s) {
    by_type(a, [&](auto x) { x.field(a, nt, sub, colour, s); });
}

cudaError_t sample(const XtalArgs& a, uint32_t nt, uint32_t per, int level, cudaStream_t s) {
    return by_type(a, [&](auto x) { return x.sample(a, nt, per, level, s); });
}

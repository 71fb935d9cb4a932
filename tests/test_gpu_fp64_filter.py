"""The FP64 Metropolis decision taken in FP32 where FP32 can take it
(boltzmann_filter, csrc/pass_impl.cuh) is the exact test's: the chain stays the
oracle's bit for bit over temperatures from almost all moves refused to almost
all accepted, where -dE/T runs from far below FP32's range to nearly 0, in free
and in constrained sweeps (whose test has a factor and takes falling energies
too)."""
import numpy as np
import pytest

import oracle
import paper_2103_03517_gb300 as mc
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2103_03517_gb300 import build as libbuild
    libbuild.build()


@pytest.mark.parametrize("T", [1e-300, 1e-39, 1e-6, 1e-3, 0.05, 0.9, 40.0, 1e6, 1e39])
@pytest.mark.parametrize("constrained", [False, True])
def test_fp64_decisions_equal_the_exact_test(T, constrained):
    dims, N = (16, 12, 10), 16 * 12 * 10
    spins = workloads.perturbed_spins(N, 3, 0.4) if constrained else workloads.random_spins(N, 3)
    kw = dict(Kc=0.1, H=(0.1, 0.0, 0.3), T=T, seed=11)
    o = oracle.Lattice(dims, J=1.0, Ku=0.2, **kw)
    o.set_spins(spins)
    h = mc.mc_create_ex(mc.make_desc(dims, K_u=0.2, K_c=kw["Kc"], H=kw["H"], T=T, seed=11, precision=mc.MC_FP64))
    try:
        mc.mc_set_spins(h, spins)
        for n, meas in ((6, False), (6, True)):
            if constrained:
                mc.mc_constrained_sweep(h, 20.0, 30.0, n, meas)
                o.constrained_sweep(20.0, 30.0, n, measure=meas)
            else:
                mc.mc_sweep(h, n, meas)
                o.sweep(n, measure=meas)
        assert np.array_equal(mc.mc_get_spins(h, N), o.spins())
        assert mc.mc_get_theta(h)[0] == o.theta
        ob, st = mc.mc_measure(h), o.stats()
        assert abs(ob.ml - st["ml"] / st["n"]) < 1e-9
    finally:
        mc.mc_destroy(h)

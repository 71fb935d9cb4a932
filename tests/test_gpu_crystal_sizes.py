"""The per-sub-lattice instances of the crystal kernels (csrc/xtal_pass.cuh) at
the sizes where their wraps and tiles can go wrong: two cells across an axis,
rows shorter than a warp that end inside a tile, odd half rows, a part-full
last tile.  FP64, bit for bit the oracle's chain."""
import numpy as np
import pytest

import oracle
import paper_2103_03517_gb300 as mc
import workloads

pytestmark = pytest.mark.gpu

KIND = {mc.MC_BCC: oracle.BCC, mc.MC_FCC: oracle.FCC, mc.MC_HCP: oracle.HCP}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2103_03517_gb300 import build as libbuild
    libbuild.build()


@pytest.mark.parametrize("lattice,J2", [(mc.MC_BCC, 0.0), (mc.MC_BCC, 0.2), (mc.MC_FCC, 0.0), (mc.MC_FCC, 0.2),
                                        (mc.MC_HCP, 0.0)])
@pytest.mark.parametrize("cells", [(2, 2, 2), (10, 6, 4), (34, 4, 2), (6, 2, 10)])
def test_crystal_instances_equal_the_oracle(lattice, J2, cells):
    N = (2 if lattice == mc.MC_BCC else 4) * cells[0] * cells[1] * cells[2]
    spins = workloads.random_spins(N, 5)
    kw = dict(Kc=0.02, H=(0.0, 0.1, 0.2), T=0.9, seed=7)
    o = oracle.Crystal(KIND[lattice], cells, J1=1.0, J2=J2, Ku=0.05, **kw)
    o.set_spins(spins)
    h = mc.mc_create_ex(mc.make_desc(cells, J2=J2, K_u=0.05, K_c=kw["Kc"], H=kw["H"], T=kw["T"], seed=kw["seed"],
                                     lattice=lattice, precision=mc.MC_FP64))
    try:
        mc.mc_set_spins(h, spins)
        for n, meas in ((3, False), (2, True)):
            mc.mc_sweep(h, n, meas)
            o.sweep(n, measure=meas)
        assert np.array_equal(mc.mc_get_spins(h, N), o.spins())
        assert mc.mc_get_theta(h)[0] == o.theta()
        ob, st = mc.mc_measure(h), o.stats()
        np.testing.assert_allclose([ob.ml, ob.e], [st["ml"], st["e"]], rtol=0, atol=1e-9)
    finally:
        mc.mc_destroy(h)


@pytest.mark.parametrize("crystal,L", [(mc.MC_FCC, 80), (mc.MC_BCC, 100)])
def test_sample_of_many_tiles_a_warp(crystal, L):
    """More than 16 tiles a warp, so that the lanes' integer parts are summed over
    several runs.  Each site's m_a is rounded once, at 2^-22: the mean is within
    2^-23 of the mean of the spins."""
    h = mc.mc_create_ex(mc.make_desc((L, L, L), K_u=0.02, T=1.2, seed=6, lattice=crystal, ring_capacity=4))
    N = L ** 3 * (4 if crystal == mc.MC_FCC else 2)
    mc.mc_sweep(h, 3)
    mc.mc_sweep(h, 1, measure=True)
    m = np.asarray(mc.mc_get_spins(h, N), dtype=np.float64).mean(axis=0)
    o = mc.mc_measure(h)
    mc.mc_destroy(h)
    assert np.max(np.abs(np.asarray(o.m) - m)) <= 2.0 ** -23

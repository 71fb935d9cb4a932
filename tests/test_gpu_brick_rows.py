"""The load and store of brick sweeps (rows of every length class: several to a
warp, one, several warps to one; numbers of rows that do not fill a warp) and the
shortest calls that a group takes as bricks."""
import numpy as np
import pytest

import paper_2103_03517_gb300 as mc
import workloads

pytestmark = pytest.mark.gpu

O = mc.MC_OPEN


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2103_03517_gb300 import build as libbuild
    libbuild.build()


@pytest.mark.parametrize("dims", [(4, 7, 9), (8, 5, 5), (16, 9, 3), (20, 7, 5), (32, 5, 7), (36, 9, 5), (64, 7, 3), (68, 6, 4),
                                  (136, 5, 5), (4096, 4, 2), (6, 7, 9), (66, 5, 3)])
def test_rows_of_every_length(dims):
    N = dims[0] * dims[1] * dims[2]
    out = []
    for path in (mc.MC_PATH_AUTO, mc.MC_PATH_ROW):
        h = mc.mc_create_ex(mc.make_desc(dims, K_u=0.05, T=0.9, seed=5, boundary=(0, O, O), kernel_path=path, ring_capacity=8))
        mc.mc_set_spins(h, workloads.random_spins(N, 11))
        for n, meas in [(3, False), (4, True), (3, True)]:
            mc.mc_sweep(h, n, meas)
        out.append((mc.mc_get_spins(h, N), mc.mc_get_theta(h), mc.mc_measure(h).asdict(), mc.mc_samples(h, 8)))
        mc.mc_destroy(h)
    a, b = out
    assert np.array_equal(a[0], b[0]) and a[1] == b[1] and a[2] == b[2] and np.array_equal(a[3], b[3])


@pytest.mark.parametrize("sizes,shortest", [((64,) * 8, 4), ((32,) * 8, 3), ((16,) * 2, 3)])
def test_shortest_call_of_a_group_that_sweeps_as_bricks(sizes, shortest):
    """Groups that gain little a sweep take a sweep more to pay for their load."""
    hs = [mc.mc_create_ex(mc.make_desc((L,) * 3, T=0.7, seed=i, ring_capacity=4)) for i, L in enumerate(sizes)]
    g = mc.mc_group_create(hs)
    for n in (2, 3, 4):
        _, kinds = mc.mc_group_time_kernels(g, n)
        assert (kinds[3] > 0) == (n >= shortest), (n, kinds)
    mc.mc_group_destroy(g)
    for h in hs:
        mc.mc_destroy(h)

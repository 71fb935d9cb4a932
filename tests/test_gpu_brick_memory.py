"""Lattices whose brick memory cannot be had sweep by launches, alone and in a
group, with the same chain, and ask for it once.  The failure is injected on the
host: MC_BRICK_INJECT_NOMEM=k, read when a lattice is created, fails its first k
requests.
"""
import numpy as np
import pytest

import paper_2103_03517_gb300 as mc
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2103_03517_gb300 import build as libbuild
    libbuild.build()


def _make(dims, path, seed):
    h = mc.mc_create_ex(mc.make_desc(dims, K_u=0.03, T=0.7, seed=seed, ring_capacity=64, kernel_path=path))
    mc.mc_set_spins(h, workloads.random_spins(dims[0] * dims[1] * dims[2], seed))
    return h


def _read(h, dims):
    return (mc.mc_get_spins(h, dims[0] * dims[1] * dims[2]), mc.mc_get_theta(h), mc.mc_measure(h).asdict(),
            mc.mc_samples(h, 64))


@pytest.mark.parametrize("dims", [[(16, 16, 16)], [(18, 10, 8)], [(16, 16, 16), (20, 12, 10), (18, 10, 8)]])
@pytest.mark.parametrize("fails", [1, 100])
def test_without_brick_memory(monkeypatch, dims, fails):
    monkeypatch.setenv("MC_BRICK_INJECT_NOMEM", str(fails))
    hs = [_make(d, mc.MC_PATH_AUTO, i) for i, d in enumerate(dims)]
    monkeypatch.delenv("MC_BRICK_INJECT_NOMEM")
    ref = [_make(d, mc.MC_PATH_ROW, i) for i, d in enumerate(dims)]
    g = mc.mc_group_create(hs)
    mc.mc_group_sweep(g, 5)
    # given up: a request that would be granted now is not made
    _, kinds = mc.mc_group_time_kernels(g, 4)
    assert kinds[3] == 0 and kinds[1] > 0, kinds
    for n, meas in [(20, True), (3, True)]:
        mc.mc_group_sweep(g, n, meas)
    mc.mc_group_sync(g)
    for r in ref:
        for n, meas in [(5, False), (4, False), (20, True), (3, True)]:
            mc.mc_sweep(r, n, meas)
    for h, r, d in zip(hs, ref, dims):
        a, b = _read(h, d), _read(r, d)
        assert np.array_equal(a[0], b[0]) and a[1] == b[1] and a[2] == b[2] and np.array_equal(a[3], b[3]), d
    mc.mc_group_destroy(g)
    for h in hs + ref:
        mc.mc_destroy(h)

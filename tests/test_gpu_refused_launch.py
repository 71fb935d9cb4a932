"""Brick launches that the device refuses (a smaller device, or one that allows no
cooperative launch): nothing of them has run, and the lattices are swept by
launches from where they stand, alone or in a group, with the chain that they
would have had.  The refusal is injected on the host: MC_BRICK_INJECT_REFUSAL=k,
read when a lattice is created, refuses its launches of fewer than k sweeps.
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


def _same(a, b):
    return np.array_equal(a[0], b[0]) and a[1] == b[1] and a[2] == b[2] and np.array_equal(a[3], b[3])


@pytest.mark.parametrize("k,runs", [(4096, [(5, False), (20, True), (3, True)]),   # every launch
                                    (3, [(4, True), (2050, False), (4, True)])])   # the second of a long run
def test_lone_lattice(monkeypatch, k, runs):
    for dims in [(16, 16, 16), (20, 12, 10), (18, 10, 8)]:
        monkeypatch.setenv("MC_BRICK_INJECT_REFUSAL", str(k))
        h = _make(dims, mc.MC_PATH_AUTO, 3)
        monkeypatch.delenv("MC_BRICK_INJECT_REFUSAL")
        ref = _make(dims, mc.MC_PATH_ROW, 3)
        for n, meas in runs:
            mc.mc_sweep(h, n, meas)
            mc.mc_sweep(ref, n, meas)
        assert _same(_read(h, dims), _read(ref, dims)), dims
        mc.mc_destroy(h)
        mc.mc_destroy(ref)


@pytest.mark.parametrize("refused", [0, 2, 4])
def test_group_with_one_refused_kernel_instance(monkeypatch, refused):
    """The lattices of a group take one launch per kernel instance (row layout,
    even rows outside it, odd rows); one of them is refused."""
    dims = [(16, 16, 16), (8, 8, 8), (20, 12, 10), (12, 8, 8), (18, 10, 8)]
    hs = []
    for i, d in enumerate(dims):
        if i == refused:
            monkeypatch.setenv("MC_BRICK_INJECT_REFUSAL", "4096")
        hs.append(_make(d, mc.MC_PATH_AUTO, i))
        monkeypatch.delenv("MC_BRICK_INJECT_REFUSAL", raising=False)
    ref = [_make(d, mc.MC_PATH_ROW, i) for i, d in enumerate(dims)]
    g = mc.mc_group_create(hs)
    for n, meas in [(5, False), (18, True), (4, True)]:
        mc.mc_group_sweep(g, n, meas)
        for h in ref:
            mc.mc_sweep(h, n, meas)
    mc.mc_group_sync(g)
    for h, r, d in zip(hs, ref, dims):
        assert _same(_read(h, d), _read(r, d)), d
    mc.mc_group_destroy(g)
    for h in hs + ref:
        mc.mc_destroy(h)

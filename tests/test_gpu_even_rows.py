"""The row kernel's LAW 1 (csrc/row_pass.cuh): FP32 lattices outside the row
layout with an even number of sites per colour and row, taken two neighbouring
sites a lane, against the general kernel (MC_PATH_GENERAL).  Same draws, same
operations in the same order, exact integer sums: the same bits.
"""
import numpy as np
import pytest

import paper_2103_03517_gb300 as mc
import workloads

pytestmark = pytest.mark.gpu

P, O, K, A = mc.MC_PERIODIC, mc.MC_OPEN, mc.MC_PINNED, mc.MC_ANTIPERIODIC


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2103_03517_gb300 import build as libbuild
    libbuild.build()


def _read(h, N, ring):
    return mc.mc_get_spins(h, N), mc.mc_get_theta(h), mc.mc_measure(h).asdict(), mc.mc_samples(h, ring)


def _run(dims, kw, spins, path):
    h = mc.mc_create_ex(mc.make_desc(dims, kernel_path=path, ring_capacity=8, **kw))
    try:
        mc.mc_set_spins(h, spins)
        mc.mc_sweep(h, 3)
        mc.mc_sweep(h, 4, True)
        mc.mc_sweep(h, 17)
        return _read(h, dims[0] * dims[1] * dims[2], 8)
    finally:
        mc.mc_destroy(h)


def _assert_same(a, b, what):
    assert np.array_equal(a[0], b[0]), (what, int(np.sum(np.any(a[0] != b[0], axis=1))))
    assert a[1] == b[1] and a[2] == b[2] and np.array_equal(a[3], b[3]), what


# rows of 2, 6, 34, 48, 50, 66 and 80 sites a colour; a last tile of 2, 32 and
# 62 sites; single rows and planes; every kind of face
CASES = [((4, 1, 1), (P, O, O)), ((4, 2, 2), (P, P, P)), ((12, 12, 12), (P, P, P)), ((68, 2, 2), (P, P, P)),
         ((132, 6, 4), (P, P, P)), ((96, 34, 20), (P, P, P)), ((160, 24, 16), (P, P, P)), ((100, 30, 50), (P, P, P)),
         ((24, 13, 11), (O, O, O)), ((100, 7, 1), (O, O, O)), ((40, 36, 30), (K, P, A)),
         ((96, 10, 12), (A, K, P)), ((64, 7, 9), (K, O, O))]


@pytest.mark.parametrize("dims,faces", CASES)
@pytest.mark.parametrize("torque", [True, False])
def test_even_rows_equal_the_general_kernel_bit_for_bit(dims, faces, torque):
    spins = workloads.random_spins(dims[0] * dims[1] * dims[2], 4)
    kw = dict(K_u=0.05, K_c=0.02, H=(0.02, 0.0, 0.05), T=0.9, seed=5, boundary=faces, sample_torque=torque)
    _assert_same(_run(dims, kw, spins, mc.MC_PATH_ROW), _run(dims, kw, spins, mc.MC_PATH_GENERAL), (dims, faces))


@pytest.mark.parametrize("dims", [(96, 40, 3), (36, 22, 5)])
def test_films_of_even_rows_equal_the_general_kernel(dims):
    gid, mask, axes = workloads.voronoi_film(*dims, 9.0, seed=3)
    spins = workloads.random_spins(dims[0] * dims[1] * dims[2], 6)
    kw = dict(K_u=0.2, T=0.6, seed=8, boundary=(P, P, O), bond_mask=mask, grain_id=gid, grain_axis=axes)
    _assert_same(_run(dims, kw, spins, mc.MC_PATH_ROW), _run(dims, kw, spins, mc.MC_PATH_GENERAL), dims)


def test_group_of_all_kinds_equals_each_alone():
    """Row layout, even rows with and without faces, odd rows: one group."""
    cells = [((32, 8, 8), (P, P, P)), ((48, 10, 12), (P, P, P)), ((24, 9, 7), (O, O, O)), ((18, 10, 6), (P, P, P)),
             ((64, 10, 16), (P, K, O))]
    def make(i):
        d, f = cells[i]
        h = mc.mc_create_ex(mc.make_desc(d, K_u=0.03, T=0.7 + 0.1 * i, seed=20 + i, boundary=f, ring_capacity=8,
                                         kernel_path=mc.MC_PATH_ROW))
        mc.mc_set_spins(h, workloads.random_spins(d[0] * d[1] * d[2], i))
        return h
    hs = [make(i) for i in range(len(cells))]
    g = mc.mc_group_create(hs)
    mc.mc_group_sweep(g, 18)
    mc.mc_group_sweep(g, 5, True)
    mc.mc_group_destroy(g)
    for i, h in enumerate(hs):
        one = make(i)
        mc.mc_sweep(one, 18)
        mc.mc_sweep(one, 5, True)
        N = int(np.prod(cells[i][0]))
        _assert_same(_read(h, N, 8), _read(one, N, 8), cells[i])
        mc.mc_destroy(one)
        mc.mc_destroy(h)

"""Brick sweeps (csrc/brick_pass.cuh): a simple cubic lattice of any shape and
boundaries held in the SMs' shared memory for a whole run of sweeps, against
the same lattice swept by launches (MC_PATH_ROW: the row kernels, or the
general kernel for sizes outside the row layout).

The draws are keyed to the same sites, the operations and their order are the
same, and counts and sample sums are exact integers, so spins, cone angle,
samples and averages must agree bit for bit.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

import paper_2103_03517_gb300 as mc
import workloads

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
P, O, K, A = mc.MC_PERIODIC, mc.MC_OPEN, mc.MC_PINNED, mc.MC_ANTIPERIODIC


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2103_03517_gb300 import build as libbuild
    libbuild.build()


def _run(dims, kw, spins, plan, path):
    ring = max(1, sum(n for n, meas in plan if meas))
    h = mc.mc_create_ex(mc.make_desc(dims, kernel_path=path, ring_capacity=ring, **kw))
    try:
        mc.mc_set_spins(h, spins)
        for n, meas in plan:
            mc.mc_sweep(h, n, measure=meas)
        N = dims[0] * dims[1] * dims[2]
        return mc.mc_get_spins(h, N), mc.mc_get_theta(h), mc.mc_measure(h).asdict(), mc.mc_samples(h, ring)
    finally:
        mc.mc_destroy(h)


def _assert_same(a, b, what):
    assert np.array_equal(a[0], b[0]), (what, int(np.sum(np.any(a[0] != b[0], axis=1))))
    assert a[1] == b[1], what
    assert a[2] == b[2], what
    assert np.array_equal(a[3], b[3]), what


# rows of the row layout (2, 4, 8, 32, 64 and 192 sites a colour), even rows
# outside it (6, 48, 50), odd rows (1, 9, 45), ragged and single-plane shapes,
# two-site axes, every kind of face
CASES = [((4, 8, 16), (P, P, P)), ((8, 8, 8), (P, P, P)), ((16, 16, 16), (P, P, P)), ((64, 64, 64), (P, P, P)),
         ((384, 8, 6), (P, P, P)), ((64, 2, 2), (P, P, P)), ((128, 20, 12), (O, P, P)), ((64, 7, 9), (O, O, O)),
         ((16, 8, 32), (A, P, P)), ((32, 16, 16), (K, A, P)), ((64, 10, 16), (P, K, O)), ((16, 4, 1), (P, A, O)),
         ((12, 12, 12), (P, P, P)), ((96, 96, 96), (P, P, P)), ((100, 30, 50), (P, P, P)), ((24, 13, 11), (O, O, O)),
         ((40, 36, 30), (K, P, A)), ((2, 2, 2), (P, P, P)), ((18, 10, 14), (P, P, P)), ((90, 75, 61), (O, O, O)),
         ((50, 50, 50), (P, P, P)), ((34, 6, 6), (A, P, K)), ((2, 5, 3), (O, O, O)), ((1026, 6, 2), (P, P, P))]


@pytest.mark.parametrize("dims,faces", CASES)
def test_brick_sweeps_equal_launched_sweeps_bit_for_bit(dims, faces):
    N = dims[0] * dims[1] * dims[2]
    spins = workloads.random_spins(N, 11)
    kw = dict(K_u=0.05, K_c=0.02, H=(0.02, 0.0, 0.05), T=0.9, seed=5, boundary=faces)
    plan = [(3, False), (4, True), (1, False), (20, True), (25, False)]
    a = _run(dims, kw, spins, plan, mc.MC_PATH_AUTO)
    _assert_same(a, _run(dims, kw, spins, plan, mc.MC_PATH_ROW), (dims, faces))
    assert np.any(a[0] != spins)


@pytest.mark.parametrize("dims", [(64, 32, 32), (48, 20, 24), (30, 20, 24)])
def test_brick_samples_without_torques_and_with_a_fixed_cone(dims):
    spins = workloads.random_spins(dims[0] * dims[1] * dims[2], 3)
    kw = dict(K_u=0.01, T=1.4, seed=2, sample_torque=0, adapt_in_measure=0)
    plan = [(5, False), (6, True), (2, False), (3, True)]
    _assert_same(_run(dims, kw, spins, plan, mc.MC_PATH_AUTO), _run(dims, kw, spins, plan, mc.MC_PATH_ROW), dims)


@pytest.mark.parametrize("sizes", [(16, 16), (8, 16, 32, 64), (12, 18, 24, 50, 64), (2, 4), (32,) * 20])
def test_group_of_small_lattices_side_by_side(sizes):
    """A group whose lattices fit the SMs together: brick launches, one per
    kernel instance, free and measured, mixed with constrained sweeps and calls
    too short for them; every lattice equals the one swept alone by launches."""
    def make(i, path):
        L = sizes[i]
        h = mc.mc_create_ex(mc.make_desc((L, L, L), K_u=0.03, T=0.5 + 0.05 * i, seed=30 + i, ring_capacity=16,
                                         kernel_path=path, init_dir=(0.1 * (i % 5), 0.0, 1.0)))
        mc.mc_set_spins(h, workloads.perturbed_spins(L ** 3, i, 0.3))
        return h

    def read(h, L):
        return mc.mc_get_spins(h, L ** 3), mc.mc_get_theta(h), mc.mc_measure(h).asdict(), mc.mc_samples(h, 16)

    n = len(sizes)
    hs = [make(i, mc.MC_PATH_AUTO) for i in range(n)]
    g = mc.mc_group_create(hs)
    _, kinds = mc.mc_group_time_kernels(g, 5)
    assert kinds[3] >= 1 and kinds[1] == 0, kinds
    mc.mc_group_sweep(g, 4, True)
    mc.mc_group_constrained_sweep(g, [10.0] * n, [0.0] * n, 3, True)
    mc.mc_group_sweep(g, 2, True)
    mc.mc_group_sweep(g, 20, True)
    mc.mc_group_sweep(g, 18)
    mc.mc_group_destroy(g)
    for i, h in enumerate(hs):
        one = make(i, mc.MC_PATH_ROW)
        mc.mc_sweep(one, 5)
        mc.mc_sweep(one, 4, True)
        mc.mc_constrained_sweep(one, 10.0, 0.0, 3, True)
        mc.mc_sweep(one, 22, True)
        mc.mc_sweep(one, 18)
        _assert_same(read(h, sizes[i]), read(one, sizes[i]), (i, sizes[i]))
        mc.mc_destroy(one)
        mc.mc_destroy(h)


def test_brick_run_longer_than_one_launch():
    """2050 sweeps take two launches; tags and epochs go on across them."""
    dims = (16, 8, 12)
    spins = workloads.random_spins(16 * 8 * 12, 5)
    kw = dict(K_u=0.02, T=0.3, seed=9, theta0_deg=90)
    plan = [(2050, False), (30, True)]
    _assert_same(_run(dims, kw, spins, plan, mc.MC_PATH_AUTO), _run(dims, kw, spins, plan, mc.MC_PATH_ROW), "two launches")


def test_brick_wait_that_runs_out_reports_timeout():
    """A host-set fault makes every block wait for a count that never comes:
    the launch ends by itself and the next synchronising call says so."""
    code = ("import paper_2103_03517_gb300 as mc\n"
            "h = mc.mc_create_ex(mc.make_desc((32, 32, 32), T=0.8))\n"
            "mc.mc_sweep(h, 5)\n"
            "try:\n    mc.mc_sync(h)\n    print('no error')\n"
            "except mc.MCError as e:\n    print('code', e.code)\n")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=120,
                       env=dict(os.environ, MC_RESIDENT_INJECT_TIMEOUT="1", PYTHONPATH=ROOT))
    assert r.stdout.strip() == f"code {mc.MC_ERR_TIMEOUT}", r.stdout + r.stderr


@pytest.mark.parametrize("dims,n,used", [((128, 16, 16), 20, False), ((128, 16, 16), 5, True), ((32, 32, 32), 5, False),
                                         ((48, 20, 24), 15, True)])
def test_sweeps_captured_by_the_caller(dims, n, used):
    """On a stream under capture the sweeps go into the caller's graph as
    launches, whether the lattice has its brick memory (used) or not; a replay
    is one more run of them.  Meanwhile another lattice's first brick launch,
    on its own stream, neither fails nor ends the capture."""
    torch = pytest.importorskip("torch")
    st = torch.cuda.Stream()
    kw = dict(K_u=0.03, T=0.7, seed=4)
    spins = workloads.random_spins(dims[0] * dims[1] * dims[2], 8)
    h = mc.mc_create_ex(mc.make_desc(dims, ring_capacity=64, stream=int(st.cuda_stream), **kw))
    other = mc.mc_create_ex(mc.make_desc((16, 16, 16), T=0.5, seed=1))
    ref = mc.mc_create_ex(mc.make_desc(dims, ring_capacity=64, kernel_path=mc.MC_PATH_ROW, **kw))
    for x in (h, ref):
        mc.mc_set_spins(x, spins)
        mc.mc_sweep(x, 4 if used else 1)
    mc.mc_sync(h)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        graph.capture_begin()
        mc.mc_sweep(h, n, measure=True)
        mc.mc_sweep(other, 5)
        graph.capture_end()
        graph.replay()
        graph.replay()
    torch.cuda.synchronize()
    mc.mc_sync(other)
    mc.mc_sweep(ref, 2 * n, measure=True)
    N = dims[0] * dims[1] * dims[2]
    assert np.array_equal(mc.mc_get_spins(h, N), mc.mc_get_spins(ref, N))
    assert mc.mc_measure(h).asdict() == mc.mc_measure(ref).asdict()
    assert np.array_equal(mc.mc_samples(h, 64), mc.mc_samples(ref, 64))
    for x in (h, other, ref):
        mc.mc_destroy(x)

"""The row kernel's launch shapes (blocks per SM, the warps of a block taking its
tiles in turn) change no bit, on lattices that really take it (MC_PATH_ROW: on the
automatic path ones of these sizes sweep as bricks): every kind of list, of the
row layout and of even rows outside it, periodic, with faces and with film tables,
and lists of long rows, which take their tiles in turn in shape 0 only."""
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


def _film(dims):
    gid, mask, axes = workloads.voronoi_film(dims[0], dims[1], dims[2], 6.0, seed=2)
    return dict(bond_mask=mask, grain_id=gid, grain_axis=axes)


# (sizes, faces, film) of each group
GROUPS = {
    "row layout": [((128, 32, 16), (P, P, P), False), ((256, 16, 8), (P, P, P), False), ((64, 64, 16), (P, P, P), False),
                   ((16, 16, 16), (P, P, P), False), ((32, 8, 8), (P, P, P), False)],
    "even rows": [((96, 20, 10), (P, P, P), False), ((12, 12, 12), (P, P, P), False), ((100, 30, 14), (P, P, P), False)],
    "faces": [((64, 16, 8), (A, P, P), False), ((32, 9, 4), (O, O, O), False), ((40, 36, 10), (K, P, A), False)],
    "films": [((64, 64, 4), (P, P, O), True), ((60, 40, 6), (P, P, O), True), ((128, 32, 3), (A, P, O), True)],
    "long rows": [((256, 64, 32), (P, P, P), False), ((512, 32, 32), (P, P, P), False)],
    "long even rows": [((400, 32, 32), (P, P, P), False)],
    "long rows with faces": [((256, 32, 40), (A, P, P), False), ((400, 30, 32), (P, O, P), False)],
    "long films": [((256, 64, 16), (P, P, O), True), ((280, 60, 16), (P, P, O), True)],
}


@pytest.mark.parametrize("name", GROUPS)
def test_row_shapes_give_the_same_chain(name):
    ref = None
    for shape in range(2):
        hs = []
        for i, (d, bc, film) in enumerate(GROUPS[name]):
            h = mc.mc_create_ex(mc.make_desc(d, K_u=0.05, K_c=0.01, H=(0.0, 0.02, 0.0), T=0.6 + 0.1 * i, seed=i + 3, boundary=bc,
                                             ring_capacity=16, kernel_path=mc.MC_PATH_ROW, **(_film(d) if film else {})))
            mc.mc_set_spins(h, workloads.random_spins(int(np.prod(d)), i))
            hs.append(h)
        g = mc.mc_group_create(hs)
        try:
            mc.mc_group_set_shapes(g, row=shape)
            _, kinds = mc.mc_group_time_kernels(g, 5)
            assert kinds[1] > 0 and kinds[3] == 0, kinds
            mc.mc_group_sweep(g, 6, measure=True)
            mc.mc_group_sync(g)
            got = [(mc.mc_get_spins(h, int(np.prod(d))), mc.mc_measure(h).asdict(), mc.mc_get_theta(h), mc.mc_samples(h, 16))
                   for h, (d, _, _) in zip(hs, GROUPS[name])]
        finally:
            mc.mc_group_destroy(g)
            for h in hs:
                mc.mc_destroy(h)
        if ref is None:
            ref = got
            continue
        for a, b in zip(ref, got):
            assert np.array_equal(a[0], b[0]) and a[1] == b[1] and a[2] == b[2] and np.array_equal(a[3], b[3])


@pytest.mark.parametrize("dims,bc", [((64, 16, 8), (A, P, P)), ((128, 8, 6), (K, P, P)), ((32, 9, 4), (O, O, O)),
                                     ((256, 6, 4), (A, K, A)), ((64, 64, 16), (P, P, P))])
def test_row_kernel_follows_the_general_kernel_over_a_few_sweeps(dims, bc):
    """As for a single sweep: the same chain on nearly every site."""
    N = int(np.prod(dims))
    spins = workloads.random_spins(N, 3)
    out = []
    for path in (mc.MC_PATH_ROW, mc.MC_PATH_GENERAL):
        h = mc.mc_create_ex(mc.make_desc(dims, K_u=0.05, K_c=0.02, H=(0.01, 0.02, 0.05), T=0.8, seed=21, boundary=bc,
                                         ring_capacity=8, kernel_path=path))
        mc.mc_set_spins(h, spins)
        mc.mc_sweep(h, 3, True)
        out.append(mc.mc_get_spins(h, N))
        mc.mc_destroy(h)
    assert np.any(out[0] != spins, axis=1).mean() > 0.2
    assert np.all(np.abs(out[0] - out[1]) < 1e-4, axis=1).mean() > 0.99


def test_two_brick_lattices_on_two_streams():
    """Brick runs of two lattices under way at the same time on streams of their
    own are each the launched sweeps' chain."""
    torch = pytest.importorskip("torch")
    dims = [(64, 64, 64), (90, 75, 61)]
    faces = [(P, P, P), (O, O, O)]
    make = lambda i, path, **kw: mc.mc_create_ex(mc.make_desc(dims[i], K_u=0.03, T=0.7, seed=i, boundary=faces[i], ring_capacity=64,
                                                              kernel_path=path, **kw))
    st = [torch.cuda.Stream() for _ in range(2)]
    hs = [make(i, mc.MC_PATH_AUTO, stream=int(st[i].cuda_stream)) for i in range(2)]
    ref = [make(i, mc.MC_PATH_ROW) for i in range(2)]
    for _ in range(5):
        for h in hs:
            mc.mc_sweep(h, 20)
            mc.mc_sweep(h, 5, True)
    for i in range(2):
        for _ in range(5):
            mc.mc_sweep(ref[i], 20)
            mc.mc_sweep(ref[i], 5, True)
        N = int(np.prod(dims[i]))
        mc.mc_sync(hs[i])
        assert np.array_equal(mc.mc_get_spins(hs[i], N), mc.mc_get_spins(ref[i], N))
        assert mc.mc_measure(hs[i]).asdict() == mc.mc_measure(ref[i]).asdict()
    for h in hs + ref:
        mc.mc_destroy(h)


def test_wait_of_a_groups_brick_sweeps_that_runs_out():
    """A host-set fault makes one lattice's blocks wait for a count that never
    comes: the launch ends by itself, its next synchronising call says so, and the
    lattices beside it, whose blocks know nothing of it, have their chain."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    code = ("import os\nimport numpy as np\nimport paper_2103_03517_gb300 as mc\n"
            "mk = lambda i, path: mc.mc_create_ex(mc.make_desc((16, 16, 16), T=0.8, seed=i, kernel_path=path))\n"
            "a = mk(0, 0)\n"
            "os.environ['MC_RESIDENT_INJECT_TIMEOUT'] = '1'\nb = mk(1, 0)\n"
            "del os.environ['MC_RESIDENT_INJECT_TIMEOUT']\nr = mk(0, mc.MC_PATH_ROW)\n"
            "g = mc.mc_group_create([a, b])\nmc.mc_group_sweep(g, 5)\n"
            "try:\n    mc.mc_sync(b)\n    print('no error')\nexcept mc.MCError as e:\n    print('code', e.code)\n"
            "mc.mc_sweep(r, 5)\nmc.mc_sync(a)\n"
            "print(np.array_equal(mc.mc_get_spins(a, 4096), mc.mc_get_spins(r, 4096)))\n")
    p = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=120,
                       env=dict(os.environ, PYTHONPATH=root))
    assert p.stdout.split("\n")[:2] == [f"code {mc.MC_ERR_TIMEOUT}", "True"], p.stdout + p.stderr

"""Calls of one measured sweep: three launches (red, black, the close that forms
the sample), with no further launch for the sample; calls of any lengths give the
chain and samples of one long call."""
import ctypes as C

import numpy as np
import pytest

import paper_2103_03517_gb300 as mc
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2103_03517_gb300 import build as libbuild
    libbuild.build()


# row layout, even rows outside it, general kernel, FP64, faces
CASES = [((16, 16, 16), {}), ((20, 12, 10), {}), ((18, 10, 8), {}), ((16, 8, 8), dict(precision=mc.MC_FP64)),
         ((32, 8, 8), dict(boundary=(mc.MC_OPEN, 0, mc.MC_PINNED)))]


@pytest.mark.parametrize("dims,kw", CASES)
def test_launches_of_one_measured_sweep(dims, kw):
    torch = pytest.importorskip("torch")
    cu = C.CDLL("libcuda.so.1")
    st = torch.cuda.Stream()
    stream, graph, nodes = C.c_void_p(st.cuda_stream), C.c_void_p(), C.c_size_t()
    h = mc.mc_create_ex(mc.make_desc(dims, T=0.7, seed=4, stream=int(st.cuda_stream), **kw))
    mc.mc_sync(h)
    assert cu.cuStreamBeginCapture_v2(stream, 2) == 0
    mc.mc_sweep(h, 1, True)
    assert cu.cuStreamEndCapture(stream, C.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, C.byref(nodes)) == 0
    assert nodes.value == 3
    cu.cuGraphDestroy(graph)
    mc.mc_destroy(h)


@pytest.mark.parametrize("dims,kw", CASES)
def test_short_calls_give_the_samples_of_a_long_one(dims, kw):
    N = dims[0] * dims[1] * dims[2]
    out = []
    for calls in ([1, 2, 1, 1, 2, 5, 1, 2], [15]):
        for torque in (1, 0):
            h = mc.mc_create_ex(mc.make_desc(dims, K_u=0.03, K_c=0.01, H=(0.0, 0.1, 0.02), T=0.7, seed=4, ring_capacity=12,
                                             sample_torque=torque, kernel_path=mc.MC_PATH_ROW, **kw))
            mc.mc_set_spins(h, workloads.random_spins(N, 8))
            for n in calls:
                mc.mc_sweep(h, n, True)
            out.append((mc.mc_get_spins(h, N), mc.mc_get_theta(h), mc.mc_measure(h).asdict(), mc.mc_samples(h, 12)))
            mc.mc_destroy(h)
    for a, b in zip(out[:2], out[2:]):
        assert np.array_equal(a[0], b[0]) and a[1] == b[1] and a[2] == b[2] and np.array_equal(a[3], b[3])


@pytest.mark.parametrize("count", [2, 18])
def test_single_measured_sweeps_of_a_group(count):
    """Few lattices, and more than are closed by blocks of one warp."""
    dims = [(16, 8, 8), (20, 6, 4), (10, 4, 4)]
    kw = dict(K_u=0.03, T=0.7, ring_capacity=4, kernel_path=mc.MC_PATH_ROW)
    make = lambda i: mc.mc_create_ex(mc.make_desc(dims[i % 3], seed=i, **kw))
    hs, ref = [make(i) for i in range(count)], [make(i) for i in range(count)]
    g = mc.mc_group_create(hs)
    for _ in range(5):
        mc.mc_group_sweep(g, 1, True)
    mc.mc_group_sync(g)
    for i, (h, r) in enumerate(zip(hs, ref)):
        N = int(np.prod(dims[i % 3]))
        mc.mc_sweep(r, 5, True)
        assert np.array_equal(mc.mc_get_spins(h, N), mc.mc_get_spins(r, N))
        assert mc.mc_measure(h).asdict() == mc.mc_measure(r).asdict()
        assert np.array_equal(mc.mc_samples(h, 4), mc.mc_samples(r, 4))
    mc.mc_group_destroy(g)
    for h in hs + ref:
        mc.mc_destroy(h)

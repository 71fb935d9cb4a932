"""Sweeps of 128-wide periodic lattices on a stream that the caller captures go
into the graph as one resident launch, whatever the lattice's size and the number
of sweeps (bricks are not captured; as launches it would take three a sweep)."""
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


@pytest.mark.parametrize("dims", [(128, 16, 16), (128, 64, 64), (128, 128, 128)])
@pytest.mark.parametrize("n,measure", [(5, False), (20, False), (20, True)])
def test_one_launch_in_the_callers_graph(dims, n, measure):
    torch = pytest.importorskip("torch")
    cu = C.CDLL("libcuda.so.1")
    st = torch.cuda.Stream()
    stream = C.c_void_p(st.cuda_stream)
    h = mc.mc_create_ex(mc.make_desc(dims, K_u=0.03, T=0.7, seed=4, ring_capacity=64, stream=int(st.cuda_stream)))
    ref = mc.mc_create_ex(mc.make_desc(dims, K_u=0.03, T=0.7, seed=4, ring_capacity=64, kernel_path=mc.MC_PATH_ROW))
    for x in (h, ref):
        mc.mc_set_spins(x, workloads.random_spins(dims[0] * dims[1] * dims[2], 8))
        mc.mc_sweep(x, 4, measure)
        mc.mc_sync(x)
    graph, ex, nodes = C.c_void_p(), C.c_void_p(), C.c_size_t()
    assert cu.cuStreamBeginCapture_v2(stream, 2) == 0
    mc.mc_sweep(h, n, measure)
    assert cu.cuStreamEndCapture(stream, C.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, C.byref(nodes)) == 0
    assert nodes.value <= 4, nodes.value  # control words, records, sweeps, samples
    assert cu.cuGraphInstantiateWithFlags(C.byref(ex), graph, C.c_ulonglong(0)) == 0
    for _ in range(2):
        assert cu.cuGraphLaunch(ex, stream) == 0
    mc.mc_sync(h)
    mc.mc_sweep(ref, 2 * n, measure)
    N = dims[0] * dims[1] * dims[2]
    assert np.array_equal(mc.mc_get_spins(h, N), mc.mc_get_spins(ref, N))
    if measure:
        assert np.array_equal(mc.mc_samples(h, 64), mc.mc_samples(ref, 64))
    cu.cuGraphExecDestroy(ex)
    cu.cuGraphDestroy(graph)
    mc.mc_destroy(h)
    mc.mc_destroy(ref)

"""mc_sweep_noalloc on spins at any float address (a slice of a larger tensor
that starts at an odd float): the row kernels move pairs of spins in 8-byte
accesses, so such spins take the general kernel, whatever the size and the
number of sweeps.  Spins that are not aligned to a float are refused before any
CUDA call.
"""
import ctypes

import numpy as np
import pytest

import paper_2103_03517_gb300 as mc

KW = dict(J=1.0, K_u=0.05, K_c=0.02, H=(0.0, 0.0, 0.1), T=0.8, seed=21)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2103_03517_gb300 import build as libbuild
    libbuild.build()


def _sweep(ptr, dims, n, samples=None):
    return mc.mc_sweep_noalloc(ptr, dims, KW["J"], KW["K_u"], (0.0, 0.0, 1.0), KW["K_c"], KW["H"], KW["T"], KW["seed"],
                               0, n, 30, samples_ptr=samples)


@pytest.mark.parametrize("off", [1, 2, 3])
def test_spins_not_aligned_to_a_float_are_refused(off):
    buf = (ctypes.c_float * 8)()  # never read: the refusal comes first
    with pytest.raises(mc.MCError) as e:
        _sweep(ctypes.addressof(buf) + off, (16, 16, 16), 2)
    assert e.value.code == mc.MC_ERR_ARG and "aligned" in str(e.value)


# row layout (16^3, 128 x 16 x 16), even rows outside it (12 x 6 x 4, 96^3: above
# the size that sweeps as bricks), odd rows; calls too short for bricks and longer
@pytest.mark.gpu
@pytest.mark.parametrize("dims,n", [((16, 16, 16), 2), ((16, 16, 16), 5), ((128, 16, 16), 2), ((12, 6, 4), 2),
                                    ((12, 6, 4), 5), ((96, 96, 96), 4), ((10, 6, 4), 2)])
def test_spins_at_an_odd_float_take_the_general_kernels_chain(dims, n):
    torch = pytest.importorskip("torch")
    h = mc.mc_create_ex(mc.make_desc(dims, ring_capacity=n, kernel_path=mc.MC_PATH_GENERAL, **KW))
    try:
        nbytes = mc.mc_state_bytes(h)
        start = np.zeros(nbytes // 4, np.float32)
        want = np.zeros_like(start)
        mc.mc_export_state(h, start.ctypes.data, nbytes)
        mc.mc_sweep(h, n, measure=True)
        mc.mc_export_state(h, want.ctypes.data, nbytes)
        theta, ref = mc.mc_get_theta(h)[0], mc.mc_samples(h, n)
    finally:
        mc.mc_destroy(h)
    buf = torch.zeros(start.size + 1, dtype=torch.float32, device="cuda")
    buf[1:] = torch.from_numpy(start)
    samples = torch.zeros(n * 14, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert buf[1:].data_ptr() % 8 == 4
    assert _sweep(buf[1:].data_ptr(), dims, n, samples.data_ptr()) == theta
    assert np.array_equal(buf[1:].cpu().numpy(), want)
    s = samples.cpu().numpy().reshape(n, 14)
    assert np.array_equal(s[:, 2].astype(np.int64), ref["accepted"])
    np.testing.assert_allclose(s[:, 3:6], ref["m"], rtol=0, atol=1e-12)
    np.testing.assert_allclose(s[:, 10:13], ref["torque"], rtol=0, atol=1e-12)

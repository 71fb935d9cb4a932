"""Energies of FP32 crystals with couplings far from 1: the exchange sum is formed
in fixed point with the couplings inside it, and must neither wrap over a lane's
tiles (96^3 cells) nor saturate at one site (J = 60).  At a temperature far below
the couplings the spins stay along the start, and the exchange energy per site is
-z J / 2 (and -3 J2 for the six next-nearest neighbours), up to the moves' small
angles."""
import numpy as np
import pytest

import paper_2103_03517_gb300 as mc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2103_03517_gb300 import build as libbuild
    libbuild.build()


# 10 sweeps from the ordered state at T = 1e-6 J move a spin by angles of about
# sqrt(T / 12 J): the energy is off by well under 1e-4 of itself
@pytest.mark.parametrize("lattice,z", [(mc.MC_BCC, 8), (mc.MC_FCC, 12), (mc.MC_HCP, 12)])
@pytest.mark.parametrize("cells,J,J2", [(96, 8.0, 0.0), (96, -4.0, 0.0), (12, 60.0, 0.0), (12, 8.0, 0.0), (12, 2.0, 100.0), (12, 1.0, 0.0),
                                        (40, 5.0, 20.0), (96, 1.0, 0.0)])
def test_exchange_energy_of_an_ordered_crystal(lattice, z, cells, J, J2):
    if lattice == mc.MC_HCP and J2:
        pytest.skip("hcp has no J2")
    e = -(z * J + 6 * J2) / 2
    scale = max(abs(J), abs(J2))
    if e > 0:  # unstable: held by a field, whose energy is taken off
        H = 1e3 * scale
    else:
        H = 0.0
    h = mc.mc_create_ex(mc.make_desc((cells,) * 3, J=J, J2=J2, H=(0.0, 0.0, H), T=1e-6 * scale, seed=1, lattice=lattice, theta0_deg=1,
                                     ring_capacity=16))
    mc.mc_sweep(h, 10, True)
    s = mc.mc_samples(h, 16)["e_parts"][:10, 0]
    mc.mc_destroy(h)
    assert np.all(np.abs(s - e) <= 1e-3 * abs(e)), (s, e)

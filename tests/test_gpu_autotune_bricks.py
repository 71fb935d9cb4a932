"""The autotuner on lattices that sweep as bricks: its row candidates are the row
kernel's launches, which such a lattice's calls of one or two sweeps take, and
their times are those of the same lattice on MC_PATH_ROW (bricks of these sizes
take 0.3 to 0.45 of them)."""
import pytest

import paper_2103_03517_gb300 as mc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2103_03517_gb300 import build as libbuild
    libbuild.build()


def _row_ms(sizes, path, alone):
    hs = [mc.mc_create_ex(mc.make_desc((L, L, L), T=0.7, seed=i, kernel_path=path)) for i, L in enumerate(sizes)]
    try:
        if alone:
            return mc.mc_autotune(hs[0], 200, mc.MC_TUNE_SWEEP)["row_ms"][:2]
        g = mc.mc_group_create(hs)
        try:
            return mc.mc_group_autotune(g, 200, mc.MC_TUNE_SWEEP)["row_ms"][:2]
        finally:
            mc.mc_group_destroy(g)
    finally:
        for h in hs:
            mc.mc_destroy(h)


@pytest.mark.parametrize("sizes,alone", [((64,), True), ((64,), False), ((32,) * 4, False), ((16, 16), False)])
def test_row_candidates_are_timed_on_the_row_kernel(sizes, alone):
    auto, row = _row_ms(sizes, mc.MC_PATH_AUTO, alone), _row_ms(sizes, mc.MC_PATH_ROW, alone)
    for a, b in zip(auto, row):
        assert 0.7 * b < a < b / 0.7, (auto, row)

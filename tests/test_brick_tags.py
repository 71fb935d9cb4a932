"""The tags of the brick sweeps' packets (brick_tag0, brick_clears in
csrc/mc_internal.h): a packet carries the tag of the pass it was written in, and
a reader waits for the tag of the pass before its own, so no older packet and no
zeroed memory may carry an awaited tag, however many launches came before.
"""
import ctypes
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2103_03517_gb300", "csrc")
EPOCHS = 1 << 19
PASSES = 2 * 2048 + 1  # the state at the start and two passes a sweep


def _tags(tmp_path):
    src, lib = tmp_path / "tags.cpp", tmp_path / "tags.so"
    src.write_text('#include "mc_internal.h"\nextern "C" unsigned tag0(unsigned e) { return mcgb::brick_tag0(e); }\n'
                   'extern "C" int clears(unsigned e) { return mcgb::brick_clears(e); }\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    d = ctypes.CDLL(str(lib))
    d.tag0.restype = ctypes.c_uint
    d.tag0.argtypes = d.clears.argtypes = [ctypes.c_uint]
    return d


def test_no_older_packet_and_no_zeroed_memory_carries_an_awaited_tag(tmp_path):
    d = _tags(tmp_path)
    near = [0, 1, 2, 77] + [k * EPOCHS + j for k in (1, 2, 8191) for j in (-3, -2, -1, 0, 1, 2, 77)] + [2 ** 32 - 2, 2 ** 32 - 1]
    for b in near:
        t = d.tag0(b)
        assert t != 0 and (t & 0x1FFF) + PASSES < 0x2000  # all of the epoch's tags nonzero and its own
    for b in near:
        for a in near:
            if a >= b:
                continue
            # the clears of launches a + 1 ... b, counted in closed form
            cleared = (b + 1) // EPOCHS - (a + 1) // EPOCHS
            same = d.tag0(a) >> 13 == d.tag0(b) >> 13
            assert not same or cleared > 0, (a, b)
    for e in near:
        assert bool(d.clears(e)) == (e % EPOCHS == EPOCHS - 1), e


CODE = """
import numpy as np
import paper_2103_03517_gb300 as mc
import workloads
dims = (20, 16, 12)
def make(i, path):
    h = mc.mc_create_ex(mc.make_desc(dims, K_u=0.03, T=0.6, seed=i, ring_capacity=64, kernel_path=path))
    mc.mc_set_spins(h, workloads.random_spins(20 * 16 * 12, i))
    return h
hs = [make(i, mc.MC_PATH_AUTO) for i in range(3)]
ref = [make(i, mc.MC_PATH_ROW) for i in range(3)]
g = mc.mc_group_create(hs)
for k in range(4):   # each lattice's epoch goes up by two a turn, through the clear
    mc.mc_group_sweep(g, 3)
    mc.mc_group_sync(g)
    for h in hs:
        mc.mc_sweep(h, 4, True)
        mc.mc_sync(h)
for h in ref:
    for k in range(4):
        mc.mc_sweep(h, 3)
        mc.mc_sweep(h, 4, True)
for a, b in zip(hs, ref):
    assert np.array_equal(mc.mc_get_spins(a, 3840), mc.mc_get_spins(b, 3840))
    assert mc.mc_measure(a).asdict() == mc.mc_measure(b).asdict()
print("ok")
"""


@pytest.mark.gpu
@pytest.mark.parametrize("first", [EPOCHS - 6, EPOCHS - 5, 2 ** 32 - 4])
def test_sweeps_through_the_epochs_wrap(first):
    """Launches alone and in a group whose epochs pass the clear (by either
    launch's preparation) and the counter's own wrap."""
    from paper_2103_03517_gb300 import build as libbuild
    libbuild.build()
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=120,
                       env=dict(os.environ, MC_BRICK_FIRST_EPOCH=str(first), PYTHONPATH=ROOT))
    assert r.stdout.strip() == "ok", r.stdout + r.stderr

"""The neighbour sort where more cells rebuild than the chip holds clusters.

A CTA then sorts a cell by itself; with few cells a cluster of eight does.  The
order of the atoms is the same (sorted by bin, stable), so a cell has the same
positions and the same lists, entry for entry, in a batch of many cells as in a
batch of one: one atom, about a CTA's and a round's worth of atoms, more bins
than one scan of the counters takes, more cells than one pass over the flags,
frozen cells among them, a second rebuild under a tilted box, and bonded beads.
"""
import numpy as np
import pytest

from paper_1902_09171_gb300 import inputs, rcell
from test_gpu_few_cells import chains
from test_gpu_list_build import TILT, gas

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    t.cuda.set_device(0)
    from paper_1902_09171_gb300 import build
    build.build()
    rcell.load()
    return t


def lists(prm, cells, look, active=None):
    """Positions and neighbour lists (slot order) of cells `look` after two rebuilds."""
    ctx = rcell.rcell_create(prm, cells)
    try:
        rcell.rcell_eval(ctx)
        if active is not None:
            rcell.rcell_set_active(ctx, np.array(active, np.int32))
        rcell.rcell_set_deformation(ctx, np.tile(TILT, (len(cells), 1, 1)))
        rcell.rcell_eval(ctx)
        on = np.ones(len(cells), int) if active is None else np.array(active)
        assert np.array_equal(rcell.rcell_get_rebuilds(ctx), 1 + on)
        out = []
        for k in look:
            n = len(cells[k]["x0"])
            out.append((rcell.rcell_get_atoms(ctx, k, n)[0], rcell.rcell_get_neighbors(ctx, k, n * 300)))
        return out
    finally:
        rcell.rcell_destroy(ctx)


def same(prm, cells, look, active=None):
    for k, got in zip(look, lists(prm, cells, look, active)):
        for a, b in zip(got, lists(prm, [cells[k]], [0], None if active is None else [active[k]])[0]):
            assert np.array_equal(a, b), (k, len(cells[k]["x0"]))


def test_sizes_and_frozen_cells():
    sizes = [1, 31, 511, 512, 513, 1024, 1025, 2049]
    box = np.array([20.0, 21.0, 22.0])
    cells = [gas(n, box, n) for n in sizes] + [gas(60 + k, box, 100 + k) for k in range(80)]
    same(rcell.params_lj_cu(), cells, [0, 1, 2, 3, 4, 5, 6, 7, 30], [k % 7 != 3 for k in range(len(cells))])


def test_more_cells_than_one_pass_over_the_flags():
    cells = [gas(20 + k % 40, np.array([13.0, 14.0, 13.5]), k) for k in range(2100)]
    same(rcell.params_lj_cu(), cells, [0, 1023, 1024, 1500, 2047, 2048, 2099])


def test_more_bins_than_one_scan():
    # 12 x 15 x 20 bins of 1.4 and more
    cells = [gas(900 + k, np.array([17.3, 21.7, 29.0]), k) for k in range(100)]
    same(rcell.params_kg(), cells, [0, 50, 99])


def test_bonded_beads():
    cells = [chains(30 + k % 5, 13, k) for k in range(120)]
    same(rcell.params_kg(), cells, [0, 1, 63, 119])

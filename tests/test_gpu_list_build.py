"""Neighbour sort and list build at the sizes where their work is split.

Random gases (every bin occupancy occurs) whose lists are compared with the
oracle's pair sets: one atom, a warp's and a tile's worth of atoms and one more
or less, more atoms than a cluster of the sort has threads, candidate counts
above the shared-memory window, lists of several hundred entries, thin boxes of
four bins, tilted boxes, uneven batches with a frozen cell, and beads with up to
four bonds.  Every pair closer than r_list by more than 1e-5 has to be there,
none that is farther by more (the set is exact up to FP32 rounding at r_list),
and none twice.
"""
import numpy as np
import pytest

import oracle
from paper_1902_09171_gb300 import inputs, rcell

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


def gas(n, box, seed):
    rng = np.random.default_rng(seed)
    return dict(H0=np.diag(box).astype(float), x0=inputs.to_f32(rng.uniform(0, 1, (n, 3)) * box * 0.999))


def check(prm, cells, F=None, active=None):
    rlist = prm.rc + prm.skin
    ctx = rcell.rcell_create(prm, cells)
    try:
        rcell.rcell_eval(ctx)
        if active is not None:
            rcell.rcell_set_active(ctx, np.array(active, np.int32))
        if F is not None:
            rcell.rcell_set_deformation(ctx, np.tile(F, (len(cells), 1, 1)))
        rcell.rcell_eval(ctx)
        expected = 1 if F is None else 2
        for k, cell in enumerate(cells):
            n = len(cell["x0"])
            x, _, _ = rcell.rcell_get_atoms(ctx, k, n)
            H, _, _ = rcell.rcell_get_box(ctx, k)
            got = [tuple(p) for p in rcell.rcell_get_neighbors(ctx, k, n * 1500)]
            b = cell.get("bonds", np.zeros((0, 2), int))
            bonded = {tuple(p) for p in b.tolist()} | {(j, i) for i, j in b.tolist()}
            near, far = ({tuple(p) for p in oracle.neighbor_pairs(x, H, rlist * f, max_pairs=n * 1500 + 64)} - bonded
                         for f in (1 - 1e-5, 1 + 1e-5))
            assert len(set(got)) == len(got)
            assert near <= set(got) <= far, (k, len(near - set(got)), len(set(got) - far))
            frozen = active is not None and not active[k]
            assert rcell.rcell_get_rebuilds(ctx)[k] == (1 if frozen else expected)
    finally:
        rcell.rcell_destroy(ctx)


TILT = np.array([[1.02, 0.13, -0.09], [0.05, 0.98, 0.11], [-0.03, 0.04, 1.01]])


@pytest.mark.parametrize("F", [None, TILT])
@pytest.mark.parametrize("n,side", [(1, 13.0), (31, 13.0), (33, 13.0), (128, 15.0), (129, 15.0), (1500, 22.0), (4097, 40.0)])
def test_sizes(n, side, F):
    check(rcell.params_lj_cu(), [gas(n, np.array([side, side * 1.1, side * 1.05]), n)], F)


@pytest.mark.parametrize("box", [(90.0, 14.5, 14.5), (14.5, 90.0, 14.5), (14.5, 14.5, 90.0)])
def test_thin_boxes(box):
    check(rcell.params_lj_cu(), [gas(1200, np.array(box), 5)], TILT)


def test_candidates_beyond_the_window_and_long_lists():
    # 0.16 atoms per cubic Angstrom within 8.72 Angstrom: lists of about 440, up to 2000 candidates
    check(rcell.params_sc_cu(skin=1.5), [gas(2500, np.array([25.0, 25.0, 25.0]), 3)], TILT)


def test_uneven_batch_with_a_frozen_cell():
    cells = [gas(n, np.array([18.0, 16.0, 17.0]), 7 + n) for n in (5, 700, 64, 1000, 257)]
    check(rcell.params_lj_cu(), cells, TILT, active=[1, 1, 0, 1, 1])


def test_beads_with_up_to_four_bonds():
    cell = gas(1300, np.array([12.0, 11.0, 12.5]), 2)
    rng = np.random.default_rng(4)
    hubs = np.arange(0, 1300, 5)  # every hub bonded to the four beads after it, most of them near neighbours
    d = rng.normal(size=(len(hubs), 4, 3))
    d *= 1.1 / np.linalg.norm(d, axis=2, keepdims=True)
    x = cell["x0"].copy()
    for m in range(4):
        x[hubs + 1 + m] = np.mod(x[hubs] + d[:, m], np.diag(cell["H0"]) * 0.9999)
    cell["x0"] = inputs.to_f32(x)
    cell["bonds"] = np.stack([np.repeat(hubs, 4), (hubs[:, None] + 1 + np.arange(4)).ravel()], 1)
    check(rcell.params_kg(), [cell], None)

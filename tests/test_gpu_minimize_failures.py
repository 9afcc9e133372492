"""Cells that fail while they are minimised, beside cells that do not.

rcell_minimize returns the first cell's error and, through the C ABI, the moves
of every cell: those that relaxed have their count, those that failed (a list
beyond its capacity, a bond beyond its length, a staging wait that ran out) -1.
"""
import ctypes as C

import numpy as np
import pytest

from paper_1902_09171_gb300 import inputs, rcell
from test_gpu_few_cells import chains

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


def minimize(ctx, n_cells, f_tol, max_iter=2000):
    """(status code, moves per cell) of the C entry point."""
    it = np.full(n_cells, 77, np.int32)
    code = rcell.load().rcell_minimize(ctx, max_iter, f_tol, 2e-3, 1e-2, 0.02, C.c_void_p(it.ctypes.data))
    return rcell.STATUS[code], it.tolist()


def crystal(a, seed):
    x, H = inputs.fcc(5, 5, 5, a)
    return dict(H0=H, x0=inputs.to_f32(inputs.jitter(x, 0.01, seed)))


@pytest.mark.parametrize("graphs", [0, 1])
@pytest.mark.parametrize("lanes", [1, 4])
def test_a_list_beyond_its_capacity(lanes, graphs):
    # r_list = 6.19: 78 neighbours at a = 3.615 (next shell 6.26), 86 at a = 3.5
    cells = [crystal(3.615, 1), crystal(3.5, 2), crystal(3.615, 3)]
    ctx = rcell.rcell_create(rcell.params_lj_cu(), cells)
    try:
        rcell.rcell_set_tuning(ctx, lanes, graphs)
        rcell.rcell_set_limits(ctx, max_neighbors=80)
        status, it = minimize(ctx, 3, 1e-3)
        assert status == "RC_EOVERFLOW"
        assert it[1] == -1 and it[0] > 0 and it[2] > 0
    finally:
        rcell.rcell_destroy(ctx)


def test_a_bond_beyond_its_length():
    cells = [chains(40, 13, 1), chains(40, 13, 2)]
    cells[1]["x0"][26:39, 2] += np.where(np.arange(13) < 6, 0.0, 1.4)  # one bond of one chain
    ctx = rcell.rcell_create(rcell.params_kg(), cells)
    try:
        status, it = minimize(ctx, 2, 0.5)
        assert status == "RC_EBOND"
        assert it[1] == -1 and it[0] > 0
    finally:
        rcell.rcell_destroy(ctx)


def test_a_staging_wait_that_runs_out():
    ctx = rcell.rcell_create(rcell.params_lj_cu(), [crystal(3.615, 1), crystal(3.615, 2)])
    try:
        rcell.rcell_set_staging(ctx, 1)
        rcell.rcell_set_limits(ctx, wait_polls=0)
        status, it = minimize(ctx, 2, 1e-3)
        assert status == "RC_ETIMEOUT"
        assert it == [-1, -1]
    finally:
        rcell.rcell_destroy(ctx)

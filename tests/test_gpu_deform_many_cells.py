"""The deformation of batches with more cells than the chip has multiprocessors.

Several cells then share a block of the kernel.  Box, rotation, stretch and the
shift tables (through the forces of atoms at the cell's faces) are those of the
same cell alone, bit for bit; cells that are switched off keep theirs, and a
deformation with a negative determinant fails its own cell only.
"""
import numpy as np
import pytest

from paper_1902_09171_gb300 import inputs, rcell
from test_gpu_list_build import gas

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_cells", [100, 153, 500, 5001])
def test_every_cell_as_alone(n_cells):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1902_09171_gb300 import build
    build.build()
    rcell.load()
    rng = np.random.default_rng(n_cells)
    cells = [gas(12, np.array([14.0, 13.5, 14.5]), k % 50) for k in range(n_cells)]
    F = np.eye(3) + rng.uniform(-0.03, 0.03, (n_cells, 3, 3))
    off, bad = n_cells // 2, n_cells - 2
    on = np.ones(n_cells, np.int32)
    on[off] = 0
    F[bad] = np.diag([1.0, 1.0, -1.0])

    def state(cs, f, mask, look):
        ctx = rcell.rcell_create(rcell.params_lj_cu(), cs)
        try:
            rcell.rcell_set_active(ctx, mask)
            rcell.rcell_set_deformation(ctx, f)
            status = rcell.rcell_sync(ctx)
            rcell.rcell_eval(ctx)
            return status, [rcell.rcell_get_box(ctx, k) + rcell.rcell_get_atoms(ctx, k, 12) for k in look]
        finally:
            rcell.rcell_destroy(ctx)

    look = sorted({0, 1, 31, 32, 99, off - 1, off, off + 1, n_cells - 3, n_cells - 1})
    status, got = state(cells, F, on, look)
    assert rcell.STATUS[status] == "RC_EDEGEN"
    for k, g in zip(look, got):
        status, alone = state([cells[k]], F[k:k + 1], on[k:k + 1], [0])
        assert status == 0
        assert all(np.array_equal(a, b) for a, b in zip(g, alone[0])), k
        if k == off:
            assert np.array_equal(g[0], cells[k]["H0"])

"""rcell_restore on a stream of the caller's that does not wait for the default one.

The shift table of a restored cell is made on the context's stream, from the box
that was copied before it: whatever the cell's box was, an evaluation right after
the restore gives the forces of the checkpointed state, bit for bit.
"""
import numpy as np
import pytest

from paper_1902_09171_gb300 import rcell
from test_gpu_few_cells import copper

pytestmark = pytest.mark.gpu


def test_evaluation_right_after_a_restore():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1902_09171_gb300 import build
    build.build()
    rcell.load()
    cells = [copper(5, 500, k) for k in range(3)]
    stream = torch.cuda.Stream()
    ctx = rcell.rcell_create(rcell.params_lj_cu(), cells, stream=stream)
    try:
        saved = rcell.rcell_checkpoint(ctx, 1)
        rcell.rcell_eval(ctx)
        f0 = rcell.rcell_get_atoms(ctx, 1, 500)[2]
        rng = np.random.default_rng(1)
        for _ in range(20):
            rcell.rcell_set_deformation(ctx, np.eye(3) + rng.uniform(-0.05, 0.05, (3, 3, 3)))
            rcell.rcell_run(ctx, 4, 0)
            rcell.rcell_restore(ctx, 1, saved)
            rcell.rcell_eval(ctx)
            assert np.array_equal(rcell.rcell_get_atoms(ctx, 1, 500)[2], f0)
        assert rcell.rcell_sync(ctx) == 0
    finally:
        rcell.rcell_destroy(ctx)

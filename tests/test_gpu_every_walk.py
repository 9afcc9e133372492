"""Every walk of the pair kernels against the oracle and against each other.

Which walk runs depends on the number of tiles the host knows to be active: up to
two per multiprocessor sixteen lanes share an atom (compiled for two CTAs per
multiprocessor, or for three beyond half a tile each), otherwise, or where only
the device knows the mask, one lane per atom, pipelined or lean.  An all-ones
device mask forces the one-lane walks on any batch; batches of more than two tiles
per multiprocessor take them without a mask, in the unmasked order of the tiles.
Forces, virial and energy follow the oracle (tolerances of the parity tests), and
trajectories and minimisations are the same on every walk, bit for bit.
"""
import numpy as np
import pytest

import oracle
from _helpers import force_err, oracle_pot
from paper_1902_09171_gb300 import inputs, rcell
from test_gpu_few_cells import copper, general_sc

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


def melt(seed):
    x, H, bonds = inputs.kg_melt(20, 50, 0.85, seed=seed, pushoff_iters=300)
    return dict(H0=H, x0=inputs.to_f32(x), v0=inputs.to_f32(0.3 * np.random.default_rng(seed).normal(size=x.shape)), bonds=bonds)


CASES = {
    "lj": (lambda: rcell.params_lj_cu(seed=7), lambda k: copper(10, 4000 - 60 * k, k)),
    "sc": (lambda: rcell.params_sc_cu(seed=7), lambda k: copper(10, 4000 - 60 * k, k)),
    "sc_general": (general_sc, lambda k: copper(10, 4000 - 60 * k, k)),
    "kg": (lambda: rcell.params_kg(seed=7), lambda k: melt(70 + k)),
}


def batch(torch, name, tiles_per_sm):
    """Cells of at least tiles_per_sm tiles per multiprocessor, two different ones in turn."""
    two = [CASES[name][1](k) for k in (0, 1)]
    per = -(-len(two[0]["x0"]) // 128)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    return [two[k % 2] for k in range(int(tiles_per_sm * n_sm / per) + 2)]


@pytest.mark.parametrize("tiles_per_sm", [0.0, 0.6, 2.1])
@pytest.mark.parametrize("name", list(CASES))
def test_forces_and_trajectories(torch, name, tiles_per_sm):
    prm, cells = CASES[name][0](), batch(torch, name, tiles_per_sm)
    ones = torch.ones(len(cells), dtype=torch.int32, device="cuda")
    last = len(cells) - 1
    first = None
    for mask, lanes in ((None, 1), (None, 0), (ones, 1), (ones, 0)):
        ctx = rcell.rcell_create(prm, cells)
        try:
            rcell.rcell_set_tuning(ctx, lanes, 1)
            if mask is not None:
                rcell.rcell_set_active(ctx, mask)
            rcell.rcell_eval(ctx)
            pe, W = rcell.rcell_get_energy(ctx)
            x, _, f = rcell.rcell_get_atoms(ctx, last, len(cells[last]["x0"]))
            H, _, _ = rcell.rcell_get_box(ctx, last)
            if first is None:
                fo, Wo, eo = oracle.forces(oracle_pot(prm), x, H, bonds=cells[last].get("bonds"))
            assert force_err(f, fo) <= 1e-5
            assert np.abs(W[last] - Wo).max() <= 1e-4 * np.abs(Wo).max()
            assert abs(pe[last] - eo) <= 1e-5 * max(abs(eo), 1.0)
            rcell.rcell_run(ctx, 13, 5)
            assert rcell.rcell_sync(ctx) == 0
            end = [rcell.rcell_get_atoms(ctx, k, len(cells[k]["x0"]))[:2] for k in (0, last)]
            if first is None:
                first = (f, end)
            assert np.array_equal(f, first[0]), lanes
            for p, q in zip(end, first[1]):
                assert all(np.array_equal(u, v) for u, v in zip(p, q)), lanes
        finally:
            rcell.rcell_destroy(ctx)


@pytest.mark.parametrize("name", list(CASES))
def test_minimisations(torch, name):
    prm, cells = CASES[name][0](), batch(torch, name, 0.0)
    ones = torch.ones(len(cells), dtype=torch.int32, device="cuda")
    first = None
    for mask, lanes in ((None, 1), (None, 0), (ones, 1), (ones, 0)):
        ctx = rcell.rcell_create(prm, cells)
        try:
            rcell.rcell_set_tuning(ctx, lanes, 1)
            if mask is not None:
                rcell.rcell_set_active(ctx, mask)
            it = rcell.rcell_minimize(ctx, 40, 1e-9, 1e-3, 1e-2, 0.02)
            assert np.all(it == -1)
            end = [rcell.rcell_get_atoms(ctx, k, len(cells[k]["x0"])) for k in range(len(cells))]
            first = first or end
            for p, q in zip(end, first):
                assert all(np.array_equal(u, v) for u, v in zip(p, q)), lanes
            assert not np.array_equal(end[0][0], cells[0]["x0"])
        finally:
            rcell.rcell_destroy(ctx)

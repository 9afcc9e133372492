"""Batches with few active cells: the cooperative walk and the masked tile order.

The pair kernels change with the number of active tiles: sixteen lanes share an
atom where it is small and known to the host, and with cells switched off the
tiles are taken from a list.  All of them sum in list order, so the same cell
has the same trajectory, bit for bit, whichever runs: alone on the cooperative
walk (host mask), on the one-lane walk of a mask only the device knows, on the
lean walk, and among all cells.  The sampled stresses differ by the order of
their FP64 sums only.
"""
import numpy as np
import pytest

from _helpers import KB, M_CU
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


def copper(edge, n, seed):
    """n atoms of a jittered crystal at 300 K."""
    x, H = inputs.fcc(edge, edge, edge, 3.615)
    x = inputs.to_f32(inputs.jitter(x, 0.05, seed))[:n]
    return dict(H0=H, x0=x, v0=inputs.to_f32(inputs.maxwell(n, M_CU, 300 * KB, 0, seed)))


def chains(n_chains, length, seed):
    """Straight chains on a cubic grid with spacing 1.05, the bonds along x."""
    rng = np.random.default_rng(seed)
    m = int(np.ceil(n_chains ** 0.5))
    y, z = np.divmod(np.arange(n_chains), m)
    x = np.stack([np.tile(np.arange(length) * 0.97, n_chains), np.repeat(y * 1.08, length), np.repeat(z * 1.08, length)], 1)
    k = np.arange(n_chains * length)
    k = k[k % length < length - 1]
    H = np.diag([max(length * 0.97 + 0.3, 6.5), max(m * 1.08, 6.5), max(m * 1.08, 6.5)])
    return dict(H0=H, x0=inputs.to_f32(x + rng.uniform(-0.02, 0.02, x.shape)), v0=inputs.to_f32(0.4 * rng.normal(size=x.shape)),
                bonds=np.stack([k, k + 1], 1))


CASES = {
    "lj": (lambda: rcell.params_lj_cu(seed=5), lambda: [copper(5, n, n) for n in (500, 33, 257, 500, 128)]),
    "sc": (lambda: rcell.params_sc_cu(seed=5, skin=0.8), lambda: [copper(6, n, n) for n in (864, 700, 861, 129, 864)]),
    "sc_general": (lambda: general_sc(), lambda: [copper(6, n, n) for n in (864, 700, 861, 129, 864)]),
    "kg": (lambda: rcell.params_kg(seed=5), lambda: [chains(n, 13, n) for n in (64, 70, 81, 100, 33)]),
}


def general_sc():
    prm = rcell.params_sc_cu(seed=5, skin=0.8)
    prm.n, prm.m = 10.0, 7.0
    return prm


@pytest.mark.parametrize("name", list(CASES))
def test_same_trajectory_on_every_walk(torch, name):
    make, cells = CASES[name][0], CASES[name][1]()
    on = np.array([0, 0, 1, 1, 0], np.int32)
    F = np.tile(np.array([[1.004, 0.003, 0.0], [0.001, 0.998, 0.002], [0.0, -0.002, 1.001]]), (len(cells), 1, 1))

    def go(mask, lanes):
        ctx = rcell.rcell_create(make(), cells)
        try:
            rcell.rcell_set_tuning(ctx, lanes, 1)
            if mask is not None:
                rcell.rcell_set_active(ctx, mask)
            for _ in range(2):
                rcell.rcell_set_deformation(ctx, F)
                rcell.rcell_run(ctx, 21, 11)
            assert rcell.rcell_sync(ctx) == 0
            s = rcell.rcell_stress(ctx)[0]
            rcell.rcell_eval(ctx)
            out = [rcell.rcell_get_atoms(ctx, k, len(cells[k]["x0"])) for k in (2, 3)]
            return s[2:4], out
        finally:
            rcell.rcell_destroy(ctx)

    s0, a0 = go(on, 1)
    device = torch.tensor(on, device="cuda")
    for mask, lanes in ((device, 1), (device, 0), (None, 1), (on, 0)):
        s, a = go(mask, lanes)
        for p, q in zip(a0, a):
            assert all(np.array_equal(u, v) for u, v in zip(p, q)), (lanes, mask is None)
        assert np.abs(s - s0).max() <= 1e-12 * np.abs(s0).max()


def test_frozen_cells_stay_and_return(torch):
    cells = CASES["lj"][1]()
    ctx = rcell.rcell_create(rcell.params_lj_cu(seed=2), cells)
    try:
        rcell.rcell_eval(ctx)
        before = rcell.rcell_get_atoms(ctx, 1, 33)[0]
        rcell.rcell_set_active(ctx, np.array([1, 0, 1, 0, 1], np.int32))
        rcell.rcell_run(ctx, 7, 3)
        assert np.array_equal(rcell.rcell_get_atoms(ctx, 1, 33)[0], before)
        rcell.rcell_set_active(ctx, np.ones(5, np.int32))
        rcell.rcell_run(ctx, 7, 3)
        assert rcell.rcell_sync(ctx) == 0
        assert not np.array_equal(rcell.rcell_get_atoms(ctx, 1, 33)[0], before)
    finally:
        rcell.rcell_destroy(ctx)

"""Sutton-Chen with general exponents, negative and zero ones among them.

Lists hold pairs beyond the cutoff (the skin), which add nothing whatever the
exponents: a power of zero is infinite for a negative one.  Forces, virial and
energy against the oracle at the tolerances of the parity tests, on the walks of
one, sixteen (few tiles) and four lanes per atom, and the static stress finite.
"""
import numpy as np
import pytest

import oracle
from _helpers import force_err, oracle_pot
from paper_1902_09171_gb300 import rcell
from test_gpu_few_cells import copper

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(10.0, 7.0), (9.0, 5.5), (9.0, -2.0), (-3.0, 6.0), (8.0, 0.0)])
def test_forces_match_oracle(n, m):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1902_09171_gb300 import build
    build.build()
    rcell.load()
    prm = rcell.params_sc_cu(skin=0.8)
    prm.n, prm.m = n, m
    cell = copper(5, 500, 3)
    for mask, lanes in ((False, 1), (False, 4), (True, 1)):
        ctx = rcell.rcell_create(prm, [cell])
        try:
            rcell.rcell_set_tuning(ctx, lanes, 1)
            if mask:
                rcell.rcell_set_active(ctx, torch.ones(1, dtype=torch.int32, device="cuda"))
            rcell.rcell_eval(ctx)
            pe, W = rcell.rcell_get_energy(ctx)
            x, _, f = rcell.rcell_get_atoms(ctx, 0, 500)
            H, _, _ = rcell.rcell_get_box(ctx, 0)  # the FP32-exact MD box
            fo, Wo, eo = oracle.forces(oracle_pot(prm), x, H)
            assert force_err(f, fo) <= 1e-5
            assert np.abs(W[0] - Wo).max() <= 1e-4 * np.abs(Wo).max()
            assert abs(pe[0] - eo) <= 1e-5 * max(abs(eo), 1.0)
            assert np.isfinite(rcell.rcell_stress_static(ctx)[1]).all()
        finally:
            rcell.rcell_destroy(ctx)

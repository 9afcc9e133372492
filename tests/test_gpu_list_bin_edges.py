"""Neighbour lists of pairs just inside r_list whose atoms sit at bin edges.

The list build leaves out the bins along z that lie wholly beyond r_list, so a
pair is placed with one atom a hair below (or above) the edge of such a bin and
the other just within r_list of it along z, over every edge of boxes 4 to 30
times as long as wide, also tilted, among a background gas that fills the bins in
between.  Every pair closer than r_list (1 - 1e-6) has to be in both atoms'
lists, none that is farther than r_list (1 + 1e-6), and none twice.  (1e-6: a
displacement is rounded once, 6e-8 of it; its square and the sum of three take
three roundings more, and r_list^2 one.)
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


def edge_cell(H, r_list, n_gas, seed):
    """Two atoms r_list (1 - 2e-6) apart along z at every bin edge, and a background gas."""
    rng = np.random.default_rng(seed)
    n_bins = int(np.floor(2 * H[2, 2] / r_list))
    edges = H[2, 2] / n_bins * np.arange(n_bins)
    d = r_list * (1 - 2e-6)
    z = []
    for side in (-1, 1):  # the atom at the edge is the lower one, then the upper one
        for off in (-3e-6, 3e-6, -1e-4):
            a = edges + off
            z.append(np.stack([a, a - side * d], 1))
    z = np.concatenate(z)
    s = rng.uniform(0.02, 0.98, (len(z), 2))  # fractional x, y of a pair
    pair = np.concatenate([np.stack([s[:, 0], s[:, 1], z[:, k] / H[2, 2]], 1) for k in (0, 1)]) @ H.T
    pair[len(z):, :2] = pair[:len(z), :2]  # straight along z
    gas = rng.uniform(0, 1, (n_gas, 3)) @ H.T
    return dict(H0=H, x0=inputs.to_f32(np.concatenate([pair, gas])))


BOXES = {
    "thin": [[14.5, 0, 0], [0, 14.5, 0], [0, 0, 90.0]],
    "long": [[13.0, 0, 0], [0, 13.0, 0], [0, 0, 400.0]],
    "tilted": [[15.0, 2.1, -3.3], [0, 14.8, 4.2], [0, 0, 200.0]],
    "wide": [[45.0, 0, 0], [0, 30.0, 0], [0, 0, 60.0]],
    "short": [[60.0, 3.0, 1.0], [0, 45.0, -2.0], [0, 0, 13.0]],
}


@pytest.mark.parametrize("name", list(BOXES))
@pytest.mark.parametrize("seed", [1, 2])
def test_pairs_just_inside_the_list_radius_at_bin_edges(name, seed):
    prm = rcell.params_lj_cu()
    r_list = prm.rc + prm.skin
    H = np.array(BOXES[name], float)
    cell = edge_cell(H, r_list, int(0.05 * np.linalg.det(H)), seed)
    n = len(cell["x0"])
    ctx = rcell.rcell_create(prm, [cell])
    try:
        rcell.rcell_eval(ctx)
        x, _, _ = rcell.rcell_get_atoms(ctx, 0, n)
        got = [tuple(p) for p in rcell.rcell_get_neighbors(ctx, 0, n * 300)]
        near, far = ({tuple(p) for p in oracle.neighbor_pairs(x, H, r_list * f, max_pairs=n * 300)}
                     for f in (1 - 1e-6, 1 + 1e-6))
        assert len(set(got)) == len(got)
        assert near <= set(got) <= far, (len(near - set(got)), len(set(got) - far))
    finally:
        rcell.rcell_destroy(ctx)

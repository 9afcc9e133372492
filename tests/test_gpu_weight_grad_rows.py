"""Weight and bias gradients, block by block, from the rows at the ends of stages.

The targets are the predictions themselves except in the first and the last row of
every 64-row stage (the row ranges of the kernel's CTAs end there too), so a row
that is lost or taken twice is a sixtieth of the sum at most: an eighth of its
norm, in every block.  Weights and biases of every layer are compared by
themselves with the oracle's, at the tolerances of the gradient tests (BF16
operands: relative 5e-2, cosine 0.999), on both tcgen05 engines.
"""
import numpy as np
import pytest

from oracle import mlp
from paper_1902_09171_gb300 import rcell
from paper_1902_09171_gb300 import surrogate as S
from test_gpu_surrogate import bf16, bf16_weights, problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("backend", [1, 2])
@pytest.mark.parametrize("B,T", [(63, 1), (130, 1), (640, 1), (1950, 1), (333, 6)])
def test_every_block_from_the_rows_at_stage_ends(B, T, backend):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1902_09171_gb300 import build
    build.build()
    rcell.load()
    theta, U, _ = problem(300 + B, B, T)
    r = np.arange(B * T)
    edge = ((r % 64 == 0) | (r % 64 == 63) | (r == B * T - 1)).reshape(T, B).T  # row t B + b
    delta = np.random.default_rng(B).standard_normal((B, T, mlp.N_OUT)) * edge[:, :, None]
    s = S.sur_create(1, B, T, 0)
    try:
        S.sur_set_backend(s, backend)
        S.sur_set_params(s, 0, theta)
        dU = torch.tensor(U, dtype=torch.float32, device="cuda")
        pred = torch.empty((1, B, T, mlp.N_OUT), dtype=torch.float32, device="cuda")
        S.sur_predict(s, dU, pred)
        _, g = S.sur_loss_grad(s, 0, dU, pred[0] + torch.tensor(delta, dtype=torch.float32, device="cuda"))
        assert S.sur_sync(s) == 0
    finally:
        S.sur_destroy(s)
    w, u = bf16_weights(theta.astype(np.float64)), bf16(U)
    _, ref = mlp.loss_and_grad(w, u, mlp.forward(w, u)[0] + delta)
    for (name, a), b in zip(mlp.unpack(g.astype(np.float64)).items(), mlp.unpack(ref).values()):
        a, b = a.ravel(), b.ravel()
        assert np.linalg.norm(a - b) <= 5e-2 * np.linalg.norm(b), (name, np.linalg.norm(a - b) / np.linalg.norm(b))
        assert a @ b > 0.999 * np.linalg.norm(a) * np.linalg.norm(b), name

"""Weight and bias gradients of the tensor-core kernel where its row ranges end.

One row, fewer rows than a 64-row stage, exactly one, one more, a few stages
(one CTA per layer) and enough for several CTAs, in a context sized for more;
against the oracle's gradient with the tolerances of the gradient tests (BF16
operands: relative 5e-2, cosine 0.999), for every member of the context.
"""
import numpy as np
import pytest

from oracle import mlp
from paper_1902_09171_gb300 import rcell
from paper_1902_09171_gb300 import surrogate as S
from test_gpu_surrogate import bf16, bf16_weights, problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T", [(1, 1), (3, 7), (64, 1), (65, 1), (50, 9), (150, 13), (333, 6)])
def test_gradient_at_the_edges_of_the_row_ranges(B, T):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1902_09171_gb300 import build
    build.build()
    rcell.load()
    s = S.sur_create(2, B + 70, T + 2, 0)
    try:
        for member in range(2):
            theta, U, Y = problem(200 + member, B, T)
            S.sur_set_params(s, member, theta)
            dU = torch.tensor(U, dtype=torch.float32, device="cuda")
            dY = torch.tensor(Y, dtype=torch.float32, device="cuda")
            _, g = S.sur_loss_grad(s, member, dU, dY)
            assert S.sur_sync(s) == 0
            _, gr = mlp.loss_and_grad(bf16_weights(theta.astype(np.float64)), bf16(U), Y)
            assert np.linalg.norm(g - gr) <= 5e-2 * np.linalg.norm(gr)
            assert g @ gr > 0.999 * np.linalg.norm(g) * np.linalg.norm(gr)
    finally:
        S.sur_destroy(s)

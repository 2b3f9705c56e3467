"""GPU: the plain FP64 product (exp_zgemm, EXP_FP64) over the shapes where its division of the work
changes -- one output per thread, per group of lanes of a warp, per several warps -- against numpy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2004_03682_gb300 import expgb  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [
    (1, 1, 1), (1, 1, 7), (1, 1, 8), (1, 1, 5000), (3, 2, 33), (10, 10, 4001), (65, 1, 9), (1, 40, 700),
    (7, 11, 511), (7, 11, 512), (64, 64, 8), (130, 70, 65), (129, 19, 16), (500, 333, 20), (2003, 401, 3),
])
@pytest.mark.parametrize("beta", [False, True])
def test_fp64_product_at_the_edges_of_its_work_division(M, N, K, beta):
    rng = np.random.default_rng(M * 7 + N * 3 + K)
    A, B, C = (rng.standard_normal(s) + 1j * rng.standard_normal(s) for s in ((M, K), (K, N), (M, N)))
    dA, dB, dC = (torch.from_numpy(x).cuda() for x in (A, B, C.copy()))
    alpha = 0.75 - 1.25j
    out = expgb.zgemm(dA, dB, dC if beta else None, alpha=alpha, beta=beta).cpu().numpy()
    ref = alpha * (A @ B) + (C if beta else 0)
    # both sums have at most K + 8 rounded complex additions and products, then alpha and C
    bound = 4.0 * (K + 8) * 2.0 ** -53 * (abs(alpha) * (np.abs(A) @ np.abs(B)) + (np.abs(C) if beta else 0))
    assert np.all(np.abs(out - ref) <= bound)

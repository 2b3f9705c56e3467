"""GPU: the emulated product at three and four slices (64-column tiles) around the edges of its
tiles, bit-exact on integer inputs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [3, 4])
@pytest.mark.parametrize("M,N,K", [(127, 31, 40), (128, 32, 255), (129, 33, 256), (5, 64, 257), (33, 65, 16), (260, 7, 515),
                                   (64, 24, 2100)])
def test_tile_edges(S, M, N, K):
    import torch
    from paper_2004_03682_gb300 import build, expgb
    build.build()
    rng = np.random.default_rng(S + M + 10 * N + 100 * K)

    def c(*shape):
        return torch.tensor(rng.integers(-8, 9, shape) + 1j * rng.integers(-8, 9, shape), dtype=torch.complex128, device="cuda")

    A, B = c(M, K), c(K, N)
    out = expgb.zgemm(A, B, precision=expgb.EXP_EMU_BF16, n_slices=S)
    np.testing.assert_array_equal(out.cpu().numpy(), A.cpu().numpy() @ B.cpu().numpy())

"""GPU: rounding error of the plain FP64 product (exp_zgemm, EXP_FP64) against sums in extended precision."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2004_03682_gb300 import expgb  # noqa: E402

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def _rms_error(M, N, K, samples=1000):
    """Over sampled outputs of standard normal operands: rms of the real and imaginary parts' errors."""
    rng = np.random.default_rng(M + 3 * N + 7 * K)
    A, B = (torch.complex(*(torch.from_numpy(rng.standard_normal(s)) for _ in range(2))).cuda() for s in ((M, K), (K, N)))
    out = expgb.zgemm(A, B)
    at = rng.choice(M * N, min(samples, M * N), replace=False)
    r, c = torch.from_numpy(at // N).cuda(), torch.from_numpy(at % N).cuda()
    a, b, got = A[r].cpu().numpy(), B[:, c].T.contiguous().cpu().numpy(), out[r, c].cpu().numpy()
    err = []
    for x, y, z in zip(a, b, got):
        xr, xi, yr, yi = (np.asarray(t, dtype=np.longdouble) for t in (x.real, x.imag, y.real, y.imag))
        err += [z.real - ((xr * yr).sum() - (xi * yi).sum()), z.imag - ((xr * yi).sum() + (xi * yr).sum())]
    return float(np.sqrt(np.mean(np.square(np.asarray(err, dtype=np.float64)))))


# A rounded number of rms size s has an error of at most 2 U s / sqrt(12) rms.  A sum of 2n products of variance
# one (n complex terms) in one sequence rounds numbers of variance 1 .. 2n.
def _sequence(n):
    return 4.0 / 12.0 * n * (2.0 * n + 1.0)


# ranges of 256 terms, added in sequence
def _ranges(K, r=256):
    m = K / r
    return U * np.sqrt(m * _sequence(r) + 4.0 / 12.0 * 2 * r * m * (m + 1) / 2)


@pytest.mark.parametrize("M,N,K", [(300, 300, 4000), (400, 400, 5000), (109, 109, 12000), (700, 130, 8000), (64, 64, 100000)])
def test_long_sums_are_as_accurate_as_ranges_of_256_terms(M, N, K):
    assert _rms_error(M, N, K) < _ranges(K)


# one warp to an output: a sequence per lane, then the lanes pairwise
def _warp(K):
    return U * np.sqrt(32 * _sequence(K / 32 if K > 32 else 1) * min(K, 32) / 32 + 4.0 / 12.0 * 2 * K * np.ceil(np.log2(min(K, 32))))


@pytest.mark.parametrize("M,N,K", [(20000, 1, 5000), (20000, 2, 2000), (1, 3000, 1000), (100000, 1, 40), (60000, 2, 16),
                                   (360, 360, 32), (290, 290, 48), (200, 200, 100), (100, 100, 400), (64, 64, 1000)])
def test_small_and_matrix_vector_products_are_as_accurate_as_a_warp_per_output(M, N, K):
    assert _rms_error(M, N, K) < _warp(K)

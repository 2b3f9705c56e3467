"""GPU: the bf16 kernels of the learned guess at the edges of their 16-sample pieces, 32-sample tiles and
128-sample groups, against the FP64 oracle with the same BF16 roundings."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from oracle import mlp as omlp  # noqa: E402
from paper_2004_03682_gb300 import expgb  # noqa: E402
from paper_2004_03682_gb300 import synthetic as syn  # noqa: E402

pytestmark = pytest.mark.gpu


def _bf(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).to(torch.bfloat16).to(torch.float64).numpy()


def _params(seed):
    p = omlp.init_params(seed)
    rng = np.random.default_rng(seed)
    k = omlp.NO * omlp.W + omlp.NO
    p[-k:] = 0.1 * rng.standard_normal(k)
    return p.astype(np.float32)


def _forward(p, x):
    W1, b1, W2, b2, W3, b3 = omlp.unflatten(p)
    h1 = _bf(np.maximum(x.astype(np.float64) @ _bf(W1).T + b1, 0.0))
    h2 = _bf(np.maximum(h1 @ _bf(W2).T + b2, 0.0))
    return h1, h2, h2 @ _bf(W3).T + b3


# an activation or gradient that lies within FP32 accumulation error of a rounding boundary takes the other
# BF16 neighbour: one part in 2^8 of one of 128 terms at worst, 2e-3 of a sum with room to spare
TOL = 2e-3


@pytest.mark.parametrize("n", [1, 15, 16, 17, 32, 33, 127, 129, 32 * 304 + 5, 4 * 32 * 304 + 17])
def test_bf16_gradient_by_sample_count(n):
    p, rng = _params(n), np.random.default_rng(n + 1)
    x = rng.uniform(0, 1, (n, 3)).astype(np.float32)
    tm = (0.05 * (rng.standard_normal(n) + 1j * rng.standard_normal(n))).astype(np.complex64).astype(complex)
    tg = (tm * (0.8 + 0.1j) + 0.002 * rng.standard_normal(n)).astype(np.complex64).astype(complex)
    m = expgb.Mlp(seed=1, bf16=True)
    m.params(set=p)
    L, g = m.loss_grad(x, tm, tg)
    W1, b1, W2, b2, W3, b3 = omlp.unflatten(p)
    h1, h2, y = _forward(p, x)
    r = (1 + y[:, 0] + 1j * y[:, 1]) * tm - tg
    c = 2.0 / (n * 0.05 ** 2)
    gy = c * np.stack([np.real(r.conj() * tm), np.real(r.conj() * 1j * tm)], -1)
    gz2 = (gy @ _bf(W3)) * (h2 > 0)
    gz1 = (_bf(gz2) @ _bf(W2)) * (h1 > 0)
    ref = [gz1.T @ x, gz1.sum(0), _bf(gz2).T @ h1, gz2.sum(0), gy.T @ h2, gy.sum(0)]
    assert abs(L - np.mean(np.abs(r) ** 2) / 0.05 ** 2) < TOL * L
    for got, want in zip(omlp.unflatten(g), ref):
        assert np.linalg.norm(got.ravel() - want.ravel()) < TOL * np.linalg.norm(want)


@pytest.mark.parametrize("o,v,g", [(2, 3, 1), (3, 11, 1), (5, 13, 3)])
def test_bf16_guess_by_element_count(o, v, g):
    prob = syn.make_problem(9, o, v, g)
    ctx = expgb.from_problems([prob])
    ctx.init_integrals([prob.seed])
    expgb.Mlp(seed=5).apply(ctx)  # untrained: the first-order amplitudes
    t = ctx.get_amplitudes(0)[1].cpu().numpy()
    m, p = expgb.Mlp(seed=1, bf16=True), _params(4)
    m.params(set=p)
    m.apply(ctx)
    got = ctx.get_amplitudes(0)[1].cpu().numpy()
    D = (prob.eps_occ[:, None, None, None] + prob.eps_occ[:, None, None] - prob.eps_virt[:, None] - prob.eps_virt)
    va = np.abs(t) * np.abs(D)
    _, _, y = _forward(p, np.stack([np.abs(t) / 0.05, -D / 10.0, va / va.max()], -1).reshape(-1, 3))
    want = (1 + y[:, 0] + 1j * y[:, 1]).reshape(t.shape) * t
    assert np.abs(got - want).max() < TOL * np.abs(want).max()


def test_bf16_guess_of_many_instances_by_element():
    """More elements to an instance than one sweep of its CTAs takes, a ragged end, a trained output layer: every
    instance against the oracle."""
    n, o, v = 64, 6, 23  # 19044 elements an instance; 8 waves of 3 CTAs on each SM are 57 CTAs of 128 an instance
    probs = [syn.make_problem(40 + k, o, v, 1) for k in range(n)]
    ctx = expgb.from_problems(probs)
    ctx.init_integrals([p.seed for p in probs], scale_mult=[0.5 + k / n for k in range(n)])
    expgb.Mlp(seed=5).apply(ctx)  # untrained: the first-order amplitudes
    first = [ctx.get_amplitudes(k)[1].cpu().numpy() for k in range(n)]
    m, p = expgb.Mlp(seed=1, bf16=True), _params(4)
    m.params(set=p)
    m.apply(ctx)
    for k, (prob, t) in enumerate(zip(probs, first)):
        got = ctx.get_amplitudes(k)[1].cpu().numpy()
        D = (prob.eps_occ[:, None, None, None] + prob.eps_occ[:, None, None] - prob.eps_virt[:, None] - prob.eps_virt)
        va = np.abs(t) * np.abs(D)
        _, _, y = _forward(p, np.stack([np.abs(t) / 0.05, -D / 10.0, va / va.max()], -1).reshape(-1, 3))
        want = (1 + y[:, 0] + 1j * y[:, 1]).reshape(t.shape) * t
        assert np.abs(want - t).max() > 0.05 * np.abs(t).max()  # the output layer counts
        assert np.abs(got - want).max() < TOL * np.abs(want).max()
    ctx.close()


def test_bf16_training_repeats_bit_for_bit():
    probs = [syn.make_problem(70 + k, 6, 22, 1) for k in range(8)]
    ctx = expgb.from_problems(probs, conv_tol=1e-6, max_iter=200)
    ctx.init_integrals([p.seed for p in probs], scale_mult=[0.4] * len(probs))
    ctx.iterate(200, raise_numeric=False)
    runs = []
    for _ in range(3):
        m = expgb.Mlp(seed=3, bf16=True)
        m.add_training_data(ctx)
        assert m.n_samples > 32 * 304
        runs.append((m.train(4, batch=16384, lr=2e-3, seed=1), m.params()))
    ctx.close()
    for losses, params in runs[1:]:
        np.testing.assert_array_equal(losses, runs[0][0])
        np.testing.assert_array_equal(params, runs[0][1])

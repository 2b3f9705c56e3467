"""GPU: the width of the emulated product's tiles at three and four slices: 48 real columns where 64 would not
save a tile, or a wave of them at short K, bit-exact either way; and (T), whose operand sets are laid out in
those tiles, on both."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from oracle import ccsd, integrals, triples  # noqa: E402
from paper_2004_03682_gb300 import expgb  # noqa: E402
from paper_2004_03682_gb300 import synthetic as syn  # noqa: E402

pytestmark = pytest.mark.gpu


def _kernels(f):
    """f() and the names of its kernels; a profile that recorded none (a process's first) is taken again."""
    for _ in range(4):
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as p:
            out = f()
            torch.cuda.synchronize()
        names = " ".join(e.key for e in p.key_averages())
        if "k_emu_gemm" in names:
            break
    return out, names


@pytest.mark.parametrize("S", [3, 4])
@pytest.mark.parametrize("M,N,K,cols", [(300, 1, 70, 48), (300, 24, 70, 48), (300, 25, 70, 48), (140, 32, 600, 64),
                                        (140, 33, 600, 48), (140, 48, 40, 48), (140, 49, 40, 48), (150, 72, 300, 48),
                                        (150, 73, 1100, 64), (600, 600, 100, 48), (4000, 150, 20, 48),
                                        (20000, 25, 100, 64), (12000, 100, 300, 64)])
def test_tile_width(S, M, N, K, cols):
    rng = np.random.default_rng(S + M + 10 * N + 100 * K)
    A, B = (torch.tensor(rng.integers(-8, 9, s) + 1j * rng.integers(-8, 9, s), dtype=torch.complex128, device="cuda")
            for s in ((M, K), (K, N)))
    out, names = _kernels(lambda: expgb.zgemm(A, B, precision=expgb.EXP_EMU_BF16, n_slices=S))
    np.testing.assert_array_equal(out.cpu().numpy(), A.cpu().numpy() @ B.cpu().numpy())
    assert f"k_emu_gemm<{S}, {cols}, false>" in names  # and without the code of the double-single outputs


# each slice fewer costs 7 bits: 1e-9 at six slices
@pytest.mark.parametrize("S,rel", [(3, 1e-9 * 2.0 ** 21), (4, 1e-9 * 2.0 ** 14)])
@pytest.mark.parametrize("no,nv,G,cols", [(4, 22, 1, 48), (4, 30, 1, 64), (4, 40, 1, 48), (5, 34, 2, 64)])
def test_triples_on_either_width(S, rel, no, nv, G, cols):
    prob = syn.make_problem(851 + nv, no, nv, G)
    t1, t2 = syn.trial_amplitudes(prob, 5)
    ctx = expgb.from_problems([prob], precision=expgb.EXP_EMU_BF16, n_slices=S)
    ctx.init_integrals([prob.seed])
    ctx.set_amplitudes(0, torch.from_numpy(t1), torch.from_numpy(t2))
    (E, _, e3), names = _kernels(lambda: ctx.ccsd_t(0, per_triple=True))
    ctx.close()
    orc = triples.per_triple(t1, t2, ccsd.Blocks(integrals.integrals(prob), integrals.fock(prob), no))
    ref = np.array([orc[i, j, k] for k in range(no) for j in range(k) for i in range(j)])
    assert np.abs(e3 - ref).max() < rel * np.abs(ref).max()
    assert f"k_emu_gemm<{S}, {cols}, true>" in names

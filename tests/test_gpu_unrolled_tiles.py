"""The unrolled decoder's on-chip path (rows and columns of degree at most 8) at
its edges: part-filled tiles of 8 shots, more tiles than blocks, rows of degree
1 to 8 at aligned and unaligned places, columns of degree up to 4 and up to 8, a
clamp that is met, checkpoint intervals that all use it.

Against the double-precision reference with the tolerances of the general passes'
tests (posteriors 1e-4, loss terms 1e-5, gradients 1e-4 of the largest plus 1e-3
of each): both paths run the same single-precision operations per message."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import unrolled as U  # noqa: E402
from paper_2512_07057_gb300 import unrolled as G  # noqa: E402
from paper_2512_07057_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _problem(max_col, M, N, seed):
    """Columns of degree 1..max_col, rows of degree at most 8."""
    rng = np.random.default_rng([max_col, M, N, seed])
    H = np.zeros((M, N), np.uint8)
    for j in range(N):
        free = np.nonzero(H.sum(1) < 8)[0]
        H[rng.choice(free, size=min(free.size, int(rng.integers(1, max_col + 1))), replace=False), j] = 1
    H[M - 1] = 0
    H[M - 1, 0] = 1                                       # a row of degree 1
    return W.problem_from_dense(H, (rng.random((2, N)) < 0.3).astype(np.uint8), rng.uniform(0.02, 0.2, N))


CASES = {
    "one": (lambda: W.bb72_code_capacity(0.05), 1, 5, 2, 1e4),
    "seven": (lambda: _problem(4, 61, 90, 0), 7, 6, 3, 1e4),
    "eight": (lambda: _problem(8, 77, 80, 1), 8, 4, 4, 1e4),
    "nine_clamped": (lambda: _problem(4, 61, 90, 2), 9, 6, 2, 6.0),
    "many_tiles": (lambda: _problem(3, 33, 60, 3), 8 * 152 * 5 + 3, 3, 2, 1e4),
    "aligned_rows": (lambda: W.bb_phenomenological(6, 6, 3, 0.03, 0.03), 70, 8, 3, 1e4),
}


@pytest.mark.parametrize("name", list(CASES))
def test_tiles_match_fp64(name):
    build, Bn, T, k, clamp = CASES[name]
    prob = build()
    w = np.random.default_rng(11).uniform(0.4, 1.1, size=(T, prob.n_edges)).astype(np.float32)
    s_t, e_t, sh = G.batch_tensors(prob, Bn, f"tiles_{name}")
    wt = torch.from_numpy(w).cuda()
    runs = []
    for ck in sorted({1, k, T}):
        tr = G.UnrolledTrainer(prob, Bn, T, ck, llr_clamp=clamp)
        llr = torch.empty((T, Bn, prob.N), dtype=torch.float32, device="cuda")
        loss = tr.forward(wt, s_t, e_t, llr).cpu().numpy().copy()
        runs.append((loss, llr.cpu().numpy(), tr.backward(wt, torch.ones(1, device="cuda")).cpu().numpy()))
        tr.close()
    for r in runs[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(runs[0], r))
    loss, llr, grad = runs[0]
    s, e = W.unpack_bits(sh.syndromes, prob.M), W.unpack_bits(sh.errors, prob.N)
    rl, rg, rpt, rtraj = U.unrolled_grad(U.Tables(prob), s, e, w.astype(np.float64), llr_clamp=clamp)
    assert np.all(np.abs(llr - rtraj) <= 1e-4 * np.maximum(1.0, np.abs(rtraj)))
    np.testing.assert_allclose(loss[1:], rpt, rtol=1e-5)
    assert abs(loss[0] - rl) <= 1e-5 * rl
    assert np.all(np.abs(grad - rg) <= 1e-4 * np.abs(rg).max() + 1e-3 * np.abs(rg))

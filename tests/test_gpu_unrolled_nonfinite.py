"""Training with a weight that is NaN or infinite, on tiles of shots: a posterior
that is not finite passes on what the clamp makes of its messages, -L_MAX of a NaN.
Posteriors against the double-precision passes with that clamp, within the tolerance
of the other tests (1e-4), infinities and NaN in the same places."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import unrolled as U  # noqa: E402
from paper_2512_07057_gb300 import unrolled as G  # noqa: E402
from paper_2512_07057_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _posteriors(prob, s_bits, w, L=1e4):
    tab = U.Tables(prob)
    sign = 1.0 - 2.0 * torch.as_tensor(s_bits, dtype=torch.float64)
    col = torch.as_tensor(tab.col_of_edge)
    E = U._initial(tab, sign.shape[0], L)
    out = []
    for wt in torch.as_tensor(w, dtype=torch.float64):
        D, _ = U._check_pass(tab, sign, E, wt, L)
        post, _, _ = U._error_pass(tab, D, L)
        E = torch.nan_to_num(post[:, col] - D, nan=-L, posinf=L, neginf=-L).clamp(-L, L)
        out.append(post)
    return torch.stack(out).numpy()


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_weights_that_are_not_finite(bad):
    prob = W.bb72_code_capacity(0.05)
    prob.priors = np.random.default_rng(1).uniform(0.02, 0.09, prob.N)      # no exact ties between columns
    T, shots = 5, 21
    w = np.random.default_rng(2).uniform(0.4, 0.9, (T, prob.n_edges)).astype(np.float32)
    w[1, 7] = w[2, 100] = bad
    synd, errs, sh = G.batch_tensors(prob, shots, "nonfinite")
    tr = G.UnrolledTrainer(prob, shots, T, 2)
    llr = torch.empty((T, shots, prob.N), dtype=torch.float32, device="cuda")
    tr.forward(torch.from_numpy(w).cuda(), synd, errs, llr)
    got = llr.cpu().numpy()
    tr.close()
    want = _posteriors(prob, W.unpack_bits(sh.syndromes, prob.M), w)
    assert np.array_equal(np.isnan(got), np.isnan(want)) and not np.isfinite(want[1]).all()
    assert np.isfinite(want[3:]).all() and np.isfinite(want).sum() > 0.9 * want.size
    ok = np.isfinite(want)
    assert np.array_equal(got[~ok], want[~ok].astype(np.float32), equal_nan=True)
    assert np.all(np.abs(got[ok] - want[ok]) <= 1e-4 * np.maximum(1.0, np.abs(want[ok])))

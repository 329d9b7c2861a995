"""Plain BP on tiles of 8 shots (rows of at most 8 edges, columns of at most 3) at
its edges: one shot, a whole tile, part-filled tiles, more tiles than blocks, one iteration, a clamp that is met.  Bit for bit the
per-candidate engine's results, which a call with ms_scale as the weight of every
edge still takes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2512_07057_gb300 import decoder as D  # noqa: E402
from paper_2512_07057_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _problem(M, N, seed):
    """Columns of degree 1..3 (and one of none), rows of degree 0..8, priors on both sides of 1/2."""
    rng = np.random.default_rng([M, N, seed])
    H = np.zeros((M, N), np.uint8)
    for j in range(1, N):
        free = np.nonzero(H.sum(1) < 8)[0]
        H[rng.choice(free, size=min(free.size, int(rng.integers(1, 4))), replace=False), j] = 1
    return W.problem_from_dense(H, (rng.random((2, N)) < 0.3).astype(np.uint8), rng.uniform(0.02, 0.6, N))


CASES = {
    "one": (lambda: _problem(61, 90, 0), 1, 5, 1e4),
    "eight": (lambda: _problem(61, 90, 0), 8, 5, 1e4),
    "ragged": (lambda: _problem(33, 60, 1), 8 * 152 * 9 + 3, 3, 1e4),
    "clamped": (lambda: _problem(61, 90, 2), 777, 9, 4.0),
    "once": (lambda: W.bb_phenomenological(6, 6, 3, 0.03, 0.03), 1001, 1, 1e4),
    "phenomenological": (lambda: W.bb_phenomenological(12, 6, 12, 0.03, 0.03), 1001, 20, 1e4),
}


@pytest.mark.parametrize("name", list(CASES))
def test_tiles_match_engine(name):
    build, Bn, T, clamp = CASES[name]
    prob = build()
    params = D.make_params(llr_clamp=clamp, max_rounds=0)
    dec = D.BeamSearchDecoder(prob, params)
    shots = W.sample_shots(prob, Bn, f"llr_tiles_{name}")
    synd = D.to_torch_words(shots.syndromes)
    got = [t.cpu().numpy() for t in dec.bp_llr(synd, T)]
    dec.set_weights(np.full((T, prob.n_edges), params.ms_scale, np.float32))
    want = [t.cpu().numpy() for t in dec.bp_llr(synd, T)]
    dec.close()
    for a, b in zip(got, want):
        assert np.array_equal(a, b)

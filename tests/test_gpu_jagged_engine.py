"""The jagged engine at its edges: rows of degree 0 to above 16 (its three
register variants and the loop), groups of columns of one degree 1 to 6 and of
mixed degrees with columns of degree 0, a last group that is not full, a clamp met
in every run, alpha 1, several results, 16-bit storage, weights, a warp and blocks
of 2 and 16 warps per candidate; shots that find the seed store full.  Bit-exact
against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2512_07057_gb300 import decoder as D  # noqa: E402
from paper_2512_07057_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _problem(M, degrees, seed):
    """32 columns of each degree in turn (0: mixed, 0 to the largest), then 5 more."""
    rng = np.random.default_rng([M, seed, *degrees])
    cols = [d for d in degrees for _ in range(32)] + [max(degrees)] * 5
    H = np.zeros((M, len(cols)), np.uint8)
    for j, d in enumerate(cols):
        d = int(rng.integers(0, max(degrees) + 1)) if d == 0 else d
        H[rng.choice(M - 1, size=d, replace=False), j] = 1      # the last row has no edge
    return W.problem_from_dense(H, (rng.random((2, len(cols))) < 0.3).astype(np.uint8),
                                rng.uniform(0.01, 0.05, len(cols)))


@pytest.mark.parametrize("M,degrees", [(30, (1, 2, 3, 0)), (60, (3, 3, 2)), (40, (4, 5, 6, 0, 2)), (110, (6, 6, 3, 0)),
                                       (70, (5, 6, 6)), (14, (3, 0))])
@pytest.mark.parametrize("alpha,clamp,storage,group_warps,results", [(0.625, 1e4, 0, 1, 1), (1.0, 5.0, 0, 2, 1),
                                                                     (0.625, 6.0, 1, 16, 1), (0.625, 6.0, 2, 1, 3)])
@pytest.mark.parametrize("weighted", [False, True])
def test_edges_of_the_jagged_engine(M, degrees, alpha, clamp, storage, group_warps, results, weighted):
    if weighted and storage:
        pytest.skip("weights take single-precision messages")
    prob = _problem(M, degrees, 1)
    shots = W.sample_shots(prob, 500, f"jagged_{M}")
    kw = dict(max_rounds=4, beam_width=5, initial_iters=7, iters_per_round=6, num_results=results)
    w = np.random.default_rng(2).uniform(0.3, 1.2, (3, prob.n_edges)).astype(np.float32) if weighted else None
    dec = D.BeamSearchDecoder(prob, D.make_params(ms_scale=alpha, llr_clamp=clamp, msg_precision=storage,
                                                  tie_guard_rel=-1.0, group_warps=group_warps, **kw))
    if weighted:
        dec.set_weights(w)
    out = dec.decode(D.to_torch_words(shots.syndromes))
    torch.cuda.synchronize()
    assert dec.sync_error() == 0
    ref = oracle.Graph(prob, "f32").decode_batch(
        shots.syndromes, oracle.Params(ms_scale=alpha, llr_clamp=clamp, msg_storage=storage, weights=w, **kw),
        nthreads=8)
    for name, got in (("corrections", out.corrections), ("status", out.status), ("iters", out.iters)):
        assert np.array_equal(D.from_torch_words(got), ref[name]), name
    dec.close()


@pytest.mark.parametrize("rounds,timed", [(3, False), (3, True), (0, False)])
def test_shots_that_find_the_seed_store_full(rounds, timed):
    """One chunk of more failing shots than the seed store holds: the others are
    decoded in windows after its beam, with and without kernel timing."""
    prob = W.bb_xyz_code_capacity(6, 6, 0.09)
    prob.priors = np.random.default_rng(4).uniform(0.02, 0.05, prob.N)
    shots = W.sample_shots(prob, 3_000, "full_store")
    kw = dict(max_rounds=rounds, beam_width=4, initial_iters=3, iters_per_round=5)
    dec = D.BeamSearchDecoder(prob, D.make_params(ms_scale=0.625, workspace_bytes=9 << 20, **kw))
    store = dec.info["chunk_shots"]
    dec.profile(timed)
    out = dec.decode(D.to_torch_words(shots.syndromes))
    torch.cuda.synchronize()
    assert dec.sync_error() == 0
    ref = oracle.Graph(prob, "f32").decode_batch(shots.syndromes, oracle.Params(ms_scale=0.625, **kw), nthreads=8)
    assert (ref["status"] != 1).sum() > 1_000 and store < 3_000
    for name, got in (("corrections", out.corrections), ("status", out.status), ("iters", out.iters)):
        assert np.array_equal(D.from_torch_words(got), ref[name]), name
    dec.close()

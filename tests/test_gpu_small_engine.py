"""The single-warp engine at the edges of what it takes: the smallest and
largest code of each of its two sizes (N = 66, 96, 130, 160), a clamp low
enough to be met in every run (the detector pass caps its minima at L_MAX
with the syndrome sign, masked nodes read as L_MAX), one and several results,
single and half precision.  Bit-exact against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2512_07057_gb300 import binding as B  # noqa: E402
from paper_2512_07057_gb300 import decoder as D  # noqa: E402
from paper_2512_07057_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [33, 48, 65, 80])
@pytest.mark.parametrize("clamp,alpha,results,storage", [(6.0, 0.625, 1, 0), (3.5, 1.0, 1, 0), (1e4, 0.625, 4, 0),
                                                         (6.0, 0.625, 1, 1)])
def test_edges_of_the_single_warp_engine(M, clamp, alpha, results, storage):
    prob = W.random_regular_36(M, 0.06, 3)
    prob.priors = np.random.default_rng(M).uniform(0.03, 0.09, prob.N)   # no exact ties between columns
    shots = W.sample_shots(prob, 1_000, f"small_edges_{M}")
    params = D.make_params(max_rounds=7, beam_width=5, initial_iters=12, iters_per_round=9, ms_scale=alpha,
                           llr_clamp=clamp, num_results=results, tie_guard_rel=-1.0,
                           msg_precision=B.BSD_FP16 if storage else B.BSD_FP32)
    dec = D.BeamSearchDecoder(prob, params)
    assert dec.shape[0] == 1
    out = dec.decode(D.to_torch_words(shots.syndromes))
    torch.cuda.synchronize()
    assert dec.sync_error() == 0
    ref = oracle.Graph(prob, "f32").decode_batch(
        shots.syndromes, oracle.Params(max_rounds=7, beam_width=5, initial_iters=12, iters_per_round=9,
                                       num_results=results, ms_scale=alpha, llr_clamp=clamp, msg_storage=storage),
        nthreads=8)
    assert (ref["status"] == 2).sum() > 20                                # the beam is used
    for name, got in (("corrections", out.corrections), ("status", out.status), ("iters", out.iters)):
        assert np.array_equal(D.from_torch_words(got), ref[name]), name
    dec.close()

"""The beam kernel's ring and window entries at their limits: one or two
entries that take shot after shot, a ring that comes round many times, the
narrowest and the widest beam, several results, warp and block candidates.
Bit-exact against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2512_07057_gb300 import decoder as D  # noqa: E402
from paper_2512_07057_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,entries", [(1, 1), (1, 2), (7, 1), (64, 2)])
@pytest.mark.parametrize("results,group_warps", [(1, 0), (3, 0), (1, 4)])
def test_few_window_entries_take_many_shots(width, entries, results, group_warps):
    prob = W.bb72_code_capacity(0.06)
    prob.priors = np.random.default_rng(5).uniform(0.06, 0.12, prob.N)   # no exact ties between columns
    shots = W.sample_shots(prob, 400, "beam_ring")
    kw = dict(max_rounds=6, beam_width=width, initial_iters=4, iters_per_round=5, num_results=results)
    # a child slot takes about 1.5 KB and a window entry has 4 w of them; the
    # window gets four fifths of the workspace, the store of waiting shots the rest
    params = D.make_params(ms_scale=0.625, group_warps=group_warps, small_batch=-1,
                           workspace_bytes=int(4 * width * 1500 * (entries + 0.2) / 0.8), **kw)
    dec = D.BeamSearchDecoder(prob, params)
    out = dec.decode(D.to_torch_words(shots.syndromes))
    torch.cuda.synchronize()
    assert dec.sync_error() == 0
    ref = oracle.Graph(prob, "f32").decode_batch(shots.syndromes, oracle.Params(ms_scale=0.625, **kw), nthreads=8)
    assert (ref["status"] == 2).sum() > 40
    for name, got in (("corrections", out.corrections), ("status", out.status), ("iters", out.iters)):
        assert np.array_equal(D.from_torch_words(got), ref[name]), name
    dec.close()

"""16-bit storage of codes whose messages do not fit on chip as floats: bit for bit
the oracle's 16-bit run, with a warp, 2 and 16 warps per candidate, column degrees up
to 3 and up to 6, one and several results; a code just below the size still runs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2512_07057_gb300 import decoder as D  # noqa: E402
from paper_2512_07057_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _problem(M, N, max_deg):
    """Columns of degree max_deg (the first ones fewer), priors low enough that part
    of the shots need the beam."""
    rng = np.random.default_rng([M, N, max_deg])
    H = np.zeros((M, N), np.uint8)
    for j in range(N):
        H[rng.choice(M, size=max_deg if j >= 40 else j % (max_deg + 1), replace=False), j] = 1
    return W.problem_from_dense(H, (rng.random((2, N)) < 0.05).astype(np.uint8),
                                np.exp(rng.uniform(np.log(3e-4), np.log(3e-3 if max_deg == 3 else 1.2e-2), N)))


# 4 E + 4 N bytes against the 227 KB of a block: 240, 288 and 224 KB
@pytest.mark.parametrize("M,N,max_deg,storage,group_warps,results",
                         [(700, 15000, 3, 1, 0, 1), (700, 15000, 3, 2, 1, 3), (900, 12000, 5, 1, 1, 1),
                          (900, 12000, 5, 2, 2, 1), (900, 12000, 5, 1, 16, 2), (700, 14000, 3, 1, 0, 1)])
def test_codes_too_large_for_floats_on_chip(M, N, max_deg, storage, group_warps, results):
    prob = _problem(M, N, max_deg)
    shots = W.sample_shots(prob, 120, f"wide_{M}_{N}")
    kw = dict(max_rounds=3, beam_width=3, initial_iters=3, iters_per_round=5, num_results=results)
    dec = D.BeamSearchDecoder(prob, D.make_params(ms_scale=0.625, msg_precision=storage, tie_guard_rel=-1.0,
                                                  group_warps=group_warps, batch_slots=-1, **kw))
    out = dec.decode(D.to_torch_words(shots.syndromes))
    torch.cuda.synchronize()
    assert dec.sync_error() == 0
    ref = oracle.Graph(prob, "f32").decode_batch(shots.syndromes,
                                                 oracle.Params(ms_scale=0.625, msg_storage=storage, **kw), nthreads=8)
    assert (ref["status"] != 1).sum() > 5
    for name, got in (("corrections", out.corrections), ("status", out.status), ("iters", out.iters)):
        assert np.array_equal(D.from_torch_words(got), ref[name]), name
    dec.close()

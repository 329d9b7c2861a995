"""The second-iteration screen of seed runs: column degrees 0 to 3, 6 and 16,
rows of degree 0 to 3 (fewer than the four entries kept per row), equal and
log-uniform priors (ties of the row minima), a clamp met at t = 1, alpha 1, 16-bit
storage, a queue too short for it, and dense syndromes whose lists overflow, some of them just.  Every
output equals the oracle's bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2512_07057_gb300 import binding as B  # noqa: E402
from paper_2512_07057_gb300 import decoder as D  # noqa: E402
from paper_2512_07057_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _problem(max_deg, M, N, errors, equal, thin):
    """Columns of degree 0..max_deg; the last `thin` rows meet at most 3 columns."""
    rng = np.random.default_rng([max_deg, M, N, thin])
    H = np.zeros((M, N), np.uint8)
    for j in range(N):
        d = int(rng.integers(0 if j % 50 == 0 else 1, max_deg + 1))
        H[rng.choice(M - thin, size=d, replace=False), j] = 1
    for i in range(M - thin, M):
        H[i, rng.choice(N, size=int(rng.integers(0, 4)), replace=False)] = 1
    keep = np.cumsum(H, 0) <= max_deg
    p = np.ones(N) if equal else np.exp(rng.uniform(np.log(0.1), np.log(8.0), N))
    p *= errors / p.sum()                                 # errors per shot
    return W.problem_from_dense(H * keep, (rng.random((3, N)) < 0.3).astype(np.uint8), p)


@pytest.mark.parametrize("max_deg,M,N,errors,equal,thin",
                         [(3, 150, 500, 1.5, True, 0), (3, 97, 333, 1.5, False, 9), (6, 160, 900, 1.0, False, 5),
                          (6, 400, 2600, 1.5, True, 0), (16, 700, 1500, 0.6, False, 3)])
@pytest.mark.parametrize("alpha,clamp,storage,group_warps", [(0.625, 1e4, 0, 16), (1.0, 9.0, 0, 16), (0.625, 1e4, 1, 16),
                                                             (0.625, 9.0, 2, 16), (0.625, 1e4, 0, 1)])
def test_second_iteration_screen(max_deg, M, N, errors, equal, thin, alpha, clamp, storage, group_warps):
    prob = _problem(max_deg, M, N, errors, equal, thin)
    shots = W.sample_shots(prob, 12_000, f"screen2_{M}")
    rng = np.random.default_rng(3)
    dense = (rng.random((200, prob.N)) < np.linspace(2.0, 60.0, 200)[:, None] / prob.N).astype(np.uint8)
    synd = np.concatenate([shots.syndromes, W.pack_bits(W.syndrome_of(prob, dense).astype(np.uint8))])
    kw = dict(max_rounds=2, beam_width=3, initial_iters=8, iters_per_round=4)
    dec = D.BeamSearchDecoder(prob, D.make_params(ms_scale=alpha, llr_clamp=clamp, msg_precision=storage,
                                                  tie_guard_rel=-1.0, group_warps=group_warps, **kw))
    dec.decode(torch.zeros((64, synd.shape[1]), dtype=torch.int32, device="cuda"))
    assert dec.profile_read()["kernel_launches"] == 5     # set-up, the two screens, seed, beam gate
    out = dec.decode(D.to_torch_words(synd))
    torch.cuda.synchronize()
    assert dec.sync_error() == 0
    ref = oracle.Graph(prob, "f32").decode_batch(
        synd, oracle.Params(ms_scale=alpha, llr_clamp=clamp, msg_storage=storage, **kw), nthreads=8)
    # more shots than two per candidate group of the seed kernel pass the first
    # screen, so the second runs, except with a warp per candidate, where they go on
    assert (ref["iters"] == 2).sum() > 40
    assert (ref["iters"] != 1).sum() > 2 * 2 * torch.cuda.get_device_properties(0).multi_processor_count
    for name, got in (("corrections", out.corrections), ("status", out.status), ("iters", out.iters)):
        assert np.array_equal(D.from_torch_words(got), ref[name]), name
    dec.close()

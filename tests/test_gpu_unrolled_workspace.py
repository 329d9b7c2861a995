"""The unrolled decoder's path follows from the code, the batch and T alone: loss and
gradient are the same bits and the workspace the same size for every checkpoint
interval, at batches of a whole number of 512 shots and between; and a T whose tiles
would take far more memory than checkpoints keeps them."""
import pytest

torch = pytest.importorskip("torch")

from paper_2512_07057_gb300 import binding as B  # noqa: E402
from paper_2512_07057_gb300 import unrolled as U  # noqa: E402
from paper_2512_07057_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shots,T", [(511, 20), (512, 20), (1024, 12), (2048, 20), (3584, 30)])
def test_no_result_depends_on_the_checkpoint_interval(shots, T):
    prob = W.bb_phenomenological(12, 6, 12, 0.002, 0.002)
    synd, errs, _ = U.batch_tensors(prob, shots, f"interval_{shots}")
    g = torch.Generator(device="cuda").manual_seed(3)
    w = 0.625 * (1 + 0.05 * torch.randn((T, prob.n_edges), generator=g, device="cuda"))
    runs = []
    for k in (1, 4, 5, T):
        tr = U.UnrolledTrainer(prob, shots, T, k)
        runs.append((tr.work.numel(), tr.forward(w, synd, errs).clone(), tr.backward(w, torch.ones(1, device="cuda"))))
        tr.close()
        del tr
    for size, loss, grad in runs[1:]:
        assert size == runs[0][0]
        assert torch.equal(loss, runs[0][1]) and torch.equal(grad, runs[0][2])


def test_many_iterations_keep_checkpoints():
    """4096 shots, T = 4000: 3.2 x 10^11 bytes on tiles, a tenth with 63 checkpoints."""
    prob = W.bb_phenomenological(12, 6, 12, 0.002, 0.002)
    tr = U.UnrolledTrainer(prob, 8, 1, 1)
    assert B.bsd_unrolled_workspace(tr.dec.h, 4096, 4000, 63) < 30 * 10 ** 9
    tr.close()

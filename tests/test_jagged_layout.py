"""The jagged engine's shared-memory placement (host logic, no GPU), the one
bsd_create builds: rows by falling degree with their k-th words side by side, every
edge in one word of its row and one slot of its column, groups of one column degree in
their first slots, and few bank conflicts on the detector error models."""
import numpy as np
import pytest

from paper_2512_07057_gb300 import binding as B
from paper_2512_07057_gb300 import workloads as W


def _check(prob):
    M, N, rp, ci = prob.M, prob.N, np.asarray(prob.H_row_ptr), np.asarray(prob.H_col_idx)
    E = int(rp[-1])
    lay = B.bsd_jagged_layout(M, N, rp, ci)
    row, word, col, slot = lay["rank_row"], lay["edge_word"], lay["column"], lay["slot_edge"]
    deg = np.diff(rp)[row]
    assert sorted(row.tolist()) == list(range(M)) and (np.diff(deg) <= 0).all()
    plane = np.concatenate([[0], np.cumsum([(deg > k).sum() for k in range(deg.max())])])
    for q, i in enumerate(row):
        assert sorted(word[rp[i]:rp[i + 1]].tolist()) == [plane[k] + q for k in range(deg[q])]
    assert sorted(word.tolist()) == list(range(E)) and sorted(col.tolist()) == list(range(N))
    k, p = np.nonzero(slot >= 0)
    assert sorted(slot[k, p].tolist()) == list(range(E)) and (ci[slot[k, p]] == col[p]).all()
    cdeg = np.bincount(ci, minlength=N)[col]
    wavefronts = ideal = 0
    for g in range(0, N, 32):
        most, sl = cdeg[g:g + 32].max(), slot[:, g:g + 32]
        assert (sl[most:] < 0).all() and (cdeg[g:g + 32].min() < most or (sl[:most] >= 0).all())
        for used in sl[:most]:
            if (used >= 0).any():
                wavefronts += np.bincount(word[used[used >= 0]] % 32).max()
                ideal += 1
    return wavefronts / max(ideal, 1)


@pytest.mark.parametrize("seed", range(4))
def test_placement_of_random_codes(seed):
    """Columns of degree 0 to 3 or 6, rows of any degree up to above 16."""
    rng = np.random.default_rng(300 + seed)
    M, N = 14 + 20 * seed, 150 + 40 * seed
    H = np.zeros((M, N), np.uint8)
    for j in range(N):
        d = int(rng.integers(0, 7 if seed % 2 else 4))
        H[rng.choice(M, size=d, replace=False), j] = 1
    _check(W.problem_from_dense(H, np.zeros((1, N), np.uint8), np.full(N, 0.05)))


@pytest.mark.parametrize("name,build,most",
                         [("phenomenological", lambda: W.bb_phenomenological(12, 6, 12, 3e-3, 3e-3), 1.85),
                          ("synthetic", W.synthetic_dem, 1.4), ("xyz", lambda: W.bb_xyz_code_capacity(12, 6, 0.05), 1.98)])
def test_placement_of_the_detector_error_models(name, build, most):
    """Wavefronts per access of the error pass: 1.76, 1.33 and 1.93; 1.94, 2.72 and
    2.00 with rows and columns as they come."""
    assert _check(build()) <= most


def test_columns_of_higher_degree_are_unsupported():
    H = np.zeros((9, 40), np.uint8)
    H[:8, 3] = 1
    H[8] = 1
    prob = W.problem_from_dense(H, np.zeros((1, 40), np.uint8), np.full(40, 0.05))
    with pytest.raises(B.BsdError) as ei:
        B.bsd_jagged_layout(prob.M, prob.N, prob.H_row_ptr, prob.H_col_idx)
    assert ei.value.code == B.BSD_ERR_UNSUPPORTED

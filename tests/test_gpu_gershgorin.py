"""The Gershgorin bound to the last bit: every row's sum runs in ascending column order, however its blocks
are staged (at most 2,048 elements and 256 blocks at a time)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2003_03868_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("bs,density", [([1], 1.0), ([32], 1.0), ([32] * 3, 1.0), ([1] * 255, 1.0), ([1] * 256, 1.0),
                                        ([1] * 257, 1.0), ([1] * 600, 0.9), ([16] * 8, 1.0), ([16] * 9, 1.0),
                                        ([13, 5, 5] * 30, 0.5), (list(range(1, 33)) * 3, 0.7), ([7, 32, 1] * 20, 0.0)])
@pytest.mark.parametrize("mu", [0.0, -0.37])
def test_gershgorin_sums_in_column_order(gb, bs, density, mu):
    m = synth.random_block_matrix(list(bs), density, 40 + len(bs), diag=density > 0.6)
    H = gb.Matrix.of(m)
    off = np.concatenate([[0], np.cumsum(bs)])
    best, at = 0.0, 0
    data, rp, col = np.asarray(m.data), np.asarray(m.row_ptr), np.asarray(m.col)
    for i in range(len(bs)):
        row, has_diag = [np.zeros((bs[i], 1))], False
        for j in col[rp[i]:rp[i + 1]]:
            n = bs[i] * bs[j]
            v = data[at:at + n].reshape(bs[i], bs[j]).copy()
            at += n
            if i == j:
                v[np.arange(bs[i]), np.arange(bs[i])] -= mu
                has_diag = True
            row.append(np.abs(v))
        s = np.add.accumulate(np.hstack(row), axis=1)[:, -1]      # one addition after the other
        if not has_diag:
            s = s + abs(mu)
        best = max(best, s.max())
    assert off[-1] == sum(bs)
    assert gb.gershgorin(H, mu) == best

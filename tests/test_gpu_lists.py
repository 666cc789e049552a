"""Block lists at the edges of the kernels that make them: prefix sums over one tile, a few tiles in one
CTA and many tiles in a chain (seen through the filter's compaction), and the lists of blocks by shape."""
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


# tiles hold 4,096 entries; up to 16,384 one CTA takes them; 400,000: more than two warps of tiles behind one
@pytest.mark.parametrize("nnzb", [1, 2, 4095, 4096, 4097, 16383, 16384, 16385, 20481, 400000])
@pytest.mark.parametrize("kept", ["some", "all", "diagonal"])
def test_filter_keeps_the_right_blocks(gb, nnzb, kept):
    rng = np.random.default_rng(nnzb)
    nblk = max(1, min(nnzb, 1000))
    bs = np.where(np.arange(nblk) % 3 == 0, 2, 1).astype(np.int32)
    off = rng.choice(nblk * nblk, size=nnzb - nblk, replace=False) if nnzb > nblk else np.zeros(0, np.int64)
    mask = np.zeros((nblk, nblk), bool)
    mask.ravel()[off] = True
    np.fill_diagonal(mask, True)
    extra = nnzb - int(mask.sum())                     # drawn diagonal places are filled up elsewhere
    free = np.flatnonzero(~mask.ravel())
    mask.ravel()[free[:extra]] = True
    rows, cols = np.nonzero(mask)
    assert len(rows) == nnzb
    rp = np.concatenate([[0], np.cumsum(mask.sum(1))]).astype(np.int64)
    area = (bs[rows] * bs[cols]).astype(np.int64)
    first = np.concatenate([[0], np.cumsum(area)])
    value = rng.uniform(0.5, 2.0, nnzb)                # every element of a block: its norm is value sqrt(area)
    data = np.repeat(value, area)
    m = gb.Matrix.of(synth.BlockMatrix(bs, rp, cols.astype(np.int32), data))
    eps = {"some": 1.6, "all": 0.0, "diagonal": 100.0}[kept]
    norm = value * np.sqrt(area)
    keep = (norm >= eps) | (rows == cols)
    assert np.all(np.abs(norm[~(rows == cols)] - eps) > 1e-9)
    m.filter(eps)
    rp2, col2, data2 = m.export()
    assert np.array_equal(rp2, np.concatenate([[0], np.cumsum(np.bincount(rows[keep], minlength=nblk))]))
    assert np.array_equal(col2, cols[keep])
    assert np.array_equal(data2, np.concatenate([data[first[b]:first[b + 1]] for b in np.flatnonzero(keep)])
                          if nnzb < 50000 else data[np.repeat(keep, area)])


# 2,048 blocks per CTA of the list kernel: just below, above and at twice that, with a few shapes and
# with hundreds; planned products list the tensor-core blocks besides
@pytest.mark.parametrize("nblk", [3, 45, 46, 64, 91])
@pytest.mark.parametrize("sizes", ["few", "many"])
@pytest.mark.parametrize("planned", [False, True])
def test_products_of_every_block_exactly_once(gb, nblk, sizes, planned):
    rng = np.random.default_rng(nblk)
    bs = np.asarray([13, 5, 5] * 31 if sizes == "few" else rng.permutation(np.arange(93) % 32 + 1), np.int32)[:nblk]
    a, b = (synth.random_block_matrix(list(bs), 1.0, nblk + t) for t in (1, 2))
    A, B = gb.Matrix.of(a), gb.Matrix.of(b)
    off = np.concatenate([[0], np.cumsum(bs)])

    def dense(M):
        rp, col, data = M.export()
        D, at = np.full((off[-1], off[-1]), np.nan), 0
        for i in range(nblk):
            for j in col[rp[i]:rp[i + 1]]:
                n = bs[i] * bs[j]
                D[off[i]:off[i + 1], off[j]:off[j + 1]] = data[at:at + n].reshape(bs[i], bs[j])
                at += n
        return D
    Ad, Bd = dense(A), dense(B)
    C = gb.Matrix(A.blk_size, A.stream)
    if planned:
        p = gb.Plan(1.0, A, B, C, 0.0)
        p.execute()
    else:
        gb.multiply(1.0, A, B, 0.0, C, 0.0)
    got, ref = dense(C), Ad @ Bd
    if planned:
        p.close()
    assert not np.isnan(got).any()
    # block by block within twice what any sum of n rounded terms keeps (both sides are rounded)
    norms = lambda D: np.sqrt(np.add.reduceat(np.add.reduceat(D * D, off[:-1], 0), off[:-1], 1))  # noqa: E731
    bound = 2 * (off[-1] + 4) * 2.0 ** -53 * (norms(Ad) @ norms(Bd))
    assert np.all(norms(got - ref) <= bound)

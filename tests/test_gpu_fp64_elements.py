"""FP64 products element by element: rows, columns and inner indices of very different size inside the blocks,
and zeros that meet large elements.

Every element is compared with a doubled-precision sum of the same terms within the bound that any summation
of n rounded FP64 terms keeps, |error_ij| <= (n + 4) 2^-53 (|A| |B|)_ij, n the matrix dimension."""
import numpy as np
import pytest

import synth
from oracle import bsr

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def gb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2003_03868_gb300 as m
    m.lib()
    return m


def _product(a, b):
    """a @ b in about twice FP64's precision (Dekker's products, Knuth's sums): (high, low)."""
    def split(x):
        c = 134217729.0 * x
        h = c - (c - x)
        return h, x - h
    hi, lo = np.zeros((a.shape[0], b.shape[1])), np.zeros((a.shape[0], b.shape[1]))
    (ah, al), (bh, bl) = split(a), split(b)
    for k in range(a.shape[1]):
        p = np.multiply.outer(a[:, k], b[k])
        e = ((np.multiply.outer(ah[:, k], bh[k]) - p) + np.multiply.outer(ah[:, k], bl[k])
             + np.multiply.outer(al[:, k], bh[k])) + np.multiply.outer(al[:, k], bl[k])
        s = hi + p
        z = s - hi
        lo += ((hi - (s - z)) + (p - z)) + e
        hi = s
    return hi, lo


def _blocks(bs, D):
    """D as a matrix of all blocks."""
    nb, off = len(bs), np.concatenate([[0], np.cumsum(bs)])
    data = np.concatenate([D[off[i]:off[i + 1], off[j]:off[j + 1]].ravel() for i in range(nb) for j in range(nb)])
    return synth.BlockMatrix(np.asarray(bs, np.int32), np.arange(nb + 1, dtype=np.int64) * nb,
                             np.tile(np.arange(nb, dtype=np.int32), nb), data)


def _error(gb, bs, a, b, planned=False):
    """(error of the library's a b, |a| |b|, tiles formed)"""
    A, B = gb.Matrix.of(_blocks(bs, a)), gb.Matrix.of(_blocks(bs, b))
    C = gb.Matrix(A.blk_size, A.stream)
    if planned:
        # made on unscaled values: the tests are repeated for those of the execution
        r = np.random.default_rng(1)
        A.put_values(r.uniform(-1.0, 1.0, a.size))
        B.put_values(r.uniform(-1.0, 1.0, b.size))
        plan = gb.Plan(1.0, A, B, C, 0.0)
        tiles = plan.stats.n_tiles
        A.put_values(_blocks(bs, a).data)
        B.put_values(_blocks(bs, b).data)
        plan.execute()
    else:
        tiles = gb.multiply(1.0, A, B, 0.0, C, 0.0).n_tiles
    got = bsr.to_dense(bsr.Mat(np.asarray(bs), *C.export()))
    if planned:
        plan.close()
    hi, lo = _product(a, b)
    return (got - hi) - lo, np.abs(a) @ np.abs(b), tiles


SIZES = [[28] * 12, [13, 5, 5] * 14]               # a little over the flops from which the tensor cores are used


@pytest.mark.parametrize("planned", [False, True])
@pytest.mark.parametrize("bits", [0, 9, 20, 66])
@pytest.mark.parametrize("kind", ["rows", "inner", "zeros"])
def test_elements_of_graded_blocks(gb, kind, bits, planned):
    for i, bs in enumerate(SIZES):
        n = sum(bs)
        r = np.random.default_rng(3000 + 10 * i + bits)
        a, b = r.uniform(-1.0, 1.0, (n, n)), r.uniform(-1.0, 1.0, (n, n))
        g, h = (2.0 ** -r.integers(0, bits + 1, n).astype(float) for _ in range(2))
        if kind == "rows":                     # weak rows of A and columns of B beside strong ones
            a, b = a * g[:, None], b * h[None, :]
        elif kind == "inner":                  # strong columns of A meet weak rows of B and the other way round
            a, b = a * g[None, :], b / g[:, None] * 2.0 ** -bits
        else:                                  # a weak inner index, and a strong one whose partner is zero
            s = r.random(n) < 0.5
            a, b = a * np.where(s, 2.0 ** -bits, 1.0)[None, :], b * np.where(s, 1.0, 0.0)[:, None]
        err, mag, tiles = _error(gb, bs, a, b, planned)
        assert tiles > 0 if bits == 0 and kind != "zeros" else True
        assert np.all(np.abs(err) <= (n + 4) * U * mag), (bs[:3], float(np.max(np.abs(err) / (U * np.maximum(mag, 1e-300)))))


def test_digits_left_out(gb):
    # four groups of 112 rows (A's couplings are twice as strong inside them).  In the first one the products
    # cancel to 2^-20, in the others B is 2^-19 smaller, where the last two of eight digits may go.  What is
    # left out of 36 digit products sums up to 2^-59.9 (root mean square: 112 terms of six digit pairs of
    # 2^12.4, 2^-78 each, at the scale 2 of the group's own rows; the others' part is below 2^-62);
    # an FP64 chain, seven digits for eight, or one digit less in the far groups leave 2^-55 and more
    n, g = 448, 112
    r = np.random.default_rng(3100)
    a, b = r.uniform(-1.0, 1.0, (n, n)), r.uniform(-1.0, 1.0, (n, n)) * 2.0 ** -19
    a[:, g // 2:g] = a[:, :g // 2]
    for x in range(0, n, g):
        a[x:x + g, x:x + g] *= 2.0
    b[:g // 2] = r.uniform(-1.0, 1.0, (g // 2, n))
    b[g // 2:g] = -(b[:g // 2] + 2.0 ** -20 * r.uniform(-1.0, 1.0, (g // 2, n)))
    for planned in (False, True):
        err, _, tiles = _error(gb, [28] * 16, a, b, planned)
        assert planned or tiles == 16             # (a plan's groups come from the values it was made with)
        assert np.sqrt(np.mean(err ** 2)) <= 2.0 ** -57

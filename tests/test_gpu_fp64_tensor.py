"""FP64 products on the tensor cores (eight-digit splitting): at the edges of the tiles and slices,
with badly scaled and non-finite operands, and in planned products whose values change.

Every block is compared with a doubled-precision sum of the same terms within the bound that any summation of
n rounded FP64 terms keeps, ||error|| <= n 2^-53 (sum_K ||A_IK|| ||B_KJ|| + |beta| ||C_IJ||), n the
matrix dimension plus 4 (two scalings, a C input, the last rounding)."""
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


def _norms(d, start):
    """Frobenius norms of the blocks of d, each scaled by its largest element before squaring."""
    n = np.maximum.reduceat(np.maximum.reduceat(np.abs(d), start[:-1], 0), start[:-1], 1)
    q = np.where(n > 0, n, 1.0)
    reps = np.diff(start)
    big = np.repeat(np.repeat(q, reps, 0), reps, 1)
    return np.where(n > 0, q * np.sqrt(np.add.reduceat(np.add.reduceat((d / big) ** 2, start[:-1], 0), start[:-1], 1)),
                    0.0)


def _check(C, Ao, Bo, alpha=1.0, beta=0.0, Co=None):
    bs = np.asarray(Ao.bs)
    start = np.concatenate([[0], np.cumsum(bs)])
    a, b = bsr.to_dense(Ao), bsr.to_dense(Bo)
    hi, lo = _product(a, b)
    rp, col, data = C.export()
    got = bsr.to_dense(bsr.Mat(bs, rp, col, data))
    mag = abs(alpha) * (_norms(a, start) @ _norms(b, start))
    # alpha and beta are short dyadic fractions: alpha * hi and beta * c round to FP64 at most
    diff = (got - alpha * hi) - alpha * lo
    if Co is not None:
        c = bsr.to_dense(Co)
        diff = ((got - beta * c) - alpha * hi) - alpha * lo
        mag = mag + abs(beta) * _norms(c, start)
    err = _norms(diff, start)
    assert np.all(err <= (start[-1] + 4) * U * mag + 1e-300)


# widths of the block groups (at most 112 rows, 16 blocks) and of the 32-column slices: full tiles
# (16 x 7, 112 = 4 x 28), one row short or over, one block per tile, slices cut inside a block
SIZES = [[7] * 64, [28] * 16, [31] * 15, [32] * 14, [23, 7, 7] * 12, [13, 5, 5] * 20, [1] * 90 + [32] * 10,
         list(range(1, 33)), [17, 16, 15, 9, 8, 24] * 5]


@pytest.mark.parametrize("si", range(len(SIZES)))
@pytest.mark.parametrize("density", [0.45, 1.0])
def test_products_at_tile_edges(gb, si, density):
    bs = SIZES[si]
    a = synth.random_block_matrix(bs, density, 1200 + si)
    b = synth.random_block_matrix(bs, density, 1300 + si)
    c = synth.random_block_matrix(bs, 0.3, 1400 + si)
    A, B, C = (gb.Matrix.of(x) for x in (a, b, c))
    st = gb.multiply(-0.75, A, B, 1.25, C, 0.0)
    if st.flops >= 64e6 and density == 1.0 and min(bs) > 1:
        assert st.n_tiles > 0
    _check(C, bsr.Mat.of(a), bsr.Mat.of(b), -0.75, 1.25, bsr.Mat.of(c))


def _scaled(m, f, seed):
    """m with every block multiplied by 10 to a uniform power in [-f, f]."""
    out = m.copy()
    rng = np.random.default_rng(seed)
    off, rows = out.blk_off(), out.rows()
    for k in range(out.nnzb):
        n = int(out.blk_size[rows[k]]) * int(out.blk_size[out.col[k]])
        out.data[off[k]:off[k] + n] *= 10.0 ** rng.uniform(-f, f)
    return out


@pytest.mark.parametrize("f", [2.0, 8.0, 60.0, 150.0])
def test_badly_scaled_blocks_keep_the_bound(gb, f):
    bs = [13, 5, 5] * 20
    a = _scaled(synth.random_block_matrix(bs, 0.9, 1500), f, 1)
    b = _scaled(synth.random_block_matrix(bs, 0.9, 1501), f, 2)
    A, B = gb.Matrix.of(a), gb.Matrix.of(b)
    C = gb.Matrix(A.blk_size, A.stream)
    gb.multiply(1.0, A, B, 0.0, C, 0.0)
    _check(C, bsr.Mat.of(a), bsr.Mat.of(b))


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e200, 1e-200, 5e-324])
def test_values_outside_the_scales(gb, bad):
    bs = [23, 7, 7] * 10
    a = synth.random_block_matrix(bs, 0.8, 1600)
    if abs(bad) < 1:
        a.data[a.blk_off()[0]:a.blk_off()[0] + 23 * 23] = bad        # a whole block
    else:
        a.data[1234] = bad
    b = synth.random_block_matrix(bs, 0.8, 1601)
    A, B = gb.Matrix.of(a), gb.Matrix.of(b)
    C = gb.Matrix(A.blk_size, A.stream)
    gb.multiply(1.0, A, B, 0.0, C, 0.0)
    ref = bsr.multiply(1.0, bsr.Mat.of(a), bsr.Mat.of(b))
    _, col, data = C.export()
    assert np.array_equal(col, ref.col)
    assert np.array_equal(np.isnan(data), np.isnan(ref.data))
    assert np.array_equal(np.isinf(data), np.isinf(ref.data))
    if np.isfinite(bad):
        _check(C, bsr.Mat.of(a), bsr.Mat.of(b))


def test_plan_with_values_that_need_the_fp64_units(gb):
    bs = [13, 5, 5] * 20
    a = synth.random_block_matrix(bs, 0.9, 1700)
    A, B = gb.Matrix.of(a), gb.Matrix.of(a)
    C = gb.Matrix(A.blk_size, A.stream)
    plan = gb.Plan(1.0, A, B, C, 0.0)
    assert plan.stats.n_tiles > 0
    for values in (a.data * 3.0, _scaled(a, 8.0, 3).data, _scaled(a, 140.0, 4).data, a.data):
        A.put_values(values)
        plan.execute()
        m = a.copy()
        m.data = values
        _check(C, bsr.Mat.of(m), bsr.Mat.of(a))
    v = a.data.copy()
    v[77] = np.nan
    A.put_values(v)
    plan.execute()
    m = a.copy()
    m.data = v
    got = bsr.to_dense(bsr.Mat(C.blk_size, *C.export()))
    # its row of the product, in the columns where B has a block
    hit = np.isnan(bsr.to_dense(bsr.Mat.of(m))).astype(float)
    there = bsr.to_dense(bsr.Mat(a.blk_size, a.row_ptr, a.col, np.ones_like(a.data)))
    assert np.array_equal(np.isnan(got), hit @ there > 0)
    plan.close()


def test_symmetric_square_equals_its_transpose_and_the_bound(gb):
    # A A of an exactly symmetric A: the mirrored products of the sign iteration, one step
    h = synth.build_hamiltonian(synth.small(40, seed=1800))
    X = gb.sign_iterate(gb.Matrix.of(h.H), 0.0, 0.0, 1e-13, max_iter=1, return_x=True).P
    D = bsr.to_dense(bsr.Mat(X.blk_size, *X.export()))
    assert np.array_equal(D, D.T)
    C = gb.Matrix(X.blk_size, X.stream)
    gb.multiply(1.0, X, X, 0.0, C, 0.0)
    _check(C, bsr.Mat(X.blk_size, *X.export()), bsr.Mat(X.blk_size, *X.export()))


@pytest.mark.parametrize("planned", [False, True])
def test_both_pipes_side_by_side_from_several_threads_and_streams(gb, planned):
    # one product's blocks run on two streams; products of several threads, each on a stream of its own
    # and one on the default stream, give the same bits as the same product by itself
    import threading

    import torch
    hs = [synth.build_hamiltonian(synth.small(40 + 8 * i, basis=b, seed=50 + i)).H
          for i, b in enumerate([(13, 5), (23, 7), (13, 7), (23, 5)])]
    alone = []
    for h in hs:
        A = gb.Matrix.of(h)
        C = gb.Matrix(A.blk_size, A.stream)
        if planned:
            p = gb.Plan(1.0, A, A, C, 1e-7)
            p.execute()
            alone.append(C.export())
            p.close()
        else:
            assert gb.multiply(1.0, A, A, 0.0, C, 1e-7).n_tiles > 0
            alone.append(C.export())
    streams = [torch.cuda.Stream() for _ in hs[1:]]
    bad = []

    def work(i):
        try:
            st = None if i == 0 else streams[i - 1].cuda_stream
            A = gb.Matrix.of(hs[i], st)
            for _ in range(6):
                C = gb.Matrix(A.blk_size, st)
                if planned:
                    p = gb.Plan(1.0, A, A, C, 1e-7)
                    for _ in range(3):
                        p.execute()
                else:
                    gb.multiply(1.0, A, A, 0.0, C, 1e-7)
                if not all(np.array_equal(x, y) for x, y in zip(C.export(), alone[i])):
                    bad.append(i)
                if planned:
                    p.close()
        except Exception as e:                       # noqa: BLE001 -- reported by the main thread
            bad.append((i, repr(e)))
    ts = [threading.Thread(target=work, args=(i,)) for i in range(len(hs))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad


@pytest.mark.parametrize("power", [-110, -75, 60, 80])
def test_badly_scaled_blocks_of_tiny_and_huge_operands(gb, power):
    # the norm products lie near the ends of FP32's range and past them, where the choice of the blocks
    # for the tensor cores is made
    bs = [13, 5, 5] * 20
    a = _scaled(synth.random_block_matrix(bs, 0.9, 1520), 8.0, 5)
    b = _scaled(synth.random_block_matrix(bs, 0.9, 1521), 8.0, 6)
    a.data *= 2.0 ** power
    b.data *= 2.0 ** power
    A, B = gb.Matrix.of(a), gb.Matrix.of(b)
    C = gb.Matrix(A.blk_size, A.stream)
    gb.multiply(1.0, A, B, 0.0, C, 0.0)
    _check(C, bsr.Mat.of(a), bsr.Mat.of(b))


def test_rows_of_subnormals(gb):
    # a block row that holds nothing but subnormals, times large elements: no element of the product is small
    bs = [23, 7, 7] * 10
    a = synth.random_block_matrix(bs, 0.9, 1620)
    b = synth.random_block_matrix(bs, 0.9, 1621)
    n = a.blk_off()[a.row_ptr[1]]
    a.data[:n] = np.ldexp(np.rint(a.data[:n] * 2.0 ** 20), -1070)
    b.data *= 2.0 ** 398
    A, B = gb.Matrix.of(a), gb.Matrix.of(b)
    C = gb.Matrix(A.blk_size, A.stream)
    gb.multiply(1.0, A, B, 0.0, C, 0.0)
    _check(C, bsr.Mat.of(a), bsr.Mat.of(b))


@pytest.mark.parametrize("kind", ["band", "random"])
def test_products_that_the_tensor_cores_would_slow_down(gb, kind):
    # many small blocks with little work each (grouping them would take longer than the product), and a pattern
    # without neighbourhoods (a block or two in every tile): both stay off the tensor cores
    nb, b = (8000, 5) if kind == "band" else (1500, 13)
    r = np.random.default_rng(1900)
    i = np.arange(nb)
    if kind == "band":
        near = i[:, None] + np.arange(-4, 5)[None, :]
        pairs = np.stack([np.repeat(i, 9), near.ravel()], 1)
        pairs = pairs[(pairs[:, 1] >= 0) & (pairs[:, 1] < nb)]
    else:
        pairs = np.concatenate([np.stack([i, i], 1), r.integers(0, nb, (20 * nb, 2))])
    key = np.unique(pairs[:, 0].astype(np.int64) * nb + pairs[:, 1])
    rp = np.concatenate([[0], np.cumsum(np.bincount(key // nb, minlength=nb))])
    a, c = (synth.BlockMatrix(np.full(nb, b, np.int32), rp, (key % nb).astype(np.int32),
                              r.uniform(-1.0, 1.0, len(key) * b * b)) for _ in range(2))
    A, B = gb.Matrix.of(a), gb.Matrix.of(c)
    C = gb.Matrix(A.blk_size, A.stream)
    st = gb.multiply(1.0, A, B, 0.0, C, 0.0)
    assert st.flops >= 64e6 and st.n_tiles == 0
    ref = bsr.multiply(1.0, bsr.Mat.of(a), bsr.Mat.of(c))
    rp2, col, data = C.export()
    assert np.array_equal(rp2, ref.rp) and np.array_equal(col, ref.col)
    # terms of a block: at most the row's blocks times b; both sums are rounded
    n = int(np.diff(rp).max()) * b
    assert np.abs(data - ref.data).max() <= 2 * (n + 2) * U * n

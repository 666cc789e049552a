"""FP64 products when the device's memory does not hold the tensor cores' digit tiles: a product that fits without
them still runs, with every block on the FP64 units."""
import numpy as np
import pytest

import synth
from oracle import bsr

pytestmark = pytest.mark.gpu


@pytest.fixture
def gb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2003_03868_gb300 as m
    m.lib()
    yield m
    m.lib().dbcsr_pool_limit(0)


def _peak(gb, work):
    gb.pool_usage(True)
    now, _ = gb.pool_usage()
    out = work()
    return out, gb.pool_usage()[1] - now


@pytest.mark.parametrize("planned", [False, True])
def test_products_without_room_for_the_digit_tiles(gb, planned):
    import ctypes as C
    bs = [23, 7, 7] * 16
    a, b = (synth.random_block_matrix(bs, 1.0, 2400 + i) for i in range(2))
    A, B = gb.Matrix.of(a), gb.Matrix.of(b)

    def product():
        M = gb.Matrix(A.blk_size, A.stream)
        if not planned:
            return M, gb.multiply(1.0, A, B, 0.0, M, 0.0).n_tiles
        p = gb.Plan(1.0, A, B, M, 0.0)
        p.execute()
        n = p.stats.n_tiles
        M.info()
        out = gb.Matrix.from_blocks(A.blk_size, *M.export())
        p.close()
        return out, n
    x, y = bsr.to_dense(bsr.Mat.of(a)), bsr.to_dense(bsr.Mat.of(b))
    bound = 2 * (x.shape[0] + 4) * 2.0 ** -53 * (np.abs(x) @ np.abs(y))
    ok = lambda M: np.all(np.abs(bsr.to_dense(bsr.Mat(A.blk_size, *M.export())) - x @ y) <= bound)  # noqa: E731
    (M, tiles), peak = _peak(gb, product)
    assert tiles > 0 and ok(M)
    del M
    lib = gb.lib()
    used = gb.pool_usage()[0]
    # the tiles' share is most of the peak: with less and less room the product first loses them, then fails
    seen = set()
    for room in (1.0, 0.9, 0.7, 0.5, 0.3, 0.2, 0.1, 0.01):
        assert lib.dbcsr_pool_limit(used + int(room * peak) + 4096) == gb._ffi.DBCSR_OK
        try:
            M, tiles = product()
        except gb.DbcsrError as e:
            assert e.status == gb._ffi.DBCSR_ENOMEM
            seen.add("none")
        else:
            assert "none" not in seen
            seen.add("tiles" if tiles else "no tiles")
            lib.dbcsr_pool_limit(0)
            assert ok(M)
            del M
        lib.dbcsr_pool_limit(0)
        assert gb.pool_usage()[0] == used
    assert seen == {"tiles", "no tiles", "none"}
    M, tiles = product()
    assert tiles > 0 and ok(M)

"""Values and patterns to and from host buffers of every kind: pinned (by the library's kernel), pinned off
16-byte boundaries, registered, pageable; nothing outside the arrays is written."""
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


def _buffer(kind, count, dtype, pad):
    """(whole array, view of count elements inside it, keep-alive)."""
    import torch
    t = torch.full((count + 2 * pad,), -7, dtype=dtype)
    if kind.startswith("pinned"):
        t = t.pin_memory()
    shift = 1 if kind == "pinned odd" else 0
    keep = None
    if kind == "registered":
        rt = torch.cuda.cudart()
        if int(rt.cudaHostRegister(t.data_ptr(), t.numel() * t.element_size(), 0)) != 0:
            pytest.skip("no host registration")
        keep = lambda: rt.cudaHostUnregister(t.data_ptr())  # noqa: E731
    return t, t[pad + shift:pad + shift + count], keep


# one block; a little below, at and above a CTA's 64 KB piece (8,192 values); many pieces
@pytest.mark.parametrize("nblk", [1, 90, 91, 92, 400])
@pytest.mark.parametrize("kind", ["pinned", "pinned odd", "registered", "pageable"])
def test_export_and_put_values(gb, kind, nblk):
    import torch
    m = synth.random_block_matrix([1] * nblk, 1.0, nblk)
    M = gb.Matrix.of(m)
    rp, col, data = M.export()
    assert np.array_equal(data, np.asarray(m.data)) and len(data) == nblk * nblk
    bufs = [_buffer(kind, n, t, 16) for n, t in ((nblk + 1, torch.int64), (len(col), torch.int32),
                                                (len(data), torch.float64))]
    try:
        M.export_to(bufs[0][1].data_ptr(), bufs[1][1].data_ptr(), len(col), bufs[2][1].data_ptr(), len(data))
        for (whole, view, _), ref in zip(bufs, (rp, col, data)):
            assert np.array_equal(view.numpy(), ref)
            out = whole.clone()
            i = (view.data_ptr() - whole.data_ptr()) // whole.element_size()
            out[i:i + len(ref)] = -7
            assert bool((out == -7).all())
        values = bufs[2][1]
        values.mul_(-3.0).add_(1.0)
        M.put_values(values.numpy())
        assert np.array_equal(M.export()[2], values.numpy())
        new = gb.Matrix.from_blocks(M.blk_size, rp, col, values.numpy())     # staged from that buffer
        assert np.array_equal(new.export()[2], values.numpy())
    finally:
        for _, _, keep in bufs:
            if keep:
                keep()


# heads and tails around the 128-byte lines of the host's side: every offset of eight bytes in a line, arrays of
# less than a line up to several
@pytest.mark.parametrize("shift", [0, 1, 2, 7, 9, 15])
def test_any_offset_in_a_line(gb, shift):
    import torch
    for nblk in (1, 2, 3, 4, 5, 9, 12, 130):
        m = synth.random_block_matrix([1] * nblk, 1.0, 100 + nblk)
        M = gb.Matrix.of(m)
        rp, col, data = M.export()
        whole = [torch.full((n + 40,), -7, dtype=t).pin_memory()
                 for n, t in ((nblk + 1, torch.int64), (len(col), torch.int32), (len(data), torch.float64))]
        view = [w[8 + shift:8 + shift + n] for w, n in zip(whole, (nblk + 1, len(col), len(data)))]
        M.export_to(view[0].data_ptr(), view[1].data_ptr(), len(col), view[2].data_ptr(), len(data))
        for w, v, ref in zip(whole, view, (rp, col, data)):
            assert np.array_equal(v.numpy(), ref)
            assert bool((w[:8 + shift] == -7).all()) and bool((w[8 + shift + len(ref):] == -7).all())
        view[2].mul_(3.0)
        M.put_values(view[2].numpy())
        assert np.array_equal(M.export()[2], view[2].numpy())

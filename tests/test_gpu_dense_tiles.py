"""Dense FP32-storage products of the submatrix method at the edges of their tiles, and the residual
of its iteration.

The products are compared with FP64 products of the same FP32 inputs within the truncation of the
operands to TF32 (2^-9 relative to |A||B| plain, 2^-18 split) plus FP32 sums over n terms and the
two operations on beta C (2^-22)."""
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


# one element; a 16-column stage and its neighbours; one and two row tiles; B^T tiles of one, two and
# three widths' edges; more tiles than SMs, at widths that the wave count narrows (432: 144 columns)
@pytest.mark.parametrize("n,nb", [(1, 3), (15, 2), (17, 1), (63, 5), (65, 400), (127, 2), (129, 3), (255, 1), (432, 58),
                                  (513, 1)])
@pytest.mark.parametrize("offset", [0, 1])
def test_dense_tiles_offsets_and_in_place(gb, n, nb, offset):
    import torch
    rng = np.random.default_rng(100 * n + nb)

    def dev(x):                       # offset 1: rows start off 16-byte boundaries
        t = torch.empty(x.size + 4, dtype=torch.float32, device="cuda")[offset:offset + x.size]
        t.copy_(torch.from_numpy(x.ravel()))
        return t
    A, B, C = (rng.uniform(-1, 1, (nb, n, n)).astype(np.float32) for _ in range(3))
    A64, B64, C64 = (torch.from_numpy(x).double().cuda() for x in (A, B, C))
    for prec, tol in ((gb.DBCSR_TF32, 2.0 ** -9), (gb.DBCSR_TF32X3, 2.0 ** -18)):
        for beta, into in ((0.0, "c"), (1.5, "c"), (0.0, "a"), (0.75, "b")):
            a, b, c = dev(A), dev(B), dev(C)
            out, C0 = {"a": (a, A64), "b": (b, B64), "c": (c, C64)}[into]
            if beta == 0.0 and into == "c":
                out.fill_(float("nan"))
            gb.dense_multiply(prec, nb, n, -0.5, a.data_ptr(), b.data_ptr(), beta, out.data_ptr())
            got = out.double().view(nb, n, n)
            ref = -0.5 * (A64 @ B64) + (beta * C0 if beta else 0.0)
            mag = 0.5 * (A64.abs() @ B64.abs()) + (beta * C0.abs() if beta else 0.0)
            assert bool(((got - ref).abs() <= (tol + n * 2.0 ** -24 + 2.0 ** -22) * mag + 1e-30).all()), (prec, into)


@pytest.mark.parametrize("scale", [1.0, 1e-12, 1e-25, 0.0])
def test_submatrix_first_residual(gb, scale):
    # full neighbourhoods: every submatrix is the whole matrix; off-diagonal elements down to and past
    # the squares that FP32 holds, and groups of zeros
    bs = [13, 5, 23, 7, 1, 32, 4]
    m = synth.random_block_matrix(bs, 1.0, 5)
    H = gb.Matrix.of(m)
    rp, col, data = H.export()
    n = sum(bs)
    off = np.concatenate([[0], np.cumsum(bs)])
    Hd = np.zeros((n, n))
    at = 0
    for i in range(len(bs)):
        for q in range(rp[i], rp[i + 1]):
            j = col[q]
            blk = data[at:at + bs[i] * bs[j]].reshape(bs[i], bs[j])
            blk *= scale                                        # (a view: the data that are uploaded)
            if i == j:
                blk += np.diag(np.linspace(-1.0, 1.5, bs[i]) + 0.01)
            Hd[off[i]:off[i + 1], off[j]:off[j + 1]] = blk
            at += bs[i] * bs[j]
    H = gb.Matrix.of(synth.BlockMatrix(np.asarray(bs, np.int32), rp, col, data))
    g = gb.submatrix_sign(H, 0.0, 1e-9, max_iter=1, prec=gb.DBCSR_MIXED)
    assert g.report.iterations == 1
    X = Hd / g.report.alpha
    n_pad = (n + 15) // 16 * 16
    ref = np.linalg.norm(X @ X - np.eye(n)) / n_pad
    bound = (2.0 ** -9 + n * 2.0 ** -24 + 2.0 ** -22) * np.linalg.norm(np.abs(X) @ np.abs(X)) / n_pad
    assert abs(g.report.residual - ref) <= bound + 1e-9 * ref

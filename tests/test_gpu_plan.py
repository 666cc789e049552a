"""Planned products on fixed patterns (dbcsr_multiply_plan / dbcsr_multiply_execute, a
CUDA graph of the numeric phase) against the one-off product and the oracle."""
import numpy as np
import pytest

import synth
from oracle import bsr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2003_03868_gb300 as m
    m.lib()
    return m


def _mat(M):
    rp, col, data = M.export()
    return bsr.Mat(M.blk_size, rp, col, data)


@pytest.mark.parametrize("prec", ["fp64", "bf16x3"])
def test_plan_equals_one_off_product(gb, prec):
    p = gb.DBCSR_FP64 if prec == "fp64" else gb.DBCSR_BF16X3
    a = synth.build_decay(synth.DECAY_32)
    eps = synth.DECAY_32.eps_filter
    A = gb.Matrix.of(a)
    C1 = gb.Matrix(A.blk_size, A.stream)
    gb.multiply(1.0, A, A, 0.0, C1, eps, prec=p)
    ref = _mat(C1)
    C2 = gb.Matrix(A.blk_size, A.stream)
    plan = gb.Plan(1.0, A, A, C2, eps, prec=p)
    for _ in range(3):              # the planned pattern holds every formed block, under-eps ones zeroed
        got = _mat(C2)
        kept = {(int(r), int(c)) for r, c in zip(ref.rows, ref.col)}
        for b in range(got.nnzb):
            I, J = int(got.rows[b]), int(got.col[b])
            blk = got.block(I, J)
            if (I, J) in kept:
                assert np.array_equal(blk, ref.block(I, J))
            else:
                assert I != J and not blk.any()
        assert kept <= {(int(r), int(c)) for r, c in zip(got.rows, got.col)}
        plan.execute()
    assert plan.stats.n_formed == got.nnzb
    plan.close()


def test_plan_with_new_values_matches_oracle(gb):
    a = synth.build_decay(synth.DECAY_32)
    eps = synth.DECAY_32.eps_filter
    A = gb.Matrix.of(a)
    B = gb.Matrix.of(a)
    C_ = gb.Matrix(A.blk_size, A.stream)
    plan = gb.Plan(-0.5, A, B, C_, eps)
    rng = np.random.default_rng(7)
    for step in range(3):
        # new values on the same patterns
        av = a.data * (0.8 + 0.4 * rng.random(a.data.shape))
        bv = a.data * (0.8 + 0.4 * rng.random(a.data.shape))
        A.put_values(av)
        B.put_values(bv)
        plan.execute()
        Ao = bsr.Mat(a.blk_size, a.row_ptr, a.col, av)
        Bo = bsr.Mat(a.blk_size, a.row_ptr, a.col, bv)
        got = _mat(C_)
        for b in range(got.nnzb):
            I, J = int(got.rows[b]), int(got.col[b])
            r = bsr.product_block(I, J, -0.5, Ao, Bo)
            nr = np.linalg.norm(r)
            if I != J and nr < eps * (1 - 1e-12):
                assert not got.block(I, J).any()
            elif I == J or nr > eps * (1 + 1e-12):
                assert np.linalg.norm(got.block(I, J) - r) <= 1e-12 * nr
    plan.close()


def test_plan_pins_its_matrices(gb):
    a = synth.random_block_matrix([13, 5, 5] * 4, 0.5, 11)
    A = gb.Matrix.of(a)
    C_ = gb.Matrix(A.blk_size, A.stream)
    plan = gb.Plan(1.0, A, A, C_, 0.0)
    with pytest.raises(gb.DbcsrError) as e:
        gb.multiply(1.0, A, A, 0.0, C_, 0.0)
    assert e.value.status == gb._ffi.DBCSR_ESTATE
    with pytest.raises(gb.DbcsrError):
        C_.filter(1.0)
    with pytest.raises(gb.DbcsrError):
        A.close()
    with pytest.raises(gb.DbcsrError):          # C may not alias an operand
        gb.Plan(1.0, A, A, A, 0.0)
    plan.close()
    gb.multiply(1.0, A, A, 0.0, C_, 0.0)         # free again once the plan is gone
    A.close()


def test_new_values_send_only_the_blocks_that_need_it_to_the_fp64_units(gb):
    # one block row of A graded by 2^-40 inside its blocks: the blocks of C in other groups' rows stay the
    # same bits, the graded row's keep an FP64 product's accuracy in every element
    bs = [28] * 16
    n, nb = sum(bs), len(bs)
    a, b = (synth.random_block_matrix(bs, 1.0, 2200 + i) for i in range(2))
    A, B = gb.Matrix.of(a), gb.Matrix.of(b)
    g_of, _, _ = A.groups()
    C = gb.Matrix(A.blk_size, A.stream)
    plan = gb.Plan(1.0, A, B, C, 0.0)
    assert plan.stats.n_tiles > 0
    dense = lambda d: np.asarray(d).reshape(nb, nb, 28, 28).transpose(0, 2, 1, 3).reshape(n, n)  # noqa: E731
    plan.execute()
    before = dense(C.export()[2])
    v = a.data.copy()
    rows = v[5 * nb * 784:6 * nb * 784].reshape(nb, 28, 28)
    rows *= 2.0 ** -np.linspace(0, 40, 28).round()[None, :, None]
    A.put_values(v)
    plan.execute()
    after = dense(C.export()[2])
    other = np.repeat(g_of != g_of[5], 28)
    assert other.any() and np.array_equal(before[other], after[other])
    x, y = dense(v)[140:168], dense(b.data)
    assert np.all(np.abs(after[140:168] - x @ y) <= 2 * (n + 4) * 2.0 ** -53 * (np.abs(x) @ np.abs(y)))
    plan.close()


def test_execution_whose_tensor_core_waits_run_out(gb):
    # the kernel stops before its first block, as after a wait that ran out: the execution's result is still
    # that of the current values (C held another one), and so is the next one
    a, b = (synth.random_block_matrix([28] * 16, 1.0, 2300 + i) for i in range(2))
    A, B = gb.Matrix.of(a), gb.Matrix.of(b)
    C = gb.Matrix(A.blk_size, A.stream)
    plan = gb.Plan(1.0, A, B, C, 0.0)
    assert plan.stats.n_tiles > 0
    test = gb.lib().dbcsr_plan_wait_selftest
    x, y = bsr.to_dense(bsr.Mat.of(a)), bsr.to_dense(bsr.Mat.of(b))
    n = x.shape[0]
    for scale, fail in ((2.0, 1), (-0.5, 1), (4.0, 0)):
        assert test(plan.handle, fail) == gb._ffi.DBCSR_OK
        A.put_values(scale * a.data)
        plan.execute()
        got = bsr.to_dense(bsr.Mat(C.blk_size, *C.export()))
        bound = 2 * (n + 4) * 2.0 ** -53 * (np.abs(scale * x) @ np.abs(y))
        assert np.all(np.abs(got - scale * (x @ y)) <= bound), (scale, fail)
    plan.close()
    assert test(None, 1) == gb._ffi.DBCSR_EINVAL

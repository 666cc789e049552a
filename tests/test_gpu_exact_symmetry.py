"""FP64 products with operands that the library knows, or once knew, to be exactly symmetric: the tensor cores
read such an operand's tiles as those of its transpose, so the knowledge must not outlive the values.

Every block is compared with a plain FP64 product within twice what any sum of n rounded terms keeps (both
sides are rounded): ||error|| <= 2 (n + 4) 2^-53 sum_K ||A_IK|| ||B_KJ||.  A transposed operand is wrong in
the first digits."""
import ctypes as C

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
WATERS = 40


@pytest.fixture(scope="module")
def gb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2003_03868_gb300 as m
    m.lib()
    return m


@pytest.fixture(scope="module")
def hamiltonian():
    return synth.build_hamiltonian(synth.small(WATERS, seed=2100)).H


def _dense(M):
    rp, col, data = M.export()
    bs = np.asarray(M.blk_size)
    off = np.concatenate([[0], np.cumsum(bs)])
    D, at = np.zeros((off[-1], off[-1])), 0
    for i in range(len(bs)):
        for j in col[rp[i]:rp[i + 1]]:
            n = bs[i] * bs[j]
            D[off[i]:off[i + 1], off[j]:off[j + 1]] = data[at:at + n].reshape(bs[i], bs[j])
            at += n
    return D


def _check(M, A, B):
    start = np.concatenate([[0], np.cumsum(M.blk_size)])[:-1]
    a, b = _dense(A), _dense(B)
    norms = lambda D: np.sqrt(np.add.reduceat(np.add.reduceat(D * D, start, 0), start, 1))  # noqa: E731
    bound = 2 * (a.shape[0] + 4) * 2.0 ** -53 * (norms(a) @ norms(b))
    assert np.all(norms(_dense(M) - a @ b) <= bound)


def _flagged(gb, h):
    """An exactly symmetric result of the library, and a copy of it."""
    X = gb.sign_iterate(gb.Matrix.of(h), 0.0, 1e-7, 1e-9, max_iter=2, return_x=True).P
    D = _dense(X)
    assert np.array_equal(D, D.T)
    return X


@pytest.mark.parametrize("which", ["b", "both", "copy"])
def test_plan_on_a_symmetric_result_takes_asymmetric_values(gb, hamiltonian, which):
    X = _flagged(gb, hamiltonian)
    B = X.copy() if which == "copy" else X
    A = X if which == "both" else gb.Matrix.of(hamiltonian)
    Cm = gb.Matrix(X.blk_size, X.stream)
    plan = gb.Plan(1.0, A, B, Cm, 0.0)
    assert plan.stats.n_tiles > 0
    _check(Cm, A, B)
    rng = np.random.default_rng(21)
    for _ in range(2):
        B.put_values(rng.uniform(-1.0, 1.0, len(B.export()[2])))
        plan.execute()
        _check(Cm, A, B)
    plan.close()


def test_submatrix_result_of_a_symmetric_matrix(gb, hamiltonian):
    # P takes its pattern from a matrix that is exactly symmetric, but is not symmetric itself
    X = _flagged(gb, hamiltonian)
    P = gb.submatrix_sign(X, 0.0, 1e-6, max_iter=40).P
    D = _dense(P)
    assert np.abs(D - D.T).max() > 1e-9
    K = gb.Matrix.of(hamiltonian)
    Cm = gb.Matrix(X.blk_size, X.stream)
    assert gb.multiply(1.0, K, P, 0.0, Cm, 0.0).n_tiles > 0
    _check(Cm, K, P)


def test_batch_into_handles_that_held_symmetric_results(gb, hamiltonian):
    # full products keep both triangles as computed: the filtered X is symmetric only up to its last bits
    H = gb.Matrix.of(hamiltonian)
    P = _flagged(gb, hamiltonian)
    mu = np.zeros(1)
    o = gb.SignOpts(1e-4, 1e-9, 3, gb.DBCSR_FP64, 1e-4, 0.5, 0, gb._ffi.DBCSR_SIGN_FULL_PRODUCTS, 2, 0)
    st = gb.lib().dbcsr_sign_iterate_batched(1, (C.c_void_p * 1)(H.handle.value), C.c_void_p(mu.ctypes.data), C.byref(o),
                                             (C.c_void_p * 1)(P.handle.value), (gb.SignReport * 1)())
    assert st in (gb._ffi.DBCSR_OK, gb._ffi.DBCSR_ENOTCONV)
    D = _dense(P)
    assert np.abs(D - D.T).max() > 1e-9
    Cm = gb.Matrix(P.blk_size, P.stream)
    assert gb.multiply(1.0, H, P, 0.0, Cm, 0.0).n_tiles > 0
    _check(Cm, H, P)

"""Operands shared between threads: the block groups of the tensor cores are kept with the matrices and shared
by the results."""
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


def test_first_products_of_several_threads_on_one_operand(gb):
    # the operand's norms are known and its groups are not: every thread's product may be the first to need them
    import threading

    import torch
    h = synth.build_hamiltonian(synth.small(40, seed=2500)).H
    ref = None
    streams = [torch.cuda.Stream() for _ in range(4)]
    for _ in range(6):
        A = gb.Matrix.of(h)
        A.groups()                                   # (its norms; the groups of this call are not kept)
        start = threading.Barrier(4)
        out, bad = [None] * 4, []

        def work(i):
            try:
                B = gb.Matrix.of(h, streams[i].cuda_stream)
                B.groups()
                C = gb.Matrix(A.blk_size, streams[i].cuda_stream)
                start.wait()
                for _ in range(3):
                    assert gb.multiply(1.0, A, B, 0.0, C, 1e-7).n_tiles > 0
                out[i] = C.export()
            except Exception as e:                   # noqa: BLE001 -- reported by the main thread
                bad.append(repr(e))
                start.abort()
        ts = [threading.Thread(target=work, args=(i,)) for i in range(4)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
        assert not bad
        ref = ref or out[0]
        for o in out:
            assert all(np.array_equal(x, y) for x, y in zip(o, ref))

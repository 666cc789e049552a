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


def test_results_outlive_their_operand_and_its_stream(gb):
    # a product's result shares its operand's groups: they stay usable, and can be freed, when the operand and
    # the stream it was made on are gone
    import torch
    rt = torch.cuda.cudart()
    h = synth.build_hamiltonian(synth.small(40, seed=2501)).H
    H = gb.Matrix.of(h)
    for _ in range(3):
        handle = torch.zeros(1, dtype=torch.int64)
        assert int(rt.cudaStreamCreate(handle.data_ptr())) == 0
        A = gb.Matrix.of(h, int(handle[0]))
        C = gb.Matrix(H.blk_size, H.stream)
        assert gb.multiply(1.0, A, H, 0.0, C, 1e-7).n_tiles > 0
        A.close()
        assert int(rt.cudaStreamDestroy(int(handle[0]))) == 0
        D, E = gb.Matrix(H.blk_size, H.stream), gb.Matrix(H.blk_size, H.stream)
        assert gb.multiply(1.0, C, H, 0.0, D, 1e-7).n_tiles > 0
        fresh = gb.Matrix.from_blocks(C.blk_size, *C.export())
        gb.multiply(1.0, fresh, H, 0.0, E, 1e-7)
        (rp, col, x), (rp2, col2, y) = D.export(), E.export()
        # the groups of the two differ (H's couplings and the product's): equal to the rounding of 920 terms
        assert np.array_equal(rp, rp2) and np.array_equal(col, col2)
        assert np.linalg.norm(x - y) <= 920 * 2.0 ** -53 * np.linalg.norm(y)
        C.close()
        D.close()


@pytest.mark.parametrize("planned", [False, True])
def test_operands_on_another_stream_whose_norms_are_not_known(gb, planned):
    # the operands' norms are formed on their stream, the product on its own, which has the higher priority while
    # a third keeps the GPU busy: the product waits for the norms
    import torch
    rows = [synth.build_hamiltonian(synth.small(40, seed=2502 + k)).H for k in range(2)]
    s, hi = torch.cuda.Stream(priority=0), torch.cuda.Stream(priority=-1)
    busy = torch.cuda.Stream()
    X = [gb.Matrix.of(h) for h in rows]
    ref = gb.Matrix(X[0].blk_size)
    gb.multiply(1.0, X[0], X[1], 0.0, ref, 1e-5)
    ref = ref.export()
    w = torch.randn(8192, 8192, device="cuda")
    torch.cuda.synchronize()
    for _ in range(5):
        A, B = (gb.Matrix.of(h, s.cuda_stream) for h in rows)
        C = gb.Matrix(A.blk_size, hi.cuda_stream)
        torch.cuda.synchronize()
        with torch.cuda.stream(busy):
            for _ in range(4):
                torch.mm(w, w)
        if planned:
            plan = gb.Plan(1.0, A, B, C, 1e-5)
            plan.execute()
            F = gb.Matrix.from_blocks(C.blk_size, *C.export())
            F.filter(1e-5)                           # (a plan keeps the blocks below eps, as zeros)
            out = F.export()
            plan.close()
        else:
            gb.multiply(1.0, A, B, 0.0, C, 1e-5)
            out = C.export()
        busy.synchronize()
        (rp, col, x), (rp2, col2, y) = out, ref
        assert np.array_equal(rp, rp2) and np.array_equal(col, col2)
        assert np.linalg.norm(x - y) <= 920 * 2.0 ** -53 * np.linalg.norm(y)

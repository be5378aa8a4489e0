"""One batched plan bound to two workspaces, to complex bins in one and real
windows in the other: each run does what its own workspace says, in any order."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pg = pytest.importorskip("paper_2405_15529_gb300")


@pytest.mark.parametrize("sizes", [[(9000, 30), (500, 70)], [(3000, 100)] * 5])
def test_bins_and_windows_of_one_plan(sizes):
    g = torch.Generator(device="cuda").manual_seed(4)
    X = [torch.randn((M, N), dtype=torch.float32, device="cuda", generator=g).t() for N, M in sizes]
    Q = [torch.randn((M, N), dtype=torch.complex64, device="cuda", generator=g).t() for N, M in sizes]
    wins = pg.BatchedPOD(X, kmodes=3, prec=pg.PREC_MIXED_3XTF32)
    bins = pg.BatchedSVD(Q, kmodes=3)
    wins.run()
    bins.run()
    SW, SB = wins.S_all.clone(), bins.S_all.clone()
    UW = [m.clone() for m in wins.modes]
    UB = [m.clone() for m in bins.modes]
    VW = [v.clone() for v in wins.VT]
    # the windows' plan, bound to the bins in a workspace of its own
    lib, n = pg.load_library(), len(sizes)
    ws = torch.empty(wins.ws.numel(), dtype=torch.uint8, device="cuda")
    ptr = lambda ts: (ctypes.c_void_p * n)(*[t.data_ptr() for t in ts])
    ld = lambda ts: (ctypes.c_int64 * n)(*[t.stride(1) for t in ts])
    assert lib.pylom_svd_batched_bind(wins.plan, ptr(bins.Q), ld(bins.Q), ptr(bins.U), ld(bins.U), ws.data_ptr(),
                                      ws.numel(), None) == pg.OK
    S2 = torch.zeros_like(SB)
    for _ in range(2):
        for t in wins.U + wins.VT + bins.U:
            t.zero_()
        wins.S_all.zero_()
        S2.zero_()
        wins.run()
        assert lib.pylom_svd_batched_run(wins.plan, ws.data_ptr(), S2.data_ptr(), 60, None) == pg.OK
        torch.cuda.synchronize()
        assert torch.equal(wins.S_all, SW) and torch.equal(S2, SB)
        for a, b in zip(wins.modes + bins.modes + wins.VT, UW + UB + VW):
            assert torch.equal(a, b)

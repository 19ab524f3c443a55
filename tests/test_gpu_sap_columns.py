"""FP32 smoother over block shapes and column counts, against oracle.smoother.sap.

The sweeps run on copies of the vectors in block order, columns copied four at a time with a
remainder; inside a stream capture they work on the caller's vectors.  Cases: a block that does
not fill a warp (2^4), uneven extents with an odd one, a full 4^4 block with more than 64 sites;
1 column, remainders of 1, 2 and 3, and a full group.

Tolerance 1e-5 relative L2: 2 cycles of 2 half sweeps, each a residual and 3 minimal-residual steps of
sums of about 100 FP32 terms per entry, well under 100 roundings of 2^-24 in sequence.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import smoother  # noqa: E402

import helpers as H  # noqa: E402
from test_gpu_fine import Fine  # noqa: E402

pytestmark = pytest.mark.gpu

SHAPES = {"2^4": ((8, 4, 4, 8), (2, 2, 2, 2)), "uneven": ((6, 8, 4, 8), (3, 4, 2, 2)),
          "flat": ((8, 4, 4, 4), (4, 2, 1, 1)), "4^4": ((8, 8, 8, 8), (4, 4, 4, 4))}


@pytest.mark.parametrize("captured", [False, True], ids=["eager", "captured"])
@pytest.mark.parametrize("nrhs", [1, 3, 6])
@pytest.mark.parametrize("shape", SHAPES)
def test_sap_fp32(shape, nrhs, captured):
    import paper_1512_04506_gb300 as amg
    L, B = SHAPES[shape]
    c = Fine(amg, L, B, 4, 811, "fp32", max_nrhs=nrhs)
    try:
        y, x0 = c.vec(nrhs, 1), c.vec(nrhs, 2)
        yd, xd = c.dev(y), c.dev(x0)
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                amg.amg_sap(c.h, yd, xd, nrhs, 2, 3, torch.cuda.current_stream())
            xd.copy_(c.dev(x0))
            g.replay()
        else:
            amg.amg_sap(c.h, yd, xd, nrhs, 2, 3, c.stream)
        torch.cuda.synchronize()
        ref = np.empty(y.shape, dtype=np.complex128)
        for r in range(nrhs):
            ref[..., r] = smoother.sap(c.U, c.C, c.m0, c.field(y[..., r].astype(np.complex128)),
                                       c.field(x0[..., r].astype(np.complex128)), B, 2, 3).reshape(c.V, 4, 3)
        got = xd.cpu().numpy()
        for r in range(nrhs):
            assert H.rel(got[..., r], ref[..., r]) < 1e-5
        assert amg.amg_sync_status(c.h) == amg.AMG_OK
    finally:
        c.close()

"""FP64 smoother with MR steps in fixed point, over block shapes, scales and non-finite input.

Tolerance against oracle.smoother.sap 1e-12 relative L2: 2 cycles of 2 half sweeps, each a residual and 3 steps of sums of
about 100 terms, well under 1000 roundings of 2^-53.  The numbers are relative to the block's largest entry, so a power of two
in y and x passes through to the last bit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import smoother  # noqa: E402

import helpers as H  # noqa: E402
from test_gpu_fine import Fine  # noqa: E402

pytestmark = pytest.mark.gpu

SHAPES = {"2^4": ((8, 4, 4, 8), (2, 2, 2, 2)), "uneven": ((6, 8, 8, 4), (3, 4, 4, 2)),
          "flat": ((8, 4, 4, 4), (4, 2, 1, 1)), "long": ((4, 14, 4, 4), (1, 7, 2, 1)), "4^4": ((8, 8, 8, 8), (4, 4, 4, 4))}


def _sap(amg, c, y, x0, nrhs, n_cycles=2, n_mr=3):
    xd = c.dev(x0)
    amg.amg_sap(c.h, c.dev(y), xd, nrhs, n_cycles, n_mr, c.stream)
    torch.cuda.synchronize()
    return xd.cpu().numpy()


@pytest.mark.parametrize("shape", SHAPES)
def test_against_oracle_and_scales(shape):
    import paper_1512_04506_gb300 as amg
    L, B = SHAPES[shape]
    nrhs = 2
    c = Fine(amg, L, B, 4, 821, "fp64", max_nrhs=nrhs)
    try:
        y, x0 = c.vec(nrhs, 1), c.vec(nrhs, 2)
        y[..., 1] *= 1e-6  # columns of different size
        x0[..., 1] = 0
        got = _sap(amg, c, y, x0, nrhs)
        for r in range(nrhs):
            ref = smoother.sap(c.U, c.C, c.m0, c.field(y[..., r]), c.field(x0[..., r]), B, 2, 3).reshape(c.V, 4, 3)
            assert H.rel(got[..., r], ref) < 1e-12
        for k in (-300, 300):
            assert np.array_equal(_sap(amg, c, y * 2.0 ** k, x0 * 2.0 ** k, nrhs), got * 2.0 ** k)
        assert np.array_equal(_sap(amg, c, y * 0, x0 * 0, nrhs), y * 0)
        assert amg.amg_sync_status(c.h) == amg.AMG_OK
    finally:
        c.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_block(bad):
    """One entry of y that is not finite: a block whose <p, p> is not positive is left as it is, so with a NaN its x
    stays, and blocks out of its reach are as without it."""
    import paper_1512_04506_gb300 as amg
    L, B = (16, 4, 4, 4), (2, 2, 2, 2)
    c = Fine(amg, L, B, 4, 823, "fp64", max_nrhs=1)
    try:
        y, x0 = c.vec(1, 1), c.vec(1, 2)
        got = _sap(amg, c, y, x0, 1, 1, 2)
        y2 = y.copy()
        y2.reshape(-1)[0] = bad  # site 0, in the block at x = 0, 1
        got2 = _sap(amg, c, y2, x0, 1, 1, 2)
        first, second = got.reshape(4, 4, 4, 16, 12), got2.reshape(4, 4, 4, 16, 12)
        if np.isnan(bad):
            assert np.array_equal(second[:2, :2, :2, :2], x0.reshape(4, 4, 4, 16, 12)[:2, :2, :2, :2])
        assert np.array_equal(second[:, :, :, 6:12], first[:, :, :, 6:12])
    finally:
        c.close()

"""FP64 smoother on vectors whose sites differ widely in size within a block.

Only block 0 (colour 0) has a right-hand side, 10^(-4 x) in size at local x, so that one cycle's result there comes from that
block alone.  Every site to 1e-12 of its own norm against oracle.smoother.sap: 2 and 4 minimal-residual steps of sums of
about 100 terms of the site's and its neighbours' sizes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import smoother  # noqa: E402

import helpers as H  # noqa: E402
from test_gpu_fine import Fine  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_mr", [2, 4])
@pytest.mark.parametrize("B", [(4, 4, 4, 2), (4, 2, 2, 1)], ids=lambda B: "x".join(map(str, B)))
def test_steep_block(B, n_mr):
    import paper_1512_04506_gb300 as amg
    L = tuple(2 * b for b in B)
    c = Fine(amg, L, B, 4, 829, "fp64", max_nrhs=2)
    try:
        site = np.arange(c.V)
        x = np.stack([site % L[0], site // L[0] % L[1], site // (L[0] * L[1]) % L[2], site // (L[0] * L[1] * L[2])])
        own = (x < np.array(B)[:, None]).all(0)
        y = c.vec(2, 1)
        y[..., 0] *= np.where(own, 10.0 ** (-4 * x[0]), 0)[:, None, None]
        xd = torch.zeros(y.shape, dtype=c.ctype, device="cuda")
        amg.amg_sap(c.h, c.dev(y), xd, 2, 1, n_mr, c.stream)
        got = xd.cpu().numpy()
        assert amg.amg_sync_status(c.h) == amg.AMG_OK
        for r in range(2):  # column 1: every site alike
            ref = smoother.sap(c.U, c.C, c.m0, c.field(y[..., r]), np.zeros_like(c.field(y[..., r])), B, 1, n_mr)
            ref = ref.reshape(c.V, 4, 3)[own]
            norm = lambda a: np.sqrt((np.abs(a) ** 2).sum((1, 2)))
            assert (norm(got[own][..., r] - ref) / norm(ref)).max() < 1e-12
    finally:
        c.close()


def test_heavy_mass():
    """A mass far above the links: the hops' share of a step keeps its own accuracy at sites where rho is 0."""
    import paper_1512_04506_gb300 as amg
    L, B = (8, 4, 4, 4), (4, 2, 2, 2)
    c = Fine(amg, L, B, 4, 831, "fp64", max_nrhs=1, m0=1e7)
    try:
        y = np.zeros((c.V, 4, 3, 1), dtype=c.np_ctype)
        y[1] = 1
        xd = torch.zeros(y.shape, dtype=c.ctype, device="cuda")
        amg.amg_sap(c.h, c.dev(y), xd, 1, 1, 2, c.stream)
        got = xd.cpu().numpy()[..., 0]
        ref = smoother.sap(c.U, c.C, c.m0, c.field(y[..., 0]), np.zeros_like(c.field(y[..., 0])), B, 1, 2).reshape(c.V, 4, 3)
        for s in (0, 2):  # neighbours of the source
            assert H.rel(got[s], ref[s]) < 1e-12
    finally:
        c.close()

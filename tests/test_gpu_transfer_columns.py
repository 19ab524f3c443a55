"""FP32 restriction and prolongation of several columns against the exported R in complex128.

Columns go in groups of 4 (restriction) and 8 (prolongation) with remainders, rows of R in groups per
warp: column counts around those groups, numbers of test vectors that fill the row groups or not, and
blocks whose dof pairs do not fill the lanes.  Tolerance 1e-5 relative L2, the library's bound for
FP32 applies (sums of at most 1536 products, rounding 2^-24 each, R rounded once).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synth import inputs as si  # noqa: E402

import helpers as H  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [((4, 4, 4, 6), (2, 2, 2, 2), 1), ((6, 8, 4, 4), (3, 4, 2, 2), 11), ((8, 8, 8, 8), (4, 4, 4, 4), 20),
         ((8, 8, 8, 8), (4, 4, 4, 4), 32)]


@pytest.mark.parametrize("L,B,ntv", CASES, ids=["2^4-1", "uneven-11", "4^4-20", "4^4-32"])
def test_columns(L, B, ntv):
    import paper_1512_04506_gb300 as amg
    sites = si.all_sites(L)
    Vc, Vb = int(np.prod(L)) // int(np.prod(B)), int(np.prod(B))
    U = torch.from_numpy(si.links(5, 0.3, sites)).cuda()
    tv = torch.from_numpy(si.test_vectors(5, ntv, sites)).cuda()
    st = torch.cuda.current_stream()
    h, _ = amg.amg_setup_coarse(amg.make_params(L, B, ntv, 17), U, tv, st)
    try:
        R = torch.empty(Vc, 2, ntv, 6 * Vb, dtype=torch.complex128, device="cuda")
        amg.amg_export_R(h, R)
        Lc = [l // b for l, b in zip(L, B)]
        order = torch.from_numpy(np.stack([H.block_sites(L, B, H.coarse_coords(Lc, i)) for i in range(Vc)])).cuda()
        for n in (1, 2, 3, 4, 5, 6, 7, 8, 9, 12, 15, 16, 17):
            y = torch.from_numpy(si.fine_rhs(6, n, sites).astype(np.complex64)).cuda()
            yc = torch.empty(Vc, 2, ntv, n, dtype=torch.complex64, device="cuda")
            amg.amg_restrict(h, y, yc, n, st)
            agg = y.to(torch.complex128)[order].reshape(Vc, Vb, 2, 6, n).transpose(1, 2).reshape(Vc, 2, 6 * Vb, n)
            assert H.rel(yc.cpu().numpy(), (R @ agg).cpu().numpy()) < 1e-5, n
            xc = torch.from_numpy(si.coarse_vector(7, ntv, n, np.arange(Vc)).astype(np.complex64)).cuda()
            x = torch.empty_like(y)
            amg.amg_prolong(h, xc, x, n, st)
            ref = (R.mH @ xc.to(torch.complex128)).reshape(Vc, 2, Vb, 6, n).transpose(1, 2).reshape(Vc, Vb, 4, 3, n)
            assert H.rel(x[order].cpu().numpy(), ref.cpu().numpy()) < 1e-5, n
    finally:
        amg.amg_destroy(h)

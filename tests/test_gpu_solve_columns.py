"""The fused Arnoldi step on grids that follow the vector's length, for every kind of column count.

Fixed numbers of FGMRES steps across a restart against oracle.krylov.fgmres with the exported D_c:
counts that divide 32 and that do not (CTAs then use a multiple of the columns), vectors of one CTA
and of several.  FP64 1e-10 (the bound of the library's fixed-step comparisons), FP32 1e-4: seven steps
of dots and updates in FP32 on a system of condition number of order 10.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import coarse, krylov, lattice as lat  # noqa: E402
from synth import inputs as si  # noqa: E402

import helpers as H  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("L", [(4, 4, 4, 4), (8, 8, 8, 8)], ids=["one-cta", "several"])
def test_columns(L, prec):
    import paper_1512_04506_gb300 as amg
    B, ntv = (2, 2, 2, 2), 8
    sites = si.all_sites(L)
    Lc = lat.coarse_dims(L, B)
    Vc = int(np.prod(Lc))
    st = torch.cuda.current_stream()
    pr = amg.AMG_FP64 if prec == "fp64" else amg.AMG_FP32
    ct = torch.complex128 if prec == "fp64" else torch.complex64
    h, _ = amg.amg_setup_coarse(amg.make_params(L, B, ntv, 16, link_prec=pr, r_prec=pr, vec_prec=pr),
                                torch.from_numpy(si.links(9, 0.3, sites)).cuda(),
                                torch.from_numpy(si.test_vectors(9, ntv, sites)).cuda(), st)
    try:
        Dc = np.empty((Vc, 9, 2 * ntv, 2 * ntv), dtype=np.complex128)
        amg.amg_export_Dc(h, Dc)
        for n in (1, 2, 3, 5, 7, 12, 16):
            b = si.coarse_vector(10, ntv, n, np.arange(Vc))
            bd = torch.from_numpy(b).to(ct).cuda()
            x = torch.empty_like(bd)
            info = amg.amg_coarse_solve(h, bd, x, n, 0.0, 4, 7, st)
            assert [k for k, _ in info] == [7] * n
            for r in range(n):
                ref = krylov.fgmres(lambda v: coarse.coarse_apply(Dc, v, Lc), b[..., r], 0.0, 4, 7)[0]
                assert H.rel(x[..., r].cpu().numpy(), ref.reshape(b[..., r].shape)) < (1e-10 if prec == "fp64" else 1e-4)
        assert amg.amg_sync_status(h) == amg.AMG_OK
    finally:
        amg.amg_destroy(h)

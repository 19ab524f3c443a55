"""The assembly of D_c by exact products of slices on the tensor cores, against the oracle.

Blocks and numbers of test vectors that take this path, where it can go wrong: an extent of 1 (no link
inside the block), sites that do not fill a group of 8 before the face, the largest block, columns that do not fill
a group of 8 or of 4, the widest accumulators (Ntv > 24), and links far from magnitude 1.  Tolerance 1e-12 relative L2
for every direction of D_c, the library's bound for the setup, and 1e-13 between the two arithmetics.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import coarse, dirac  # noqa: E402
from synth import inputs as si  # noqa: E402

import helpers as H  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [((2, 3, 3, 3), 16, 1.0), ((1, 3, 3, 7), 17, 1.0), ((4, 3, 3, 3), 9, 1.0), ((4, 4, 4, 2), 24, 1.0),
         ((3, 3, 3, 3), 25, 1.0), ((3, 3, 3, 3), 32, 1.0), ((11, 31, 1, 1), 3, 1.0), ((4, 4, 4, 4), 6, 1.0),
         ((4, 3, 3, 3), 12, 3e-21), ((2, 4, 3, 3), 20, 2.5e5)]


@pytest.mark.parametrize("B,ntv,scale", CASES, ids=["%s-%d-%g" % ("x".join(map(str, c[0])), c[1], c[2]) for c in CASES])
def test_assembly(B, ntv, scale):
    import paper_1512_04506_gb300 as amg
    L = tuple(2 * b for b in B)
    sites = si.all_sites(L)
    Uh, tvh = si.links(37, 0.3, sites) * scale, si.test_vectors(37, ntv, sites)
    U = np.moveaxis(Uh.reshape(H.field_shape(L) + (4, 3, 3)), 4, 0)
    Q = coarse.orthonormalize(tvh.reshape(H.field_shape(L) + (4, 3, ntv)), B)
    ref = coarse.coarse_operator(U, dirac.clover_field(U, H.CSW), H.M0, Q, L, B)
    got = []
    for arith in (amg.AMG_SETUP_FP64, amg.AMG_SETUP_F32PAIR):
        p = amg.make_params(L, B, ntv, m0=H.M0, csw=H.CSW, link_prec=amg.AMG_FP64, r_prec=amg.AMG_FP64,
                            vec_prec=amg.AMG_FP64, setup_arith=arith)
        h, _ = amg.amg_setup_coarse(p, torch.from_numpy(Uh).cuda(), torch.from_numpy(tvh).cuda(),
                                    torch.cuda.current_stream())
        try:
            Dc = np.empty_like(ref)
            amg.amg_export_Dc(h, Dc)
            for d in range(9):
                assert H.rel(Dc[:, d], ref[:, d]) < 1e-12, d
            got.append(Dc)
            assert amg.amg_sync_status(h) == amg.AMG_OK
        finally:
            amg.amg_destroy(h)
    for d in range(9):
        assert H.rel(got[1][:, d], got[0][:, d]) < 1e-13, d


def test_non_finite_links():
    """A NaN in one link leaving its block: F_mu of that block and what follows from it is NaN, the block's
    other directions and the other blocks' are as without it."""
    import paper_1512_04506_gb300 as amg
    B, ntv = (4, 4, 4, 2), 20
    L = tuple(2 * b for b in B)
    sites = si.all_sites(L)
    Uh, tvh = si.links(39, 0.3, sites), si.test_vectors(39, ntv, sites)
    bad = Uh.copy().reshape(H.field_shape(L) + (4, 3, 3))
    bad[0, 0, 0, 3, 0, 1, 2] = np.nan  # x = 3, direction 0
    bad = bad.reshape(Uh.shape)
    got = []
    for links in (Uh, bad):
        p = amg.make_params(L, B, ntv, m0=H.M0, csw=0.0, link_prec=amg.AMG_FP64, r_prec=amg.AMG_FP64,
                            vec_prec=amg.AMG_FP64, setup_arith=amg.AMG_SETUP_FP64)
        h, _ = amg.amg_setup_coarse(p, torch.from_numpy(links).cuda(), torch.from_numpy(tvh).cuda(),
                                    torch.cuda.current_stream())
        try:
            Dc = np.empty((16, 9, 2 * ntv, 2 * ntv), dtype=np.complex128)
            amg.amg_export_Dc(h, Dc)
            got.append(Dc)
        finally:
            amg.amg_destroy(h)
    assert np.isfinite(got[0]).all()
    assert np.isnan(got[1][0, 1]).all() and np.isnan(got[1][1, 2]).all()
    for i in range(16):
        for d in range(1, 9):
            if (i, d) not in ((0, 1), (1, 2)):
                np.testing.assert_array_equal(got[1][i, d], got[0][i, d])

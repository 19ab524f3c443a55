"""The setup over numbers of test vectors, in both arithmetics, against the oracle.

The assembly's tile shape and its groups of warps follow 2 ntv, and the Gram-Schmidt works on column
blocks of 4 and a number of elements per thread that follows the aggregate: every tile shape, full and
partial column blocks, and extents that leave an uneven number of sites before the face.  Tolerance
1e-12 relative L2 for R and for every direction of D_c, the library's bound for the setup.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import coarse, dirac  # noqa: E402
from synth import inputs as si  # noqa: E402

import helpers as H  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [((4, 4, 4, 4), (2, 2, 2, 2), n) for n in (1, 2, 4, 7, 8, 11, 16, 24)] + \
        [((6, 4, 4, 4), (3, 2, 2, 1), n) for n in (6, 12, 20)] + [((6, 6, 4, 8), (3, 3, 2, 4), 32)]


@pytest.mark.parametrize("L,B,ntv", CASES, ids=["%s-%d" % ("x".join(map(str, c[1])), c[2]) for c in CASES])
def test_setup(L, B, ntv):
    import paper_1512_04506_gb300 as amg
    sites = si.all_sites(L)
    Uh, tvh = si.links(31, 0.3, sites), si.test_vectors(31, ntv, sites)
    U = np.moveaxis(Uh.reshape(H.field_shape(L) + (4, 3, 3)), 4, 0)
    Q = coarse.orthonormalize(tvh.reshape(H.field_shape(L) + (4, 3, ntv)), B)
    ref = coarse.coarse_operator(U, dirac.clover_field(U, H.CSW), H.M0, Q, L, B)
    for arith in (amg.AMG_SETUP_FP64, amg.AMG_SETUP_F32PAIR):
        p = amg.make_params(L, B, ntv, m0=H.M0, csw=H.CSW, link_prec=amg.AMG_FP64, r_prec=amg.AMG_FP64,
                            vec_prec=amg.AMG_FP64, setup_arith=arith)
        h, _ = amg.amg_setup_coarse(p, torch.from_numpy(Uh).cuda(), torch.from_numpy(tvh).cuda(),
                                    torch.cuda.current_stream())
        try:
            R = np.empty((ref.shape[0], 2, ntv, Q.shape[2]), dtype=np.complex128)
            Dc = np.empty_like(ref)
            amg.amg_export_R(h, R)
            amg.amg_export_Dc(h, Dc)
            assert H.rel(R, H.q_to_lib_R(Q)) < 1e-12
            for d in range(9):
                assert H.rel(Dc[:, d], ref[:, d]) < 1e-12, d
            assert amg.amg_sync_status(h) == amg.AMG_OK
        finally:
            amg.amg_destroy(h)

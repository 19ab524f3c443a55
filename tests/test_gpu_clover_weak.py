"""The clover term of links close to 1: C is then much smaller than the links it is formed from.

Tolerance 1e-13 of C's own size against the oracle's sums in doubles: Q - Q^dagger keeps only parts that every product
carries relative to their own size (imaginary parts and off-diagonals of the size of eps), some hundred
roundings.  Also lattices that are weak only in part.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import dirac  # noqa: E402
from synth import inputs as si  # noqa: E402

import helpers as H  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps", [1e-2, 1e-4, 1e-7])
@pytest.mark.parametrize("part", [False, True], ids=["all", "part"])
def test_weak_links(eps, part):
    import paper_1512_04506_gb300 as amg
    L, B = (4, 6, 4, 4), (2, 2, 2, 2)
    sites = si.all_sites(L)
    Uh = si.links(61, eps, sites)
    if part:  # strong links for y >= 3
        Uh = np.where((sites // 4 % 6 >= 3)[:, None, None, None], si.links(61, 0.3, sites), Uh)
    U = np.moveaxis(Uh.reshape(H.field_shape(L) + (4, 3, 3)), 4, 0)
    ref = H.clover_to_lib(dirac.clover_field(U, 1.0))
    p = amg.make_params(L, B, 1, m0=H.M0, csw=1.0, link_prec=amg.AMG_FP64, r_prec=amg.AMG_FP64, vec_prec=amg.AMG_FP64)
    h, _ = amg.amg_setup_coarse(p, torch.from_numpy(np.ascontiguousarray(Uh)).cuda(),
                                torch.from_numpy(si.test_vectors(61, 1, sites)).cuda(), torch.cuda.current_stream())
    try:
        C = np.empty(ref.shape, dtype=np.complex128)
        amg.amg_export_clover(h, C)
    finally:
        amg.amg_destroy(h)
    norm = lambda a: np.sqrt((np.abs(a) ** 2).sum((1, 2, 3)))
    assert (norm(C - ref) / norm(ref)).max() < 1e-13
    assert np.array_equal(C, np.conj(np.swapaxes(C, -1, -2)))
    assert np.array_equal(C[..., :3, :3], -C[..., 3:, 3:])


def test_unit_links():
    """Links 1 everywhere: the clover is 0."""
    import paper_1512_04506_gb300 as amg
    L, B = (4, 4, 4, 4), (2, 2, 2, 2)
    V = 256
    Uh = np.ascontiguousarray(np.broadcast_to(np.eye(3, dtype=np.complex128), (V, 4, 3, 3)))
    p = amg.make_params(L, B, 1, m0=H.M0, csw=1.0, link_prec=amg.AMG_FP64, r_prec=amg.AMG_FP64, vec_prec=amg.AMG_FP64)
    h, _ = amg.amg_setup_coarse(p, torch.from_numpy(Uh).cuda(), torch.from_numpy(si.test_vectors(61, 1, si.all_sites(L))).cuda(),
                                torch.cuda.current_stream())
    try:
        C = np.empty((V, 2, 6, 6), dtype=np.complex128)
        amg.amg_export_clover(h, C)
        assert not C.any()
    finally:
        amg.amg_destroy(h)

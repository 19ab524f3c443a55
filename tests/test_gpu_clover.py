"""The clover term, formed in fixed point, against the oracle.

Lattices with an extent of 2 (both neighbours the same site) and odd extents; links of magnitude 1, scaled far up
and down, and with directions of very different magnitude, so that the leaves of a plane and the planes carry
different exponents.  Tolerance 1e-14 relative L2 (1e-13 where the scaled directions mix): three products of 60-bit
numbers in sequence, each 3 units of 2^-58 of the factors' bounds, against FP64 sums in the oracle of 36 terms.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import dirac  # noqa: E402
from synth import inputs as si  # noqa: E402

import helpers as H  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [(4, 4, 4, 4), (2, 6, 3, 5), (7, 2, 4, 2)], ids=lambda L: "x".join(map(str, L)))
@pytest.mark.parametrize("scale", [(1, 1, 1, 1), (1e-25,) * 4, (3e30,) * 4, (1, 1e-3, 1e4, 1e-9)],
                         ids=["unit", "down", "up", "mixed"])
def test_clover(L, scale):
    import paper_1512_04506_gb300 as amg
    sites = si.all_sites(L)
    Uh = si.links(41, 0.6, sites).reshape(-1, 4, 3, 3) * np.array(scale).reshape(1, 4, 1, 1)
    csw = 1.0 / max(scale) ** 4
    U = np.moveaxis(Uh.reshape(H.field_shape(L) + (4, 3, 3)), 4, 0)
    ref = H.clover_to_lib(dirac.clover_field(U, csw))
    B = tuple(2 if n in (4, 6) else 1 for n in L)
    p = amg.make_params(L, B, 1, m0=H.M0, csw=csw, link_prec=amg.AMG_FP64, r_prec=amg.AMG_FP64, vec_prec=amg.AMG_FP64)
    tv = si.test_vectors(41, 1, sites)
    h, _ = amg.amg_setup_coarse(p, torch.from_numpy(np.ascontiguousarray(Uh)).cuda(), torch.from_numpy(tv).cuda(),
                                torch.cuda.current_stream())
    try:
        C = np.empty(ref.shape, dtype=np.complex128)
        amg.amg_export_clover(h, C)
        assert H.rel(C, ref) < (1e-13 if max(scale) != min(scale) else 1e-14)
        # Hermitian per chirality to the last bit, the diagonal blocks opposite
        assert np.array_equal(C, np.conj(np.swapaxes(C, -1, -2)))
        assert np.array_equal(C[..., :3, :3], -C[..., 3:, 3:])
    finally:
        amg.amg_destroy(h)

"""Setup from test vectors whose sites differ widely in size within a block.

Sites of both faces of direction x scaled by 1e-9 (with blocks of 4 in x), every site by a power of ten between 1e-9
and 1, or only the sites of one block.  R against the oracle's orthonormalisation: every site of every aggregate to 1e-12
of its own norm, in both arithmetics: sums and updates in doubles, and in pairs of floats (2^-47 per number), are good to
some hundred roundings of the site's own entries.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import coarse, dirac  # noqa: E402
from synth import inputs as si  # noqa: E402

import helpers as H  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [((4, 4, 4, 1), 20, "faces"), ((4, 4, 4, 2), 16, "faces"), ((2, 2, 2, 2), 16, "spread"),
         ((3, 3, 3, 3), 12, "spread"), ((4, 4, 4, 1), 17, "one_block")]


def _inputs(B, ntv, kind):
    L = tuple(2 * b for b in B)
    sites = si.all_sites(L)
    c = np.stack([sites % L[0], sites // L[0] % L[1], sites // (L[0] * L[1]) % L[2], sites // (L[0] * L[1] * L[2])])
    scale = 10.0 ** (-9 * np.random.default_rng(47).random(len(sites)))
    if kind == "faces":
        lx = c[0] % B[0]
        scale = np.where((lx == 0) | (lx == B[0] - 1), 1e-9, 1.0)
    elif kind == "one_block":
        scale[(c >= np.array(B)[:, None]).any(0)] = 1.0
    return L, si.links(47, 0.3, sites), np.ascontiguousarray(si.test_vectors(47, ntv, sites) * scale[:, None, None, None])


def _setup(amg, L, B, ntv, Uh, tv, arith):
    p = amg.make_params(L, B, ntv, m0=H.M0, csw=H.CSW, link_prec=amg.AMG_FP64, r_prec=amg.AMG_FP64,
                        vec_prec=amg.AMG_FP64,
                        setup_arith=amg.AMG_SETUP_FP64 if arith == "fp64" else amg.AMG_SETUP_F32PAIR)
    h, _ = amg.amg_setup_coarse(p, torch.from_numpy(Uh).cuda(), torch.from_numpy(tv).cuda(), torch.cuda.current_stream())
    try:
        R = np.empty((16, 2, ntv, 6 * int(np.prod(B))), dtype=np.complex128)
        Dc = np.empty((16, 9, 2 * ntv, 2 * ntv), dtype=np.complex128)
        amg.amg_export_R(h, R)
        amg.amg_export_Dc(h, Dc)
        assert amg.amg_sync_status(h) == amg.AMG_OK
        return R, Dc
    finally:
        amg.amg_destroy(h)


@pytest.mark.parametrize("arith", ["fp64", "pair"])
@pytest.mark.parametrize("B,ntv,kind", CASES, ids=["%s-%d-%s" % ("x".join(map(str, c[0])), c[1], c[2]) for c in CASES])
def test_R(B, ntv, kind, arith):
    import paper_1512_04506_gb300 as amg
    L, Uh, tv = _inputs(B, ntv, kind)
    ref = H.q_to_lib_R(coarse.orthonormalize(tv.reshape(H.field_shape(L) + (4, 3, ntv)), B))
    R, _ = _setup(amg, L, B, ntv, Uh, tv, arith)
    site = (16, 2, ntv, -1, 6)
    err = np.sqrt((np.abs(R - ref) ** 2).reshape(site).sum((2, 4)))
    assert (err / np.sqrt((np.abs(ref) ** 2).reshape(site).sum((2, 4)))).max() < 1e-12


# also an extent of 1 (no link inside), and more columns than the pair tiles with builder warps take
MORE = CASES + [((1, 4, 4, 5), 12, "spread"), ((4, 3, 3, 3), 26, "faces")]


@pytest.mark.parametrize("arith", ["fp64", "pair"])
@pytest.mark.parametrize("B,ntv,kind", MORE, ids=["%s-%d-%s" % ("x".join(map(str, c[0])), c[1], c[2]) for c in MORE])
def test_Dc(B, ntv, kind, arith):
    """Every direction of every site's D_c to 1e-12 of its own norm, the library's bound for a direction."""
    import paper_1512_04506_gb300 as amg
    L, Uh, tv = _inputs(B, ntv, kind)
    U = np.moveaxis(Uh.reshape(H.field_shape(L) + (4, 3, 3)), 4, 0)
    Q = coarse.orthonormalize(tv.reshape(H.field_shape(L) + (4, 3, ntv)), B)
    ref = coarse.coarse_operator(U, dirac.clover_field(U, H.CSW), H.M0, Q, L, B)
    _, Dc = _setup(amg, L, B, ntv, Uh, tv, arith)
    err = np.sqrt((np.abs(Dc - ref) ** 2).sum((2, 3)) / (np.abs(ref) ** 2).sum((2, 3)))
    assert err.max() < 1e-12

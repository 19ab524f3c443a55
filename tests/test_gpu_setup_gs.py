"""Gram-Schmidt on aggregates in fixed point: sizes of its dispatch, near-dependent and non-finite columns.

The columns' scales run over many powers of two.  R against the oracle's orthonormalisation 1e-12 relative L2, the library's
bound for the setup.  For columns that depend on earlier ones up to a part of 1e-9, R itself is only determined to
the part's share of the rounding, but rows are orthonormal to 1e-12 where the column is the first of its block of 4 or
depends on its own block only (two projections, 2^-53 of the column's norm at the second).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import coarse  # noqa: E402
from synth import inputs as si  # noqa: E402

import helpers as H  # noqa: E402

pytestmark = pytest.mark.gpu

# entries per aggregate: 6, 48, 252, 258, 510, 516, 1020, 1026, 1536, 2046 (the last beyond it)
CASES = [((1, 1, 1, 1), 6), ((2, 2, 2, 1), 24), ((7, 3, 2, 1), 9), ((43, 1, 1, 1), 5), ((17, 5, 1, 1), 13),
         ((43, 2, 1, 1), 6), ((17, 5, 2, 1), 12), ((19, 3, 3, 1), 7), ((4, 4, 4, 4), 11), ((31, 11, 1, 1), 5)]


def _run(amg, B, ntv, tv, arith, allow=False):
    L = tuple(2 * b for b in B)
    U = si.links(43, 0.3, si.all_sites(L))
    p = amg.make_params(L, B, ntv, m0=H.M0, csw=H.CSW, link_prec=amg.AMG_FP64, r_prec=amg.AMG_FP64,
                        vec_prec=amg.AMG_FP64, setup_arith=arith)
    h, status = amg.amg_setup_coarse(p, torch.from_numpy(U).cuda(), torch.from_numpy(tv).cuda(),
                                     torch.cuda.current_stream(), allow_rank_deficient=allow)
    try:
        R = np.empty((16, 2, ntv, 6 * int(np.prod(B))), dtype=np.complex128)
        amg.amg_export_R(h, R)
        return R, status
    finally:
        amg.amg_destroy(h)


def _arith(amg, name):
    return amg.AMG_SETUP_FP64 if name == "fp64" else amg.AMG_SETUP_F32PAIR


@pytest.mark.parametrize("arith", ["fp64", "pair"])
@pytest.mark.parametrize("B,ntv", CASES, ids=["%s-%d" % ("x".join(map(str, c[0])), c[1]) for c in CASES])
def test_sizes(B, ntv, arith):
    import paper_1512_04506_gb300 as amg
    L = tuple(2 * b for b in B)
    scale = 2.0 ** (np.arange(ntv) * 7 % 31 - 15)
    tv = np.ascontiguousarray(si.test_vectors(43, ntv, si.all_sites(L)) * scale)
    Q = coarse.orthonormalize(tv.reshape(H.field_shape(L) + (4, 3, ntv)), B)
    R, _ = _run(amg, B, ntv, tv, _arith(amg, arith))
    assert H.rel(R, H.q_to_lib_R(Q)) < 1e-12


@pytest.mark.parametrize("part", [1e-5, 1e-9])
@pytest.mark.parametrize("B", [(2, 2, 2, 2), (4, 4, 4, 4)], ids=["2^4", "4^4"])
def test_near_dependent(B, part):
    import paper_1512_04506_gb300 as amg
    ntv, L = 10, tuple(2 * b for b in B)
    tv = si.test_vectors(44, ntv, si.all_sites(L)).copy()
    for j in (1, 4, 8):
        tv[..., j] = tv[..., 0] - 2 * tv[..., j - 1] + part * tv[..., j]
    R, _ = _run(amg, B, ntv, np.ascontiguousarray(tv), amg.AMG_SETUP_FP64)
    gram = np.einsum("ahin,ahjn->ahij", R, R.conj())
    assert np.abs(gram - np.eye(ntv)).max() < 1e-12


@pytest.mark.parametrize("B", [(2, 2, 2, 2), (4, 4, 4, 4)], ids=["2^4", "4^4"])
@pytest.mark.parametrize("kind", ["dependent", "zero", "nan", "inf"])
def test_refused(B, kind):
    import paper_1512_04506_gb300 as amg
    ntv, L = 7, tuple(2 * b for b in B)
    tv = si.test_vectors(45, ntv, si.all_sites(L)).copy()
    if kind == "dependent":
        tv[..., 5] = tv[..., 1] + tv[..., 2]
    elif kind == "zero":
        tv[..., 5] = 0
    else:
        tv[3, ..., 5] = np.nan if kind == "nan" else np.inf
    tv = np.ascontiguousarray(tv)
    for arith in (amg.AMG_SETUP_FP64,) + ((amg.AMG_SETUP_F32PAIR,) if kind in ("dependent", "zero") else ()):
        with pytest.raises(amg.AmgError) as e:
            _run(amg, B, ntv, tv, arith)
        assert e.value.status == amg.AMG_ERR_RANK_DEFICIENT

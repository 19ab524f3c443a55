"""FP32 fine operator and smoother at sizes where their larger launch shapes serve.

D of one column in tiles of blocks (as many tiles as SMs or more): 4^4 blocks (one per CTA), 3^4 (three per CTA, 243 of 256
threads, a last CTA with two) and 2^4 (sixteen, a last CTA with eight); 1e-5 relative L2 against oracle.dirac as for the other
shapes, every site to 1e-4 of its norm (sums of about 100 terms, 2^-24 each).  The y - D x form through a restarted outer solve:
the residual that it reports is the true one to 1e-3 of itself.  The smoother with several columns per CTA, a short last
group and even and odd numbers of steps, and in more than one set of copies: every column as alone, to the last bit (a
column's arithmetic does not depend on the others).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import dirac  # noqa: E402

import helpers as H  # noqa: E402
from test_gpu_fine import Fine  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,B", [((16, 16, 16, 16), (4, 4, 4, 4)), ((12, 12, 12, 24), (3, 3, 3, 3)),
                                 ((14, 14, 14, 16), (2, 2, 2, 2))], ids=["4^4", "3^4", "2^4"])
def test_dirac_one_column(L, B):
    import paper_1512_04506_gb300 as amg
    c = Fine(amg, L, B, 1, 851, "fp32", max_nrhs=1)
    try:
        psi = c.vec(1, 1)
        out = torch.empty_like(c.dev(psi))
        amg.amg_dirac_apply(c.h, c.dev(psi), out, 1, c.stream)
        ref = dirac.apply_dirac(c.U, c.C, c.m0, c.field(psi[..., 0].astype(np.complex128))).reshape(c.V, 12)
        err = out.cpu().numpy().reshape(c.V, 12) - ref
        assert H.rel(err + ref, ref) < 1e-5
        assert (np.linalg.norm(err, axis=1) / np.linalg.norm(ref, axis=1)).max() < 1e-4
        assert amg.amg_sync_status(c.h) == amg.AMG_OK
    finally:
        c.close()


def test_residual_form():
    import paper_1512_04506_gb300 as amg
    c = Fine(amg, (16, 16, 16, 16), (4, 4, 4, 4), 4, 853, "fp32", max_nrhs=1)
    try:
        f = c.vec(1, 1)
        u = torch.empty_like(c.dev(f))
        vp = amg.make_vcycle_params(0.05, 30, 50, 1, 2)
        info = amg.amg_solve(c.h, vp, c.dev(f), u, 1, tol=0.0, restart=2, max_applies=7, stream=c.stream)
        f64 = c.field(f[..., 0].astype(np.complex128))
        r = f64 - dirac.apply_dirac(c.U, c.C, c.m0, c.field(u.cpu().numpy()[..., 0].astype(np.complex128)))
        true = np.linalg.norm(r.ravel()) / np.linalg.norm(f64.ravel())
        assert 1e-4 < true < 0.9  # far above the rounding of u
        assert abs(info[0][1] / true - 1) < 1e-3
    finally:
        c.close()


@pytest.mark.parametrize("n_mr", [3, 4])
@pytest.mark.parametrize("B", [(4, 4, 4, 4), (2, 2, 2, 2)], ids=["4^4", "2^4"])
@pytest.mark.parametrize("L,nrhs", [((16, 16, 16, 16), 3), ((16, 16, 16, 16), 12), ((8, 16, 16, 16), 5)],
                         ids=["whole", "many", "short"])
def test_sap_columns(L, nrhs, B, n_mr):
    import paper_1512_04506_gb300 as amg
    c = Fine(amg, L, B, 1, 857, "fp32", max_nrhs=nrhs)
    try:
        y, x0 = c.dev(c.vec(nrhs, 1)), c.dev(c.vec(nrhs, 2))
        x = x0.clone()
        amg.amg_sap(c.h, y, x, nrhs, 2, n_mr, c.stream)
        for r in range(nrhs):
            one = x0[..., r:r + 1].contiguous()
            amg.amg_sap(c.h, y[..., r:r + 1].contiguous(), one, 1, 2, n_mr, c.stream)
            assert torch.equal(one[..., 0], x[..., r])
        assert amg.amg_sync_status(c.h) == amg.AMG_OK
    finally:
        c.close()


def test_sap_two_sets_of_copies():
    """12 columns at 32^4: the copies of x and y take 2.4 GB, more than one set may."""
    import paper_1512_04506_gb300 as amg
    from synth import device as sd
    L, B, nrhs = (32, 32, 32, 32), (4, 4, 4, 4), 12
    V, st = 32 ** 4, torch.cuda.current_stream()
    U = sd.links(859, 0.3, L)
    p = amg.make_params(L, B, 1, nrhs, H.M0, H.CSW, amg.AMG_FP32, amg.AMG_FP32, amg.AMG_FP32)
    h, _ = amg.amg_setup_coarse(p, U, sd.test_vectors(859, 1, L), st)
    try:
        amg.amg_setup_fine(h, U, st)
        y = sd.fine_rhs(860, nrhs, L)
        x = torch.zeros(V, 4, 3, nrhs, dtype=torch.complex64, device="cuda")
        assert 2 * y.numel() * 8 > 2 << 30
        amg.amg_sap(h, y, x, nrhs, 1, 2, st)
        for r in (0, 9, 10, 11):
            one = torch.zeros(V, 4, 3, 1, dtype=torch.complex64, device="cuda")
            amg.amg_sap(h, y[..., r:r + 1].contiguous(), one, 1, 1, 2, st)
            assert torch.equal(one[..., 0], x[..., r])
        assert amg.amg_sync_status(h) == amg.AMG_OK
    finally:
        amg.amg_destroy(h)


@pytest.mark.parametrize("L,B,cycles", [((12, 16, 16, 16), (3, 4, 4, 2), 1), ((12, 16, 16, 16), (3, 4, 4, 2), 2),
                                        ((8, 8, 8, 8), (2, 2, 2, 2), 3), ((8, 8, 8, 8), (4, 4, 4, 4), 1)])
def test_with_and_without_copies(L, B, cycles):
    """Few columns or cycles work on the caller's vectors, more on copies: the same bits."""
    import paper_1512_04506_gb300 as amg
    c = Fine(amg, L, B, 1, 861, "fp32", max_nrhs=17)
    try:
        n = 4 if c.V > 20000 else 17
        y, x0 = c.dev(c.vec(n, 1)), c.dev(c.vec(n, 2))
        x = x0.clone()
        amg.amg_sap(c.h, y, x, n, cycles, 3, c.stream)
        for k in (1, 2, 3):
            part = x0[..., :k].contiguous()
            amg.amg_sap(c.h, y[..., :k].contiguous(), part, k, cycles, 3, c.stream)
            assert torch.equal(part, x[..., :k])
    finally:
        c.close()


@pytest.mark.parametrize("L,B,nrhs", [((8, 8, 8, 8), (4, 4, 4, 4), 2), ((8, 8, 8, 16), (4, 4, 4, 2), 12),
                                      ((12, 12, 12, 12), (3, 3, 3, 3), 6), ((16, 16, 16, 8), (2, 4, 4, 4), 16)],
                         ids=["one-2", "two-12", "one-6", "two-16"])
def test_dirac_even_columns(L, B, nrhs):
    """One or two columns per thread, by the waves they take."""
    import paper_1512_04506_gb300 as amg
    c = Fine(amg, L, B, 1, 863, "fp32", max_nrhs=nrhs)
    try:
        psi = c.vec(nrhs, 1)
        out = torch.empty_like(c.dev(psi))
        amg.amg_dirac_apply(c.h, c.dev(psi), out, nrhs, c.stream)
        got = out.cpu().numpy()
        for r in range(nrhs):
            ref = dirac.apply_dirac(c.U, c.C, c.m0, c.field(psi[..., r].astype(np.complex128))).reshape(c.V, 4, 3)
            assert H.rel(got[..., r], ref) < 1e-5
    finally:
        c.close()

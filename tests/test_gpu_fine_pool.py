"""The FP32 smoother's copies stay in the handle's pool from call to call, also on small lattices.

Device memory right after a sweep (copies in the pool) and after a synchronisation is the same: a pool whose threshold lies
below what it holds, in pieces of 32 MB, gives memory back there and the next sweep allocates it again.
"""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,nrhs", [((8, 8, 8, 8), 1), ((16, 16, 16, 16), 5), ((24, 24, 24, 24), 12)])
def test_nothing_given_back(L, nrhs):
    import paper_1512_04506_gb300 as amg
    V = L[0] * L[1] * L[2] * L[3]
    st = torch.cuda.current_stream()
    U = torch.eye(3, dtype=torch.complex128, device="cuda").expand(V, 4, 3, 3).contiguous()
    tv = torch.ones(V, 4, 3, 1, dtype=torch.complex128, device="cuda")
    p = amg.make_params(L, (4, 4, 4, 4), 1, nrhs, -0.3, 1.0, amg.AMG_FP32, amg.AMG_FP32, amg.AMG_FP32)
    h, _ = amg.amg_setup_coarse(p, U, tv, st)
    try:
        amg.amg_setup_fine(h, U, st)
        y = torch.ones(V, 4, 3, nrhs, dtype=torch.complex64, device="cuda")
        x = torch.zeros_like(y)
        ev = torch.cuda.Event()
        free = []
        for _ in range(3):
            amg.amg_sap(h, y, x, nrhs, 1, 1, st)
            ev.record()
            while not ev.query():  # not a synchronisation
                pass
            before = torch.cuda.mem_get_info()[0]
            torch.cuda.synchronize()
            free.append((before, torch.cuda.mem_get_info()[0]))
        assert free[-1][0] == free[-1][1]
    finally:
        amg.amg_destroy(h)


def test_links_set_again():
    """amg_setup_fine with other links on the same handle: no more memory held, and results of a new handle."""
    import paper_1512_04506_gb300 as amg
    from synth import device as sd
    L, nrhs, st = (16, 16, 16, 16), 5, torch.cuda.current_stream()
    Us, tv, y = [sd.links(s, 0.3, L) for s in (81, 82)], sd.test_vectors(81, 2, L), sd.fine_rhs(81, nrhs, L)
    p = amg.make_params(L, (4, 4, 4, 4), 2, nrhs, -0.3, 1.0, amg.AMG_FP32, amg.AMG_FP32, amg.AMG_FP32)
    out, held = [], []
    for first in (0, 1):
        h, _ = amg.amg_setup_coarse(p, Us[1], tv, st)
        try:
            for k in range(first, 2):
                amg.amg_setup_fine(h, Us[k], st)
                x = torch.zeros_like(y)
                amg.amg_sap(h, y, x, nrhs, 2, 3, st)
                torch.cuda.synchronize()
                held.append(torch.cuda.mem_get_info()[0])
            out.append(x)
        finally:
            amg.amg_destroy(h)
    assert torch.equal(out[0], out[1])
    assert abs(held[0] - held[1]) < 16 << 20

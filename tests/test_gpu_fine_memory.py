"""Device memory that amg_setup_fine holds.

FP32: links and clover (288 and 224 bytes per site) and, where the smoother can run, its copies of max_nrhs columns of x
and y (192 bytes per site and column, at most 2 GB unless one column takes more), kept between calls.
"""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SLACK = 64 << 20  # granularity of pools and allocations, and what the setup's own pool gives back meanwhile


def _held(L, B, max_nrhs, use):
    import paper_1512_04506_gb300 as amg
    V = L[0] * L[1] * L[2] * L[3]
    st = torch.cuda.current_stream()
    U = torch.eye(3, dtype=torch.complex128, device="cuda").expand(V, 4, 3, 3).contiguous()
    tv = torch.ones(V, 4, 3, 1, dtype=torch.complex128, device="cuda")
    p = amg.make_params(L, B, 1, max_nrhs, -0.3, 1.0, amg.AMG_FP32, amg.AMG_FP32, amg.AMG_FP32)
    h, _ = amg.amg_setup_coarse(p, U, tv, st)
    try:
        del tv
        y = torch.ones(V, 4, 3, 1, dtype=torch.complex64, device="cuda") if use else None
        x = torch.zeros_like(y) if use else None
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        amg.amg_setup_fine(h, U, st)
        torch.cuda.synchronize()
        if use:
            amg.amg_sap(h, y, x, 1, 1, 1, st)
            torch.cuda.synchronize()
        held = free - torch.cuda.mem_get_info()[0]
        assert amg.amg_sync_status(h) == amg.AMG_OK
        return held, V
    finally:
        amg.amg_destroy(h)
        torch.cuda.empty_cache()


def test_no_copies_without_the_smoother():
    """An odd coarse extent: only D can run, and nothing is held for the smoother."""
    held, V = _held((12, 16, 16, 16), (4, 4, 4, 4), 64, False)
    assert held < 512 * V + SLACK


def test_copies_kept():
    held, V = _held((16, 16, 16, 16), (4, 4, 4, 4), 16, True)
    assert abs(held - (512 * V + 192 * 16 * V)) < SLACK


def test_large_lattice_keeps_one_column():
    """Above 11.2 million sites one column's copies exceed 2 GB; they are kept between calls all the same."""
    held, V = _held((48, 48, 48, 112), (4, 4, 4, 4), 1, True)
    assert 192 * V > 2 << 30
    assert abs(held - (512 * V + 192 * V)) < SLACK


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_outer_solve_gets_the_smoothers_memory(prec):
    """Free memory that holds the outer solve's workspace only together with what the smoother holds for its speed."""
    import paper_1512_04506_gb300 as amg
    L, B, restart, max_nrhs = (24, 24, 24, 24), (4, 4, 4, 4), 30, 32 if prec == "fp32" else 1
    V, z = 24 ** 4, 8 if prec == "fp32" else 16
    pr, ct = (amg.AMG_FP32, torch.complex64) if prec == "fp32" else (amg.AMG_FP64, torch.complex128)
    need, held = (2 * restart + 2) * V * 12 * z, 192 * 32 * V if prec == "fp32" else 1056 * V
    from synth import device as sd
    st = torch.cuda.current_stream()
    U, tv, f = sd.links(71, 0.3, L), sd.test_vectors(71, 4, L), sd.fine_rhs(71, 1, L, ct)
    vp, out = amg.make_vcycle_params(0.05, 30, 50, 1, 2), []
    for full in (False, True):
        h, _ = amg.amg_setup_coarse(amg.make_params(L, B, 4, max_nrhs, -0.3, 1.0, pr, pr, pr), U, tv, st)
        try:
            amg.amg_setup_fine(h, U, st)
            u = torch.empty_like(f)
            amg.amg_vcycle(h, vp, f, u, 1, st)
            torch.cuda.synchronize()
            torch.cuda.empty_cache()
            fill = None
            if full:
                fill = torch.empty(torch.cuda.mem_get_info()[0] - need + held // 2, dtype=torch.uint8, device="cuda")
                assert torch.cuda.mem_get_info()[0] < need
            info = amg.amg_solve(h, vp, f, u, 1, tol=0.0, restart=restart, max_applies=3, stream=st)
            del fill
            out.append((info[0][1], u))
            assert amg.amg_sync_status(h) == amg.AMG_OK
        finally:
            amg.amg_destroy(h)
            torch.cuda.empty_cache()
    assert abs(out[1][0] / out[0][0] - 1) < 1e-5
    assert torch.linalg.vector_norm(out[1][1] - out[0][1]) < 1e-5 * torch.linalg.vector_norm(out[0][1])


def test_out_of_memory_is_reported_once():
    """An outer solve without memory for its workspace: the call fails, the next one does not."""
    import paper_1512_04506_gb300 as amg
    from synth import device as sd
    L, st = (24, 24, 24, 24), torch.cuda.current_stream()
    U, f = sd.links(73, 0.3, L), sd.fine_rhs(73, 1, L, torch.complex128)
    pr = amg.AMG_FP64
    h, _ = amg.amg_setup_coarse(amg.make_params(L, (4, 4, 4, 4), 2, 1, -0.3, 1.0, pr, pr, pr), U, sd.test_vectors(73, 2, L), st)
    try:
        amg.amg_setup_fine(h, U, st)
        vp, u = amg.make_vcycle_params(0.05, 30, 50, 1, 2), torch.empty_like(f)
        amg.amg_vcycle(h, vp, f, u, 1, st)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        fill = torch.empty(torch.cuda.mem_get_info()[0] - (1 << 30), dtype=torch.uint8, device="cuda")
        with pytest.raises(amg.AmgError) as e:  # 3.9 GB
            amg.amg_solve(h, vp, f, u, 1, tol=0.0, restart=30, max_applies=3, stream=st)
        assert e.value.status == amg.AMG_ERR_OOM
        amg.amg_dirac_apply(h, f, u, 1, st)
        amg.amg_vcycle(h, vp, f, u, 1, st)
        assert amg.amg_sync_status(h) == amg.AMG_OK
        del fill
    finally:
        amg.amg_destroy(h)
        torch.cuda.empty_cache()

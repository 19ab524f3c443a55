"""FP32 fine operator and smoother near the ends of the FP32 range.

D is linear and a minimal-residual step does not depend on the scale, so a power of two in the vectors passes through
to the last bit as long as D psi, D x and the sums of squares of the block stay finite.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from test_gpu_fine import Fine  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [1, 2, 3])
def test_dirac_large(nrhs):
    """A source whose D psi reaches the upper half of the FP32 range."""
    import paper_1512_04506_gb300 as amg
    c = Fine(amg, (8, 8, 8, 8), (4, 4, 4, 4), 1, 841, "fp32", max_nrhs=nrhs)
    try:
        psi = torch.zeros(c.V, 4, 3, nrhs, dtype=c.ctype, device="cuda")
        psi[5, 1, 2] = 1.5
        out, big = torch.empty_like(psi), torch.empty_like(psi)
        amg.amg_dirac_apply(c.h, psi, out, nrhs, c.stream)
        top = float(torch.view_as_real(out).abs().max())
        k = 2.0 ** np.floor(np.log2(3.4e38 / top))
        amg.amg_dirac_apply(c.h, psi * k, big, nrhs, c.stream)
        assert torch.isfinite(torch.view_as_real(big)).all()
        assert torch.equal(big, out * k)
    finally:
        c.close()


@pytest.mark.parametrize("B", [(4, 4, 4, 4), (2, 2, 2, 2)], ids=["4^4", "2^4"])
def test_sap_large(B):
    """<B rho, B rho> up to the power of two below the largest FP32 number."""
    import paper_1512_04506_gb300 as amg
    c = Fine(amg, (8, 8, 8, 8), B, 1, 843, "fp32", max_nrhs=1)
    try:
        y = torch.zeros(c.V, 4, 3, 1, dtype=c.ctype, device="cuda")
        y[0, 1, 2] = 1.0
        x = torch.zeros_like(y)
        amg.amg_sap(c.h, y, x, 1, 1, 1, c.stream)
        d = torch.empty_like(y)
        amg.amg_dirac_apply(c.h, y, d, 1, c.stream)
        # 1.001 |D y|^2 k^2 < 2^128 bounds |B y k|^2
        k = 2.0 ** np.floor((128 - np.log2(1.001 * float((d.abs() ** 2).sum()))) / 2)
        big = torch.zeros_like(y)
        amg.amg_sap(c.h, y * k, big, 1, 1, 1, c.stream)
        assert torch.equal(big, x * k)
    finally:
        c.close()

"""Launch geometry and fused diagnostics at the heights and sizes they can be given."""
import numpy as np
import pytest

from tests.conftest import has_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module")
def P():
    import paper_1802_01272_gb300 as P
    P.lib()
    return P


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("Lx,Ly,row_block", [(112, 1024, 1024), (112, 1024, 256), (113, 1000, 512)])
def test_fused_mass_is_as_exact_for_any_row_block(P, precision, Lx, Ly, row_block):
    """Mass of a uniform state from step_diag.  A partial FP32 sum of n values c is off by at
    most n 2^-24 of itself; a lane adds up at most 64 nodes, so the bar is 64 x 2^-24 of the sum
    of rho - rho_ref.  c = 1 + 2^-16 - 2^-19: sums of 256 and more lose almost half a unit in
    the last place with every node, all in one direction."""
    c = 1.0 + 2.0 ** -16 - 2.0 ** -19
    prec = {"fp32": P.LBM_FP32_SHIFTED, "fp16": P.LBM_FP16_SHIFTED}[precision]
    p = P.Params(Lx=Lx, Ly=Ly, T=1.0, rho_ref=1.0, precision=prec)
    with P.Lattice(p) as L:
        L.set_launch(row_block, 1)
        L.init_rho_u(np.full((Ly, Lx), 1.0 + c), np.zeros((Ly, Lx)), np.zeros((Ly, Lx)))
        fused = L.step_diag(1, 0.5)
        # FP16 rounds what it stores: the state before the stored rounding is what is summed
        exact = L.diagnostics(0.5)["mass"] if precision == "fp32" else None
        if exact is None:
            q = P.Params(Lx=Lx, Ly=4, T=1.0, rho_ref=1.0, precision=prec)
            with P.Lattice(q) as M:
                M.init_rho_u(np.full((4, Lx), 1.0 + c), np.zeros((4, Lx)), np.zeros((4, Lx)))
                exact = M.step_diag(1, 0.5)["mass"] * Ly / 4
    excess = exact - Lx * Ly
    assert abs(fused["mass"] - exact) <= 64 * 2.0 ** -24 * excess

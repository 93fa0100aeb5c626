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


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
def test_set_launch_is_what_runs_on_a_small_lattice(P, precision):
    """A geometry that was asked for is launched and reported: one CTA per strip and row block
    (three strips of 56 columns here, fewer items than SMs).  The state does not depend on it."""
    prec = {"fp32": P.LBM_FP32_SHIFTED, "fp16": P.LBM_FP16_SHIFTED}[precision]
    p = P.Params(Lx=128, Ly=64, rho_ref=1.0, precision=prec)
    y, x = np.mgrid[0:64, 0:128]
    rho = 1.0 + 0.01 * (((x * 31 + y * 17) % 29) / 29.0)
    want = None
    for row_block, ctas in ((0, 0), (16, 1), (24, 0), (32, 1), (64, 2), (8, 1), (4, 1)):
        with P.Lattice(p) as L:
            if row_block:
                k = L.set_launch(row_block, ctas)
                assert k["row_block"] == row_block and k["grid"] == 3 * -(-64 // row_block), k
            L.init_rho_u(rho, 0.02 * rho, -0.01 * rho)
            L.step(35)
            f = L.get_f()
            if row_block:
                assert L.kernel_info() == k
        want = f if want is None else want
        assert np.array_equal(f, want)


def test_tune_keeps_a_geometry_it_timed(P):
    """lbm_tune on a small lattice: either the geometry it began with or one of its candidates,
    which are launched undivided; set_launch with the reported row blocks then runs the same."""
    p = P.Params(Lx=128, Ly=64, rho_ref=1.0)
    with P.Lattice(p) as L:
        L.init_rho_u(np.ones((64, 128)), np.zeros((64, 128)), np.zeros((64, 128)))
        begun = L.kernel_info()
        k = L.tune(2)
        assert k == begun or k["grid"] == 3 * -(-64 // k["row_block"]), (begun, k)
        k = L.set_launch(16, 1)
        assert k["grid"] == 12
        t = L.tune(2)
        assert t["grid"] == 3 * -(-64 // t["row_block"]), t


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("regularize", [0, 1])
@pytest.mark.parametrize("Lx", [128, 113])
def test_set_launch_takes_three_ctas_per_sm(P, precision, regularize, Lx):
    """One, two or three CTAs per SM are accepted for every FP32 and FP16 kernel, four are not."""
    prec = {"fp32": P.LBM_FP32_SHIFTED, "fp16": P.LBM_FP16_SHIFTED}[precision]
    with P.Lattice(P.Params(Lx=Lx, Ly=4096, precision=prec, regularize=regularize)) as L:
        for ctas in (1, 2, 3):
            assert L.set_launch(4, ctas)["row_block"] == 4
        with pytest.raises(Exception):
            L.set_launch(4, 4)
        L.init_rho_u(np.ones((4096, Lx)), np.zeros((4096, Lx)), np.zeros((4096, Lx)))
        L.step(2)
        L.sync()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("row_block", [41, 1025, 2 ** 31 - 1])
def test_row_blocks_higher_than_the_lattice(P, precision, row_block):
    """Any row block from the lattice's height on is one block: the state is the default's."""
    prec = {"fp64": P.LBM_FP64, "fp32": P.LBM_FP32_SHIFTED, "fp16": P.LBM_FP16_SHIFTED}[precision]
    p = P.Params(Lx=130, Ly=41, rho_ref=1.0, precision=prec)
    y, x = np.mgrid[0:41, 0:130]
    rho = 1.0 + 0.01 * (((x * 31 + y * 17) % 29) / 29.0)
    out = []
    for rb in (0, row_block):
        with P.Lattice(p) as L:
            if rb:
                assert L.set_launch(rb, 1)["row_block"] == rb
            L.init_rho_u(rho, 0.02 * rho, -0.01 * rho)
            L.step(5)
            L.sync()
            out.append(L.get_f())
    assert np.array_equal(*out)

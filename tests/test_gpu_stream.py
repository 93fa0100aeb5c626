"""The step kernels at the sizes where their staging, rings, hand-overs and tiles
can go wrong, against the FP64 oracle: the narrowest lattices with tensor copies
(68, 72) and widths whose last strip holds 4 columns (116) or all of its 56
(112); heights under a batch, not a multiple of a batch or of half a batch; row
blocks that end in mid-batch; lattices staged value by value (odd widths, widths
under a strip); walls, reservoir, regularisation and every scheme."""
import numpy as np
import pytest

import synth
from tests.conftest import has_gpu
from tests.helpers import oracle_params

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]

STEPS = 3

# (Lx, Ly, order, limiter, walls, reservoir, regularize, row_block)
CASES = [
    (68, 4, 2, 0, 0, 0, 0, 0),
    (72, 5, 2, 0, 0, 0, 0, 0),
    (112, 18, 2, 0, 0, 0, 0, 0),
    (116, 19, 2, 0, 1, 0, 0, 0),
    (128, 8, 2, 0, 0, 0, 0, 0),
    (240, 33, 2, 0, 0, 0, 0, 7),      # row blocks that are no multiple of a batch
    (240, 34, 2, 0, 1, 0, 0, 6),
    (300, 300, 2, 0, 0, 1, 0, 0),     # R_BC = 22 nodes
    (300, 290, 2, 0, 0, 1, 1, 0),
    (176, 21, 2, 0, 1, 0, 1, 0),
    (176, 22, 1, 0, 1, 0, 0, 0),
    (176, 23, 2, 1, 0, 0, 0, 0),
    (176, 23, 2, 2, 0, 0, 0, 0),
    (37, 23, 2, 0, 0, 0, 0, 0),       # value by value
    (8, 3, 2, 0, 0, 0, 0, 0),
    (113, 2, 2, 0, 1, 0, 0, 0),
    (57, 30, 1, 0, 0, 0, 1, 5),
    (16, 8, 2, 0, 0, 0, 0, 0),        # one tile of the FP64 collision, and one node more
    (17, 9, 2, 0, 0, 0, 0, 0),
    (84, 40, 2, 0, 1, 0, 0, 33),      # a half strip of the FP64 advection without columns
    (128, 70, 2, 0, 0, 0, 0, 21),
]


@pytest.fixture(scope="module")
def P():
    import paper_1802_01272_gb300 as P
    P.lib()
    return P


def _fields(Lx, Ly):
    rho, ux, uy = synth.bubble(Lx, Ly, 1.55, 0.55, R=min(Lx, Ly) / 4 + 1, W=2.0)
    rho = rho * (1.0 + 1e-3 * synth.normal(3, Lx * Ly).reshape(Ly, Lx))
    ux = ux + 0.05 * synth.fourier_mode(Lx, Ly, 0.0, 1.0, 1, 2)
    uy = uy - 0.04 * synth.fourier_mode(Lx, Ly, 0.0, 1.0, 2, 1)
    return rho, ux, uy


def _params(P, case, precision):
    Lx, Ly, order, lim, walls, res, reg, _ = case
    lp = P.Params(Lx=Lx, Ly=Ly, precision=precision, ctu_order=order, limiter=lim, boundary=walls,
                  reservoir=res, regularize=reg, T=0.85, tau=2e-3, rho_ext=1.55, rho_ref=1.5)
    if walls:
        lp.shear_rate = 2 * 0.3 / (Ly * lp.ds)
    return lp


def _weights(P, O, op):
    return O.init_feq(op, np.ones((op.Ly, op.Lx)), np.zeros((op.Ly, op.Lx)),
                      np.zeros((op.Ly, op.Lx)))


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_against_oracle(P, oracle_mod, case, precision):
    """f after three steps.  FP32: a step rounds each stored value about ten times
    (advection, collision), the limited differences pass an error on at most
    threefold, and the force adds rounding of the same size: 3 steps x 10 x 3 x
    2^-24 = 5.4e-6 of the largest |f|; bar 1e-5.  FP16: one more rounding of every
    stored deviation per step, 2^-11 of the largest deviation each (and of the
    start's), passed on at most threefold.  FP64: 3 x 30 x 2^-53 = 1e-14; bar 1e-13."""
    O = oracle_mod
    prec = {"fp64": P.LBM_FP64, "fp32": P.LBM_FP32_SHIFTED, "fp16": P.LBM_FP16_SHIFTED}[precision]
    lp = _params(P, case, prec)
    rho, ux, uy = _fields(lp.Lx, lp.Ly)
    op = oracle_params(O, lp)
    f0 = O.init_feq(op, rho, ux, uy)
    with P.Lattice(lp) as L:
        if case[7]:
            L.set_launch(case[7], 0)
        L.init_rho_u(rho, ux, uy)
        L.step(STEPS)
        L.sync()
        fg = L.get_f()
    fo = O.step(op, f0, STEPS)
    err = np.abs(fg - fo).max()
    bar = (1e-13 if precision == "fp64" else 1e-5) * np.abs(fo).max()
    if precision == "fp16":
        # f - w rho_ref with w from f^eq at rest at T = 1 (= w rho)
        op1 = oracle_params(O, lp)
        op1.T = 1.0
        dev = np.abs(f0 - lp.rho_ref * _weights(P, O, op1)).max()
        bar += 3 * (STEPS + 1) * 2.0 ** -11 * dev
    assert err <= bar, (err, bar)


def test_many_lattices_in_one_launch(P, oracle_mod):
    """The batched kernel on lattices of the sizes above, each against the oracle."""
    from paper_1802_01272_gb300.binding import step_many
    O = oracle_mod
    cases = [c for c in CASES if c[2] == 2 and c[3] == 0 and not c[6] and c[0] % 4 == 0 and c[0] >= 68]
    lats, want = [], []
    for c in cases:
        lp = _params(P, c, P.LBM_FP32_SHIFTED)
        rho, ux, uy = _fields(lp.Lx, lp.Ly)
        op = oracle_params(O, lp)
        L = P.Lattice(lp)
        L.init_rho_u(rho, ux, uy)
        lats.append(L)
        want.append(O.step(op, O.init_feq(op, rho, ux, uy), STEPS))
    step_many(lats, STEPS)
    for c, L, fo in zip(cases, lats, want):
        fg = L.get_f()
        assert np.abs(fg - fo).max() <= 1e-5 * np.abs(fo).max(), c
        L.close()

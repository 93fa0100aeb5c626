"""The step kernels plane by plane, and over several work items per CTA.

Each plane of f is judged against its own scale: the planes of the fast velocities
hold a hundredth of the slow ones' values, so that one bar over all planes would
pass almost anything in them.  The bars are checked on the CPU to fail for a wrong
scheme, a plane group that was not advected, and a toggled regularisation."""
import numpy as np
import pytest

from tests.conftest import has_gpu
from tests.helpers import oracle_params
from tests.test_gpu_stream import CASES, STEPS, _fields, _params

gpu = [pytest.mark.gpu, pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module")
def P():
    import paper_1802_01272_gb300 as P
    return P


def _weights(O, op):
    one, zero = np.ones((op.Ly, op.Lx)), np.zeros((op.Ly, op.Lx))
    T, op.T = op.T, 1.0
    w = O.init_feq(op, one, zero, zero)  # f^eq at rest at T = 1 is w rho
    op.T = T
    return w


def _bars(O, op, f0, fo, rho_ref, precision):
    """Per plane.  FP32: a step rounds each value about ten times at the size of its plane's
    largest |f| (differences and sums of its own values, then the collision, whose terms are
    w_k times the same few numbers) and passes an error on at most threefold: 3 steps x 10 x 3
    x 2^-24 = 5.4e-6, bar 1e-5 of max |f_k|.  FP16: each stored deviation from w_k rho_ref is
    rounded once more per step and at the start, 2^-11 of the plane's largest, passed on at
    most threefold."""
    bar = 1e-5 * np.abs(fo).max(axis=(1, 2))
    if precision == "fp16":
        dev = np.abs(f0 - rho_ref * _weights(O, op)).max(axis=(1, 2))
        bar = bar + 3 * (STEPS + 1) * 2.0 ** -11 * dev
    return bar


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("case", CASES[::2], ids=lambda c: "x".join(map(str, c)))
def test_bars_tell_wrong_steps_apart(P, oracle_mod, case, precision):
    O = oracle_mod
    lp = _params(P, case, P.LBM_FP32_SHIFTED)
    op = oracle_params(O, lp)
    f0 = O.init_feq(op, *_fields(lp.Lx, lp.Ly))
    fo = O.step(op, f0, STEPS)
    bar = _bars(O, op, f0, fo, lp.rho_ref, precision)

    def seen(f):
        return (np.abs(f - fo).max(axis=(1, 2)) > bar).any()
    wrong = oracle_params(O, lp)
    wrong.ctu_order = 3 - wrong.ctu_order
    if lp.limiter == 0 or lp.ctu_order == 1:
        assert seen(O.step(wrong, f0, STEPS)), "order"
    wrong = oracle_params(O, lp)
    wrong.regularize = 1 - wrong.regularize
    if precision == "fp32":  # (in three steps it may stay below the rounding of FP16 storage)
        assert seen(O.step(wrong, f0, STEPS)), "regularisation"
    for group in range(4):
        stuck = fo.copy()
        stuck[4 * group:4 * group + 4] = f0[4 * group:4 * group + 4]
        assert seen(stuck), "group %d not stepped" % group


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
class TestPlanes:
    pytestmark = gpu

    def test_against_oracle(self, P, oracle_mod, case, precision):
        O = oracle_mod
        lp = _params(P, case, {"fp32": P.LBM_FP32_SHIFTED, "fp16": P.LBM_FP16_SHIFTED}[precision])
        rho, ux, uy = _fields(lp.Lx, lp.Ly)
        op = oracle_params(O, lp)
        f0 = O.init_feq(op, rho, ux, uy)
        fo = O.step(op, f0, STEPS)
        with P.Lattice(lp) as L:
            if case[7]:
                L.set_launch(case[7], 0)
            L.init_rho_u(rho, ux, uy)
            L.step(STEPS)
            L.sync()
            fg = L.get_f()
        err, bar = np.abs(fg - fo).max(axis=(1, 2)), _bars(O, op, f0, fo, lp.rho_ref, precision)
        assert (err <= bar).all(), (err / bar).round(2)


# (Lx, Ly, walls, reservoir, regularize, precision): six or seven strips, 60 row blocks and more
# of two rows, on one CTA per SM: every CTA takes two or three items, in other strips
SEVERAL = [(300, 121, 0, 0, 0, "fp32"), (300, 121, 1, 0, 0, "fp32"), (301, 120, 0, 0, 0, "fp32"),
           (301, 120, 1, 0, 0, "fp32"), (336, 333, 0, 1, 0, "fp32"), (300, 121, 1, 0, 1, "fp32"),
           (296, 121, 0, 0, 0, "fp16"), (296, 121, 1, 0, 0, "fp16"), (301, 121, 1, 0, 0, "fp16"),
           (300, 121, 1, 0, 0, "fp64"), (301, 121, 0, 0, 0, "fp64")]


@pytest.mark.parametrize("case", SEVERAL, ids=lambda c: "x".join(map(str, c)))
class TestSeveralItems:
    pytestmark = gpu

    def test_state_does_not_depend_on_the_launch(self, P, case):
        """Work items one after the other in a CTA (staging, rings and roles carried over from
        strip to strip and across the x seam) against one item per CTA: the same bits."""
        Lx, Ly, walls, res, reg, precision = case
        prec = {"fp64": P.LBM_FP64, "fp32": P.LBM_FP32_SHIFTED, "fp16": P.LBM_FP16_SHIFTED}[precision]
        lp = _params(P, (Lx, Ly, 2, 0, walls, res, reg, 0), prec)
        rho, ux, uy = _fields(Lx, Ly)
        out = []
        for launch in (None, (2, 1), (3, 1), (5, 2)):
            with P.Lattice(lp) as L:
                if launch:
                    L.set_launch(*launch)
                L.init_rho_u(rho, ux, uy)
                L.step(5)
                L.sync()
                out.append(L.get_f())
        for f in out[1:]:
            assert np.array_equal(f, out[0])


class TestManyItems:
    pytestmark = gpu

    @pytest.mark.parametrize("order,limiter,regularize",
                             [(2, 0, 0), (1, 0, 0), (2, 1, 0), (2, 2, 0), (2, 0, 1), (1, 0, 1)])
    def test_more_strips_than_ctas_in_one_launch(self, P, order, limiter, regularize):
        """One batched launch over lattices of 60 to 61 strips each, 483 in all: more items than
        resident CTAs, whose segments come from lattices of different widths, heights and walls.
        The plain collision gives the bits of each lattice stepped alone, the regularised one
        the same to FP32 rounding of its moments (bar 1e-6 of the largest |f|)."""
        from paper_1802_01272_gb300.binding import step_many
        specs = [(3360, 24, 0), (3364, 23, 1), (3416, 24, 0), (3372, 21, 1), (3360, 24, 1), (3376, 22, 0),
                 (3380, 24, 0), (3408, 23, 1)]
        alone, many = [], []
        for Lx, Ly, walls in specs:
            lp = _params(P, (Lx, Ly, order, limiter, walls, 0, regularize, 0), P.LBM_FP32_SHIFTED)
            for lats in (alone, many):
                L = P.Lattice(lp)
                L.init_rho_u(*_fields(Lx, Ly))
                lats.append(L)
        for L in alone:
            L.step(4)
        step_many(many, 4)
        for A, B in zip(alone, many):
            a, b = A.get_f(), B.get_f()
            if regularize:
                assert np.abs(a - b).max() <= 1e-6 * np.abs(a).max()
            else:
                assert np.array_equal(a, b)
            A.close()
            B.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("Lx,Ly", [(128, 24), (37, 22)])
class TestUnalignedFields:
    pytestmark = gpu

    def test_device_fields_on_odd_addresses(self, P, precision, Lx, Ly):
        """Device fields need only the alignment of a double: fields that start 8 bytes past a
        16-byte boundary give the state and the moments of aligned ones."""
        import torch
        prec = {"fp64": P.LBM_FP64, "fp32": P.LBM_FP32_SHIFTED, "fp16": P.LBM_FP16_SHIFTED}[precision]
        lp = _params(P, (Lx, Ly, 2, 0, 0, 0, 0, 0), prec)
        fields = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in _fields(Lx, Ly)]
        n = Lx * Ly
        got = []
        for odd in ((0, 0, 0), (1, 0, 0), (0, 0, 1), (1, 1, 1)):
            src = [torch.empty(n + 2, device="cuda", dtype=torch.float64)[o:o + n].view(Ly, Lx) for o in odd]
            dst = [torch.empty(n + 2, device="cuda", dtype=torch.float64)[o:o + n].view(Ly, Lx) for o in odd]
            for s, v in zip(src, fields):
                s.copy_(v)
            torch.cuda.synchronize()
            with P.Lattice(lp) as L:
                L.init_rho_u_device(*src)
                L.step(2)
                L.moments_device(*dst)
                L.sync()
                got.append([L.get_f()] + [d.cpu().numpy() for d in dst])
        for g in got[1:]:
            for a, b in zip(g, got[0]):
                assert np.array_equal(a, b)

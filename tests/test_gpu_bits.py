"""The FP32 and FP16 steps, the start from equilibrium and the read-outs, bit for bit:
digests of their results as recorded on a GB300 with the step kernel of commit a50bef1
(one kernel body in which all warps advect, then collide).  A kernel laid out otherwise
does the same operations on every node in the same order, so that runs can be compared
and continued across versions, and no output moves away from the FP64 step's.

The inputs are made of sums, products and quotients only, which every machine rounds
alike."""
import hashlib
import json
import os

import numpy as np
import pytest

from tests.conftest import has_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not has_gpu(), reason="needs a CUDA GPU")]

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "step_bits.json")

# name: (precision, Lx, Ly, steps, parameters)
SHEARED = dict(T=0.8, tau=1e-2, boundary=1, uw=0.6)
CASES = {
    "ctu2": ("fp32", 240, 97, 40, dict()),
    "ctu2-ragged": ("fp32", 113, 70, 21, dict()),
    "ctu2-low": ("fp32", 128, 3, 17, dict()),
    "ctu2-walls": ("fp32", 176, 64, 33, dict(boundary=1, uw=0.4)),
    "ctu1": ("fp32", 300, 83, 20, dict(ctu_order=1)),
    "ctu1-ragged-walls": ("fp32", 67, 30, 20, dict(ctu_order=1, boundary=1, uw=0.4)),
    "limiter-1": ("fp32", 124, 40, 20, dict(limiter=1)),
    "limiter-2-walls": ("fp32", 124, 41, 20, dict(limiter=2, boundary=1, uw=0.2)),
    "reservoir": ("fp32", 400, 384, 12, dict(reservoir=1, T=0.8)),
    "reservoir-ctu1-ragged": ("fp32", 401, 390, 12, dict(reservoir=1, T=0.8, ctu_order=1)),
    "sheared-bubble": ("fp32", 1024, 512, 100, SHEARED),
    "fp16": ("fp16", 240, 97, 40, dict()),
    "fp16-walls": ("fp16", 512, 256, 20, SHEARED),
    "fp16-ragged-ctu1": ("fp16", 113, 70, 20, dict(ctu_order=1)),
    "fp16-reservoir": ("fp16", 400, 384, 12, dict(reservoir=1, T=0.8)),
}


def fields(Lx, Ly):
    """A bubble (a rational profile), density noise, a flow of triangle waves."""
    y, x = np.mgrid[0:Ly, 0:Lx].astype(np.int64)
    d2 = ((x - Lx // 2) ** 2 + (y - Ly // 2) ** 2).astype(np.float64)
    r2 = float(max(min(Lx, Ly) // 4, 1)) ** 2
    noise = ((x * 7919 + y * 104729 + (x * y) % 9973) % 10007).astype(np.float64) / 10007.0 - 0.5
    rho = (0.25 + 1.6 * d2 * d2 / (d2 * d2 + r2 * r2)) * (1.0 + 0.004 * noise)

    def wave(i, n):
        t = (i % n).astype(np.float64) / n
        return np.where(t < 0.5, 4.0 * t - 1.0, 3.0 - 4.0 * t)
    ux = 0.15 * wave(x + 2 * y, max(Lx, 8)) + 0.05
    uy = 0.15 * wave(2 * x + y, max(Ly, 8)) - 0.04
    return rho, ux, uy


def params(P, precision, Lx, Ly, kw):
    kw = dict(kw)
    uw = kw.pop("uw", 0.0)
    p = P.Params(Lx=Lx, Ly=Ly, **{**dict(T=0.85, tau=2e-3, rho_ext=1.85, rho_ref=1.85), **kw},
                 precision={"fp32": P.LBM_FP32_SHIFTED, "fp16": P.LBM_FP16_SHIFTED}[precision])
    p.shear_rate = 2.0 * uw / (Ly * p.ds)
    return p


def digest(*arrays):
    h = hashlib.sha256()
    for a in arrays:
        h.update((np.ascontiguousarray(a, dtype="<f8") + 0.0).tobytes())  # (-0 as 0)
    return h.hexdigest()[:24]


def record(P, name):
    """Digests of the state at the start, after the first and after all steps, of its moments
    and of the bubble record's densities."""
    precision, Lx, Ly, steps, kw = CASES[name]
    with P.Lattice(params(P, precision, Lx, Ly, kw)) as L:
        L.init_rho_u(*fields(Lx, Ly))
        start = L.get_f()
        L.step(1)
        first = L.get_f()
        L.step(steps - 1)
        L.sync()
        d = L.diagnostics(1.0)
        return {"start": digest(start), "first": digest(first), "f": digest(L.get_f()),
                "moments": digest(*L.moments()),
                "record": [float(d[k]).hex() for k in ("rho_center", "rho_min", "rho_max")] + [int(d["nb"])]}


def record_many(P):
    from paper_1802_01272_gb300.binding import step_many
    lats = []
    for Lx, Ly, kw in ((256, 256, {}), (128, 64, {}), (512, 100, dict(boundary=1, uw=0.3)), (68, 300, {}),
                       (400, 384, dict(reservoir=1, T=0.8))):
        L = P.Lattice(params(P, "fp32", Lx, Ly, kw))
        L.init_rho_u(*fields(Lx, Ly))
        lats.append(L)
    step_many(lats, 19)
    out = [digest(L.get_f()) for L in lats]
    for L in lats:
        L.close()
    return out


@pytest.fixture(scope="module")
def P():
    import paper_1802_01272_gb300 as P
    P.lib()
    return P


@pytest.fixture(scope="module")
def golden():
    with open(GOLDEN) as f:
        return json.load(f)


@pytest.mark.parametrize("name", list(CASES))
def test_step_bits(P, golden, name):
    assert record(P, name) == golden[name]


def test_step_many_bits(P, golden):
    assert record_many(P) == golden["many"]

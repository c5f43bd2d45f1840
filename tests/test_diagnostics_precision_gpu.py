"""Diagnostics carry the precision of FP64 sums.

The state has rho = 1 and no colour gradient, and a few nodes whose moving
populations are one link each, so that the momentum of a node and its u are FP32
values the test knows exactly.  Tolerances: an FP64 sum of eight terms rounds
eight times, each by at most 2^-53 of the sum of their magnitudes (additions of
zero are exact); max|u| is the square root (2^-53) of an FP64 sum of two exact
squares (2^-53, halved by the root)."""
import math

import numpy as np
import pytest

from paper_2005_04642_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines too
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2005_04642_gb300 import cmrt as cm  # noqa: E402

cm.load()

NX, NY = 4, 8192  # a column of many rows per CTA


def _lattice(order):
    return cm.Lattice(I.base_params(NX, NY, stencil_order=order), None, None)


def _state():
    pops = np.zeros((2, 9, NY, NX), np.float32)
    pops[0, 0] = 1.0
    return pops


# eight momenta whose cancelling FP32 pair sum is off by 2^-46 of their magnitudes
TERMS = np.array([2.4680748555994114e-09, -0.13798120617866516, 1.6285359834000701e-06, 2.423831801934284e-09,
                  -0.0006519687594845891, -0.004335709381848574, -7.539885700680315e-05, -2.4680748555994114e-09],
                 np.float32)


@pytest.mark.parametrize("order", [2, 6])
@pytest.mark.parametrize("axis", [0, 1], ids=["x", "y"])
def test_momentum_of_terms_of_unequal_size(axis, order):
    plus, minus = ((8, 4), (2, 6))[axis]
    want = math.fsum(TERMS.tolist())
    bound = 8 * 2.0**-53 * math.fsum(abs(v) for v in TERMS.tolist())
    lat = _lattice(order)
    for shift in range(16):  # wherever the rows of a CTA and its groups of rows begin
        pops = _state()
        for k, v in enumerate(TERMS):
            pops[0, plus if v > 0 else minus, 200 + shift + k, 1] = abs(v)
        lat.set_populations(pops)
        got = lat.diagnostics()
        assert abs(got["mom_" + "xy"[axis]] - want) <= bound, shift
        assert got["mom_" + "yx"[axis]] == 0.0
    lat.close()


# pairs of velocities with |u|^2 within 2^-47 of each other
CLOSE = [("0x1.d767840000000p-26", "0x1.3419520000000p-32", "0x1.d767860000000p-26", "0x1.33e8580000000p-32"),
         ("0x1.abfcea0000000p-26", "0x1.933d600000000p-33", "0x1.abfcec0000000p-26", "0x1.92b56e0000000p-33")]


@pytest.mark.parametrize("order", [2, 6])
@pytest.mark.parametrize("swap", [False, True])
@pytest.mark.parametrize("pair", CLOSE, ids=["first_faster", "second_faster"])
def test_fastest_of_two_nodes_of_nearly_one_speed(pair, swap, order):
    v = [float.fromhex(x) for x in pair]
    nodes = [(v[0], v[1]), (v[2], v[3])]
    want = max(math.sqrt(x * x + y * y) for x, y in nodes)
    pops = _state()
    for k, (x, y) in enumerate(nodes[::-1] if swap else nodes):
        pops[0, 8, 201 + k, 1] = x
        pops[0, 2, 201 + k, 1] = y
    lat = _lattice(order)
    lat.set_populations(pops)
    f = lat.fields()
    assert sorted(f["ux"].unique().tolist()) == sorted({0.0, v[0], v[2]})  # u is the momentum
    assert lat.diagnostics()["umax"] == pytest.approx(want, rel=2.0**-51, abs=0.0)
    lat.close()

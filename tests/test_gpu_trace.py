"""Traced curves against the CPU oracle where the tracing takes its different
routes: 4 lanes per curve and 2 (many curves), field magnitudes inside and
outside the range of the fast unit direction (|beta|^2 in 2^-60 .. 2^60),
flows almost along a grid axis, and points on grid lines.

Discrete structure exactly; coordinates to 1e-12 in index units, as in
test_gpu_parity.py (the operations are the same, correctly rounded)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_11041_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _field(nx, ny, kind, scale):
    X, Y = W.node_coords(nx, ny)
    if kind == "sheared":
        b1, b2 = W.sheared_beta(nx, ny)
    elif kind == "axis":      # along x to one part in 10^3, on grid lines at the left
        b1, b2 = np.ones((ny, nx)), 1e-3 * np.sin(3.0 * X) ** 2
    else:                     # rotating
        b1, b2 = -5.0 * (Y + 1.0), 5.0 * (X + 1.0)
    return b1 * scale, b2 * scale


@pytest.mark.parametrize("nx,ny,kind,scale", [
    (65, 65, "sheared", 1.0), (3000, 40, "sheared", 1.0), (90, 70, "axis", 1.0), (61, 61, "rotating", 1.0),
    (48, 48, "sheared", 1e-12), (48, 48, "sheared", 1e12), (48, 48, "rotating", 2.0 ** 29),
    (48, 48, "rotating", 2.0 ** -31),
])
def test_traced_curves_match_oracle(nx, ny, kind, scale):
    from paper_2411_11041_gb300 import Solver
    b1, b2 = _field(nx, ny, kind, scale)
    p = W.Problem(nx, ny, 1e-2, 1.0, b1, b2, np.ones((ny, nx)), W.make_mask("square", nx, ny),
                  y1=(ny - 1) / (nx - 1))
    o, s = O.Oracle(p), Solver(p)
    for fam in (0, 1):
        a, b = o.lines(fam), s.lines(fam)
        assert np.array_equal(a["off"], b["off"])
        assert np.abs(a["xi"] - b["xi"]).max() <= 1e-12
        assert np.abs(a["eta"] - b["eta"]).max() <= 1e-12
        np.testing.assert_allclose(b["h"], a["h"], rtol=1e-13)
    if (nx, ny) == (3000, 40):  # enough curves for two lanes each
        assert len(o.lines(0)["off"]) + len(o.lines(1)["off"]) > 8 * 3 * 152

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


KERNEL = r"""
#include <cuda_runtime.h>
#include "unit_component.cuh"
__global__ void k_unit(const double* num, const double* s, double* out, unsigned char* bad, long n)
{
    const long k = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (k >= n) return;
    bool b = false;
    out[k] = unit_component(num[k], s[k], b);
    bad[k] = b;
}
extern "C" int unit(const double* num, const double* s, double* out, unsigned char* bad, long n)
{
    k_unit<<<(unsigned)((n + 255) / 256), 256>>>(num, s, out, bad, n);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? (int)e : (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def unit(tmp_path_factory):
    """unit_component of the tracing on arrays, compiled with its flags."""
    import ctypes as C
    import subprocess

    import torch

    from paper_2411_11041_gb300 import build as B
    d = tmp_path_factory.mktemp("unit")
    (d / "unit.cu").write_text(KERNEL)
    subprocess.run([B.NVCC, *B.ARCH, *B.COMMON, *B.UNITS["geometry.cu"], "-I", B.CSRC, "-shared", "-o",
                    str(d / "unit.so"), str(d / "unit.cu")], check=True)
    f = C.CDLL(str(d / "unit.so")).unit
    f.argtypes = [C.c_void_p] * 4 + [C.c_long]

    def call(num, s):
        a = [torch.as_tensor(v, dtype=torch.float64, device="cuda:0").contiguous() for v in (num, s)]
        out = torch.empty_like(a[0])
        bad = torch.empty(a[0].shape, dtype=torch.uint8, device="cuda:0")
        torch.cuda.synchronize()
        assert f(*(t.data_ptr() for t in (*a, out, bad)), out.numel()) == 0
        return out.cpu().numpy(), bad.cpu().numpy()

    return call


@pytest.mark.parametrize("case", ["random", "range", "edges"])
def test_unit_component_is_num_over_sqrt(unit, case):
    """num / sqrt(s) as numpy's correctly rounded sqrt and / give it: the two
    roundings' arguments are within 2^-85, so of 2^24 values 2^-6 are expected to
    differ and more than one is a fault; a difference is one ulp at most."""
    rng = np.random.default_rng(11)
    n = 1 << 24
    if case == "random":    # a field's components: num^2 is a part of s
        v, w = rng.normal(size=n), rng.normal(size=n)
        num, s = v, v * v + w * w
    elif case == "range":   # the whole fast range and beyond both ends of it
        s = rng.uniform(1.0, 2.0, n) * 2.0 ** rng.integers(-64, 64, n)
        num = rng.uniform(-1.0, 1.0, n) * np.sqrt(s)
    else:                   # neighbours of powers of two, both ends of the range, squares
        e = 2.0 ** np.arange(-62, 63)
        s = e.copy()
        up, dn = e.copy(), e.copy()
        for _ in range(2000):
            up, dn = np.nextafter(up, np.inf), np.nextafter(dn, 0.0)
            s = np.concatenate([s, up, dn]) if s.size < 2_000_000 else s
        q = rng.integers(1, 1 << 26, 200000).astype(np.float64)
        s = np.concatenate([s, q * q])
        num = rng.uniform(-1.0, 1.0, s.size) * np.sqrt(s)
        num[::7] = 0.0
    got, bad = unit(num, s)
    want = num / np.sqrt(s)
    assert not bad.any()
    diff = np.flatnonzero(got != want)
    assert diff.size <= 1, (diff.size, num[diff[:5]], s[diff[:5]])
    assert (np.abs(got - want)[diff] <= np.spacing(np.abs(want[diff]))).all()


def test_unit_component_of_no_direction(unit):
    inf, nan = np.inf, np.nan
    num = np.array([0.0, 1.0, 1.0, 1.0, 1.0, inf, 0.0])
    s = np.array([0.0, -1.0, nan, inf, 5e-324, inf, -0.0])
    got, bad = unit(num, s)
    with np.errstate(all="ignore"):
        want = num / np.sqrt(s)
    assert bad.tolist() == [1, 1, 1, 0, 0, 0, 1]
    assert np.array_equal(got, want, equal_nan=True)

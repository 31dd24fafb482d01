"""The mass sums (mclbm_mass) of given populations: no fewer bits than nine FP64 additions per node, and
the infinities and large values that those can hold."""
import ctypes as C
import math

import numpy as np
import pytest

from tests import _parity as P

pytestmark = pytest.mark.gpu

N = 2  # the smallest lattice: every thread that has a node has one


@pytest.fixture(scope="module", autouse=True)
def _built():
    P.ensure_built()


def _mass(planes):
    """Return code and sums of a lattice whose node (1, 0) holds the given 18 values, the others 0."""
    import torch
    import paper_1511_04552_gb300 as m
    c = m.Cavity(N, N, 1e3, 6.2, 0.02, 20e-9)
    s = np.zeros((27, N, N), np.float32)
    s[:18, 0, 1] = planes
    c.state_set(torch.from_numpy(s).cuda())
    w, p = C.c_double(), C.c_double()
    rc = m.lib().mclbm_mass(c._h, C.byref(w), C.byref(p))
    k = c.consts()
    return rc, (w.value, p.value), (N * N * k["rho_w0"], N * N * k["rho_p0"])


@pytest.mark.parametrize("seed", range(8))
def test_sums_that_fp64_holds_are_exact(seed):
    """Values whose FP64 sum is exact in any order (all bits within 2^0 .. 2^-52): the two largest errors
    of an FP32 sum are themselves too long for their sum in FP32."""
    r = np.random.default_rng(seed)
    v = np.zeros((2, 9), np.float32)
    for s in range(2):
        odd = (r.integers(1 << 22, 1 << 23, size=2) * 2 + 1).astype(np.float64)  # 24 bits
        v[s, 0], v[s, 1] = 1.0, odd[0] * 2.0 ** -49
        v[s, 2], v[s, 3] = 0.25, odd[1] * 2.0 ** -51
    rc, got, offset = _mass(v.reshape(18))
    want = [math.fsum(x.astype(np.float64)) for x in v]
    assert rc == 0
    assert got[0] == want[0] + offset[0] and got[1] == want[1] + offset[1]


def test_values_whose_fp32_sum_overflows():
    v = np.zeros(18, np.float32)
    v[:9], v[9:] = 2e38, 1.0
    v[0] = -3e38
    rc, got, offset = _mass(v)
    assert rc == 0
    assert got[0] == math.fsum(v[:9].astype(np.float64)) + offset[0] and got[1] == 9.0 + offset[1]


@pytest.mark.parametrize("value,other", [(np.inf, 1.0), (-np.inf, 1.0), (np.inf, -np.inf),
                                         (np.nan, 1.0)])
def test_infinities_and_nan(value, other):
    import paper_1511_04552_gb300 as m
    v = np.zeros(18, np.float32)
    v[3], v[5], v[12] = value, other, 0.5
    rc, got, offset = _mass(v)
    assert rc == m.binding.EDIVERGED
    with np.errstate(invalid="ignore"):
        want = float(np.float64(value) + np.float64(other))
    assert got[0] == want or (math.isnan(got[0]) and math.isnan(want))
    assert got[1] == 0.5 + offset[1]

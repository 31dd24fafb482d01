"""The initial fill from caller fields: its pairs of FP32 numbers with an FP64 second way store the
values that an FP64 evaluation of Eqs 26-27 rounds to."""
import numpy as np
import pytest

import workloads
from tests import _parity as P

pytestmark = pytest.mark.gpu

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)


@pytest.fixture(scope="module", autouse=True)
def _built():
    P.ensure_built()


def _fp64_state(w, nx, c, fr, sets):
    w = w.astype(np.float64)
    ux, uy, th, phi = w[:4]
    drw = (w[4] if len(w) == 5 else 1.0 - phi) - c["rho_w0"]
    drp = phi / fr - c["rho_p0"]
    dth = th - (0.5 - (np.arange(nx) + 0.5) / nx)
    parts = [(drw, c["rho_w0"] + drw), (drp, c["rho_p0"] + drp)] + [(dth, th)] * sets
    usq = 1.5 * (ux * ux + uy * uy)
    out = []
    for d, r in parts:
        for q in range(9):
            eu = EX[q] * ux + EY[q] * uy
            out.append((P.W[q] * (d + r * (eu * (3.0 + 4.5 * eu) - usq))).astype(np.float32))
    return np.stack(out)


@pytest.mark.parametrize("sets", [1, 2])
@pytest.mark.parametrize("density", [False, True])
@pytest.mark.parametrize("nx,ny,phi,kind", [
    (67, 33, 0.03, "noise"),
    (128, 40, 0.02, "smooth"),
    (33, 32, 0.04, "conduction"),  # theta and phi as close to the rest state as FP32 gets
    (40, 40, 0.0, "noise"),        # no particles: exact zeros
    (40, 31, 0.03, "tiny"),        # terms whose low parts underflow FP32
    (50, 50, 0.03, "huge"),        # squares that overflow FP32, and a NaN
])
def test_warm_fill_rounds_like_fp64(nx, ny, phi, kind, density, sets):
    import torch
    import paper_1511_04552_gb300 as m
    w = workloads.perturbed_rest_fields(nx, ny, phi, seed=3)
    x, y = np.meshgrid(np.linspace(0, 1, nx), np.linspace(0, 1, ny))
    if kind == "smooth":
        w[0], w[1], w[3] = 0.03 * np.sin(6 * y + x), 0.02 * np.cos(5 * x), phi * (1 + x * y / 100)
    elif kind == "conduction":
        w[0], w[1], w[2], w[3] = 0.01, -0.02, 0.5 - (np.arange(nx) + 0.5) / nx, phi
    elif kind == "tiny":
        w[0] *= 1e-33
        w[1] *= 1e-20
    elif kind == "huge":
        w[0] *= 1e22
        w[2, 4, 5] = np.nan
    if density:
        w = np.concatenate([w, (1.0 - w[3:4]) * (1.0 + 1e-3 * np.sin(7 * x))[None]])
    w = np.ascontiguousarray(w, dtype=np.float32)
    cav = m.Cavity(nx, ny, 1e4, 6.2, phi, 30e-9, thermal_sets=sets)
    got = cav.init(warm=torch.from_numpy(w).cuda()).state_get().cpu().numpy()
    with np.errstate(all="ignore"):
        exp = _fp64_state(w, nx, cav.consts(), cav.props.rho_f / cav.props.rho_p, sets)
    # numpy and the device may contract FP64 products differently (2^-53): a rounding to FP32
    # then differs in one of 2^28 values
    np.testing.assert_array_equal(got, exp)

"""States at the limits of the approximations, in the mixed and the FP64 form:
far from the origin, groups on a line, a strong vortex at the facing end of a
group, domains many core sizes wide, tiny circulations.

References are the FP64 form (fewer than 256 particles, or the full-jet flag:
no approximation) or the oracle.  Tolerances, unless stated at a test: mixed
velocities 2e-6 and moment rates 5e-6 (growing with the order beyond 6) as
everywhere, each particle against the scale of its own pair terms; FP64 1e-12.
"""
import math

import numpy as np
import pytest

import mmvm_inputs
from oracle.rhs import rhs_regrouped
from tests.parity_util import (abs_scale_rows, rhs_error, rhs_error_cond, rhs_error_rows,
                               vel_error, vel_error_cond, vel_error_rows, weights)

pytestmark = pytest.mark.gpu

X_FAR = (20.0, 32.0, 40.0, 50.0, 58.0, 66.0, 74.0, 80.0, 88.0)  # near/far threshold by order
LAM = math.sqrt(0.5)  # core units are the units of length


@pytest.fixture(scope="module")
def mm():
    import paper_1010_2475_gb300 as mm

    mm.load_library()
    return mm


def _rhs(mm, order, lam, x, m, precision, flags=0):
    with mm.Context(order, lam, 1e-3, precision, flags=flags) as ctx:
        ctx.set_state(x, m, 0.0)
        return ctx.rhs()


def _moments(gamma, order, lam, rng, amp=0.1):
    """Circulations gamma, moments of order >= 2 `amp` of them in the weighted norm."""
    m = np.zeros((len(gamma), mmvm_inputs.n_moments(order)))
    m[:, 0] = gamma
    if order >= 2:
        m[:, 3:] = amp * rng.normal(size=m[:, 3:].shape) * gamma[:, None] \
            / np.sqrt(weights(order, lam)[3:])
    return m


def _tol(order):
    return 5e-6 * max(1.0, order / 6.0)


@pytest.mark.parametrize("order", [0, 2, 4, 6, 8])
@pytest.mark.parametrize("state", ["disk", "patches", "clusters"])
def test_fp64_shortcut_far_from_the_origin(mm, order, state):
    """The test for the point-vortex form works on differences of positions:
    at 2e8 units one FP32 step of a coordinate is 16 units, wider than the far
    threshold.  `clusters`: the targets of one warp lie in several clusters 1e8
    units apart, each around a value half way between two FP32 numbers."""
    rng = np.random.default_rng(order)
    n = 504
    if state == "disk":
        x = 8.0 * rng.uniform(-1.0, 1.0, size=(n, 2)) + [2e8 + 8.0, -2e8]
    elif state == "patches":
        x = mmvm_inputs.two_patches(n=n, order=order, sigma=0.1, seed=order).x * 7.0 + [-4e8, 3e6]
    else:
        x = 4.0 * rng.uniform(-1.0, 1.0, size=(n, 2))
        c = (2.0 ** 27 * (1 + np.arange(24))).astype(np.float32)
        x[:, 0] += np.repeat(c.astype(np.float64) + 0.5 * np.spacing(c), 21)
    m = _moments(rng.normal(size=n), order, LAM, rng)
    gx, gM = _rhs(mm, order, LAM, x, m, mm.MMVM_FP64)
    rx, rM = _rhs(mm, order, LAM, x, m, mm.MMVM_FP64, mm.MMVM_FLAG_NO_FAR_FIELD)
    assert vel_error_rows(gx, rx) <= 1e-12
    if order >= 2:
        assert rhs_error_rows(gM, rM, order, LAM) <= 1e-12

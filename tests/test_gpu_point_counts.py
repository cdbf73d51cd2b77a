"""Point counts of curves with any coordinates: settled in FP32, in whole numbers or by the FP64
sequence, the oracle's number on every input."""
import numpy as np
import pytest

import oracle
from gpu_util import bezier
from paper_2201_02789_gb300 import nestpar as npb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = npb.Context(0)
    yield c
    c.close()


def _coordinates(kind, n):
    rng = np.random.default_rng(len(kind))
    u = rng.random((n, 6))
    if kind == "pixels":
        u *= 4000
    elif kind == "far from the origin":
        u = 1e6 + 100 * u
    elif kind == "whole numbers":           # (many ties: t a whole number)
        u = rng.integers(-64, 64, (n, 6))
    elif kind == "all scales":
        u = rng.normal(size=(n, 6)) * 2.0 ** rng.integers(-100, 100, (n, 1))
    elif kind == "straight":
        u[:, 2:4] = (u[:, :2] + u[:, 4:]) / 2 + u[:, 2:4] * 2.0 ** -rng.integers(1, 40, (n, 1))
    elif kind == "closed":
        u[:, 4:] = u[:, :2] + u[:, 4:] * 2.0 ** -rng.integers(1, 60, (n, 1))
    elif kind == "extremes":
        u = rng.choice([0.0, -0.0, 1.0, 1e-45, -3e-39, 1e-30, 2.0 ** 50, 3e38, -3e38], (n, 6))
    return np.ascontiguousarray(u.astype(np.float32).reshape(n, 3, 2))


@pytest.mark.parametrize("kind", ["uniform", "pixels", "far from the origin", "whole numbers", "all scales", "straight",
                                  "closed", "extremes"])
def test_counts_of_any_coordinates(ctx, kind):
    ctrl = _coordinates(kind, 20000)
    ref = oracle.bezier_offsets(ctrl)
    status, off, _, _ = bezier(ctx, ctrl, npb.config("tca"), cap=1, check=False)
    assert status == npb.NP_ERR_CAPACITY
    np.testing.assert_array_equal(off, ref)

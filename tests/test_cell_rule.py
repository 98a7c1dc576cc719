"""The rule by which a cell index is found without a divide, against subtract, divide, floor in fp32 (CPU).

The rule is the kernels' own: csrc/rules.cuh compiled for the host."""
import ctypes

import numpy as np
import pytest

F, I = ctypes.POINTER(ctypes.c_float), ctypes.POINTER(ctypes.c_int32)


def by_divide(p, mn, vs, dim):
    with np.errstate(all="ignore"):
        f = np.floor((p - mn) / vs)
    ok = (f >= 0) & (f < np.float32(dim))
    return np.where(ok, f, -1).astype(np.int64)


def by_rule(rules, p, mn, vs, dim, axis):
    """Index of `p` along one axis, and the share found without a divide; the point is at the centre of the other axes' only cell."""
    pts = np.full((len(p), 3), 0.5, np.float32)
    pts[:, axis] = p
    lo, size, dims = np.zeros(3, np.float32), np.ones(3, np.float32), np.ones(3, np.int32)
    lo[axis], size[axis], dims[axis] = mn, vs, dim
    out = np.empty((len(p), 3), np.int32)
    pts = np.ascontiguousarray(pts)
    sure = rules.cells(pts.ctypes.data_as(F), len(p), lo.ctypes.data_as(F), size.ctypes.data_as(F), dims.ctypes.data_as(I),
                       out.ctypes.data_as(I))
    return out[:, axis].astype(np.int64), sure / len(p)


def points(rng, mn, vs, dim, n=200_000):
    """Points anywhere around the axis, points a few ulps around multiples of the cell size, far and odd values."""
    with np.errstate(all="ignore"):
        p = (mn + rng.integers(-3, dim + 3, n).astype(np.float32) * vs).astype(np.float32)
        p[: n // 2] = (mn + (rng.random(n // 2) * (dim + 2) - 1).astype(np.float32) * vs).astype(np.float32)
        for _ in range(3):
            p = np.where(rng.random(n) < 0.5, np.nextafter(p, np.float32(np.inf)), np.nextafter(p, np.float32(-np.inf)))
        odd = [np.nan, np.inf, -np.inf, 3e38, -3e38, 1e-45, -1e-45, 0.0, -0.0, 4.1e6, 4.2e6, 8.4e6, 1.26e7, 1.7e7, -4.2e6,
               -1.26e7, -1.7e7, -1e9, -1e20]
        return np.concatenate([p, np.array(odd, np.float32), (np.array(odd, np.float32) * vs + mn).astype(np.float32)]).astype(np.float32)


@pytest.mark.parametrize("dim", [1, 7, 40, 1366, 1600, 65536, 1_200_000, 1_300_000, 5_000_000, 1 << 24])
def test_same_cells_as_subtract_divide_floor(rules, dim):
    rng = np.random.default_rng(dim)
    for i, (mn, vs) in enumerate(((0.0, 0.05), (-51.2, 0.075), (-3.0, 0.1), (-5.0, 8.0), (1e-3, 1 / 3), (0.0, 1e-30), (1e-39, 1e30),
                                  (-1e6, 1e-3))):
        mn, vs = np.float32(mn), np.float32(vs)
        p = points(rng, mn, vs, dim)
        got, _ = by_rule(rules, p, mn, vs, dim, i % 3)
        assert np.array_equal(got, by_divide(p, mn, vs, dim))
        if dim < 100_000 and vs == np.float32(0.05):
            _, sure = by_rule(rules, p[: len(p) // 2 - 100], mn, vs, dim, i % 3)
            assert sure > 0.9                                      # the divide is the exception

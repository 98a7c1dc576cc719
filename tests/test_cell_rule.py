"""The rule by which a cell index is found without a divide, against subtract, divide, floor in fp32 (CPU)."""
import numpy as np
import pytest


def by_divide(p, mn, vs, dim):
    with np.errstate(all="ignore"):
        f = np.floor((p - mn) / vs)
    ok = (f >= 0) & (f < np.float32(dim))
    return np.where(ok, f, -1).astype(np.int64)


def without_divide(p, mn, vs, dim):
    """The arithmetic of cell_xyz, operation by operation; the divide where the margin does not decide."""
    magic = np.float32(12582912.0)
    with np.errstate(all="ignore"):
        inv = np.float32(1.0) / vs
        if not np.isfinite(inv) or abs(inv) < np.finfo(np.float32).tiny:
            inv = np.float32(np.nan)
        q = (p - mn) * inv
        t = q + magic
        e = q - (t - magic)
        sure = np.abs(e) > np.float32(4e-7) * np.float32(dim + 2)
    i = t.view(np.int32).astype(np.int64) - int(magic.view(np.int32)) + (e.view(np.int32) >> 31)
    i = ((i + 2**31) % 2**32 - 2**31)
    fast = np.where((i >= 0) & (i < dim), i, -1)
    return np.where(sure, fast, by_divide(p, mn, vs, dim)), sure


@pytest.mark.parametrize("dim", [1, 7, 40, 1366, 1600, 65536, 1_200_000, 1_300_000, 5_000_000, 1 << 24])
def test_same_cells_as_subtract_divide_floor(dim):
    rng = np.random.default_rng(dim)
    for mn, vs in ((0.0, 0.05), (-51.2, 0.075), (-3.0, 0.1), (-5.0, 8.0), (1e-3, 1 / 3), (0.0, 1e-30), (1e-39, 1e30), (-1e6, 1e-3)):
        mn, vs = np.float32(mn), np.float32(vs)
        n = 200_000
        with np.errstate(all="ignore"):
            p = (mn + rng.integers(-3, dim + 3, n).astype(np.float32) * vs).astype(np.float32)
            p[: n // 2] = (mn + (rng.random(n // 2) * (dim + 2) - 1).astype(np.float32) * vs).astype(np.float32)
            for _ in range(3):
                p = np.where(rng.random(n) < 0.5, np.nextafter(p, np.float32(np.inf)), np.nextafter(p, np.float32(-np.inf)))
        odd = [np.nan, np.inf, -np.inf, 3e38, -3e38, 1e-45, -1e-45, 0.0, -0.0, 4.1e6, 4.2e6, 8.4e6, 1.26e7, 1.7e7, -4.2e6, -1.26e7, -1.7e7]
        with np.errstate(all="ignore"):
            p = np.concatenate([p, np.array(odd, np.float32), (np.array(odd, np.float32) * vs + mn).astype(np.float32)]).astype(np.float32)
        got, sure = without_divide(p, mn, vs, dim)
        assert np.array_equal(got, by_divide(p, mn, vs, dim))
        if dim < 100_000 and vs == np.float32(0.05):
            assert sure[: n // 2].mean() > 0.9                     # the divide is the exception

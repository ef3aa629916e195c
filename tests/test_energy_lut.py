"""Table of grid-segment bounds by an energy's leading bits: for every energy
inside the grid the segment lies within the bounds (host code, no GPU)."""
import ctypes as C

import numpy as np
import pytest

from paper_2110_09214_gb300 import inputs, obem

SHIFT, SIZE = 18, 8192


def _lut(grid):
    grid = np.ascontiguousarray(grid, np.float32)
    out = np.zeros(SIZE, np.uint32)
    fn = getattr(obem.load(), "_Z15obem_energy_lutPKfiPj")     # void obem_energy_lut(const float *, int, uint32_t *)
    fn.restype = None
    fn(grid.ctypes.data_as(C.c_void_p), C.c_int(len(grid)), out.ctypes.data_as(C.c_void_p))
    return out


@pytest.mark.parametrize("name", ["argon", "maxwell", "two", "from_zero", "negative", "dense", "coarse", "tiny"])
def test_bounds(name):
    rng = np.random.default_rng(5)
    grid = {"argon": inputs.argon_like_gas().egrid, "maxwell": inputs.maxwell_gas().egrid,
            "two": np.float32([1.0, 1.0000001]), "from_zero": np.linspace(0, 50, 301, dtype=np.float32),
            "negative": np.float32([-3.0, -1.0, 0.5, 7.0]),
            "dense": np.unique(np.float32(1.0) + np.arange(4096, dtype=np.float32) * np.float32(1.2e-7))[:4096],
            "coarse": np.sort(rng.uniform(0.01, 1e4, 17)).astype(np.float32),
            "tiny": np.float32([1e-44, 1e-40, 3e-39, 1e-37])}[name]
    lut = _lut(grid)
    inside = rng.uniform(max(grid[0], 0), grid[-1], 20000).astype(np.float32)
    e = np.concatenate([inside, grid, np.nextafter(grid, np.float32(-np.inf)), np.nextafter(grid, np.float32(np.inf)),
                        np.float32(10.0) ** rng.uniform(-44, 4, 5000).astype(np.float32)]).astype(np.float32)
    e = e[(e >= grid[0]) & (e < grid[-1]) & (e >= 0)]
    seg = np.searchsorted(grid, e, side="right") - 1           # last grid point <= e
    b = lut[(e.view(np.uint32) >> SHIFT) & (SIZE - 1)]
    lo, hi = (b & 0xFFFF).astype(int), (b >> 16).astype(int)
    assert np.all(lo <= seg) and np.all(seg < hi) and np.all(hi <= len(grid) - 1)

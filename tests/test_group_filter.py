"""The threshold of the tensor-core candidate test (csrc/radius_group.cuh), restated in numpy: operands cut to TF32, sums in fp32.
No pair within the cutoff may fail it, whatever the group's extent, place and unit of length."""
import os
import re

import numpy as np
import pytest

F32 = np.float32


def _tf32(v):
    return (np.asarray(v, F32).view(np.uint32) & np.uint32(0xFFFFE000)).view(F32)


@pytest.mark.parametrize("unit", [1.0, 2.0 ** -20, 2.0 ** 40])
@pytest.mark.parametrize("extent", [0.0, 0.3, 1.0, 4.0, 16.0])          # of the group, in cutoffs
@pytest.mark.parametrize("place", [0.0, 1.0, 1000.0])                    # of the group in the box, in cutoffs
def test_no_neighbour_fails_the_filter(unit, extent, place):
    rng = np.random.default_rng(int(extent * 10 + place))
    r = F32(unit)
    for _ in range(60):
        q = ((place + (rng.random((16, 3)) - 0.5) * extent * [1.0, 0.2, 0.2]) * unit).astype(F32)
        d = rng.normal(size=(16, 64, 3))
        d *= (1.0 - rng.random((16, 64, 1)) ** 4 * 0.01) * unit / np.linalg.norm(d, axis=2, keepdims=True)      # close to the cutoff
        c = (q[:, None, :] + d).astype(F32)
        near = ((q[:, None, :].astype(np.float64) - c) ** 2).sum(2) <= float(r) ** 2
        o = q[8]
        ql, cl = q - o, c - o
        norm = (ql * ql).sum(1, dtype=F32)
        far = np.sqrt(norm.max())
        reach = F32(far + F32(1.001) * r)
        r2_hi = F32(r * r * F32(1 + 32 * 2.0 ** -24))
        thr = F32(r2_hi + F32(3.95e-3) * far * reach + F32(4e-6) * reach * reach)
        t = (norm - thr)[:, None] + (_tf32(F32(-2) * ql)[:, None, :] * _tf32(cl)).sum(2, dtype=F32) + _tf32(cl * cl).sum(2, dtype=F32)
        assert not np.any(near & (t >= 0))
        assert np.any(near)


def _threshold_constants():
    """(product, reach, sums) of the threshold as the kernel's source has them."""
    with open(os.path.join(os.path.dirname(__file__), "..", "paper_2609_24802_b200", "csrc", "radius_group.cuh")) as f:
        src = f.read()
    return [F32(re.search(r"constexpr float %s = ([0-9.e+-]+)f;" % name, src).group(1)) for name in ("FILTER_PRODUCT", "FILTER_REACH", "FILTER_SUMS")]


@pytest.mark.parametrize("unit", [1.0, 2.0 ** -20, 2.0 ** 40])
@pytest.mark.parametrize("cells", [1, 2, 5, 16])                         # along x, of the group
@pytest.mark.parametrize("place", [0.0, 7.0, 1000.0])                    # of the group in the box, in cells
def test_no_neighbour_fails_the_filter_about_the_middle_of_the_cells(unit, cells, place):
    """The same with the kernel's own constants and origin, queries up to the faces of their cells."""
    product, reach_of, sums = _threshold_constants()
    rng = np.random.default_rng(int(cells * 10 + place))
    r = F32(unit)
    edge = F32(1.002 * unit)                                             # a cell is at least this long
    for _ in range(60):
        q = ((place + rng.random((16, 3)) * [cells, 1.0, 1.0]) * edge).astype(F32)
        q[:2] = ((place + np.array([[0.0, 0.0, 0.0], [cells, 1.0, 1.0]])) * edge).astype(F32)
        d = rng.normal(size=(16, 64, 3))
        d[:2] = np.abs(d[:2]) * np.array([-1.0, 1.0])[:, None, None]      # away from the middle, where the operands are largest
        d *= (1.0 - rng.random((16, 64, 1)) ** 4 * 0.01) * unit / np.linalg.norm(d, axis=2, keepdims=True)
        c = (q[:, None, :] + d).astype(F32)
        near = ((q[:, None, :].astype(np.float64) - c) ** 2).sum(2) <= float(r) ** 2
        o = (F32(place) + F32(0.5) * np.array([cells, 1, 1], F32)) * edge
        ql, cl = q - o, c - o
        norm = (ql * ql).sum(1, dtype=F32)
        far = np.sqrt(norm.max())
        reach = F32(far + reach_of * r)
        r2_hi = F32(r * r * F32(1 + 32 * 2.0 ** -24))
        thr = F32(r2_hi + product * far * reach + sums * reach * reach)
        t = (norm - thr)[:, None] + (_tf32(F32(-2) * ql)[:, None, :] * _tf32(cl)).sum(2, dtype=F32) + _tf32(cl * cl).sum(2, dtype=F32)
        assert not np.any(near & (t >= 0))
        assert np.any(near)

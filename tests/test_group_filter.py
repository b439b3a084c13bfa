"""The threshold of the tensor-core candidate test (csrc/radius_group.cuh), restated in numpy: operands cut to TF32, sums in fp32.
No pair within the cutoff may fail it, whatever the group's extent, place and unit of length."""
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
        o = (np.array([place, place, place]) * unit).astype(F32)                      # the middle of the cells
        ql, cl = q - o, c - o
        norm = (ql * ql).sum(1, dtype=F32)
        far = np.sqrt(norm.max())
        reach = F32(far + F32(1.001) * r)
        r2_hi = F32(r * r * F32(1 + 32 * 2.0 ** -24))
        thr = F32(r2_hi + F32(3.95e-3) * far * reach + F32(4e-6) * reach * reach)
        t = (norm - thr)[:, None] + (_tf32(F32(-2) * ql)[:, None, :] * _tf32(cl)).sum(2, dtype=F32) + _tf32(cl * cl).sum(2, dtype=F32)
        assert not np.any(near & (t >= 0))
        assert np.any(near)

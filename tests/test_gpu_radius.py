"""GPU parity: cell binning and the fused radius traversal (through the C ABI) against the
fp64 CPU oracle.  Cells, offsets, order and neighbour counts must match bit-exactly; sums
within 1e-5 and gradients within 1e-4 of the sum of absolute contributions."""
import numpy as np
import pytest

import gen
import oracle
from parity import GRAD_TOL, SUM_TOL, Guard, dev, host, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tiga():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2609_24802_b200 import api
    return api


def _check_bin(tiga, pos, r, box, per):
    ref = oracle.bin_points(pos, r, box, per)
    got = tiga.tiga_radius_bin(dev(pos, torch), r, box, per)
    assert got["ncell"] == ref["ncell"].tolist()
    assert np.array_equal(host(got["cell"]), ref["cell"])
    assert np.array_equal(host(got["cell_start"]), ref["cell_start"])
    assert np.array_equal(host(got["order"]), ref["order"])


def _check_gauss(tiga, pos, x, gy, r, box, per, sigma, kind=None, use_cells=False, backward=True):
    kind = tiga.MSG_GAUSS if kind is None else kind
    y, A, cnt = oracle.radius_forward(pos, x, r, box, per, kind, p0=sigma, use_cells=use_cells)
    pd, xd = dev(pos, torch), dev(x, torch)
    guard = Guard(torch)
    n, F = x.shape
    ws = guard.workspace(tiga.tiga_radius_workspace_bytes(n, F, r, box, per))
    out, count, ws = tiga.tiga_apply_radius(pd, xd, r, box, per, kind, p0=sigma, out=guard.empty((n, F)),
                                            count=guard.empty((n,), torch.int32), ws=ws)
    guard.check()
    assert np.array_equal(host(count), cnt), "neighbour counts must be bit exact"
    assert rel_err(host(out), y, A) <= SUM_TOL
    if backward and kind == tiga.MSG_GAUSS:
        ref = oracle.radius_backward_gauss(pos, x, gy, r, box, per, sigma, use_cells=use_cells)
        gyd = dev(gy, torch)
        gx, gp = tiga.tiga_apply_radius_backward(pd, xd, gyd, r, box, per, sigma, ws=ws, reuse_plan=True,
                                                 grad_feat=guard.empty((n, F)), grad_pos=guard.empty((n, 3)))
        guard.check()
        assert rel_err(host(gx), ref["gx"], ref["Agx"]) <= GRAD_TOL
        assert rel_err(host(gp), ref["gp"], ref["Agp"]) <= GRAD_TOL
        gx2, gp2 = tiga.tiga_apply_radius_backward(pd, xd, gyd, r, box, per, sigma)      # rebuilds the bins
        assert torch.equal(gx, gx2) and torch.equal(gp, gp2)
    return out, count


# ------------------------------------------------------------------------------ binning
def test_binning_is_bit_exact(tiga):
    ones = np.ones(3, np.float32)
    for n, r, per, seed in [(4096, 0.06, [0, 0, 0], 1), (50_000, 0.05, [1, 1, 1], 2), (128, 0.35, [0, 0, 0], 7),
                            (3000, 0.3, [1, 0, 1], 3), (1000, 0.45, [1, 1, 1], 4), (7, 0.2, [0, 0, 0], 5),
                            (200_000, 0.004, [1, 1, 1], 6)]:
        pos = gen.uniform_points(n, seed)
        pos[0] = 0.0
        pos[-1] = 1.0                     # on the upper faces: clamped into the last cell
        _check_bin(tiga, pos, np.float32(r), ones, per)
    # everything in one cell; clustered points (a few very full cells)
    _check_bin(tiga, gen.uniform_points(500, 9) * np.float32(0.01), np.float32(0.1), ones, [0, 0, 0])
    p = gen.uniform_points(20_000, 10)
    p[:15_000] = p[:15_000] * np.float32(0.02) + np.float32(0.5)
    _check_bin(tiga, p, np.float32(0.05), ones, [1, 1, 1])
    # cell occupancies on both sides of the limits of the dense-cell ordering (256 by rank counting,
    # above that a sorting network: in shared memory up to 2048 ids, in place beyond), ids interleaved
    rng = np.random.default_rng(12)
    sizes = [256, 257, 2048, 2049, 8193]
    parts = [gen.uniform_points(m, 13 + k) * np.float32(0.2) + np.float32([0.25 * (k % 4), 0.25 * (k // 4), 0.0])
             for k, m in enumerate(sizes)]
    p = np.concatenate(parts)[rng.permutation(sum(sizes))]
    _check_bin(tiga, p, np.float32(0.25), ones, [0, 0, 0])
    # anisotropic box
    box = np.array([1.0, 2.5, 0.3], np.float32)
    _check_bin(tiga, gen.uniform_points(5000, 11) * box[None, :], np.float32(0.07), box, [1, 0, 0])
    c = gen.config("cfg3", m=20)
    _check_bin(tiga, c["pos"], c["r"], c["box"], c["periodic"])


@pytest.mark.parametrize("n,r", [(1, 0.3), (4096, 0.06), (4096, 0.049), (4096, 0.047), (4095, 0.051), (4097, 0.06), (4096, 0.4), (1024, 0.2)])
def test_one_launch_binning_at_its_limits(tiga, n, r):
    """At most 4096 points and 8192 cells are binned by one CTA: both limits, and cells fuller than the ranking limit."""
    ones = np.ones(3, np.float32)
    pos = gen.uniform_points(n, 18)
    _check_bin(tiga, pos, np.float32(r), ones, [0, 0, 0])
    pos[n // 3:] = pos[n // 3:] * np.float32(0.04) + np.float32(0.3)
    _check_bin(tiga, pos, np.float32(r), ones, [0, 1, 0])


# ------------------------------------------------------------------------------ Gaussian
@pytest.mark.parametrize("n,r,box,cells", [(4046, 0.99, (31, 24, 11), 8184), (4095, 0.99, (31, 24, 11), 8184), (4096, 0.06, (2, 1, 1), 8192),
                                           (4096, 0.99, (32, 32, 8), 8192), (4096, 0.99, (32, 16, 16), 8192), (4096, 0.96, (32, 16, 17), 8704)])
def test_one_launch_binning_of_anisotropic_boxes(tiga, n, r, box, cells):
    """Grids of up to 8192 cells, the most that one CTA bins (no cubic grid comes nearer than 8000), with point counts
    around what fits the default 48 KB of shared memory, and one grid beyond them."""
    box = np.array(box, np.float32)
    assert np.prod(tiga.tiga_radius_grid(n, r, box, [0, 0, 0])[0]) == cells
    pos = gen.uniform_points(n, 7) * box
    _check_bin(tiga, pos, np.float32(r), box, [0, 0, 0])
    x = gen.normal_features(n, 4, 8)
    _check_gauss(tiga, pos, x, x, np.float32(r), box, [0, 0, 0], np.float32(r / 2), backward=False)
    idx, d2, y, A = oracle.knn(pos, x, 1)
    out, nbr, nd2, _ = tiga.tiga_apply_knn(dev(pos, torch), dev(x, torch), 1, box)
    assert np.array_equal(host(nbr), idx) and np.array_equal(host(nd2), d2) and rel_err(host(out), y, A) <= SUM_TOL


@pytest.mark.parametrize("counts", [(64, 65, 63, 0, 1, 128, 2), (4096,), (2000, 2001), (65,) * 63, (256, 257, 255, 1000, 66, 31, 32, 33), (64,) * 64])
def test_one_launch_binning_of_dense_cells(tiga, counts):
    """Cells on both sides of the 64 points that are ordered by counting, up to all points in one cell and as many denser cells
    as there can be (63)."""
    rng = np.random.default_rng(len(counts))
    cell = rng.permutation(np.repeat(rng.permutation(64)[:len(counts)], counts))
    corner = np.stack([cell % 4, cell // 4 % 4, cell // 16], 1)
    pos = ((corner + rng.uniform(0.02, 0.98, corner.shape)) * 0.25).astype(np.float32)
    assert tiga.tiga_radius_grid(len(pos), 0.24, np.ones(3, np.float32), [0, 0, 0])[0] == [4, 4, 4]
    _check_bin(tiga, pos, np.float32(0.24), np.ones(3, np.float32), [0, 0, 0])


def test_cfg0_tiny_forward_and_backward(tiga):
    c = gen.config("cfg0")
    _check_gauss(tiga, c["pos"], c["x"], c["gy"], c["r"], c["box"], c["periodic"], c["sigma"])


@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("F", [4, 16, 32, 64, 128])
def test_gaussian_small(tiga, periodic, F):
    n = 6000
    pos = gen.uniform_points(n, 20 + F)
    x = gen.normal_features(n, F, 20 + F, 31)
    gy = gen.normal_features(n, F, 20 + F, 32)
    r = gen.radius_for_expected_neighbours(n, 24.0)
    _check_gauss(tiga, pos, x, gy, r, np.ones(3, np.float32), [periodic] * 3, np.float32(float(r) / 2))


@pytest.mark.parametrize("F", [1, 3, 6])
def test_forward_widths_that_are_not_multiples_of_four(tiga, F):
    n = 5000
    pos = gen.uniform_points(n, 40 + F)
    x = gen.normal_features(n, F, 40 + F, 31)
    r = gen.radius_for_expected_neighbours(n, 32.0)
    ones = np.ones(3, np.float32)
    _check_gauss(tiga, pos, x, None, r, ones, [0, 0, 0], np.float32(float(r) / 2), backward=False)
    _check_gauss(tiga, pos, x, None, r, ones, [1, 1, 1], np.float32(float(r) / 2), kind=tiga.MSG_DIST)
    with pytest.raises(tiga.TigaError) as ei:      # the backward needs 128-bit rows
        tiga.tiga_apply_radius_backward(dev(pos, torch), dev(x, torch), dev(x, torch), r, ones, [0, 0, 0], 0.1)
    assert ei.value.status == 2


@pytest.mark.parametrize("per_cell", [1, 3, 4, 5, 6, 7, 8, 9, 16, 17, 33, 64, 65, 130])
@pytest.mark.parametrize("F", [1, 2, 3, 4, 8])
def test_narrow_features_at_every_split_of_the_lanes(tiga, F, per_cell):
    """Forwards with at most four features share the warp's lanes out by the number of queries of a cell (and
    F = 8 shares lists between lane groups): occupancies on both sides of every split, of the query batch (16), of
    what makes a cell dense at these sizes (more than 6 points, cut into slices of 4) and of the staged chunk (256
    candidates), with wrapped faces (four cells) and with the explicit minimum image (three cells)."""
    ones = np.ones(3, np.float32)
    for cells, periodic in ((3, 1), (4, 1), (3, 0)):
        n = per_cell * cells ** 3
        pos = gen.uniform_points(n, 60 + F + per_cell)
        x = gen.normal_features(n, F, 60 + F + per_cell, 31)
        r = np.float32(1.0 / cells / 1.002)
        for kind in (tiga.MSG_GAUSS, tiga.MSG_DIST):
            _check_gauss(tiga, pos, x, None, r, ones, [periodic] * 3, np.float32(float(r) / 2), kind=kind, backward=False)


@pytest.mark.parametrize("per_cell", [22, 24, 25, 27, 40])
def test_narrow_features_on_both_sides_of_the_largest_slices(tiga, per_cell):
    """From 100 k points on slices have 16 queries and a cell is cut above 24."""
    cells = 17
    n = per_cell * cells ** 3
    pos, x = gen.uniform_points(n, 90 + per_cell), gen.normal_features(n, 3, 91, 31)
    ones, r = np.ones(3, np.float32), np.float32(1.0 / cells / 1.002)
    _check_gauss(tiga, pos, x, None, r, ones, [1, 1, 1], np.float32(float(r) / 2), use_cells=True, backward=False)


@pytest.mark.parametrize("F", [1, 4, 16])
@pytest.mark.parametrize("cells", [(5, 60, 61), (11, 41, 41), (64, 24, 24), (41, 30, 30)])
def test_runs_of_sparse_cells(tiga, cells, F):
    """Sparse inputs join neighbouring cells along x: every run length from 1 to 8 (limited by the grid where the faces
    wrap), runs that touch the lower or the upper face, a remainder run at the end of a row."""
    box = np.array(cells, np.float32)
    r = np.float32(1.0 / 1.002)
    n = int(np.prod(cells))
    for share, periodic in ((1.0, 1), (0.4, 1), (0.4, 0), (3.0, 0)):
        m = int(share * n)
        pos = gen.uniform_points(m, 70 + F) * box[None, :]
        pos = np.minimum(pos, box[None, :])
        x, gy = gen.normal_features(m, F, 71, 31), gen.normal_features(m, F, 71, 32)
        _check_gauss(tiga, pos, x, gy, r, box, [periodic] * 3, np.float32(0.5), use_cells=True, backward=F >= 4)


@pytest.mark.parametrize("sigma", [1e14, 1e20, np.inf])
@pytest.mark.parametrize("F", [1, 2, 3, 4, 8])
def test_gaussian_as_wide_as_fp32_allows(tiga, F, sigma):
    """Every accepted pair weighs one: the message becomes a plain neighbour sum (the oracle's with a weight that is one
    to the last bit).  Cutoff of a lattice spacing's multiple, so that pairs sit on the cutoff and are refused in fp64."""
    i = np.arange(12, dtype=np.float32) * np.float32(0.08) + np.float32(0.05)
    pos = np.stack([t.reshape(-1) for t in np.meshgrid(i, i, i, indexing="ij")], 1)
    pos = np.concatenate([pos, gen.uniform_points(1777, 33)]).astype(np.float32)
    x = gen.normal_features(len(pos), F, 34)
    ones = np.ones(3, np.float32)
    r = np.float32(0.08)
    y, A, cnt = oracle.radius_forward(pos, x, r, ones, [0, 0, 0], oracle.MSG_GAUSS, p0=1e9)
    out, count, _ = tiga.tiga_apply_radius(dev(pos, torch), dev(x, torch), r, ones, [0, 0, 0], tiga.MSG_GAUSS, p0=sigma, want_count=True)
    assert np.array_equal(host(count), cnt) and rel_err(host(out), y, A) <= SUM_TOL


@pytest.mark.parametrize("message", ["gauss", "dist"])
@pytest.mark.parametrize("F", [1, 2, 3, 4])
def test_infinite_features_reach_their_neighbours_only(tiga, F, message):
    """A row with an infinite source among its neighbours is that infinity, any other row is what it is without it."""
    pos, x = gen.uniform_points(2000, 35), gen.normal_features(2000, F, 36)
    ones, r, per = np.ones(3, np.float32), np.float32(0.11), [1, 1, 1]
    kind = tiga.MSG_GAUSS if message == "gauss" else tiga.MSG_DIST
    P = dev(pos, torch)
    plain = host(tiga.tiga_apply_radius(P, dev(x, torch), r, ones, per, kind, p0=0.1)[0])
    x[1234] = np.inf
    got = host(tiga.tiga_apply_radius(P, dev(x, torch), r, ones, per, kind, p0=0.1)[0])
    d = pos.astype(np.float64) - pos[1234].astype(np.float64)
    d2 = ((d - np.rint(d)) ** 2).sum(1)
    assert abs(d2 - np.float64(r) ** 2).min() > 1e-7          # no pair of this point is near the cutoff
    near = d2 <= np.float64(r) ** 2
    near[1234] = False
    assert 3 < near.sum() < 30
    assert np.all(got[near] == np.inf) and np.array_equal(got[~near], plain[~near])


def test_few_cells_mixed_periodicity_and_anisotropic_box(tiga):
    # the paper's tiny radius shape: 128 points, cutoff 0.35 (two cells per dimension)
    pos = gen.uniform_points(128, 7)
    x = gen.normal_features(128, 8, 7); gy = gen.normal_features(128, 8, 7, 32)
    ones = np.ones(3, np.float32)
    _check_gauss(tiga, pos, x, gy, np.float32(0.35), ones, [0, 0, 0], np.float32(0.2))
    _check_gauss(tiga, pos, x, gy, np.float32(0.35), ones, [1, 1, 1], np.float32(0.2))   # one cell, minimum image
    _check_gauss(tiga, pos, x, gy, np.float32(0.3), ones, [1, 0, 1], np.float32(0.2))    # three cells where periodic
    box = np.array([1.0, 2.5, 0.3], np.float32)
    n = 4000
    pos = gen.uniform_points(n, 12) * box[None, :]
    x = gen.normal_features(n, 16, 12); gy = gen.normal_features(n, 16, 12, 32)
    _check_gauss(tiga, pos, x, gy, np.float32(0.09), box, [1, 0, 1], np.float32(0.05))
    # the paper's own message: distance-weighted sum
    _check_gauss(tiga, pos, x, gy, np.float32(0.09), box, [1, 0, 1], np.float32(0.05), kind=tiga.MSG_DIST)


def test_pairs_exactly_on_the_cutoff_are_neighbours(tiga):
    # binary-grid coordinates: many pairs at distance exactly r (inclusive predicate)
    k = np.arange(16, dtype=np.float32) / 16
    X, Y, Z = np.meshgrid(k, k, k, indexing="ij")
    pos = np.stack([X.ravel(), Y.ravel(), Z.ravel()], 1).astype(np.float32)
    n = pos.shape[0]
    x = gen.normal_features(n, 8, 5); gy = gen.normal_features(n, 8, 5, 32)
    for per in ([0, 0, 0], [1, 1, 1]):
        out, count = _check_gauss(tiga, pos, x, gy, np.float32(3.0 / 16), np.ones(3, np.float32), per, np.float32(0.1))
        if per[0]:
            # |v| <= 3 on the integer lattice: 123 points minus the origin
            assert np.all(host(count) == 122)


def test_no_neighbours_and_coincident_points(tiga):
    pos = np.array([[0.1, 0.1, 0.1], [0.9, 0.9, 0.9], [0.5, 0.5, 0.5], [0.5, 0.5, 0.5], [0.5, 0.5, 0.5]], np.float32)
    x = gen.normal_features(5, 4, 1); gy = gen.normal_features(5, 4, 1, 32)
    out, count = _check_gauss(tiga, pos, x, gy, np.float32(0.05), np.ones(3, np.float32), [0, 0, 0], np.float32(0.02))
    assert host(count).tolist() == [0, 0, 2, 2, 2]
    assert np.all(host(out)[:2] == 0.0)


def test_clustered_points_overflow_the_pair_list(tiga):
    n = 3000
    pos = gen.uniform_points(n, 15) * np.float32(0.1) + np.float32(0.3)       # ~500 neighbours each
    x = gen.normal_features(n, 32, 15); gy = gen.normal_features(n, 32, 15, 32)
    _check_gauss(tiga, pos, x, gy, np.float32(0.05), np.ones(3, np.float32), [0, 0, 0], np.float32(0.03))


def test_gaussian_mid_replica(tiga):
    """A 131,072-point replica of the 1M-point periodic workload (32 expected neighbours, F=32),
    every row against the oracle's cell-directory variant (itself pinned to all pairs)."""
    c = gen.config("cfg2", n=131_072)
    _check_gauss(tiga, c["pos"], c["x"], c["gy"], c["r"], c["box"], c["periodic"], c["sigma"], use_cells=True)


# ------------------------------------------------------------------------------ Lennard-Jones
def _check_lj(tiga, pos, r, box, per, eps=1.0, s=1.0, use_cells=False, tol=SUM_TOL):
    y, A, cnt = oracle.radius_forward(pos, None, r, box, per, oracle.MSG_LJ, eps, s, use_cells=use_cells)
    guard = Guard(torch)
    n = len(pos)
    out, count, _ = tiga.tiga_apply_radius(dev(pos, torch), None, r, box, per, tiga.MSG_LJ, p0=eps, p1=s,
                                           out=guard.empty((n, 4)), count=guard.empty((n,), torch.int32),
                                           ws=guard.workspace(tiga.tiga_radius_workspace_bytes(n, 4, r, box, per)))
    guard.check()
    assert np.array_equal(host(count), cnt)
    err = rel_err(host(out), y, A)
    print(f"Lennard-Jones: largest normalised error {err:.3e} (tolerance {tol:.1e})")
    assert err <= tol
    return host(out), A


def test_lennard_jones_lattices(tiga):
    c = gen.config("cfg3", m=12)
    out, A = _check_lj(tiga, c["pos"], c["r"], c["box"], c["periodic"])
    assert np.max(np.abs(out[:, :3].astype(np.float64).sum(0))) < 1e-6 * A[:, :3].sum()   # Newton's third law
    # perfect lattice: 56 neighbours, zero force, closed-form energy per particle
    pos, L = gen.jittered_lattice(10, 0.8, 0.0)
    out, A = _check_lj(tiga, pos, np.float32(2.5), np.full(3, L, np.float32), [1, 1, 1])
    assert np.max(np.abs(out[:, 3] - (-5.264771118950892))) < 2e-4
    # other eps / s, non-periodic
    pos = gen.uniform_points(2000, 3) * np.float32(12.0)
    keep = np.ones(len(pos), bool)
    d = np.linalg.norm(pos[:, None, :].astype(np.float64) - pos[None, :, :], axis=2) + np.eye(len(pos)) * 9
    keep[np.unique(np.nonzero(d < 0.7)[0])] = False          # no overlapping particles
    _check_lj(tiga, pos[keep], np.float32(2.0), np.full(3, 12.0, np.float32), [0, 0, 0], eps=1.5, s=0.8)


def test_lennard_jones_at_any_unit_of_length(tiga):
    """Lengths of 1e16 (squares beyond 1e30): the forces scale with eps / s, the energies and counts stay."""
    c = gen.config("cfg3", m=10)
    unit = np.float32(2.0 ** 53)                               # a power of two: every quotient of lengths stays the same bits
    pos, r, box = c["pos"] * unit, np.float32(c["r"]) * unit, np.asarray(c["box"], np.float32) * unit
    P = lambda a: dev(a, torch)
    out, count, _ = tiga.tiga_apply_radius(P(c["pos"]), None, c["r"], c["box"], c["periodic"], tiga.MSG_LJ, p0=1.0, p1=1.0, want_count=True)
    big, count2, _ = tiga.tiga_apply_radius(P(pos), None, r, box, c["periodic"], tiga.MSG_LJ, p0=1.0, p1=float(unit), want_count=True)
    assert torch.equal(count, count2)
    assert torch.equal(big[:, 3], out[:, 3]) and torch.equal(big[:, :3] * float(unit), out[:, :3])


def test_lennard_jones_replica(tiga):
    c = gen.config("cfg3", m=40)          # 64,000 particles
    out, A = _check_lj(tiga, c["pos"], c["r"], c["box"], c["periodic"], use_cells=True)
    assert np.max(np.abs(out[:, :3].astype(np.float64).sum(0))) < 1e-6 * A[:, :3].sum()


def _separated_points(n, box, seed, dmin):
    """Uniform points in the box with no pair closer than dmin (Lennard-Jones inputs never overlap)."""
    pos = (gen.uniform_points(n, seed).astype(np.float64) * np.asarray(box, np.float64)).astype(np.float32)
    d = pos[:, None, :].astype(np.float64) - pos[None, :, :]
    d -= np.asarray(box, np.float64) * np.rint(d / np.asarray(box, np.float64))      # strictest reading: periodic in all
    dist = np.sqrt((d * d).sum(2)) + np.eye(n) * 1e9
    keep = np.ones(n, bool)
    for i in range(n):
        if keep[i]:
            keep[(dist[i] < dmin) & (np.arange(n) > i)] = False
    return pos[keep]


def _box_of(cells):
    return np.array([c * 1.05 + 0.3 for c in cells], np.float32)       # floor(len / (r (1 + 2^-10))) = cells at r = 1


# a periodic dimension must be longer than twice the cutoff: such combinations are left out
_SMALL_GRIDS = [(cells, per) for cells in [(1, 1, 1), (2, 2, 2), (3, 3, 3), (4, 3, 2), (1, 5, 3), (6, 1, 1), (3, 4, 1)]
                for per in [(0, 0, 0), (1, 1, 1), (1, 0, 1), (0, 1, 0)]
                if not any(p and b <= 2.0 for p, b in zip(per, _box_of(cells)))]


@pytest.mark.parametrize("cells,periodic", _SMALL_GRIDS)
def test_lennard_jones_small_grids(tiga, cells, periodic):
    """Every unordered pair must be visited exactly once whatever the grid: one, two or three
    cells per dimension, wrapped or clipped (a periodic dimension with fewer than three cells
    collapses to one cell with the explicit minimum image)."""
    r = np.float32(1.0)
    box = _box_of(cells)
    pos = _separated_points(600, box, 40 + sum(cells), 0.45)
    grid, _ = tiga.tiga_radius_grid(len(pos), r, box, list(periodic))
    expect = [1 if (p and c < 3) else c for c, p in zip(cells, periodic)]
    cap = int(round((8 * len(pos)) ** (1 / 3) - 0.5))
    assert list(grid) == [min(e, cap) for e in expect]
    out, A = _check_lj(tiga, pos, r, box, list(periodic), eps=0.7, s=0.5)
    assert np.max(np.abs(out[:, :3].astype(np.float64).sum(0))) < 1e-5 * max(A[:, :3].sum(), 1e-30)


def test_lennard_jones_dense_cells_span_several_stage_chunks(tiga):
    """Hundreds of points per cell: the cell's own points alone overflow the stage, so the
    stencil is processed in several chunks and a query is left out across chunk borders."""
    box = np.array([6.0, 6.0, 6.0], np.float32)
    pos = _separated_points(2600, box, 77, 0.25)
    assert len(pos) > 1800
    # The pair force goes like d^-14 and the closest pairs (0.25 apart in cells of edge 3) dominate the
    # sums: a displacement formed from coordinates relative to a cell corner would carry an fp32
    # rounding of the CELL size and miss the tolerance here.  The kernel subtracts stored original
    # coordinates (periodic images by exact shifts), so the plain tolerance holds.
    for periodic in ([0, 0, 0], [1, 1, 1]):
        grid, _ = tiga.tiga_radius_grid(len(pos), np.float32(2.0), box, periodic)
        assert max(grid) <= 2
        _check_lj(tiga, pos, np.float32(2.0), box, periodic, eps=0.3, s=0.3)


def test_lennard_jones_is_reproducible(tiga):
    """Every row adds up its own neighbourhood in an order of its own: two runs give the same bits, with and without counts."""
    c = gen.config("cfg3", m=24)
    pd = dev(c["pos"], torch)
    a, ca, _ = tiga.tiga_apply_radius(pd, None, c["r"], c["box"], c["periodic"], tiga.MSG_LJ, p0=1.0, p1=1.0, want_count=True)
    b, cb, _ = tiga.tiga_apply_radius(pd, None, c["r"], c["box"], c["periodic"], tiga.MSG_LJ, p0=1.0, p1=1.0, want_count=True)
    assert torch.equal(ca, cb) and torch.equal(a, b)
    y, A, cnt = oracle.radius_forward(c["pos"], None, c["r"], c["box"], c["periodic"], oracle.MSG_LJ, 1.0, 1.0, use_cells=True)
    nocount, none, _ = tiga.tiga_apply_radius(pd, None, c["r"], c["box"], c["periodic"], tiga.MSG_LJ, p0=1.0, p1=1.0)
    assert none is None and torch.equal(nocount, a) and rel_err(host(nocount), y, A) <= SUM_TOL


# ------------------------------------------------------------------------------ full size
def test_cfg2_full_size_sampled_rows(tiga):
    """1M points, periodic, F=32: 4096 sampled rows against all-pairs brute force, all rows
    against the oracle's cell-directory variant, plus global invariants."""
    c = gen.config("cfg2")
    n = c["n"]
    pd, xd, gyd = dev(c["pos"], torch), dev(c["x"], torch), dev(c["gy"], torch)
    out, count, ws = tiga.tiga_apply_radius(pd, xd, c["r"], c["box"], c["periodic"], tiga.MSG_GAUSS,
                                            p0=c["sigma"], want_count=True)
    gx, gp = tiga.tiga_apply_radius_backward(pd, xd, gyd, c["r"], c["box"], c["periodic"], c["sigma"], ws=ws, reuse_plan=True)
    out, count, gx, gp = host(out), host(count), host(gx), host(gp)
    rows = np.sort(gen.rng(1, 77).choice(n, 4096, replace=False))
    y, A, cnt = oracle.radius_forward(c["pos"], c["x"], c["r"], c["box"], c["periodic"], oracle.MSG_GAUSS,
                                      p0=c["sigma"], rows=rows)
    assert np.array_equal(count[rows], cnt)
    assert rel_err(out[rows], y, A) <= SUM_TOL
    b = oracle.radius_backward_gauss(c["pos"], c["x"], c["gy"], c["r"], c["box"], c["periodic"], c["sigma"], rows=rows)
    assert rel_err(gx[rows], b["gx"], b["Agx"]) <= GRAD_TOL
    assert rel_err(gp[rows], b["gp"], b["Agp"]) <= GRAD_TOL
    y, A, cnt = oracle.radius_forward(c["pos"], c["x"], c["r"], c["box"], c["periodic"], oracle.MSG_GAUSS,
                                      p0=c["sigma"], use_cells=True)
    assert np.array_equal(count, cnt) and count.sum() % 2 == 0
    assert rel_err(out, y, A) <= SUM_TOL
    assert abs(count.mean() - 32.0) < 0.1
    b = oracle.radius_backward_gauss(c["pos"], c["x"], c["gy"], c["r"], c["box"], c["periodic"], c["sigma"], use_cells=True)
    assert rel_err(gx, b["gx"], b["Agx"]) <= GRAD_TOL
    assert rel_err(gp, b["gp"], b["Agp"]) <= GRAD_TOL
    assert np.max(np.abs(gp.astype(np.float64).sum(0))) < 1e-5 * b["Agp"].sum()     # translation invariance


def test_cfg3_full_size(tiga):
    """160^3 = 4,096,000 jittered-lattice particles, periodic, cutoff 2.5: 2048 sampled rows against
    all-pairs brute force, every row against the oracle's cell-directory variant, and Newton's
    third law over the whole system."""
    c = gen.config("cfg3")
    n = c["n"]
    assert n == 4_096_000
    out, count, _ = tiga.tiga_apply_radius(dev(c["pos"], torch), None, c["r"], c["box"], c["periodic"], tiga.MSG_LJ,
                                           p0=1.0, p1=1.0, want_count=True)
    out, count = host(out), host(count)
    rows = np.sort(gen.rng(3, 78).choice(n, 2048, replace=False))
    y, A, cnt = oracle.radius_forward(c["pos"], None, c["r"], c["box"], c["periodic"], oracle.MSG_LJ, 1.0, 1.0, rows=rows)
    assert np.array_equal(count[rows], cnt)
    assert rel_err(out[rows], y, A) <= SUM_TOL
    y, A, cnt = oracle.radius_forward(c["pos"], None, c["r"], c["box"], c["periodic"], oracle.MSG_LJ, 1.0, 1.0, use_cells=True)
    assert np.array_equal(count, cnt) and count.sum() % 2 == 0
    assert rel_err(out, y, A) <= SUM_TOL
    assert 50 < count.mean() < 58
    assert np.max(np.abs(out[:, :3].astype(np.float64).sum(0))) < 1e-6 * A[:, :3].sum()


def test_sparse_periodic_box_pairs_at_the_cutoff_across_a_face(tiga):
    """Few points, small cutoff: the grid is capped (cells eleven times the cutoff), and pairs sit
    within a few ulps of r on both sides of it across the lower x face and inside the box.  The
    neighbour counts must equal the fp64 predicate's, pair by pair."""
    r = np.float32(0.01)
    ones = np.ones(3, np.float32)
    rows = []
    for k in range(24):
        y, z = np.float32(0.04 * k + 0.013), np.float32(0.9 - 0.031 * k)
        xa = np.float32(0.003 + 0.0001 * k)
        xb = np.float32(1.0) - (r - xa)                      # across the face, about r away
        xb = np.nextafter(xb, np.float32(2.0 if k % 2 else 0.0), dtype=np.float32)
        for _ in range(k % 5):
            xb = np.nextafter(xb, np.float32(2.0 if k % 2 else 0.0), dtype=np.float32)
        rows += [[xa, y, z], [xb, y, z]]
        xc = np.float32(0.4 + 0.01 * k)                      # the same inside the box
        xd = xc + r
        for _ in range(k % 4):
            xd = np.nextafter(xd, np.float32(2.0 if k % 2 else 0.0), dtype=np.float32)
        rows += [[xc, y, np.float32(z * 0.5)], [xd, y, np.float32(z * 0.5)]]
    pos = np.array(rows, np.float32)
    assert tiga.tiga_radius_grid(len(pos), float(r), ones, [1, 1, 1])[0][0] < 12      # capped grid
    x = gen.normal_features(len(pos), 8, 5)
    gy = gen.normal_features(len(pos), 8, 6)
    _, cnt = _check_gauss(tiga, pos, x, gy, r, ones, [1, 1, 1], float(r) / 2)
    c = host(cnt)
    assert 0 < c.sum() < len(pos)                            # some of the pairs are inside, some outside


# ------------------------------------------------------------------------------ validation
def test_point_validation(tiga):
    box = np.array([1.0, 2.0, 0.5], np.float32)
    pos = gen.uniform_points(10_000, 3) * box[None, :]
    pos[17] = box                                              # the upper faces belong to the box
    tiga.tiga_validate_points(dev(pos, torch), box)            # passes
    for bad in (np.float32(-1e-6), np.float32(np.nan), np.float32(np.inf), np.float32(0.5000001)):
        q = pos.copy()
        q[4321, 2] = bad
        with pytest.raises(tiga.TigaError) as e:
            tiga.tiga_validate_points(dev(q, torch), box)
        assert e.value.status == 7
        tiga.tiga_validate_points(dev(q, torch), box, level=0)     # metadata only: nothing is read
    tiga.tiga_validate_points(dev(pos[:0], torch), box)


# ------------------------------------------------------------------------------ uneven density
def test_clustered_points_are_spread_over_many_warps(tiga):
    """Most points in a dozen tight blobs: some cells hold hundreds of points, which are cut into slices of 16 queries and
    shared out to many warps.  Parity as usual, and the call must stay within 5x of a uniform cloud with the same number of accepted pairs."""
    n, F = 200_000, 8
    pos = gen.clustered_points(n, 21)
    x = gen.normal_features(n, F, 21, 31); gy = gen.normal_features(n, F, 21, 32)
    ones = np.ones(3, np.float32)
    r = np.float32(0.01)
    grid, _ = tiga.tiga_radius_grid(n, r, ones, [0, 0, 0])
    cell = np.minimum((pos * np.float32(grid)).astype(np.int64), np.array(grid) - 1)
    occupancy = np.bincount((cell[:, 2] * grid[1] + cell[:, 1]) * grid[0] + cell[:, 0])
    assert occupancy.max() > 4 * 64                                   # several slices per cell
    out, count = _check_gauss(tiga, pos, x, gy, r, ones, [0, 0, 0], np.float32(0.005), use_cells=True)
    pairs = int(host(count).sum())
    # Lennard-Jones on the same cloud (scaled): the length s lies below the smallest distance of any pair, so no pair
    # energy is a difference of two nearly equal powers (the normalisation by |contributions| would not cover that)
    # (cutoff 0.8: a few dozen neighbours per particle as in the workload, while the cells -- their number is capped
    # by the point count -- still hold hundreds of points; rows of a thousand terms that cancel would exceed what
    # fp32 accumulation can promise)
    _check_lj(tiga, pos * np.float32(300.0), np.float32(0.8), np.full(3, 300.0, np.float32), [0, 0, 0], eps=1e-3, s=0.005, use_cells=True)

    def timed(p, rr):
        pd, xd = dev(p, torch), dev(x, torch)
        o, c, ws = tiga.tiga_apply_radius(pd, xd, rr, ones, [0, 0, 0], tiga.MSG_GAUSS, p0=float(rr) / 2, want_count=True)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for _ in range(5):
            tiga.tiga_apply_radius(pd, xd, rr, ones, [0, 0, 0], tiga.MSG_GAUSS, p0=float(rr) / 2, out=o, count=c, ws=ws)
        b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b) / 5, int(c.sum().item())

    r_uniform = np.float32((pairs * 3.0 / (4.0 * np.pi * n * n)) ** (1.0 / 3.0))
    t_c, p_c = timed(pos, r)
    t_u, p_u = timed(gen.uniform_points(n, 22), r_uniform)
    print(f"clustered: {p_c} pairs in {t_c:.3f} ms; uniform: {p_u} pairs in {t_u:.3f} ms")
    assert 0.7 * p_c < p_u < 1.4 * p_c
    assert t_c < 5.0 * t_u


# (points, cutoff, box, periodic): units of 4, 8 and 16 points, sparse and dense cells on both sides of the two stages (fewer and more than
# three points per cell), rows of cells that end inside a group, a run that nearly closes around the box (4 and 5 cells), explicit
# minimum image (3 cells), more accepted candidates than the lists hold, a stencil of many stages (one cell, all points), lengths
# far from one
_GROUPS = [(8192, 0.05, (1, 1, 1), [0, 0, 0]), (11841, 0.05, (1, 1, 1), [0, 1, 1]), (24001, 0.035, (1, 1, 1), [0, 0, 0]),
           (24001, 0.045, (1, 1, 1), [1, 1, 1]), (24001, 0.05, (1, 1, 1), [1, 0, 1]), (24001, 0.19, (1, 1, 1), [1, 1, 1]),
           (11999, 0.24, (1, 1, 1), [1, 1, 1]), (11999, 0.3, (1, 1, 1), [1, 0, 1]), (8192, 0.9, (1, 1, 1), [0, 0, 0]),
           (30011, 0.05, (4, 0.5, 0.5), [1, 1, 0]), (30011, 0.05, (0.23, 4, 1), [1, 0, 1]),
           (24001, 50.0, (1024, 1024, 1024), [1, 1, 1]), (24001, 0.04 / 4096, (1 / 4096,) * 3, [0, 1, 0])]


@pytest.mark.parametrize("n,r,box,periodic", _GROUPS)
@pytest.mark.parametrize("F", [1, 4])
def test_groups_of_queries(tiga, F, n, r, box, periodic):
    box = np.asarray(box, np.float32)
    pos = np.minimum(gen.uniform_points(n, 71) * box, np.nextafter(box, np.float32(0))).astype(np.float32)
    x = gen.normal_features(n, F, 71, 31)
    for kind in (tiga.MSG_GAUSS, tiga.MSG_DIST):
        _check_gauss(tiga, pos, x, None, np.float32(r), box, periodic, np.float32(r) / 2, kind=kind, use_cells=r < 0.2 * box.min(), backward=False)


@pytest.mark.parametrize("L", [4e18, 2e17, 1e-14, 1e-17])
@pytest.mark.parametrize("F", [1, 3])
def test_narrow_features_at_lengths_near_the_ends_of_fp32(tiga, F, L):
    """A box that holds the place of the padding, one just short of it, squared cutoffs near and below the smallest normal number."""
    box = np.full(3, L, np.float32)
    pos = np.minimum(gen.uniform_points(24001, 73) * box, np.nextafter(box, np.float32(0))).astype(np.float32)
    x = gen.normal_features(len(pos), F, 73, 31)
    r = np.float32(0.045 * L)
    for kind in (tiga.MSG_GAUSS, tiga.MSG_DIST):
        _check_gauss(tiga, pos, x, None, r, box, [0, 0, 0], r / np.float32(2), kind=kind, use_cells=True, backward=False)


def test_long_sums_are_added_up_in_pieces(tiga):
    """24 k neighbours per point, positive terms.  A running sum of m terms is off by 2^-24 sqrt(m / 9) of itself, rms (half an ulp of the running
    value at most, each time): 1.9e-7 for 94 pieces of 256 candidates, 7.7e-7 for four running sums of a term at a time."""
    n = 24001
    pos = gen.uniform_points(n, 74)
    x = np.abs(gen.normal_features(n, 1, 74, 31))
    rows = np.sort(gen.rng(74, 1).choice(n, 512, replace=False))
    box, r = np.ones(3, np.float32), np.float32(1.8)
    y, A, cnt = oracle.radius_forward(pos, x, r, box, [0, 0, 0], oracle.MSG_DIST, rows=rows)
    out, count, _ = tiga.tiga_apply_radius(dev(pos, torch), dev(x, torch), r, box, [0, 0, 0], tiga.MSG_DIST, want_count=True)
    assert np.array_equal(host(count)[rows], cnt)
    err = float(np.sqrt(np.mean(((host(out)[rows] - y) / A) ** 2)))
    print(f"rms error {err:.2e}")
    assert err <= 2.2e-7


# (points, cutoff, periodic, shape): inputs of less than three points per cell on average whose points crowd together: units of full cells (above 20
# points) beside units of groups, more accepted candidates than the sparse stage's lists hold (a slab of about 8 points a cell), every unit length
_CROWDED = [(8192, 0.05, [0, 0, 0], "blobs"), (15001, 0.04, [1, 1, 0], "blobs"), (24001, 0.035, [0, 0, 0], "blobs"), (24001, 0.0341, [0, 0, 0], "slab"),
            (24001, 0.0341, [1, 1, 1], "slab"), (300_007, 0.014, [1, 0, 1], "blobs"), (300_007, 0.0152, [0, 1, 0], "slab")]


@pytest.mark.parametrize("n,r,periodic,shape", _CROWDED)
@pytest.mark.parametrize("message", ["sum1", "sum4", "lj"])
def test_groups_and_full_cells_side_by_side(tiga, message, n, r, periodic, shape):
    ones = np.ones(3, np.float32)
    pos = gen.clustered_points(n, 75) if shape == "blobs" else gen.uniform_points(n, 75) * np.array([1.0, 1.0, 0.1], np.float32)
    grid, _ = tiga.tiga_radius_grid(n, r, ones, periodic)
    cell = np.minimum((pos * np.float32(grid)).astype(np.int64), np.array(grid) - 1)
    held = np.bincount((cell[:, 2] * grid[1] + cell[:, 1]) * grid[0] + cell[:, 0])
    assert 0.7 <= n / np.prod(grid) < 3 and (held > 20).any() and ((held > 0) & (held <= 20)).any()
    if message == "lj":
        _check_lj(tiga, pos * np.float32(300.0), np.float32(300.0 * r), np.full(3, 300.0, np.float32), periodic, eps=1e-3, s=0.001, use_cells=True)
    else:
        x = gen.normal_features(n, 1 if message == "sum1" else 4, 75, 31)
        _check_gauss(tiga, pos, x, None, np.float32(r), ones, periodic, np.float32(r) / 2, kind=tiga.MSG_DIST, use_cells=True, backward=False)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("message", ["sum1", "sum4", "lj"])
def test_a_coordinate_that_is_not_finite_affects_its_own_point_only(tiga, message, bad):
    """What a diverging simulation hands over: every other point has the neighbours that it has without the bad ones."""
    c = gen.config("cfg3", m=21)
    r, box, periodic = (c["r"], c["box"], c["periodic"]) if message == "lj" else (np.float32(0.08), np.ones(3, np.float32), [0, 0, 0])
    pos = c["pos"].copy() if message == "lj" else gen.uniform_points(24001, 72)
    n, F = len(pos), 1 if message == "sum1" else 4
    x = gen.normal_features(n, F, 72, 31)
    which = np.sort(gen.rng(72, 3).choice(n, 300, replace=False))
    pos[which, np.arange(300) % 3] = bad
    good = np.delete(np.arange(n), which)
    kind, p0, p1 = (tiga.MSG_LJ, 1.0, 1.0) if message == "lj" else (tiga.MSG_DIST, 0.0, 0.0)
    y, A, cnt = oracle.radius_forward(pos[good], None if message == "lj" else x[good], r, box, periodic, kind, p0, p1, use_cells=True)
    out, count, _ = tiga.tiga_apply_radius(dev(pos, torch), None if message == "lj" else dev(x, torch), r, box, periodic, kind, p0=p0, p1=p1, want_count=True)
    assert np.array_equal(host(count)[good], cnt)
    assert rel_err(host(out)[good], y, A) <= SUM_TOL
    assert not host(count)[which].any() and not host(out)[which].any()


@pytest.mark.parametrize("m", [21, 29])
def test_groups_decide_pairs_at_the_cutoff_exactly(tiga, m):
    """Lattices whose neighbours lie exactly at the cutoff, just inside and just outside."""
    h = np.float32(1.0 / 32.0)
    grid = (np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3) * h).astype(np.float32)
    box = np.full(3, m, np.float32) * h
    x = gen.normal_features(len(grid), 2, 5, 31)
    for r in (h, np.nextafter(h, np.float32(0)), np.nextafter(h, np.float32(1)), np.float32(np.sqrt(2.0)) * h, 2 * h):
        for periodic in ([0, 0, 0], [1, 1, 1]):
            _check_gauss(tiga, grid, x, None, r, box, periodic, r, use_cells=True, backward=False)


@pytest.mark.parametrize("n", [8, 9, 15, 16, 17, 33, 700])
def test_lennard_jones_in_one_cell(tiga, n):
    pos = _separated_points(n, np.full(3, 6.0, np.float32), 9, 0.45)
    _check_lj(tiga, pos, np.float32(5.9), np.full(3, 6.0, np.float32), [0, 0, 0])


@pytest.mark.parametrize("n", [8200, 40_000, 500_000, 600_000])
def test_binning_at_every_form_of_the_scan(tiga, n):
    """Cells as fine as the grid allows: 32, 154, 1926 and 2316 chunks of cells (the last above the limit of the folded totals)."""
    _check_bin(tiga, gen.uniform_points(n, 17), np.float32(1e-4), np.ones(3, np.float32), [0, 0, 0])


@pytest.mark.parametrize("n,r", [(9001, 0.05), (9001, 0.12), (24001, 0.9)])
@pytest.mark.parametrize("F", [1, 2, 3, 4])
def test_groups_with_infinite_features_and_widest_gaussian(tiga, F, n, r):
    """Sparse and dense stages, many stages: a row with an infinite source among its neighbours is that infinity, any other row is what it is
    without it; with a Gaussian that gives every distance the weight one the sums are the plain neighbour sums."""
    pos, x = gen.uniform_points(n, 76), gen.normal_features(n, F, 77)
    ones, r, per = np.ones(3, np.float32), np.float32(r), [0, 0, 0]
    rows = np.sort(gen.rng(76, 1).choice(n, 512, replace=False))
    y, A, cnt = oracle.radius_forward(pos, x, r, ones, per, oracle.MSG_GAUSS, p0=1e9, rows=rows)
    P = dev(pos, torch)
    for sigma in (1e14, np.inf):
        out, count, _ = tiga.tiga_apply_radius(P, dev(x, torch), r, ones, per, tiga.MSG_GAUSS, p0=sigma, want_count=True)
        assert np.array_equal(host(count)[rows], cnt) and rel_err(host(out)[rows], y, A) <= SUM_TOL
    d2 = ((pos.astype(np.float64) - pos[1234].astype(np.float64)) ** 2).sum(1)
    near = d2 <= np.float64(r) ** 2
    near[1234] = False
    sure = abs(d2 - np.float64(r) ** 2) > 1e-7
    x[1234] = 0.0
    plain = {kind: host(tiga.tiga_apply_radius(P, dev(x, torch), r, ones, per, kind, p0=0.1)[0]) for kind in (tiga.MSG_GAUSS, tiga.MSG_DIST)}
    x[1234] = np.inf
    for kind in plain:
        got = host(tiga.tiga_apply_radius(P, dev(x, torch), r, ones, per, kind, p0=0.1)[0])
        assert np.all(got[near & sure] == np.inf) and np.array_equal(got[~near & sure], plain[kind][~near & sure])


@pytest.mark.parametrize("F,n,r,periodic", [(1, 300_007, 0.0294, [0, 0, 0]), (4, 300_007, 0.0294, [1, 1, 1]), (4, 300_007, 0.0147, [1, 0, 1])])
def test_groups_in_units_of_32_points(tiga, F, n, r, periodic):
    pos, x = gen.uniform_points(n, 78), gen.normal_features(n, F, 78, 31)
    for kind in (tiga.MSG_GAUSS, tiga.MSG_DIST):
        _check_gauss(tiga, pos, x, None, np.float32(r), np.ones(3, np.float32), periodic, np.float32(r) / 2, kind=kind, use_cells=True, backward=False)


@pytest.mark.parametrize("per_cell", [22, 24, 25, 27, 40])
def test_narrow_features_in_slices_of_sixteen(tiga, per_cell):
    """Cells' form (the box holds the place of the padding) with more than 100 k points: slices of 16 queries, cells cut above 24."""
    cells, L = 17, 4e18
    n = per_cell * cells ** 3
    box = np.full(3, L, np.float32)
    pos = np.minimum(gen.uniform_points(n, 90 + per_cell) * box, np.nextafter(box, np.float32(0))).astype(np.float32)
    r = np.float32(L / cells / 1.002)
    _check_gauss(tiga, pos, gen.normal_features(n, 3, 91, 31), None, r, box, [1, 1, 1], r / np.float32(2), use_cells=True, backward=False)


@pytest.mark.parametrize("n,mean,periodic", [(1500, 9.0, [0, 0, 0]), (8192, 3.2, [0, 1, 0]), (24001, 1.0, [1, 1, 1]), (24001, 5.0, [0, 0, 0]), (94719, 3.5, [0, 0, 0]), (94721, 3.5, [1, 0, 0])])
@pytest.mark.parametrize("message", ["sum1", "sum4", "lj"])
def test_clustered_inputs_on_both_sides_of_the_rule(tiga, message, n, mean, periodic):
    """Sparse and dense on average, up to the size (94,720 points) that is done as cells and slices when more than a quarter of the points lie in cells
    that stand out from the mean, and above it; the smallest goes through the one-launch binning."""
    ones, r = np.ones(3, np.float32), float((mean / n) ** (1 / 3) / 1.002)
    pos = gen.clustered_points(n, 79)
    grid, _ = tiga.tiga_radius_grid(n, np.float32(r), ones, periodic)
    cell = np.minimum((pos * np.float32(grid)).astype(np.int64), np.array(grid) - 1)
    held = np.bincount((cell[:, 2] * grid[1] + cell[:, 1]) * grid[0] + cell[:, 0])
    per = n / np.prod(grid)
    assert 0.7 <= per and held[held > max(48, per + 6 * per ** 0.5 + 6)].sum() > n / 4 and min(grid) > 3
    rows = np.sort(gen.rng(79, 1).choice(n, 512, replace=False))
    kind = tiga.MSG_LJ if message == "lj" else tiga.MSG_DIST
    x = None if message == "lj" else gen.normal_features(n, 1 if message == "sum1" else 4, 79, 31)
    s = 2e-6 if message == "lj" else 0.0                      # below the smallest distance
    y, A, cnt = oracle.radius_forward(pos, x, np.float32(r), ones, periodic, kind, 1e-3, s, rows=rows)
    out, count, _ = tiga.tiga_apply_radius(dev(pos, torch), None if x is None else dev(x, torch), np.float32(r), ones, periodic, kind, p0=1e-3, p1=s, want_count=True)
    assert np.array_equal(host(count)[rows], cnt)
    assert rel_err(host(out)[rows], y, A) <= SUM_TOL

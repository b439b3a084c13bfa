"""GPU parity of the edge-network message over the radius relation (paper Appendix A) against the
fp64 oracle: outputs within 1e-5 and every gradient (features, positions, W1, b1, W2, b2) within
1e-4 of the sum of absolute contributions; neighbour counts bit-exact."""
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


def _check(tiga, pos, x, gy, r, box, per, params, use_cells=True, backward=True, kink_eps=1e-5, min_keep=0.95):
    y, A, cnt = oracle.radius_mlp_forward(pos, x, r, box, per, *params, use_cells=use_cells)
    pd, xd = dev(pos, torch), dev(x, torch)
    P = [dev(a, torch) for a in params]
    guard = Guard(torch)
    n = len(pos)
    out, count, ws = tiga.tiga_apply_radius_mlp(pd, xd, r, box, per, *P, out=guard.empty((n, params[2].shape[0])),
                                                count=guard.empty((n,), torch.int32),
                                                ws=guard.workspace(tiga.tiga_radius_workspace_bytes(n, x.shape[1], r, box, per)))
    guard.check()
    assert np.array_equal(host(count), cnt), "neighbour counts must be bit exact"
    assert rel_err(host(out), y, A) <= SUM_TOL
    if backward:
        # rows that touch a pre-activation within kink_eps of the ReLU kink are left out of the per-row
        # comparison: fp32 and fp64 may take different sides there and the derivative jumps
        ref = oracle.radius_mlp_backward(pos, x, gy, r, box, per, *params, use_cells=use_cells, kink_eps=kink_eps)
        keep = ref["kink"] == 0
        assert keep.mean() > min_keep
        g = tiga.tiga_apply_radius_mlp_backward(pd, xd, dev(gy, torch), r, box, per, *P, ws=ws, reuse_plan=True)
        for ours, name in (("grad_feat", "gx"), ("grad_pos", "gp")):
            assert rel_err(host(g[ours])[keep], ref[name][keep], ref["A" + name][keep]) <= GRAD_TOL, name
        for ours, name in (("grad_W1", "gW1"), ("grad_b1", "gb1"), ("grad_W2", "gW2"), ("grad_b2", "gb2")):
            assert rel_err(host(g[ours]), ref[name], ref["A" + name]) <= GRAD_TOL, name
        g2 = tiga.tiga_apply_radius_mlp_backward(pd, xd, dev(gy, torch), r, box, per, *P)      # rebuilds the bins
        assert torch.equal(g["grad_feat"], g2["grad_feat"]) and torch.equal(g["grad_pos"], g2["grad_pos"])


@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("dims", [(8, 16, 4), (8, 8, 4), (8, 32, 4), (1, 8, 1), (5, 16, 3), (13, 32, 2)])
def test_small_clouds(tiga, periodic, dims):
    f_in, hidden, f_out = dims
    n = 3000
    pos = gen.uniform_points(n, 60 + hidden)
    x = gen.normal_features(n, f_in, 61, 31)
    gy = gen.normal_features(n, f_out, 61, 32)
    r = gen.radius_for_expected_neighbours(n, 12.0)
    _check(tiga, pos, x, gy, r, np.ones(3, np.float32), [periodic] * 3, gen.mlp_params(f_in, hidden, f_out, 7))


def test_paper_example_shape(tiga):
    # Appendix A: 128 points, 8 node features, hidden 16, 4 outputs, cutoff 0.35
    pos = gen.uniform_points(128, 7)
    x = gen.normal_features(128, 8, 7, 31)
    gy = gen.normal_features(128, 4, 7, 32)
    params = gen.mlp_params(8, 16, 4, 7)
    ones = np.ones(3, np.float32)
    _check(tiga, pos, x, gy, np.float32(0.35), ones, [0, 0, 0], params, use_cells=False)
    _check(tiga, pos, x, gy, np.float32(0.35), ones, [1, 1, 1], params, use_cells=False)     # single cell, minimum image


def test_dense_cluster_overflows_the_lists(tiga):
    n = 2500
    pos = gen.uniform_points(n, 15) * np.float32(0.1) + np.float32(0.3)
    x = gen.normal_features(n, 8, 15, 31)
    gy = gen.normal_features(n, 4, 15, 32)
    # about 400 neighbours per point: many pre-activations per row, so a tighter kink margin
    _check(tiga, pos, x, gy, np.float32(0.04), np.ones(3, np.float32), [0, 0, 0], gen.mlp_params(8, 16, 4, 9),
           kink_eps=3e-6, min_keep=0.9)      # 93 % of the rows are kept with this margin


@pytest.mark.parametrize("hidden", [8, 32])
def test_surface_stand_in(tiga, hidden):
    """35,947 points on a closed surface with cutoff 0.015 (the size and radius of the paper's
    differentiated edge-network study; the geometry itself is synthetic)."""
    n = 35_947
    pos = gen.surface_points(n, 3)
    x = gen.normal_features(n, 8, 3, 31)
    gy = gen.normal_features(n, 4, 3, 32)
    _check(tiga, pos, x, gy, np.float32(0.015), np.ones(3, np.float32), [0, 0, 0], gen.mlp_params(8, hidden, 4, 3))


@pytest.mark.parametrize("hidden", [8, 16, 32])
@pytest.mark.parametrize("f_in", [1, 4, 5, 9, 12, 13])
def test_every_split_of_lanes_and_staged_features(tiga, f_in, hidden):
    """32 / hidden pairs advance together and features are staged four at a time: every combination, on a cloud of 30 to
    250 neighbours that spans slices, several stage chunks (144 candidates), list batches (176 pairs) and wrapped
    faces.  (No query has only a few neighbours: a single message, or a single pair's gradient, may cancel to nearly
    nothing, and a tolerance relative to it would test the rounding of the terms it is formed from.  The thin background of
    test_messages_that_cancel_lose_no_precision has such queries, in a norm over all rows.)"""
    n = 1500
    pos = (gen.uniform_points(n, 70 + f_in) * np.float32(0.35) + np.float32(0.8)) % np.float32(1.0)
    x, gy = gen.normal_features(n, f_in, 72, 31), gen.normal_features(n, 3, 72, 32)
    _check(tiga, pos, x, gy, np.float32(0.12), np.ones(3, np.float32), [1, 1, 1], gen.mlp_params(f_in, hidden, 3, 8), min_keep=0.5)


@pytest.mark.parametrize("f_in,hidden", [(8, 32), (13, 16)])
def test_backward_calls_share_a_plan(tiga, f_in, hidden):
    """A reused plan is only read: two cotangents of the same points, on two streams at once, give what each gives alone."""
    n = 30_000
    pos, x = dev(gen.surface_points(n, 5), torch), dev(gen.normal_features(n, f_in, 6, 31), torch)
    P = [dev(a, torch) for a in gen.mlp_params(f_in, hidden, 4, 7)]
    r, ones = np.float32(0.016), np.ones(3, np.float32)
    gys = [dev(gen.normal_features(n, 4, 8, 32 + i), torch) for i in range(2)]
    _, _, ws = tiga.tiga_apply_radius_mlp(pos, x, r, ones, [0, 0, 0], *P)
    plan = ws.clone()
    alone = [tiga.tiga_apply_radius_mlp_backward(pos, x, gy, r, ones, [0, 0, 0], *P, ws=ws, reuse_plan=True) for gy in gys]
    torch.cuda.synchronize()
    assert torch.equal(ws, plan)
    streams = [torch.cuda.Stream() for _ in gys]
    for _ in range(5):
        got = [None, None]
        for i, s in enumerate(streams):
            with torch.cuda.stream(s):
                got[i] = tiga.tiga_apply_radius_mlp_backward(pos, x, gys[i], r, ones, [0, 0, 0], *P, ws=ws, reuse_plan=True)
        torch.cuda.synchronize()
        for a, b in zip(alone, got):
            assert torch.equal(a["grad_feat"], b["grad_feat"]) and torch.equal(a["grad_pos"], b["grad_pos"])
            for name in ("grad_W1", "grad_b1", "grad_W2", "grad_b2"):      # sums of 450 k pairs in any order
                assert float((a[name] - b[name]).norm()) <= 1e-4 * float(a[name].norm()), name


def test_infinite_inputs_stay_where_they_belong(tiga):
    """An infinite feature makes its neighbours' outputs infinite (not NaN: every first-layer feature weight and every
    second-layer weight is positive); an isolated point with an infinite feature or cotangent adds nothing to any other
    gradient and keeps zeros; a cotangent that is not finite does not reach the parameters of units that are off."""
    n, f_in, hidden, f_out = 1500, 8, 16, 2
    pos = gen.uniform_points(n, 44) * np.float32(0.8)
    pos[:2] = [[0.95, 0.95, 0.95], [0.95, 0.05, 0.95]]
    x, gy = gen.normal_features(n, f_in, 45, 31), gen.normal_features(n, f_out, 46, 32)
    W1, b1, W2, b2 = gen.mlp_params(f_in, hidden, f_out, 7)
    W1, W2 = np.abs(W1) + np.float32(0.01), np.abs(W2) + np.float32(0.01)
    W1[5], b1[5] = 0, -1                                        # this unit is never on
    P = [dev(a, torch) for a in (W1, b1, W2, b2)]
    r, ones, per = np.float32(0.09), np.ones(3, np.float32), [0, 0, 0]

    def both(x, gy):
        X = dev(x, torch)
        out, count, ws = tiga.tiga_apply_radius_mlp(dev(pos, torch), X, r, ones, per, *P, want_count=True)
        g = tiga.tiga_apply_radius_mlp_backward(dev(pos, torch), X, dev(gy, torch), r, ones, per, *P, ws=ws, reuse_plan=True)
        return host(out), host(count), {k: host(v) for k, v in g.items()}

    out, count, g = both(x, gy)
    assert count[0] == count[1] == 0 and count[7] > 2
    d2 = ((pos.astype(np.float64) - pos[7].astype(np.float64)) ** 2).sum(1)
    near = d2 <= np.float64(r) ** 2
    near[7] = False
    assert near.sum() == count[7]
    far, lone, odd = x.copy(), x.copy(), gy.copy()
    far[7] = np.inf
    out2, _, _ = both(far, gy)
    assert np.all(out2[near] == np.inf) and np.array_equal(out2[~near], out[~near])
    lone[0] = np.inf
    odd[1] = np.nan
    out3, _, g3 = both(lone, odd)
    assert np.array_equal(out3, out) and np.all(out3[:2] == 0)
    for k in ("grad_feat", "grad_pos"):
        assert np.array_equal(g3[k], g[k]) and np.all(g3[k][:2] == 0)
    for k in ("grad_W1", "grad_b1", "grad_W2", "grad_b2"):      # added up in any order
        assert np.allclose(g3[k], g[k], rtol=1e-4, atol=1e-4 * np.abs(g[k]).max()), k
    odd = gy.copy()
    odd[7] = np.inf
    g4 = both(x, odd)[2]
    assert np.all(g4["grad_W1"][5] == 0) and g4["grad_b1"][5] == 0
    assert np.all(np.isinf(g4["grad_W1"][0, 3:]) | np.isnan(g4["grad_W1"][0, 3:]))


@pytest.mark.parametrize("weight", ["W1", "b1", "W2", "b2"])
def test_isolated_points_keep_the_zero_vector_for_any_weights(tiga, weight):
    pos = (np.stack(np.meshgrid(*[np.arange(5)] * 3, indexing="ij"), -1).reshape(-1, 3) * 0.2 + 0.1).astype(np.float32)
    n = len(pos)
    params = dict(zip(("W1", "b1", "W2", "b2"), gen.mlp_params(3, 8, 2, 7)))
    params[weight] = np.full_like(params[weight], np.inf)
    P = [dev(a, torch) for a in params.values()]
    X, G = dev(gen.normal_features(n, 3, 1, 31), torch), dev(gen.normal_features(n, 2, 1, 32), torch)
    out, _, ws = tiga.tiga_apply_radius_mlp(dev(pos, torch), X, np.float32(0.1), np.ones(3, np.float32), [0, 0, 0], *P)
    g = tiga.tiga_apply_radius_mlp_backward(dev(pos, torch), X, G, np.float32(0.1), np.ones(3, np.float32), [0, 0, 0], *P, ws=ws, reuse_plan=True)
    assert not host(out).any() and not any(host(v).any() for v in g.values())


@pytest.mark.parametrize("dims", [(8, 32, 4), (13, 16, 3), (5, 32, 2), (1, 8, 1)])
def test_messages_that_cancel_lose_no_precision(tiga, dims):
    """Output bias chosen so that the messages average to zero: behind the ReLU the sums over a query's pairs are then far
    larger than the result.  2-norm errors relative to the sums of |contributions|: what remains is the rounding of the
    pre-activations and of the result.  Measured: messages added one by one 1.3e-8 to 2.4e-8 (positions 2.5e-8 to 7e-8),
    this form 0.8e-8 to 2.3e-8 (1.6e-8 to 4.1e-8), the same sums rounded to fp32 before W2 and W1^T 4.4e-8 to 17e-8."""
    f_in, hidden, f_out = dims
    n = 3000
    pos, r, ones, per = gen.clustered_points(n, 1), np.float32(0.03), np.ones(3, np.float32), [0, 0, 0]
    x, gy = gen.normal_features(n, f_in, 73, 31), gen.normal_features(n, f_out, 73, 32)
    W1, b1, W2, b2 = gen.mlp_params(f_in, hidden, f_out, 9)
    y0, _, cnt = oracle.radius_mlp_forward(pos, x, r, ones, per, W1, b1, W2, 0 * b2, use_cells=True)
    params = (W1, b1, W2, (-y0.sum(0) / cnt.sum()).astype(np.float32))
    y, A, _ = oracle.radius_mlp_forward(pos, x, r, ones, per, *params, use_cells=True)
    P = [dev(a, torch) for a in params]
    out, _, ws = tiga.tiga_apply_radius_mlp(dev(pos, torch), dev(x, torch), r, ones, per, *P)
    ref = oracle.radius_mlp_backward(pos, x, gy, r, ones, per, *params, use_cells=True, kink_eps=1e-5)
    keep = ref["kink"] == 0
    g = tiga.tiga_apply_radius_mlp_backward(dev(pos, torch), dev(x, torch), dev(gy, torch), r, ones, per, *P, ws=ws, reuse_plan=True)
    error = lambda got, want, A: np.linalg.norm(got - want) / np.linalg.norm(A)
    assert error(host(out), y, A) <= 3.5e-8
    assert error(host(g["grad_feat"])[keep], ref["gx"][keep], ref["Agx"][keep]) <= 3e-8
    assert error(host(g["grad_pos"])[keep], ref["gp"][keep], ref["Agp"][keep]) <= 6e-8

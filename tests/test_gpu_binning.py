"""The binning rule on the GPU at its edges: pixels and ranges of points aimed at cell borders, range limits, the
octant borders, the axis and the ends of the FP32 range, bit for bit against the oracle's plain rule."""
import math

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _edge_points(pp, rng, n):
    """Points within a few roundings of a column border, a row border, a range limit or an octant border."""
    cols, rows = int(pp.cols), int(pp.rows)
    az = math.pi - rng.integers(0, cols + 1, n) / float(pp.s_az)
    el = float(pp.el_top) - rng.integers(0, rows + 1, n) / float(pp.s_el)
    kind = rng.integers(0, 5, n)
    az = np.where(kind == 1, rng.uniform(-math.pi, math.pi, n), az)
    el = np.where(kind == 0, rng.uniform(-0.8, 0.8, n), el)
    az = np.where(kind == 4, rng.integers(-4, 5, n) * math.pi / 4, az)
    el = np.where(kind == 4, rng.integers(-1, 2, n) * math.pi / 4, el)
    r = np.exp(rng.uniform(math.log(0.5), math.log(90.0), n))
    r = np.where(kind == 3, np.where(rng.random(n) < 0.5, float(pp.r_min), float(pp.r_max)), r)
    p = np.stack([r * np.cos(el) * np.cos(az), r * np.cos(el) * np.sin(az), r * np.sin(el)], 1).astype(np.float32)
    for k in range(3):  # a few units in the last place either way
        p[:, k] = p[:, k] * (1 + rng.integers(-3, 4, n) * 2.0 ** -24).astype(np.float32)
    special = [0.0, -0.0, 1e-40, -1e-40, 1e-20, 1e19, -1e19, 3e38, np.inf, -np.inf, np.nan, 1.0, -1.0]
    m = n // 16
    p[:m] = rng.choice(np.array(special, np.float32), (m, 3))
    return np.concatenate([p, np.ones((n, 1), np.float32)], 1)


@pytest.mark.parametrize("rows,cols,half_deg,r_min,r_max", [
    (3, 5, 30.0, 0.1, 100.0), (16, 512, 15.0, 0.3, 30.0), (64, 1024, 16.6, 0.5, 120.0), (333, 1777, 45.0, 0.3, 150.0),
    (1024, 4096, 45.0, 0.3, 150.0), (7, 2000, 80.0, 0.0, 1e19), (5, 130000, 1.0, 0.5, 1e30)])
def test_projection_at_cell_edges_is_the_rule_bit_for_bit(rows, cols, half_deg, r_min, r_max):
    torch = pytest.importorskip("torch")
    import paper_2101_00585_gb300 as up
    h = math.radians(half_deg)
    pp = synth.Pano.make(rows, cols, h, -h, r_min, r_max)
    for rep in range(4):
        rng = np.random.default_rng((rows, cols, rep))
        pts = _edge_points(pp, rng, min(60000, 8 * rows * cols))
        with np.errstate(all="ignore"):
            d_ref, i_ref = oracle.project(pts, pp)
        depth, idx, _ = up.project(torch.from_numpy(pts).cuda(), pp)
        assert np.array_equal(idx.cpu().numpy(), i_ref)
        assert np.array_equal(depth.cpu().numpy().view(np.uint32), d_ref.view(np.uint32))


@pytest.mark.parametrize("sw,kf", [((64, 512, 20.0), (32, 256, 20.0)), ((64, 512, 20.0), (96, 768, 60.0)),
                                   ((31, 901, 15.0), (62, 1802, 15.0)), ((16, 512, 15.0), (45, 90, 80.0)),
                                   ((128, 2048, 22.5), (64, 1024, 22.5)), ((5, 120000, 1.0), (40, 3000, 1.0))])
def test_association_at_cell_corners_is_the_rule_point_for_point(sw, kf):
    """Keyframe pixel centres that fall on sweep cell corners (sizes in ratios of two) and near them (small turns),
    steep points beyond 45 degrees, ranges at both limits: with the gates open a candidate's score counts the
    samples whose sweep cell holds a point, and a random half of the cells do, so it equals the oracle's count
    only if every sample's cell is the rule's."""
    torch = pytest.importorskip("torch")
    import paper_2101_00585_gb300 as up
    pano = lambda p: synth.Pano.make(p[0], p[1], math.radians(p[2]), -math.radians(p[2]), 0.5, 40.0)  # noqa: E731
    sp, kp = pano(sw), pano(kf)
    rng = np.random.default_rng((sw[1], kf[1]))
    depth = np.exp(rng.uniform(math.log(0.4), math.log(50.0), kf[:2])).astype(np.float32)
    depth[rng.random(kf[:2]) < 0.1] = 0.5
    depth[rng.random(kf[:2]) < 0.1] = 40.0
    depth[rng.random(kf[:2]) < 0.1] = 0.0
    kn = np.zeros(kf[:2] + (4,), np.float32)
    kn[..., 2], kn[..., 3] = 1.0, 1.0
    sp4 = np.zeros(sw[:2] + (4,), np.float32)
    sn4 = np.zeros_like(sp4)
    held = rng.random(sw[:2]) < 0.5
    sp4[held] = [1.0, 2.0, 3.0, 1.0]
    sn4[held] = [0.0, 0.0, 1.0, 1.0]
    twists = np.zeros((12, 6))
    for i in range(1, 12):
        twists[i] = rng.standard_normal(6) * 10.0 ** -rng.uniform(1, 7)
    poses = np.stack([oracle.se3_exp_left(t, np.hstack([np.eye(3), np.zeros((3, 1))])).reshape(12) for t in twists])
    gate = dict(d_max=1e3, cos_theta_max=-2.0)
    ref, _ = oracle.grid_score(depth, kn, kp, sp4, sn4, sp, poses, 1, oracle.Params(**gate))
    k, s = up.KeyframeBuffer(kp), up.SweepFrame(sp)
    k.set(torch.from_numpy(depth).cuda(), torch.from_numpy(kn).cuda())
    s.set(torch.from_numpy(sp4).cuda(), torch.from_numpy(sn4).cuda())
    scores, _, _ = up.grid_score(k, s, torch.from_numpy(poses).cuda(), up.Params(**gate), 1)
    assert np.array_equal(scores.cpu().numpy(), ref)
    # the registration's and the batched form's association of the same candidates
    state = up.IcpState(k)
    prm = up.Params(**gate, max_iters=1)
    batch = up.Batch(s, [k], 12)
    batch.run(torch.from_numpy(poses).cuda(), prm)
    recs = batch.read_stats()
    for i in range(12):
        state.pose.copy_(torch.from_numpy(poses[i]).cuda())
        up.icp(k, s, state, prm)
        assert state.read_stats()["inliers"] == ref[i] and recs[i]["inliers"] == ref[i]

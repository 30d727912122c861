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

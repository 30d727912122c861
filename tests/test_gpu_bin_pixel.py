"""The registration's fast binning against the plain rule, cell for cell: points anywhere on the sphere, points within a
few roundings of cell borders, range limits, the 45-degree borders and the axis, the ends of the FP32 range, and
panoramas that reach the zenith, look only up or down, or take every range."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

import synth
from tests.test_gpu_binning import _edge_points

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2101_00585_gb300 import api, build
    so = str(tmp_path_factory.mktemp("probe") / "libprobe.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "bin_probe.cu")
    subprocess.run([build._nvcc()] + build.ARCH + build.NVCC_FLAGS + ["-shared", "-o", so, src, "-lcudart"], check=True)
    fn = ctypes.CDLL(so).probe_bin
    fn.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]

    def cells(pts, pp):
        import torch
        t = torch.from_numpy(np.ascontiguousarray(pts, np.float32)).cuda()
        out = torch.full((2, len(t)), -7, dtype=torch.int32, device="cuda")
        ps = api.pano_struct(pp)
        torch.cuda.synchronize()
        assert fn(t.data_ptr(), len(t), ctypes.addressof(ps), out[0].data_ptr(), out[1].data_ptr()) == 0
        return out.cpu().numpy()
    return cells


def _steep_edges(pp, rng, n):
    """Points within a few roundings of a row border, a column border or 45 degrees, anywhere up or down."""
    top, s_el, rows = float(pp.el_top), float(pp.s_el), int(pp.rows)
    el = np.where(rng.random(n) < 0.7, top - rng.integers(0, rows + 1, n) / s_el, rng.uniform(-1.6, 1.6, n))
    el = np.where(rng.random(n) < 0.2, rng.choice([-1.0, 1.0], n) * (math.pi / 4 + rng.integers(-4, 5, n) * 2.0 ** -24),
                  el)
    az = rng.uniform(-math.pi, math.pi, n)
    az = np.where(rng.random(n) < 0.3, math.pi - rng.integers(0, int(pp.cols) + 1, n) / float(pp.s_az), az)
    r = np.exp(rng.uniform(math.log(0.2), math.log(200.0), n))
    p = np.stack([r * np.cos(el) * np.cos(az), r * np.cos(el) * np.sin(az), r * np.sin(el)], 1).astype(np.float32)
    p *= (1 + rng.integers(-3, 4, p.shape) * 2.0 ** -24).astype(np.float32)
    return np.concatenate([p, np.ones((n, 1), np.float32)], 1)


@pytest.mark.parametrize("rows,cols,top_deg,bottom_deg,r_min,r_max", [
    (64, 1024, 16.6, -16.6, 0.5, 120.0), (512, 2048, 45.0, -45.0, 0.3, 150.0), (1024, 4096, 60.0, -60.0, 0.3, 150.0),
    (333, 1777, 80.0, -80.0, 0.3, 150.0), (64, 1024, 90.0, 0.0, 0.0, 120.0), (64, 1024, 89.0, 46.0, 0.3, 120.0),
    (37, 901, -50.0, -90.0, 0.3, 120.0), (2000, 2000, 90.0, -90.0, 0.0, 1e19), (7, 300, 90.0, -90.0, 1e-30, 1e30),
    (3, 5, 70.0, -80.0, 0.0, math.inf), (16, 512, 15.0, -15.0, 0.3, math.inf), (1, 1, 1.0, -1.0, 1.0, 1.0),
    (60000, 8, 60.0, 59.0, 0.1, 50.0), (5, 130000, 80.0, -1.0, 0.5, 40.0)])
def test_cells_are_the_rules(probe, rows, cols, top_deg, bottom_deg, r_min, r_max):
    pp = synth.Pano.make(rows, cols, math.radians(top_deg), math.radians(bottom_deg), r_min, r_max)
    seen = 0
    for rep in range(3):
        rng = np.random.default_rng((rows, cols, rep))
        d = rng.standard_normal((200000, 3))
        d *= np.exp(rng.uniform(-2, 5, (200000, 1))) / np.linalg.norm(d, axis=1, keepdims=True)
        pts = np.concatenate([d, np.ones((len(d), 1))], 1).astype(np.float32)
        with np.errstate(over="ignore", invalid="ignore"):
            pts = np.concatenate([pts, _edge_points(pp, rng, 200000), _steep_edges(pp, rng, 600000)])
        cell, rule = probe(pts, pp)
        assert np.array_equal(cell, rule)
        assert rule.min() >= -1 and rule.max() < rows * cols
        seen += (rule >= 0).sum()
    assert seen > 0

"""Keyframes with more samples than the persistent launch holds in shared memory: what does not fit goes to tensor
memory and, past that, to global memory.  A box seen from inside, so every keyframe pixel can hold a sample.

Tolerance: the launch and the single-step kernel add the same FP32 products in different orders, at most about a
hundred to a partial sum before exact or compensated sums take over: 100 * 2^-24 = 6e-6 in the worst case,
1e-6 with random signs; the counts are integers and equal."""
import math

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _box(pp, half=(6.0, 4.0, 3.0)):
    el = float(pp.el_top) - (np.arange(pp.rows) + 0.5) / float(pp.s_el)
    az = math.pi - (np.arange(pp.cols) + 0.5) / float(pp.s_az)
    d = np.stack([np.cos(el)[:, None] * np.cos(az), np.cos(el)[:, None] * np.sin(az),
                  np.broadcast_to(np.sin(el)[:, None], (pp.rows, pp.cols))], -1)
    t = np.array(half) / np.maximum(np.abs(d), 1e-9)
    k = t.argmin(-1)
    n = np.zeros_like(d)
    np.put_along_axis(n, k[..., None], -np.sign(np.take_along_axis(d, k[..., None], -1)), -1)
    return np.take_along_axis(t, k[..., None], -1)[..., 0].astype(np.float32), n.astype(np.float32), d


@pytest.mark.parametrize("rows,cols,fill,f16,loss", [
    (1024, 4096, 1.0, False, 0), (1024, 4096, 1.0, True, 1), (1024, 4096, 0.6, False, 1), (1024, 4096, 0.6, True, 0),
    (777, 3001, 0.9, False, 0), (700, 2350, 1.0, True, 0), (512, 2400, 1.0, False, 0)])
def test_dense_keyframe_steps_and_update(rows, cols, fill, f16, loss):
    torch = pytest.importorskip("torch")
    import paper_2101_00585_gb300 as up
    rng = np.random.default_rng((rows, cols))
    kp = synth.Pano.make(rows, cols, math.radians(45.0), -math.radians(45.0), 0.3, 150.0)
    sp = synth.Pano.make(64, 1024, math.radians(40.0), -math.radians(40.0), 0.3, 120.0)
    kd, kn, _ = _box(kp)
    held = rng.random(kd.shape) < fill
    nw = np.concatenate([kn, rng.integers(1, 11, kd.shape + (1,)).astype(np.float32)], -1) * held[..., None]
    sd, sn, sdir = _box(sp)
    pix = np.concatenate([(sd[..., None] * sdir), np.ones(sd.shape + (1,))], -1).astype(np.float32)
    snv = np.concatenate([sn, np.ones(sd.shape + (1,), np.float32)], -1)
    prec = up.F16 if f16 else up.F32
    off = synth.pose(synth.rot_axis_angle([0.2, 0.1, 1.0], 0.01), [0.05, -0.03, 0.02])

    def make(**kw):
        t = up.Tracker(sp, kp, up.Params(loss=loss, max_iters=4), precision=prec, constant_velocity=False, **kw)
        t.kf.set(torch.from_numpy(kd * held).cuda(), torch.from_numpy(nw).cuda().to(t.kf.nw.dtype))
        t.sw.set(torch.from_numpy(pix).cuda(), torch.from_numpy(snv).cuda().to(t.sw.nrm.dtype))
        return t

    t = make()
    one = up.Params(loss=loss, max_iters=1)
    states = []
    for call in (up.icp, up.icp_step):
        st = up.IcpState(t.kf)
        st.pose.copy_(torch.from_numpy(off.reshape(12)).cuda())
        call(t.kf, t.sw, st, one)
        states.append(st.read_stats())
    a, b = states
    assert a["status"] == 0 and a["inliers"] == b["inliers"] > 0.5 * held.sum() * 0.8
    for key in ("A", "b"):
        x, y = np.array(a[key]), np.array(b[key])
        assert np.linalg.norm(x - y) <= 6e-6 * max(np.linalg.norm(y), np.sqrt(b["sse"] * np.array(b["A"]).max()))
    # the update inside the launch against the update as a call of its own, at the pose the launch registered
    from paper_2101_00585_gb300 import _abi
    import ctypes
    ks, ss = t.kf.struct(), t.sw.struct()
    before = t.kf.depth.clone(), t.kf.nw.clone()
    s = torch.cuda.current_stream().cuda_stream
    p = lambda v: ctypes.c_void_p(v.data_ptr())  # noqa: E731
    t.prev.copy_(torch.from_numpy(off.reshape(12)).cuda())
    _abi.check("upslam_track", _abi.lib().upslam_track(
        ctypes.byref(ks), ctypes.byref(ss), p(t.prev), p(t.motion), p(t.state.pose), 1, ctypes.byref(t._ip),
        ctypes.byref(t._fp), p(t.state.stats), p(t.state.ws), t.state.ws_bytes, p(t.kf.zbuf), s))
    after = t.kf.depth.clone(), t.kf.nw.clone()
    assert t.state.read_stats()["accepted"] == 1
    t.kf.depth.copy_(before[0])
    t.kf.nw.copy_(before[1])
    up.fuse(t.kf, t.sw, t.state.pose, t.params, t.state.stats)
    assert torch.equal(t.kf.depth.view(torch.int32), after[0].view(torch.int32))
    assert torch.equal(t.kf.nw, after[1])
    # a second launch finds the tensor memory free again and gives the same bits
    st2 = up.IcpState(t.kf)
    for _ in range(2):
        t.kf.depth.copy_(before[0])
        t.kf.nw.copy_(before[1])
        st2.pose.copy_(torch.from_numpy(off.reshape(12)).cuda())
        up.icp(t.kf, t.sw, st2, one)
        assert st2.read_stats()["A"] == a["A"]

"""The batched form's FP64 solve on systems of any scale: an IRLS weight 1 / max(|r|, loss_delta) with a large
loss_delta is the least-squares weight times a constant, so the normal equations are those of the squared error scaled
down, to where products of many of their elements are no longer normal numbers.

Tolerance of xi against LAPACK on the recorded system: reciprocals good to 2^-44 (6e-14) and sums of FP64 products,
amplified by at most the condition number of these systems (below 1e5): 1e-16 * 1e5 * 10 terms = 1e-10, taken as 1e-9
relative."""
import math

import numpy as np
import pytest

import synth
from tests.helpers import room_sweep_and_keyframe

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("loss_delta", [2.0 ** 20, 2.0 ** 70, 2.0 ** 80, 2.0 ** 90, 2.0 ** 100, 1e30, 2.0 ** 110,
                                        3.0e38])
def test_batched_step_solves_scaled_systems(loss_delta):
    torch = pytest.importorskip("torch")
    import paper_2101_00585_gb300 as up
    c, prm, sp4, sn4, kd, kn = room_sweep_and_keyframe(noise=True)
    kf = up.KeyframeBuffer(c.kf)
    kf.set(torch.from_numpy(kd).cuda(), torch.from_numpy(kn).cuda())
    sw = up.SweepFrame(c.sweep)
    sw.set(torch.from_numpy(sp4).cuda(), torch.from_numpy(sn4).cuda())
    off = [synth.pose(synth.rot_axis_angle([0.3, -0.2, 1.0], math.radians(a)), [t, -t, 0.2 * t])
           for a, t in ((0.0, 0.0), (0.3, 0.01), (3.0, 0.05))]
    T0 = torch.from_numpy(np.stack([synth.pose_mul(c.T_true, o).reshape(12) for o in off])).cuda()
    one = dict(max_iters=1, d_max=2.0, eps_rot=0.0, eps_trans=0.0)
    batch = up.Batch(sw, [kf], len(off))
    batch.run(T0, up.Params(loss=1, loss_delta=loss_delta, **one))
    for st in batch.read_stats():
        assert st["status"] == 0 and st["iters"] == 1
        A = np.zeros((6, 6))
        A[np.triu_indices(6)] = st["A"]
        A = A + np.triu(A, 1).T
        assert A[3, 3] <= 1.01 * st["inliers"] / loss_delta  # the weight is the constant
        assert np.linalg.cond(A) < 1e5
        ref = np.linalg.solve(A, -np.array(st["b"]))
        assert np.linalg.norm(np.array(st["xi"]) - ref) <= 1e-9 * np.linalg.norm(ref)

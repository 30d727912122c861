"""The persistent launch's FP64 solve and SE(3) update against LAPACK and expm on the record it writes: both forms
(3 x 3 blocks; elimination, taken when pivot_eps asks for more than the blocks certify), small and large steps.

Tolerance of xi: reciprocals good to 2^-44 (6e-14) and sums of FP64 products, amplified by at most the condition
number of these systems (below 1e5): 1e-16 * 1e5 * 10 terms = 1e-10, taken as 1e-9 relative."""
import math

import numpy as np
import pytest
from scipy.linalg import expm

import synth
from tests.helpers import IDENTITY, room_sweep_and_keyframe

pytestmark = pytest.mark.gpu


def _twist(xi):
    M = np.zeros((4, 4))
    w = xi[:3]
    M[:3, :3] = [[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]]
    M[:3, 3] = xi[3:]
    return M


@pytest.mark.parametrize("pivot_eps", [1e-12, 2.9e-8, 1e-7])  # blocks, blocks at their limit, elimination
@pytest.mark.parametrize("angle_deg,trans", [(0.0, 0.0), (0.003, 1e-4), (0.3, 0.01), (3.0, 0.05), (8.0, 0.1)])
def test_step_solves_the_recorded_system(pivot_eps, angle_deg, trans):
    torch = pytest.importorskip("torch")
    import paper_2101_00585_gb300 as up
    c, prm, sp4, sn4, kd, kn = room_sweep_and_keyframe(noise=True)
    kf = up.KeyframeBuffer(c.kf)
    kf.set(torch.from_numpy(kd).cuda(), torch.from_numpy(kn).cuda())
    sw = up.SweepFrame(c.sweep)
    sw.set(torch.from_numpy(sp4).cuda(), torch.from_numpy(sn4).cuda())
    off = synth.pose(synth.rot_axis_angle([0.3, -0.2, 1.0], math.radians(angle_deg)), [trans, -trans, 0.2 * trans])
    T0 = synth.pose_mul(c.T_true, off)
    state = up.IcpState(kf)
    state.pose.copy_(torch.from_numpy(T0.reshape(12)).cuda())
    up.icp(kf, sw, state, up.Params(max_iters=1, pivot_eps=pivot_eps, d_max=2.0, eps_rot=0.0, eps_trans=0.0))
    st = state.read_stats()
    assert st["status"] == 0 and st["iters"] == 1 and st["converged"] == 0
    A = np.zeros((6, 6))
    A[np.triu_indices(6)] = st["A"]
    A = A + np.triu(A, 1).T
    assert np.linalg.cond(A) < 1e5
    ref = np.linalg.solve(A, -np.array(st["b"]))
    xi = np.array(st["xi"])
    assert np.linalg.norm(xi - ref) <= 1e-9 * np.linalg.norm(ref)
    # T <- exp(xi^) T: entries of order one and a few metres, sums of a dozen FP64 roundings
    T = state.pose.cpu().numpy().reshape(3, 4)
    want = expm(_twist(xi)) @ np.vstack([T0, [0, 0, 0, 1]])
    assert np.abs(T - want[:3]).max() < 1e-13 * 8


@pytest.mark.parametrize("pivot_eps", [1e-12, 1e-7])
def test_convergence_thresholds_are_both_needed(pivot_eps):
    torch = pytest.importorskip("torch")
    import paper_2101_00585_gb300 as up
    c, prm, sp4, sn4, kd, kn = room_sweep_and_keyframe(noise=True)
    kf = up.KeyframeBuffer(c.kf)
    kf.set(torch.from_numpy(kd).cuda(), torch.from_numpy(kn).cuda())
    sw = up.SweepFrame(c.sweep)
    sw.set(torch.from_numpy(sp4).cuda(), torch.from_numpy(sn4).cuda())
    for er, et, conv in ((1.0, 1.0, 1), (0.0, 1.0, 0), (1.0, 0.0, 0)):
        state = up.IcpState(kf)
        state.pose.copy_(torch.from_numpy(IDENTITY.reshape(12)).cuda())
        up.icp(kf, sw, state, up.Params(max_iters=3, pivot_eps=pivot_eps, eps_rot=er, eps_trans=et))
        st = state.read_stats()
        assert st["converged"] == conv and st["iters"] == (1 if conv else 3)

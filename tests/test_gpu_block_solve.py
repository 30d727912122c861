"""The warps' FP64 6x6 solve (3 x 3 blocks, or elimination where the blocks would lose digits) on systems chosen for
it: spectra down to 1e-9 in random bases, rows of unlike scale, any overall scale, and systems without a solution.

Tolerance: with the rows and columns scaled to a unit diagonal (what the solve's products and the certificate see)
either form's reciprocals are good to 2^-44 and its sums to a few units of 2^-53, amplified by at most the scaled
matrix's condition number; eight of the first are allowed, 2^-41 times that number.  The reference is rational."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

IU = np.triu_indices(6)


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2101_00585_gb300 import build
    so = str(tmp_path_factory.mktemp("probe") / "libprobe.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "solve_probe.cu")
    subprocess.run([build._nvcc()] + build.ARCH + build.NVCC_FLAGS + ["-shared", "-o", so, src, "-lcudart"], check=True)
    fn = ctypes.CDLL(so).probe_solve
    fn.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_double, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]

    def solve(systems, pivot_eps=1e-12, elim=False):
        import torch
        t = torch.from_numpy(np.ascontiguousarray(systems, np.float64)).cuda()
        xi = torch.zeros(len(t), 6, dtype=torch.float64, device="cuda")
        ok = torch.zeros(len(t), dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert fn(t.data_ptr(), len(t), pivot_eps, int(elim), xi.data_ptr(), ok.data_ptr()) == 0
        return xi.cpu().numpy(), ok.cpu().numpy().astype(bool)
    return solve


def _exact(t):
    U = [[None] * 6 for _ in range(6)]
    for v, i, j in zip(t[:21], *IU):
        U[i][j] = U[j][i] = Fraction(float(v))
    y = [-Fraction(float(v)) for v in t[21:]]
    for j in range(6):
        for i in range(j + 1, 6):
            m = U[i][j] / U[j][j]
            y[i] -= m * y[j]
            for k in range(j, 6):
                U[i][k] -= m * U[j][k]
    x = [None] * 6
    for i in range(5, -1, -1):
        x[i] = (y[i] - sum(U[i][k] * x[k] for k in range(i + 1, 6))) / U[i][i]
    return np.array([float(v) for v in x])


def _systems(cond, graded, scale, n, seed):
    rng = np.random.default_rng(seed)
    out = np.empty((n, 27))
    for i in range(n):
        ev = np.exp(rng.uniform(-np.log(cond), 0.0, 6))
        ev[:2] = 1.0, 1.0 / cond
        Q, _ = np.linalg.qr(rng.standard_normal((6, 6)))
        D = 2.0 ** rng.uniform(-graded, graded, 6)
        A = (Q * ev @ Q.T) * D[:, None] * D
        out[i, :21], out[i, 21:] = A[IU], rng.standard_normal(6) * D
    return out * 2.0 ** scale


def _scaled(t):
    A = np.zeros((6, 6))
    A[IU] = t[:21]
    A = A + np.triu(A, 1).T
    d = np.sqrt(np.diag(A))
    return d, np.linalg.cond(A / d[:, None] / d)


@pytest.mark.parametrize("cond", [3.0, 1e2, 1e3, 1e4, 1e5, 1e6, 1e7])
@pytest.mark.parametrize("graded,scale", [(0, 16), (3, 0), (0, -55), (0, -60), (0, -75), (0, -84), (0, -100),
                                          (0, 80), (0, 84), (0, 120)])
def test_solution_is_good_to_the_condition_of_the_system(probe, cond, graded, scale):
    systems = _systems(cond, graded, scale, 60, (int(cond), graded, scale + 1000))
    xi, ok = probe(systems)
    xe, oke = probe(systems, elim=True)
    assert np.array_equal(ok, oke)
    for t, x, good in zip(systems, xi, ok):
        d, c = _scaled(t)
        if not good:  # a pivot that rounding may put below 1e-12 of the diagonal
            assert c * 2.0 ** (4 * graded) > 1e9
            continue
        want = _exact(t)
        assert np.linalg.norm((x - want) * d) <= 2.0 ** -41 * c * np.linalg.norm(want * d)
    if cond == 3.0 and graded == 0 and -55 <= scale <= 80:  # well-conditioned systems take the blocks, whose bits are their own
        assert (xi != xe).any(1).mean() > 0.5
    if not -59 <= scale <= 86:  # outside the blocks' range
        assert np.array_equal(xi, xe)


@pytest.mark.parametrize("pivot_eps", [0.0, 1e-12, 2.9e-8, 1e-7, 1e-3])
def test_verdict_is_the_eliminations(probe, pivot_eps):
    """Zero, rank-deficient, indefinite, infinite and undefined systems, and definite ones, at several pivot limits."""
    rng = np.random.default_rng(7)
    base = _systems(10.0, 0, 10, 40, 5)
    cases = [base, np.zeros((1, 27))]
    for rank in (1, 2, 3, 4, 5):
        J = rng.integers(-9, 10, (20, rank, 6)).astype(float)
        A = np.einsum("nri,nrj->nij", J, J)  # integers: exactly singular
        cases.append(np.concatenate([A[:, IU[0], IU[1]], rng.standard_normal((20, 6))], 1))
    for value in (0.0, -1.0, -1e5, np.inf, -np.inf, np.nan, 1e300, 1e-300):
        t = np.repeat(base[:1], 27, 0)
        t[np.arange(27), np.arange(27)] = value
        cases.append(t)
    systems = np.concatenate(cases)
    xi, ok = probe(systems, pivot_eps)
    xe, oke = probe(systems, pivot_eps, elim=True)
    assert np.array_equal(ok, oke)
    assert np.isfinite(xi[ok]).all()
    if pivot_eps > 0.0:
        assert not ok[40:141].any()  # the zero system and those of low rank
    if 0.0 < pivot_eps < 1e-6:
        assert ok[:40].all()

"""Lane-mode steps with their products on the integer pipes: the plain kernel's bits, also where operands are exactly
zero (motion in a coordinate plane or along an axis) and for masses, depths and tolerances far from the usual (needs
a GB300)."""
import numpy as np
import pytest

from paper_2509_15117_gb300 import binding as Bd
from paper_2509_15117_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _both(descs, y0, phi0, sid):
    pytest.importorskip("torch")
    with Bd.System(descs) as S:
        a = Bd.to_numpy(S.run(y0, phi0, sid, kernel=Bd.IA_KERNEL_PLAIN, y_final=True))
        b = Bd.to_numpy(S.run(y0, phi0, sid, y_final=True))
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)


@pytest.mark.parametrize("zeros", ["none", "some", "all"])
def test_motion_in_planes_and_along_axes(zeros, n=20001):
    """Above 16 trajectories per warp, so that lane mode runs: directions in the xy plane and along each axis keep
    components exactly zero throughout."""
    sysd = I.make_system("Rb", E_K=1e-3, max_attempts=700)
    rng = np.random.default_rng(4)
    u = np.abs(rng.normal(size=(n, 3)))
    pick = {"none": np.zeros(n, bool), "some": rng.random(n) < 0.02, "all": np.ones(n, bool)}[zeros]
    kind = rng.integers(0, 4, n)
    for axis in range(3):
        m = pick & (kind == axis)
        u[m] = 0.0
        u[m, axis] = 1.0
    u[pick & (kind == 3), 2] = 0.0
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    y0 = np.zeros((n, 12))
    y0[:, 6:9] = sysd.r0 * u
    y0[:, 9:12] = -I.speed_for_energy(I.kelvin(1e-3), sysd.m_atom) * u
    _both([sysd.as_dict()], y0, rng.random(n) * 6.28, np.zeros(n, dtype=np.int32))


def test_unusual_systems(n=20001):
    """No interaction, no trap, tiny and huge masses and lengths: operands of zero, or beyond 2^+-500, on some lanes."""
    base = I.make_system("Rb", E_K=1e-3, max_attempts=200).as_dict()
    descs = [base, dict(base, alpha=0.0), dict(base, q=(0.0, 0.0, 0.0)), dict(base, m_atom=1e-140, m_ion=1e-140),
             dict(base, m_atom=1e200), dict(base, rtol=1e-3, atol_pos=1e-160), dict(base, De=1e-30)]
    rng = np.random.default_rng(8)
    th, ph = I.octant_random(n, 8)
    y0 = I.head_on(th, ph, base["r0"], I.speed_for_energy(I.kelvin(1e-3), base["m_atom"]))
    y0[::11, 0:6] = 1e-170 * rng.normal(size=(len(y0[::11]), 6))
    _both(descs, y0, rng.random(n) * 6.28, rng.integers(0, len(descs), n).astype(np.int32))

"""The sampler's integer square root, division and uniform conversion are the correctly rounded ones: head-on and
disk states recomputed from the raw generator words with numpy's IEEE operations agree to the bit wherever no
transcendental function enters (needs a GB300)."""
import numpy as np
import pytest

from paper_2509_15117_gb300 import binding as Bd
from paper_2509_15117_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,first", [(1, 0), (33, 7), (100003, 2 ** 33)])
def test_head_on_z_and_radius(n, first):
    torch = pytest.importorskip("torch")
    d = I.make_system("Rb").as_dict()
    y = torch.empty((12, n), dtype=torch.float64, device="cuda")
    ph = torch.empty(n, dtype=torch.float64, device="cuda")
    E = I.kelvin(1.5e-6)
    Bd.ia_sample_ics(Bd.make_sampler(Bd.IA_SAMPLE_HEAD_ON, d, 77, E=E), first, y, ph)
    w = torch.empty((n, 4), dtype=torch.int64, device="cuda")
    Bd.ia_philox4x64(77, Bd.IA_SAMPLE_HEAD_ON, 0, first, w)
    u = ((w.cpu().numpy().view(np.uint64) >> np.uint64(11)) | np.uint64(1)).astype(np.float64) * 2.0 ** -53
    y = y.cpu().numpy()
    np.testing.assert_array_equal(ph.cpu().numpy(), 2.0 * np.pi * u[:, 0])
    np.testing.assert_array_equal(y[8], d["r0"] * u[:, 1])
    v0 = np.sqrt(2.0 * E / d["m_atom"])
    np.testing.assert_array_equal(y[11], -v0 * u[:, 1])
    # x = r0 (st cos a), y = r0 (st sin a): the radius from st, to the rounding of the products (4 ulp)
    st = np.sqrt((1.0 - u[:, 1]) * (1.0 + u[:, 1]))
    np.testing.assert_allclose(np.hypot(y[6], y[7]), d["r0"] * st, rtol=4 * 2.0 ** -52, atol=0)


def test_disk_geometry(n=200003):
    """|v_hat| = 1 and x_a . v_hat = -sqrt(r0^2 - b^2) to a few roundings, over all directions of v."""
    torch = pytest.importorskip("torch")
    d = I.make_system("Rb").as_dict()
    y = torch.empty((12, n), dtype=torch.float64, device="cuda")
    ph = torch.empty(n, dtype=torch.float64, device="cuda")
    Bd.ia_sample_ics(Bd.make_sampler(Bd.IA_SAMPLE_DISK, d, 5, kT=I.kelvin(1e-3), kT_ion=0.0, b_max=2000.0), 0, y, ph)
    w = torch.empty((n, 4), dtype=torch.int64, device="cuda")
    Bd.ia_philox4x64(5, Bd.IA_SAMPLE_DISK, 0, 0, w)
    u1 = ((w.cpu().numpy().view(np.uint64)[:, 1] >> np.uint64(11)) | np.uint64(1)).astype(np.float64) * 2.0 ** -53
    x, v = y[6:9].cpu().numpy(), y[9:12].cpu().numpy()
    back = np.sqrt(d["r0"] ** 2 - (2000.0 * np.sqrt(u1)) ** 2)
    along = np.sum(x * v, axis=0) / np.sqrt(np.sum(v * v, axis=0))
    # products and sums of order r0 with unit vectors good to 3 ulp: 16 eps r0
    assert np.abs(along + back).max() <= 16 * 2.0 ** -52 * d["r0"]
    assert np.abs(np.sqrt(np.sum(x * x, axis=0)) - d["r0"]).max() <= 16 * 2.0 ** -52 * d["r0"]

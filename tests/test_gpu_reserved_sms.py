"""SMs reserved for the tail: a caller's number is honoured at any batch size, the last part of a batch keeps them for
trajectories that the part before left in group mode, and the plain kernel's bits come out where tail workers, their
batches of the lane phase and local trajectories meet (needs a GB300)."""
import numpy as np
import pytest

from paper_2509_15117_gb300 import binding as Bd
from tests.test_gpu_local_groups import batch  # noqa: F401  (40 systems, 3 to 2,500 attempts, and plain results)

pytestmark = pytest.mark.gpu


def _same(ref, out, n):
    for k in ref:
        np.testing.assert_array_equal(out[k], ref[k][:n], err_msg=k)


@pytest.mark.parametrize("n,kw,reserved", [(7001, {}, 0), (7001, {"tail_sms": 8}, 8), (1, {"tail_sms": 1}, 1),
                                           (609, {"tail_sms": 76}, 76), (40001, {"tail_sms": 32}, 32),
                                           (7001, {"tail_sms": -1}, 0)])
def test_the_callers_number(batch, n, kw, reserved):  # noqa: F811
    torch, descs, y0, phi0, sid, ref = batch
    with Bd.System(descs) as S:
        out = Bd.to_numpy(S.run(y0[:n], phi0[:n], sid[:n], y_final=True, **kw))
        assert Bd.ia_launch_phases(S.handle)[2] == 0
        assert Bd.ia_test_tail(S.handle)[1] == reserved
    _same(ref, out, n)


@pytest.mark.parametrize("last", [1, 501, 7001])
def test_last_part_keeps_them_for_carried_trajectories(batch, last):  # noqa: F811
    """The first part has more trajectories than lanes and a budget of 3, so that it ends with the tail at work."""
    torch, descs, y0, phi0, sid, ref = batch
    y0, phi0, sid = (np.concatenate([a, a]) for a in (y0, phi0, sid))
    ref = {k: np.concatenate([v, v]) for k, v in ref.items()}
    n = len(phi0)
    with Bd.System(descs) as S:
        Bd.ia_test_limits(S.handle, 3)
        y, p, d = Bd.to_device_soa(y0, phi0, sid)
        out = Bd.alloc_obs(n, y_final=True)
        with Bd.Queue(S.handle, n) as Q:
            Q.launch(y, p, d, out, n - last)
            Q.launch(y, p, d, out, last)
            torch.cuda.synchronize()
            assert Q.phases()[2] == 0
            assert Bd.ia_test_tail(S.handle, Q)[1] == 32
    _same(ref, Bd.to_numpy(out), n)


@pytest.mark.parametrize("n", [33, 3041, 9121, 19457, 40001])
@pytest.mark.parametrize("kw", [{}, {"tail_warps": 1}, {"block": 256, "tail_warps": 8}, {"tail_group": 8}, {"block": 64},
                                {"suspend_capacity": 40}])
def test_workers_beside_local_trajectories(batch, n, kw):  # noqa: F811
    torch, descs, y0, phi0, sid, ref = batch
    with Bd.System(descs) as S:
        Bd.ia_test_limits(S.handle, 300, 0)
        out = Bd.to_numpy(S.run(y0[:n], phi0[:n], sid[:n], y_final=True, **kw))
        assert Bd.ia_launch_phases(S.handle)[2] == 0
        assert Bd.ia_test_tail(S.handle)[1] == 32
    _same(ref, out, n)

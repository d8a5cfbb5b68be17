"""Trajectories that a warp took to group mode when the queue ran empty pass the slice budget: they go to suspend
records while the warp has more than a batch of them, and every result keeps the plain kernel's bits. A small budget
(a test hook) brings short trajectories there (needs a GB300)."""
import numpy as np
import pytest

from paper_2509_15117_gb300 import binding as Bd
from tests.test_gpu_local_groups import batch  # noqa: F401  (40 systems, 3 to 2,500 attempts, and plain results)

pytestmark = pytest.mark.gpu


def _same(ref, out, n):
    for k in ref:
        np.testing.assert_array_equal(out[k], ref[k][:n], err_msg=k)


# two warps of 12; 12 and 15 per warp on one warp of every sub-partition; lane mode first, then group mode; and every
# form of the launch, with too few records among them
@pytest.mark.parametrize("n,kw", [(24, {"grid": 1, "block": 64}), (7001, {}), (9120, {}), (19457, {}), (40001, {}),
                                  (7001, {"tail_group": 8}), (7001, {"block": 256}), (9121, {"regs_variant": 3}),
                                  (7001, {"suspend_capacity": 5}), (40001, {"suspend_capacity": 700})])
@pytest.mark.parametrize("budget", [3, 300])
def test_past_the_budget(batch, n, kw, budget):  # noqa: F811
    torch, descs, y0, phi0, sid, ref = batch
    with Bd.System(descs) as S:
        Bd.ia_test_limits(S.handle, budget)
        out = Bd.to_numpy(S.run(y0[:n], phi0[:n], sid[:n], y_final=True, **kw))
        assert Bd.ia_launch_phases(S.handle)[2] == 0
        records = Bd.ia_test_tail(S.handle)[0]
    _same(ref, out, n)
    assert records > n // 32


@pytest.mark.parametrize("counts", [[7001], [3000, 4001], [40000, 0, 1], [15000, 15000, 7001]])
def test_parts_past_the_budget(batch, counts):  # noqa: F811
    """Carry records, suspend records, group-mode carry records and local trajectories in the last part."""
    torch, descs, y0, phi0, sid, ref = batch
    n = sum(counts)
    with Bd.System(descs) as S:
        Bd.ia_test_limits(S.handle, 300)
        y, p, d = Bd.to_device_soa(y0[:n], phi0[:n], sid[:n])
        out = Bd.alloc_obs(n, y_final=True)
        with Bd.Queue(S.handle, n) as Q:
            for c in counts:
                Q.launch(y, p, d, out, c)
                torch.cuda.synchronize()
                assert Q.phases()[2] == 0
            assert Bd.ia_test_tail(S.handle, Q)[0] > 0
    _same(ref, Bd.to_numpy(out), n)


def test_capped_below_the_budget_publishes_nothing(batch):  # noqa: F811
    torch, descs, y0, phi0, sid, ref = batch
    n = 7001
    with Bd.System(descs) as S:
        Bd.ia_test_limits(S.handle, 2501)  # one more than the longest trajectory
        out = Bd.to_numpy(S.run(y0[:n], phi0[:n], sid[:n], y_final=True))
        assert Bd.ia_test_tail(S.handle)[0] == 0
    _same(ref, out, n)

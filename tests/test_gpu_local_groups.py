"""Batches around the sizes where the persistent launch changes how it spreads trajectories over warps and when
the last of them move to group mode: the plain kernel's bits at every size (needs a GB300)."""
import numpy as np
import pytest

from paper_2509_15117_gb300 import binding as Bd
from paper_2509_15117_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def batch():
    """Trajectories of all 40 sweep systems in random order, of 3 to 2,500 attempted steps, some unusable; and the
    plain kernel's results."""
    torch = pytest.importorskip("torch")
    systems, y0, phi0, sid = I.c2_workload(33)
    perm = np.random.default_rng(9).permutation(len(sid))[:40001]
    y0, phi0, sid = y0[perm], phi0[perm], sid[perm].copy()
    for k, s in enumerate(systems):
        s.max_attempts = 3 if k % 7 == 0 else 2500
    sid[::997] = 40          # outside the table
    y0[5::1009, 2] = np.nan  # BAD_IC
    descs = [s.as_dict() for s in systems]
    with Bd.System(descs) as S:
        ref = Bd.to_numpy(S.run(y0, phi0, sid, kernel=Bd.IA_KERNEL_PLAIN, y_final=True))
    return torch, descs, y0, phi0, sid, ref


# 152 SMs have 608 sub-partitions: five trajectories on each, one warp more, five on each of 1,216 warps, three
# batches, full warps on every sub-partition, more than every lane
@pytest.mark.parametrize("n", [1, 4, 6, 33, 609, 3040, 3041, 6081, 9121, 19457, 40001])
def test_sizes_give_plain_bits(batch, n):
    torch, descs, y0, phi0, sid, ref = batch
    with Bd.System(descs) as S:
        g = Bd.to_numpy(S.run(y0[:n], phi0[:n], sid[:n], y_final=True))
        assert Bd.ia_launch_phases(S.handle)[2] == 0
    for k in ref:
        np.testing.assert_array_equal(g[k], ref[k][:n], err_msg=k)


@pytest.mark.parametrize("kw", [{"tail_group": 8}, {"block": 64}, {"block": 256}, {"blocks_per_sm": 1},
                                {"refill": 16}, {"regs_variant": 3}, {"grid": 7}, {"tail_sms": -1}])
def test_options_give_plain_bits(batch, kw):
    torch, descs, y0, phi0, sid, ref = batch
    n = 5003
    with Bd.System(descs) as S:
        g = Bd.to_numpy(S.run(y0[:n], phi0[:n], sid[:n], y_final=True, **kw))
        assert Bd.ia_launch_phases(S.handle)[2] == 0
    for k in ref:
        np.testing.assert_array_equal(g[k], ref[k][:n], err_msg=k)


@pytest.mark.parametrize("counts", [[2000, 1, 2002], [0, 4003]])
def test_parts_give_plain_bits(batch, counts):
    torch, descs, y0, phi0, sid, ref = batch
    n = sum(counts)
    with Bd.System(descs) as S:
        y, p, d = Bd.to_device_soa(y0[:n], phi0[:n], sid[:n])
        out = Bd.alloc_obs(n, y_final=True)
        with Bd.Queue(S.handle, n) as Q:
            for c in counts:
                Q.launch(y, p, d, out, c)
            torch.cuda.synchronize()
            assert Q.phases()[2] == 0
        g = Bd.to_numpy(out)
    for k in ref:
        np.testing.assert_array_equal(g[k], ref[k][:n], err_msg=k)

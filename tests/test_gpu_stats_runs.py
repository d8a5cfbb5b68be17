"""Statistics of synthetic observables whose cells come in runs: rows of one cell, rows with a cell boundary
inside, skipped trajectories, ragged ends (needs a GB300)."""
import math

import numpy as np
import pytest

from paper_2509_15117_gb300 import binding as Bd
from paper_2509_15117_gb300 import inputs as I
from tests.test_gpu_batch import _bounce_bin_np, _lifetime_bin_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,cells", [(1, 1), (31, 1), (33, 2), (1024, 3), (4097, 5), (200003, 7), (70001, 1024)])
def test_counts_and_sums_of_cell_runs(n, cells):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n)
    nb = np.where(rng.random(n) < 0.3, (1 + rng.random(n) ** -0.9).astype(np.int32), rng.integers(0, 2, n)).astype(np.int32)
    status = np.where(nb >= 2, Bd.ST_COMPLEX, 0) | np.where(rng.random(n) < 0.05, 1 << rng.integers(0, 6, n), 0)
    steps, rej = rng.integers(0, 2 ** 31 - 1, n), rng.integers(0, 10 ** 6, n)
    dE, t1 = rng.normal(size=n), rng.random(n) * 1e9
    tau = np.where(nb >= 2, 10.0 ** rng.uniform(4, 14, n), 0.0)
    cell = (np.arange(n) * cells // n).astype(np.int32)  # runs of about n / cells
    cell[rng.random(n) < 1e-3] = -1                      # skipped
    if n > 2000:
        cell[1000:1500] = rng.integers(-1, cells + 1, 500)  # rows of many cells, some out of range
    z = np.zeros(n)
    host = {"theta_s": z, "dp": z, "dE_ion": dE, "t_final": z, "t_first_bounce": t1, "t_last_bounce": t1 + tau,
            "n_bounce": nb, "status": status.astype(np.int32), "n_steps": steps.astype(np.int32),
            "n_rej": rej.astype(np.int32)}
    out = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in host.items()}
    with Bd.System([I.make_system("Rb").as_dict()]) as S:
        a, b = Bd.alloc_stats(cells), Bd.alloc_stats(cells)
        cd = torch.from_numpy(cell).cuda()
        Bd.ia_reduce_stats(S.handle, out, n, cd, cells, a)
        Bd.ia_reduce_stats(S.handle, out, n, cd, cells, b)
        torch.cuda.synchronize()
        r, r2 = Bd.stats_to_numpy(a), Bd.stats_to_numpy(b)
    assert r.tobytes() == r2.tobytes()
    life = host["t_last_bounce"] - t1
    for c in range(0, cells, max(1, cells // 16)):
        m = cell == c
        cm = m & (nb >= 2)
        assert r[c]["n"] == m.sum() and r[c]["n_complex"] == cm.sum()
        assert r[c]["attempts"] == np.sum(steps[m] + rej[m])
        np.testing.assert_array_equal(r[c]["bounce_hist"],
                                      np.bincount(_bounce_bin_np(nb[m]), minlength=Bd.STATS_BOUNCE_BINS))
        np.testing.assert_array_equal(r[c]["lifetime_hist"],
                                      np.bincount(_lifetime_bin_np(life[cm]), minlength=Bd.STATS_LIFETIME_BINS))
        assert r[c]["n_status"][Bd.STATS_EXIT_SLOT] == np.sum((status[m] & 0xFF) == 0)
        for bit in range(6):
            assert r[c]["n_status"][bit] == np.sum((status[m] >> bit) & 1)
        # any order of summation: at most n eps sum |x|
        k, eps = max(1, int(m.sum())), 2.0 ** -53
        assert abs(r[c]["sum_dE"] - math.fsum(dE[m])) <= k * eps * np.abs(dE[m]).sum()
        assert abs(r[c]["sum_dE2"] - math.fsum(dE[m] ** 2)) <= (k + 2) * eps * np.sum(dE[m] ** 2)

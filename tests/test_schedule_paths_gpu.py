"""The ways through the subsets of MaxUtil (up to 10 members, few left out, halves) at their borders, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import eb_oracle as O

pytestmark = pytest.mark.gpu


# members of the pool, members that may stay out: 5 | 6 members, 10 | 11, few left out (from 3 for 11 members, 2 for 12, 1 for 13) up to 4 | 5,
# the least and the most of each
@pytest.mark.parametrize("members,out", [(2, 1), (4, 3), (5, 2), (5, 4), (6, 1), (6, 5), (8, 2), (9, 8), (10, 1), (10, 5), (10, 9), (11, 1), (11, 2),
                                         (11, 3), (11, 4), (11, 5), (12, 1), (12, 2), (13, 1), (13, 3), (14, 4), (14, 5), (16, 1), (16, 4), (16, 5)])
@pytest.mark.parametrize("D", [1, 3, 8, 16])
def test_maxutil_takes_the_oracles_subset(members, out, D):
    from paper_2608_07964_b200 import binding as B
    rng = np.random.default_rng(members * 1000 + out * 100 + D)
    step = B.MoEStep(1, 16, 1, 0, 64, 64, D, [e % D for e in range(16)], 64)
    where = sorted(rng.choice(16, size=members, replace=False).tolist())
    pool = sum(1 << j for j in where)
    batch = B.Batch([0] * 17, [0] * 16, pool)
    # no work at all, ties, sums below and above 2048 (where quotients alone decide no more), loads beyond 2^22 (64-bit sums)
    for top in (1, 3, 120, 5000, 1 << 23):
        loads = rng.integers(0, top, size=(16, D)).astype(np.int32)
        loads[where[0]] = 0
        if top == 5000:
            loads[where[-1]] = loads[where[1]]   # equal members, so equal quotients among large numbers
        got = step.eb_schedule(batch, members - out, O.POLICY_MAXUTIL, to_host=True, mb_load=torch.from_numpy(loads).cuda())
        ref = O.schedule(loads, pool, members - out, O.POLICY_MAXUTIL)
        for k in ("run_mask", "defer_mask", "n_run", "joint_load", "util_num", "util_den"):
            assert got[k] == ref[k], (top, k, got[k], ref[k], loads.tolist())

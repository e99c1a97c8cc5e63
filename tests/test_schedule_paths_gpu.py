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


def _both(B, step, batch, loads, m, policy):
    """The schedule of these loads by eb_schedule and by a whole step in which every micro-batch keeps its routing."""
    dev = torch.from_numpy(loads).cuda()
    yield "eb_schedule", step.eb_schedule(batch, m, policy, to_host=True, mb_load=dev)
    step.mb_load.copy_(dev)
    step.eb_step(batch, m, policy, route_mask=0)
    yield "eb_step", step.sched_result()
    assert step.device_status() == 0


def _small_step(D, tokens=1):
    from paper_2608_07964_b200 import binding as B
    step = B.MoEStep(1, 16, 1, 0, 64, 64, D, [e % D for e in range(16)], 16 * tokens)
    w = [torch.zeros(1, 16, 64, 64, dtype=torch.bfloat16, device="cuda") for _ in range(3)]
    step.bind_weights(*w)
    step.logits.normal_(generator=torch.Generator(device="cuda").manual_seed(3))
    step.x.zero_()
    step.eb_route(B.Batch([tokens * j for j in range(17)], [0] * 16))
    return B, step


def _same(got, ref, *what):
    for k in ("run_mask", "defer_mask", "n_run", "joint_load", "util_num", "util_den"):
        assert got[k] == ref[k], (what, k, got[k], ref[k])


@pytest.mark.parametrize("members,m", [(n, m) for n in (14, 15, 16) for m in (1, 2, n // 2 - 1, n // 2, n - 6, n - 5)] + [(11, 6), (13, 1), (13, 8)])
def test_halves_by_one_block_and_by_several(members, m):
    """Loads of few values, so that equal subsets lie in the shares of different blocks."""
    rng = np.random.default_rng(members * 100 + m)
    for D, top in ((4, 3), (4, 40), (16, 2), (3, 7)):
        B, step = _small_step(D)
        where = sorted(rng.choice(16, size=members, replace=False).tolist())
        pool = sum(1 << j for j in where)
        batch = B.Batch(list(range(17)), [0] * 16, pool)
        loads = rng.integers(0, top, size=(16, D)).astype(np.int32)
        ref = O.schedule(loads, pool, m, O.POLICY_MAXUTIL)
        for by, got in _both(B, step, batch, loads, m, O.POLICY_MAXUTIL):
            _same(got, ref, by, D, top, loads.tolist())


@pytest.mark.parametrize("members,out", [(3, 1), (5, 4), (8, 2), (10, 0), (10, 3), (10, 9), (11, 0), (11, 1), (11, 2), (12, 4), (16, 0), (16, 4), (11, 5), (16, 6)])
@pytest.mark.parametrize("top", [1 << 11, 1 << 21, 1 << 22, (1 << 22) + 1, 1 << 25])
def test_subsets_that_are_nearly_equal(members, out, top):
    """Members that are equal or differ by one on one device: quotients that floating point cannot tell apart, or rounds the wrong way
    round, among loads up to the limit of 32-bit sums and beyond it.  In a whole step these are loads of micro-batches that keep their
    routing."""
    D = 16
    rng = np.random.default_rng(members * 1000 + out * 10 + top % 7)
    B, step = _small_step(D)
    where = sorted(rng.choice(16, size=members, replace=False).tolist())
    pool = sum(1 << j for j in where)
    batch = B.Batch(list(range(17)), [0] * 16, pool)
    for trial in range(3):
        base = rng.integers(top - max(2, top >> (4 + 6 * trial)), top, size=D)
        loads = np.tile(base, (16, 1))
        for j in range(16):
            loads[j, rng.integers(0, D)] += rng.integers(-1, 2)
        loads = np.minimum(loads, top).astype(np.int32)
        loads[where[0], 0] = top
        ref = O.schedule(loads, pool, members - out, O.POLICY_MAXUTIL)
        for by, got in _both(B, step, batch, loads, members - out, O.POLICY_MAXUTIL):
            _same(got, ref, by, trial, loads[where].tolist())


@pytest.mark.parametrize("policy", [O.POLICY_CUMUTIL, O.POLICY_DIFFPEAK])
@pytest.mark.parametrize("top", [5, 1 << 22, (1 << 22) + 1])
def test_the_linear_policies_of_a_step_with_kept_loads(policy, top):
    rng = np.random.default_rng(top + policy)
    for D, members, m in ((1, 4, 2), (5, 9, 7), (16, 16, 12)):
        B, step = _small_step(D)
        pool = sum(1 << j for j in sorted(rng.choice(16, size=members, replace=False).tolist()))
        loads = rng.integers(0, top + 1, size=(16, D)).astype(np.int32)
        loads[3, 0] = top
        ref = O.schedule(loads, pool, m, policy)
        for by, got in _both(B, step, B.Batch(list(range(17)), [0] * 16, pool), loads, m, policy):
            _same(got, ref, by, D, loads.tolist())


def test_a_step_of_more_assignments_than_32_bit_sums_are_used_for():
    """16 x 32769 tokens to 8 experts each, 4194432 assignments: 64-bit sums whatever the loads are."""
    from paper_2608_07964_b200 import binding as B
    T, D = 32769, 5
    step = B.MoEStep(1, 12, 8, 0, 64, 64, D, [e % D for e in range(12)], 16 * T)
    step.bind_weights(*[torch.zeros(1, 12, 64, 64, dtype=torch.bfloat16, device="cuda") for _ in range(3)])
    step.logits.normal_(generator=torch.Generator(device="cuda").manual_seed(9))
    step.logits[:5 * T, 0] += 9   # skewed loads of some micro-batches
    step.x.zero_()
    for members, m in ((16, 12), (9, 5), (16, 8)):
        pool = (1 << members) - 1
        step.eb_step(B.Batch([T * j for j in range(17)], [0] * 16, pool), m)
        loads = step.mb_load.cpu().numpy()
        device_of = torch.tensor([e % D for e in range(12)], device="cuda")
        for j in (0, 7, 15):
            want = torch.bincount(device_of[step.topk_idx[j * T:(j + 1) * T].long().flatten()], minlength=D)
            assert want.tolist() == loads[j].tolist()
        _same(step.sched_result(), O.schedule(loads, pool, m, O.POLICY_MAXUTIL), members, m, loads.tolist())
    assert step.device_status() == 0

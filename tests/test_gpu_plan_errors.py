"""The planning kernel of the tiled path: what it reports of a batch with several faults, a range
of the whole batch that adds to the status words, and more groups than one of its blocks holds
threads (it plans 1024 groups at a time, in every block).  Bar of the parity tests."""
import dataclasses

import numpy as np
import pytest

from batches import from_rollouts
from paper_2606_18954_gb300 import workloads as W
from test_gpu_parity import batch_of, compare, gp_mod, oracle_params, oracle_run, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPE, BAD_REWARD, UNSUPPORTED = 2, 3, 5


def test_layout_errors_come_first(gp_mod):
    """A group above the declared largest one is UNSUPPORTED only in an otherwise sound batch: an
    error of the layout is found late (at the end of a rollout of 4000 steps, by a block other
    than the first) and reported all the same."""
    rng = np.random.default_rng(3)
    rows = rng.standard_normal((4040, 8))
    groups = [[(rows[r:r + 1], [2], r % 2) for r in range(40)], [(rows[40:4000], [1] * 3960, 1)]]
    b = from_rollouts(groups, dtype="bf16")
    gp = gp_mod.GraphPO(kappa=0.9, flags=gp_mod.binding.FLAG_TILED)
    db = gp_mod.Batch.from_arrays(b, device="cuda")
    db.max_states_per_group = 32
    out = gp.alloc_outputs(db)
    for fault, code in ((None, UNSUPPORTED), ("tokens", SHAPE), ("reward", BAD_REWARD), (None, UNSUPPORTED)):
        good = db.rollout_token_off.clone(), db.reward.clone()
        if fault == "tokens":
            db.step_len[-1] = 2  # the rollout's steps no longer fill its token span
        if fault == "reward":
            db.reward[-1] = 7
        for _ in range(3):
            gp.compute_into(db, out)
            with pytest.raises(gp_mod.GraphPOError) as e:
                gp.check()
            assert e.value.code == code, fault
        db.step_len[-1] = 1
        db.rollout_token_off.copy_(good[0])
        db.reward.copy_(good[1])


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_whole_range_without_clearing(gp_mod, dtype):
    import torch
    b = W.make_batch(dataclasses.replace(W.CONFIGS["math"].scaled(3), dtype=dtype)) if dtype == "f32" else batch_of("math", 3)
    p = oracle_params(b)
    gp = gp_mod.GraphPO(kappa=p["kappa"], w=p["w"], lambda_eff=p["lambda_eff"], flags=gp_mod.binding.FLAG_TILED)
    db = gp_mod.Batch.from_arrays(b, device="cuda")
    out, ws, stream = gp.alloc_outputs(db, nodes=True), gp.workspace(db), torch.cuda.current_stream()
    ws.fill_(0xFF)
    for clear in (True, False, False):
        for t in out.values():
            t.fill_(-1)
        gp.compute_groups(db, out, 0, db.num_groups, clear, ws, stream)
        gp.check()
        compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, p), f"{dtype} {clear}")
    db.reward[0] = 7
    gp.compute_groups(db, out, 0, db.num_groups, False, ws, stream)
    db.reward[0] = 0
    gp.compute_groups(db, out, 0, db.num_groups, False, ws, stream)
    with pytest.raises(gp_mod.GraphPOError) as e:
        gp.check()
    assert e.value.code == BAD_REWARD


@pytest.mark.parametrize("groups", [1023, 1024, 1025, 2100])
def test_many_groups(gp_mod, groups):
    spec = dataclasses.replace(W.CONFIGS["agentic"], groups=groups, rollouts=4, d=32, centroids=6, sigma=0.05, kappa=0.9,
                               steps=("uniform", 1, 4), lengths=("per_step", 1, 5))
    b = dict(W.make_batch(spec, seed=groups))
    b["group_rollout_off"] = np.repeat(b["group_rollout_off"], [1 + (k % 9 == 4) for k in range(groups + 1)])
    p = oracle_params(b)
    gp = gp_mod.GraphPO(kappa=p["kappa"], w=p["w"], lambda_eff=p["lambda_eff"], flags=gp_mod.binding.FLAG_TILED)
    db = gp_mod.Batch.from_arrays(b, device="cuda")
    out = gp(db, components=True, nodes=True)
    gp.check()
    compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, p), f"{groups} groups")

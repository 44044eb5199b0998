"""The group-resident bf16 kernel's token scatter put off to the next group of the CTA: more groups
than CTAs (a group may follow on every one), groups without states among them, step lengths below and
far above a half-warp's 16-byte chunks, one- and two-pass groups, branching batches; with the
per-token components (not put off) too.  Same bar as the parity tests."""
import dataclasses

import numpy as np
import pytest

from paper_2606_18954_gb300 import workloads as W
from test_gpu_parity import compare, gp_mod, oracle_params, oracle_run, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("components", [False, True])
@pytest.mark.parametrize("kind,steps,tokens", [("chain", (15, 24), 9), ("chain", (21, 24), 300), ("chain", (9, 12), 70),
                                               ("tree", None, 90)])
def test_deferred_scatter(gp_mod, kind, steps, tokens, components):
    if kind == "tree":
        spec = W.TreeSpec("defer", 330, (2, 5, 4, 2, 2), 64, "bf16", 32, 0.05, 0.92, ("per_step", 1, tokens),
                          ("beta", 2.0, 2.0))
        b = dict(W.make_tree_batch(spec, seed=5))
    else:
        spec = dataclasses.replace(W.CONFIGS["math"], groups=330, rollouts=16, d=64, centroids=24, sigma=0.05, kappa=0.9,
                                   steps=("uniform", *steps), lengths=("per_step", 1, tokens))
        b = dict(W.make_batch(spec, seed=5))
        # a group without states after every seventh
        b["group_rollout_off"] = np.repeat(b["group_rollout_off"], [1 + (k % 7 == 3) for k in range(331)])
    params = oracle_params(b)
    gp = gp_mod.GraphPO(kappa=params["kappa"], w=params["w"], lambda_eff=params["lambda_eff"])
    db = gp_mod.Batch.from_arrays(b, device="cuda")
    assert 128 < db.max_states_per_group <= 384
    out = gp(db, components=components, nodes=True)
    gp.check()
    compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, params), f"{kind} {steps}")


@pytest.mark.parametrize("tree", [False, True])
@pytest.mark.parametrize("d", [504, 512])
def test_deferred_before_two_passes(gp_mod, d, tree):
    """Put off only before a group of two passes (289 to 384 states) and with rows of at least 512:
    groups of one and of two passes in turn on every CTA that has several."""
    if tree:
        spec = W.TreeSpec("defer", 340, (4, 5, 4, 3), d, "bf16", 24, 0.05, 0.9, ("per_step", 1, 60), ("beta", 2.0, 2.0))
        b = dict(W.make_tree_batch(spec, seed=6))
        n = np.diff(b["group_state_off"])
    else:
        spec = dataclasses.replace(W.CONFIGS["math"], groups=340, rollouts=16, d=d, centroids=24, sigma=0.05, kappa=0.9,
                                   steps=("uniform", 15, 22), lengths=("per_step", 1, 60))
        b = dict(W.make_batch(spec, seed=6))
        n = np.diff(np.asarray(b["rollout_step_off"])[np.asarray(b["group_rollout_off"])])
    assert (n > 288).any() and (n <= 288).any() and n.max() <= 384
    params = oracle_params(b)
    gp = gp_mod.GraphPO(kappa=params["kappa"], w=params["w"], lambda_eff=params["lambda_eff"])
    out = gp(gp_mod.Batch.from_arrays(b, device="cuda"), nodes=True)
    gp.check()
    compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, params), f"d={d} tree={tree}")

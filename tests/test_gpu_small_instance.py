"""The group-resident bf16 kernel's 128-state instance (two CTAs per SM) with several groups on every
CTA, over the placements of the compensated row statistics: while a CTA's first group streams in,
by a launch before for the later groups (rows of d <= 256, branching batches and many small groups
with wider ones, widths that are a multiple of 32), or after the classes, of the needed rows; with
and without prompt embeddings.  Same bar as the parity tests."""
import dataclasses

import numpy as np
import pytest

from paper_2606_18954_gb300 import workloads as W
from test_gpu_parity import compare, gp_mod, oracle_params, oracle_run, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def batch(d, tree, groups):
    if tree:
        spec = W.TreeSpec("small", groups, (3, 4, 3), d, "bf16", 8, 0.05, 0.9, ("per_step", 1, 9), ("beta", 2.0, 2.0))
        return W.make_tree_batch(spec, seed=41 + d)
    spec = dataclasses.replace(W.CONFIGS["agentic"], groups=groups, rollouts=6, d=d, centroids=8, sigma=0.05, kappa=0.9,
                               steps=("uniform", 2, 7), lengths=("per_step", 1, 9))
    return W.make_batch(spec, seed=41 + d)


@pytest.mark.parametrize("prompt", [False, True])
@pytest.mark.parametrize("d", [64, 72, 256, 264, 320, 1024, 1032])
@pytest.mark.parametrize("tree,groups", [(False, 340), (False, 1250), (True, 330)])
def test_later_groups(gp_mod, tree, groups, d, prompt):
    import torch
    b = dict(batch(d, tree, groups))
    if prompt:
        b["root_emb"] = W.f32_to_bf16_bits(np.random.default_rng(d).standard_normal((groups, d)).astype(np.float32))
    params = oracle_params(b)
    gp = gp_mod.GraphPO(kappa=params["kappa"], w=params["w"], lambda_eff=params["lambda_eff"])
    db = gp_mod.Batch.from_arrays(b, device="cuda")
    assert db.max_states_per_group <= 128
    assert groups > 2 * torch.cuda.get_device_properties(0).multi_processor_count
    out = gp(db, components=prompt, nodes=True)
    gp.check()
    compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, params), f"d={d} tree={tree}")

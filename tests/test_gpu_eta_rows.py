"""The group-resident bf16 kernel's compensated row statistics: of every row while it streams in
(a CTA's first group of a branching batch or with d < 1024), else of the rows whose eta(p(v), v)
can reach a result, by half-warps in stages of 64 chunks of 16 bytes.  More groups than CTAs (156
groups of more than 128 states), rows that are no multiple of a stage, of a half-warp or of a
chunk, with and without prompt embeddings, and rows whose norms span many binades (each sum's
bias comes from its rows' own norms).  Same bar as the
parity tests: class ids exact, |gpu - ref| <= 1e-5 |ref| + 1e-6."""
import dataclasses

import numpy as np
import pytest

from paper_2606_18954_gb300 import workloads as W
from test_gpu_parity import compare, gp_mod, oracle_params, oracle_run, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def batch(d, tree):
    if tree:
        spec = W.TreeSpec("eta", 156, (4, 5, 3, 2), d, "bf16", 12, 0.05, 0.9, ("per_step", 1, 9), ("beta", 2.0, 2.0))
        return W.make_tree_batch(spec, seed=31 + d)
    spec = dataclasses.replace(W.CONFIGS["math"], groups=156, rollouts=16, d=d, centroids=12, sigma=0.05, kappa=0.9,
                               steps=("uniform", 8, 12), lengths=("per_step", 1, 9))
    return W.make_batch(spec, seed=31 + d)


@pytest.mark.parametrize("tree", [False, True])
@pytest.mark.parametrize("d,prompt,scaled", [(24, False, False), (60, True, False), (264, False, True),
                                             (1000, True, True), (1028, False, False)])
def test_eta_rows(gp_mod, d, prompt, scaled, tree):
    import torch
    b = dict(batch(d, tree))
    rng = np.random.default_rng(d)
    if scaled:  # exact: powers of two
        f = W.bf16_bits_to_f32(b["emb"]) * np.exp2(rng.integers(-30, 31, (len(b["emb"]), 1))).astype(np.float32)
        b["emb"] = W.f32_to_bf16_bits(f)
    if prompt:
        b["root_emb"] = W.f32_to_bf16_bits(rng.standard_normal((156, d)).astype(np.float32))
    params = oracle_params(b)
    gp = gp_mod.GraphPO(kappa=params["kappa"], w=params["w"], lambda_eff=params["lambda_eff"])
    dp = (d + 7) // 8 * 8

    def padded(bits):  # rows of whole 16-byte chunks, the padding never read
        x = torch.full((len(bits), dp), float("nan"), dtype=torch.bfloat16, device="cuda")
        x[:, :d] = torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)
        return x

    db = gp_mod.Batch.from_arrays({k: v for k, v in b.items() if k != "root_emb"}, device="cuda")
    db.emb = padded(b["emb"])[:, :d]
    db.root_emb = padded(b["root_emb"]) if prompt else None
    assert 128 < db.max_states_per_group <= 384
    out = gp(db, components=True, nodes=True)
    gp.check()
    compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, params), f"d={d}")

"""The compensated row sums behind eta where the other tests do not reach: rows whose squared norm
is finite but four times it is not in fp32, so that the sums' biases are infinite and the sums
start over with TwoSum (half_warp_row_sums after the classes, eight_rows_sums beside the tiled
similarities); and the tiled kernel's statistics at widths that are no multiple of a chunk, a
quarter-warp's stage or a k-slice.  Same bar as the parity tests."""
import dataclasses

import numpy as np
import pytest

from paper_2606_18954_gb300 import workloads as W
from test_gpu_parity import PATH_FLAGS, compare, gp_mod, oracle_params, oracle_run, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def run(P, b, d, flags, prompt=None):
    """The batch with rows padded to whole 16-byte chunks, the padding NaN (never read)."""
    import torch
    params = oracle_params(b)
    gp = P.GraphPO(kappa=params["kappa"], w=params["w"], lambda_eff=params["lambda_eff"], flags=flags)
    dp = (d + 7) // 8 * 8

    def padded(bits):
        x = torch.full((len(bits), dp), float("nan"), dtype=torch.bfloat16, device="cuda")
        x[:, :d] = torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)
        return x[:, :d]

    db = P.Batch.from_arrays({k: v for k, v in b.items() if k != "root_emb"}, device="cuda")
    db.emb = padded(b["emb"])
    db.root_emb = padded(b["root_emb"]) if "root_emb" in b else None
    out = gp(db, components=True, nodes=True)
    gp.check()
    return {k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, params)


def depths(b):
    if b.get("parent") is None:
        return np.concatenate([np.arange(n) for n in np.diff(b["rollout_step_off"])])
    par, gs = np.asarray(b["parent"]), np.asarray(b["group_state_off"])
    dep = np.zeros(len(par), int)
    for g in range(len(gs) - 1):
        for v in range(gs[g], gs[g + 1]):
            dep[v] = 0 if par[v] < 0 else dep[gs[g] + par[v]] + 1
    return dep


def batch(d, tree, groups):
    if tree:
        spec = W.TreeSpec("sums", groups, (4, 5, 3, 2), d, "bf16", 12, 0.05, 0.9, ("per_step", 1, 9), ("beta", 2.0, 2.0))
        return dict(W.make_tree_batch(spec, seed=51 + d))
    spec = dataclasses.replace(W.CONFIGS["math"], groups=groups, rollouts=16, d=d, centroids=12, sigma=0.05, kappa=0.9,
                               steps=("uniform", 8, 12), lengths=("per_step", 1, 9))
    return dict(W.make_batch(spec, seed=51 + d))


@pytest.mark.parametrize("tree,d,path,groups", [(False, 1032, "fused", 4), (True, 1032, "fused", 160),
                                                (False, 264, "fused", 160), (False, 1028, "tiled", 4),
                                                (True, 136, "tiled", 4)])
def test_restart(gp_mod, tree, d, path, groups):
    b = batch(d, tree, groups)
    f = W.bf16_bits_to_f32(b["emb"])
    # every other step: squared norms around 2^126, of which four times is above fp32; the steps
    # between small enough for the product of the two norms (exact: powers of two)
    f = f * np.where(depths(b) % 2 == 1, 2.0 ** 63, 2.0 ** -20)[:, None].astype(np.float32)
    n2 = (f.astype(np.float64) ** 2).sum(1)
    assert (4.04 * n2 > 3.4e38).sum() > len(n2) // 5 and n2.max() < 3.4e38
    b["emb"] = W.f32_to_bf16_bits(f)
    gpu, ref = run(gp_mod, b, d, PATH_FLAGS[path])
    compare(gpu, ref, f"{path} d={d}")


@pytest.mark.parametrize("prompt", [False, True])
@pytest.mark.parametrize("d", [20, 63, 99, 321, 1030])
@pytest.mark.parametrize("tree", [False, True])
def test_tiled_widths(gp_mod, tree, d, prompt):
    b = batch(d, tree, 5)
    if prompt:
        b["root_emb"] = W.f32_to_bf16_bits(np.random.default_rng(d).standard_normal((5, d)).astype(np.float32))
    gpu, ref = run(gp_mod, b, d, PATH_FLAGS["tiled"])
    compare(gpu, ref, f"tree={tree} d={d} prompt={prompt}")

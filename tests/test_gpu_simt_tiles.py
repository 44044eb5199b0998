"""The CUDA-core similarity kernel (64 x 32 tiles, k in stages of 32 split between two halves of
a CTA) at the edges of its tiles and stages: groups one below, at and one above multiples of
16, 32, 64, 128 and 256 states in one batch, widths that are no multiple of a stage or of a
16-byte chunk, fp32 (cp.async) and bf16 (converted) rows, chain and tree layouts.  Same bar as
the parity tests."""
import numpy as np
import pytest

from batches import from_rollouts
from paper_2606_18954_gb300 import workloads as W
from test_gpu_parity import _group, _margin_ok, compare, gp_mod, oracle_params, oracle_run, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu
SIZES = [1, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 257, 321]


def steps(n):
    """n states in rollouts of 1 to 9 steps."""
    out = []
    while sum(out) < n:
        out.append(min(1 + len(out) % 9, n - sum(out)))
    return out


@pytest.mark.parametrize("tree", [False, True])
@pytest.mark.parametrize("dtype,d", [("f32", 64), ("f32", 90), ("f32", 131), ("bf16", 72), ("bf16", 99)])
def test_tile_edges(gp_mod, dtype, d, tree):
    import torch
    rng = np.random.default_rng(d)
    groups = [_group(rng, len(steps(n)), steps(n), d, lambda r, h: (r + h) % 5 if (r * 7 + h) % 3 else None)
              for n in SIZES]
    b = from_rollouts(groups, dtype=dtype)
    assert _margin_ok(b, 0.9)
    if tree:
        b = W.as_tree(b)
    params = oracle_params(b)
    flags = gp_mod.binding.FLAG_TILED | (gp_mod.binding.FLAG_SIMT_SIMILARITY if dtype == "bf16" else 0)
    gp = gp_mod.GraphPO(kappa=0.9, w=0.7, lambda_eff=1.0, flags=flags)
    unit = 4 if dtype == "f32" else 8
    dp = (d + unit - 1) // unit * unit
    emb = b["emb"] if dtype == "f32" else b["emb"].view(np.int16)
    wide = np.full((len(emb), dp), -1, emb.dtype)  # (bf16: -1 is a NaN pattern)
    if dtype == "f32":
        wide[:] = np.nan
    wide[:, :d] = emb
    db = gp_mod.Batch.from_arrays(b, device="cuda")
    t = torch.from_numpy(wide).cuda()
    db.emb = (t if dtype == "f32" else t.view(torch.bfloat16))[:, :d]  # row stride dp, the padding never read
    out = gp(db, components=True, nodes=True)
    gp.check()
    compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, params), f"{dtype} d={d} tree={tree}")


@pytest.mark.parametrize("most", [4, 33, 65])
def test_many_small_groups(gp_mod, most):
    """Tiles only where some group has states for them (row halves x column chunks by the declared
    largest group), and more work items than one launch takes."""
    G = 40000 if most == 4 else 300
    rng = np.random.default_rng(most)
    n = rng.integers(1, 3, 2 * G)  # two rollouts per group
    n[:2] = [1, most - 1]
    so = np.concatenate([[0], np.cumsum(n)]).astype(np.int32)
    N = int(so[-1])
    emb = np.zeros((N, 8), np.float32)
    emb[np.arange(N), rng.integers(0, 8, N)] = rng.uniform(0.5, 2.0, N).astype(np.float32)  # cosines 0 or 1
    lens = rng.integers(1, 4, N).astype(np.int32)
    to = np.concatenate([[0], np.cumsum(lens)])[so].astype(np.int64)
    b = dict(group_rollout_off=(2 * np.arange(G + 1)).astype(np.int32), rollout_step_off=so, step_len=lens,
             rollout_token_off=to, emb=emb, emb_dtype="f32", reward=rng.integers(0, 2, 2 * G).astype(np.uint8),
             kappa=0.9, w=0.7, lambda_eff=1.0)
    gp = gp_mod.GraphPO(kappa=0.9, w=0.7, lambda_eff=1.0, flags=gp_mod.binding.FLAG_TILED)
    db = gp_mod.Batch.from_arrays(b, device="cuda")
    assert db.max_states_per_group == most
    out = gp(db, components=True, nodes=True)
    gp.check()
    compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, oracle_params(b)), f"{most}")

"""The per-group kernel of the tiled path where a group's spanning-forest edges exceed its list in
shared memory (10 words per state): few classes, so that nearly every slot of every work item has
an edge, 10 to 24 per state: about as many as the list holds (1578 and 1579 states), fewer (300),
more (1700, 2048) and the largest group.  Same bar as the parity tests."""
import numpy as np
import pytest

from paper_2606_18954_gb300 import workloads as W
from test_gpu_parity import compare, gp_mod, oracle_params, oracle_run, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(1578, 1579), (1700, 300, 2048), (4096,)])
def test_more_edges_than_the_list(gp_mod, sizes):
    rng = np.random.default_rng(sizes[0])
    n, go = [], [0]
    for s in sizes:
        left = s
        while left:
            k = min(left, int(rng.integers(5, 30)))
            n.append(k)
            left -= k
        go.append(len(n))
    so = np.concatenate([[0], np.cumsum(n)]).astype(np.int32)
    N = int(so[-1])
    emb = np.zeros((N, 8), np.float32)
    emb[np.arange(N), rng.integers(0, 3, N)] = np.exp2(rng.integers(-2, 3, N)).astype(np.float32)  # cosines 0 or 1
    lens = rng.integers(1, 4, N).astype(np.int32)
    b = dict(group_rollout_off=np.asarray(go, np.int32), rollout_step_off=so, step_len=lens,
             rollout_token_off=np.concatenate([[0], np.cumsum(lens)])[so].astype(np.int64),
             emb=W.f32_to_bf16_bits(emb), emb_dtype="bf16", reward=rng.integers(0, 2, len(n)).astype(np.uint8),
             kappa=0.9, w=0.7, lambda_eff=1.0)
    gp = gp_mod.GraphPO(kappa=0.9, w=0.7, lambda_eff=1.0)
    db = gp_mod.Batch.from_arrays(b, device="cuda")
    out = gp(db, components=True, nodes=True)
    gp.check()
    compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, oracle_params(b)), str(sizes))

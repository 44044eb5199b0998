"""The policy loss at the edges of its tiles (512 tokens, one warp each; 4-token chunks with up to
three edge boundaries inside): token counts around one tile and one chunk, edges of one to five
tokens, edges that end on, before and after tile and chunk boundaries, edges over many tiles.
Tolerances of test_gpu_loss_eff.py (loss_tolerances)."""
import numpy as np
import pytest

from batches import from_rollouts
from oracle import loss as OL
from paper_2606_18954_gb300 import workloads as W
from test_gpu_loss_eff import check_loss, gp_mod, loss_inputs, loss_tolerances, run_loss, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def lens_of(kind):
    rng = np.random.default_rng(5)
    return {"one": [1], "t3": [1, 2], "t511": [511], "t512": [512], "t513": [512, 1], "ones": [1] * 1027,
            "short": list(rng.integers(1, 6, 700)), "twos": [2] * 512 + [3] * 343, "chunk": [4] * 300 + [1],
            "around": [509, 3, 1, 511, 513, 2, 1, 1, 508], "long": [5000, 1, 1, 1, 3001, 2, 40, 9000, 3]}[kind]


@pytest.mark.parametrize("form,beta", [("dual", 0.0), ("split", 0.1)])
@pytest.mark.parametrize("kind", ["one", "t3", "t511", "t512", "t513", "ones", "short", "twos", "chunk", "around", "long"])
def test_loss_tiles(gp_mod, kind, form, beta):
    lens = lens_of(kind)
    rng = np.random.default_rng(len(lens))
    cut = max(1, len(lens) // 3)  # two rollouts where there are edges enough
    parts = [lens[:cut], lens[cut:]] if len(lens) > 1 else [lens]
    b = from_rollouts([[([rng.standard_normal(8) for _ in p], p, r) for r, p in enumerate(parts)]], dtype="bf16")
    lp, A, cor, eff, mask = loss_inputs(b, 11)
    lam = 0.7
    ref = OL.token_loss(b, lp["logp"], lp["old_logp"], lp["ref_logp"], edge_adv=A, edge_cor=cor, edge_eff=eff,
                        edge_mask=mask, beta=beta, lambda_eff=lam, form=form, norm="edge")
    gpu = run_loss(gp_mod, b, lp, form, "edge", beta, lam, A=A, cor=cor, eff=eff, mask=mask)
    A1, A2 = (A, None) if form == "dual" else (cor, eff)
    scale, gscale = loss_tolerances(b, lp, A1, A2, mask, lam, beta, "edge")
    check_loss(gpu, ref, scale, gscale, f"{kind}/{form}")

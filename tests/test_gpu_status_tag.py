"""The status words of a call: the one-kernel paths mark their errors with a tag of the call's own
instead of clearing the words first.  Whatever the workspace held before, an earlier call's error
is no error of a later one, and an error of the call itself is reported; a captured graph, whose
replays share one call's parameters, clears the words instead."""
import pytest

from test_gpu_parity import batch_of, compare, gp_mod, oracle_params, oracle_run, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

NAMES = [("math", 2), ("tiny", 4)]  # the bf16 and the fp32 one-kernel paths


def setup(P, name, groups):
    b = batch_of(name, groups)
    p = oracle_params(b)
    gp = P.GraphPO(kappa=p["kappa"], w=p["w"], lambda_eff=p["lambda_eff"])
    db = P.Batch.from_arrays(b, device="cuda")
    return b, p, gp, db, gp.alloc_outputs(db, nodes=True)


@pytest.mark.parametrize("name,groups", NAMES)
@pytest.mark.parametrize("fill", [0, 1, 0xFF, "noise"])
def test_words_of_earlier_use(gp_mod, name, groups, fill):
    import torch
    b, p, gp, db, out = setup(gp_mod, name, groups)
    ws = gp.workspace(db)
    ws.copy_(torch.randint(0, 256, ws.shape, dtype=torch.uint8, device="cuda")) if fill == "noise" else ws.fill_(fill)
    good = db.reward.clone()
    for bad in (False, True, False):
        db.reward.copy_(good)
        if bad:
            db.reward[0] = 7
        gp.compute_into(db, out)
        if bad:
            with pytest.raises(gp_mod.GraphPOError) as e:
                gp.check()
            assert e.value.code == 3  # GPO_ERR_BAD_REWARD
        else:
            gp.check()
            compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, p), f"{name} {fill}")
    # two calls without a look between them: the status is the last one's
    db.reward[0] = 7
    gp.compute_into(db, out)
    db.reward.copy_(good)
    gp.compute_into(db, out)
    gp.check()


@pytest.mark.parametrize("name,groups", NAMES)
def test_captured_replays(gp_mod, name, groups):
    import torch
    b, p, gp, db, out = setup(gp_mod, name, groups)
    gp.compute_into(db, out)
    gp.check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gp.compute_into(db, out)
    good = db.reward.clone()
    db.reward[0] = 7
    graph.replay()
    with pytest.raises(gp_mod.GraphPOError):
        gp.check()
    db.reward.copy_(good)
    out["adv"].zero_()
    graph.replay()
    gp.check()
    compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, p), f"{name} replay")


def test_ranges_after_a_whole_call(gp_mod):
    """Ranges without a clearing call join the whole call before them; a clearing one starts over."""
    import torch
    b, p, gp, db, out = setup(gp_mod, "math", 4)
    ws, stream = gp.workspace(db), torch.cuda.current_stream()
    good = db.reward.clone()
    db.reward[0] = 7  # in group 0
    gp.compute_into(db, out)
    gp.compute_groups(db, out, 2, 1, False, ws, stream)
    with pytest.raises(gp_mod.GraphPOError):
        gp.check()
    gp.compute_groups(db, out, 2, 2, True, ws, stream)
    gp.check()
    gp.compute_groups(db, out, 0, 1, False, ws, stream)
    with pytest.raises(gp_mod.GraphPOError):
        gp.check()
    db.reward.copy_(good)
    gp.compute_into(db, out)
    gp.check()


def other_work(P, gp, kind):
    """A whole call of another batch in a workspace of its own, on a one-kernel path."""
    import torch
    from paper_2606_18954_gb300 import workloads as W
    b = W.make_tree_batch(W.TREE_CONFIGS["tree"].scaled(2)) if kind == "budget" else batch_of("math", 2)
    db = P.Batch.from_arrays(b, device="cuda")
    ws = torch.empty(gp.workspace_size(db), dtype=torch.uint8, device="cuda")
    if kind == "budget":
        gp.layer_budget(db, 2, 2, workspace=ws)
    else:
        gp.compute_into(db, gp.alloc_outputs(db), workspace=ws)


@pytest.mark.parametrize("kind", ["compute", "budget"])
def test_ranges_around_a_call_elsewhere(gp_mod, kind):
    """A workspace's ranges share their first error whatever the context does elsewhere between."""
    import torch
    b, p, gp, db, out = setup(gp_mod, "math", 4)
    ws, stream = gp.workspace(db), torch.cuda.current_stream()
    good, length = db.reward.clone(), db.step_len.clone()
    db.reward[0] = 7    # group 0: GPO_ERR_BAD_REWARD
    db.step_len[-1] = 0  # group 3: GPO_ERR_SHAPE
    gp.compute_groups(db, out, 0, 1, True, ws, stream)
    other_work(gp_mod, gp, kind)
    gp.compute_groups(db, out, 2, 2, False, ws, stream)
    with pytest.raises(gp_mod.GraphPOError) as e:
        gp.check()
    assert e.value.code == 3  # the first range's
    db.reward.copy_(good)
    db.step_len.copy_(length)
    gp.compute_groups(db, out, 0, 2, True, ws, stream)
    other_work(gp_mod, gp, kind)
    gp.compute_groups(db, out, 2, 2, False, ws, stream)
    gp.check()
    compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, p), kind)


def test_ranges_of_two_contexts(gp_mod):
    """Two contexts that add ranges to one workspace, one of them after a whole call of its own."""
    import torch
    _, _, gp, db, out = setup(gp_mod, "math", 4)
    gp2 = setup(gp_mod, "math", 2)[2]
    other_work(gp_mod, gp2, "compute")
    ws, stream = gp.workspace(db), torch.cuda.current_stream()
    db.reward[0] = 7
    db.step_len[-1] = 0
    gp.compute_groups(db, out, 0, 1, True, ws, stream)
    gp2.compute_groups(db, out, 1, 3, False, ws, stream)
    for g in (gp, gp2):
        with pytest.raises(gp_mod.GraphPOError) as e:
            g.check()
        assert e.value.code == 3
    db.reward[0] = 0
    gp.compute_groups(db, out, 0, 1, True, ws, stream)
    gp2.compute_groups(db, out, 1, 3, False, ws, stream)
    for g in (gp, gp2):  # the second context's error
        with pytest.raises(gp_mod.GraphPOError) as e:
            g.check()
        assert e.value.code == 2


@pytest.mark.parametrize("name,groups", NAMES)
def test_replays_after_an_eager_call(gp_mod, name, groups):
    import torch
    b, p, gp, db, out = setup(gp_mod, name, groups)
    gp.compute_into(db, out)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gp.compute_into(db, out)
    good = db.reward.clone()
    for _ in range(2):
        db.reward.copy_(good)
        gp.compute_into(db, out)  # eager, same context and workspace
        db.reward[0] = 7
        graph.replay()
        with pytest.raises(gp_mod.GraphPOError) as e:
            gp.check()
        assert e.value.code == 3
        db.reward.copy_(good)
        gp.compute_into(db, out)
        gp.check()
        db.reward[0] = 7
        gp.compute_into(db, out)
        db.reward.copy_(good)
        out["adv"].zero_()
        graph.replay()
        gp.check()
        compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, p), f"{name} replay")

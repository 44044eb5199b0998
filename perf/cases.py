"""The work that programs have this framework do, as measurable cases.

A case names one call (or one training step's calls) and the shape of its batch; `prepare`
draws a batch of that shape on the GPU, `run` is one pass through the package's public entry
points, `exact` the same results from plain torch in 64 bits.  Kinds of case:

  advantages  GraphPO.__call__: a batch of rollout groups to per-token advantages
  step        a trainer's whole step on a new batch: advantages, loss plan, policy loss and
              its gradient
  loss        GraphPO.token_loss on a batch whose plan is at hand: the policy loss and its
              gradient, once per optimiser step
  budget      GraphPO.layer_budget: classes and next-layer budgets of a tree being grown
  host        GraphPO.compute_host: a batch in pinned host memory to advantages there

Batches follow paper_2606_18954_gb300.workloads (the shapes of its CONFIGS and TREE_CONFIGS,
centroid recipe, lengths and rewards), drawn on the GPU.  Its margin filter has nothing to do
here: two states of one centroid have a cosine near 1 / (1 + sigma^2) >= 0.99 and any other
two one near 0, both far from the threshold.
"""
import math
import zlib

import numpy as np
import torch

import paper_2606_18954_gb300 as P

KAPPA, W_POOL, LAMBDA, EPS = 0.92, 0.7, 1.0, 1e-6


def _chain(name, groups, rollouts, steps, tokens, d, centroids, **kw):
    """A chain-layout batch: steps = (lo, hi) per rollout, tokens = (lo, hi) per step, or
    (median, cap) of the whole response with response=True."""
    c = dict(name=name, kind="advantages", tree=False, groups=groups, rollouts=rollouts, steps_lo=steps[0],
             steps_hi=steps[1], tok_lo=tokens[0], tok_hi=tokens[1], response=False, d=d, dtype="bf16",
             centroids=centroids, sigma=0.08, reward="beta2", outputs="adv", prompt=False, rule="noncausal",
             beta_kl=0.0, form="dual", norm="edge")
    c.update(kw)
    return c


def _tree(name, groups, schedule, tokens, d, centroids, **kw):
    """A tree-layout batch expanded by the branching schedule, tokens = (lo, hi) per edge."""
    c = _chain(name, groups, 0, (0, 0), tokens, d, centroids, tree=True, schedule=schedule, b_next=2)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call in use: a debugging run or a small trainer, fp32 embeddings (CONFIGS["tiny"])
        _chain("tiny_fp32", 8, 8, (6, 6), (32, 256), 256, 12, dtype="f32", sigma=0.05, reward="half"),
        # one trainer rank's share of prompts: the whole step on a new batch, bound by latency and launches
        _chain("step_small", 16, 8, (4, 10), (64, 1024), 1024, 16, kind="step", reward="rare"),
        # RLVR on math problems: the ordinary training batch (CONFIGS["math"])
        _chain("math", 128, 16, (12, 20), (2048, 8192), 1024, 32, response=True),
        # search agents: many short rollouts (CONFIGS["agentic"]), every optional output asked for
        _chain("agentic_all", 256, 8, (4, 10), (64, 1024), 1024, 16, reward="rare", outputs="all"),
        # branching rollouts with the paper's best schedule (TREE_CONFIGS["tree"]), per-edge outputs
        _tree("tree", 128, "2,5,4,2,2", (64, 512), 1024, 32, outputs="edges"),
        # a whole global batch at once, several groups for each SM (CONFIGS["full"])
        _chain("full", 512, 16, (15, 25), (4096, 16384), 1024, 48, response=True, reward="uniform"),
        # wide groups, the quadratic similarity work: 2048 states per prompt (CONFIGS["wide"])
        _chain("wide", 64, 64, (32, 32), (32, 512), 2048, 64, sigma=0.06, reward="half", outputs="nodes"),
        # an encoder that hands over fp32 embeddings at an ordinary batch's group size
        _chain("math_fp32", 64, 16, (12, 20), (2048, 8192), 1024, 32, dtype="f32", response=True),
        # the optimiser steps on an ordinary batch: the clipped loss and its gradient
        _chain("loss_math", 128, 16, (12, 20), (2048, 8192), 1024, 32, kind="loss", response=True),
        # the same over a global batch: split form with the KL term
        _chain("loss_full_split_kl", 512, 16, (15, 25), (4096, 16384), 1024, 48, kind="loss", response=True,
               form="split", beta_kl=0.01),
        # growing a tree layer by layer: the budgets after layer 4 of the branching schedule
        _tree("budget", 128, "2,5,4,2", (64, 512), 1024, 32, kind="budget"),
        # rollouts and embeddings that arrive in host memory, end to end
        _chain("math_host", 128, 16, (12, 20), (2048, 8192), 1024, 32, kind="host", response=True),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["advantages", "advantages", "advantages", "tree", "step", "loss", "budget", "host"])
    if kind in ("tree", "budget"):
        sched = rng.choice(["2,5,4,2,2", "4,5,3,2", "5,4,2,2,2", "2,4,3,2,2,2", "7,6,5", "3,3,3"])
        c = _tree("", log(2, 128), sched, (rng.choice([1, 32, 64]), rng.choice([100, 512])), log(64, 1100),
                  rng.choice([8, 16, 32, 48]), kind="budget" if kind == "budget" else "advantages",
                  dtype="f32" if rng.random() < 0.15 else "bf16", b_next=rng.randint(1, 6),
                  outputs=rng.choice(["adv", "nodes", "edges", "all"]), reward=rng.choice(["half", "rare", "beta2"]),
                  prompt=kind == "tree" and rng.random() < 0.25)
        if c["dtype"] == "f32":
            c.update(groups=min(c["groups"], 32), d=min(c["d"], 512))
        return c
    f32 = kind == "advantages" and rng.random() < 0.3
    d = log(64, 2048)
    if kind == "host":  # compute_host keeps the rows as they are: whole 16-byte chunks
        d = d // 8 * 8
    n = log(24, 2048 if kind == "advantages" else 384)  # states of a group, about
    rollouts = min(log(4, 64), n)
    steps = max(1, n // rollouts)
    lo, hi = max(1, (2 * steps) // 3), max(1, steps + steps // 3)
    n = rollouts * hi
    cap = 16e6 if f32 else (64e6 if kind in ("step", "host") else 150e6)
    most = min(512, cap / (n * d), (4e9 if f32 else 400e9) / (float(n) * n * d))  # embeddings, pair products
    groups = max(1, min(log(1, 512), int(most)))
    response = rng.random() < 0.4
    tok = (log(100, 4096), 16384) if response else (log(1, 64), log(65, 1024))
    mean = tok[0] * 1.2 * rollouts if response else 0.5 * (tok[0] + tok[1]) * n
    groups = max(1, min(groups, int((12e6 if kind == "host" else 30e6) / mean)))
    return _chain("", groups, rollouts, (lo, hi), tok, d, rng.choice([8, 16, 32, 64]), kind=kind, response=response,
                  dtype="f32" if f32 else "bf16", reward=rng.choice(["half", "rare", "beta2", "uniform"]),
                  outputs=rng.choice(["adv", "nodes", "edges", "all"]),
                  rule="same_depth" if rng.random() < 0.15 else "noncausal",
                  prompt=kind == "advantages" and rng.random() < 0.15,
                  form=rng.choice(["dual", "split"]), norm=rng.choice(["edge", "token"]),
                  beta_kl=rng.choice([0.0, 0.0, 0.01]))


# ---------------------------------------------------------------------------- inputs


def _structure(case, seed):
    """Offsets, depths, step lengths, parents and rewards of one batch (numpy).  The sizes are
    the case's own, so that passes over batches of other seeds can be compared; the rewards
    are drawn from the seed."""
    text = repr(sorted((k, v) for k, v in case.items() if k != "name"))
    rng = np.random.default_rng([zlib.crc32(text.encode()), 20261202])
    G = case["groups"]
    p = {"half": lambda: np.full(G, 0.5), "rare": lambda: np.full(G, 0.3), "beta2": lambda: rng.beta(2.0, 2.0, G),
         "uniform": lambda: rng.beta(1.0, 1.0, G)}[case["reward"]]()
    drawn = np.random.default_rng([seed, 20261202])
    if case["tree"]:
        sched = [int(x) for x in case["schedule"].split(",")]
        H = len(sched)
        par, dep, gs, stop = [], [], [0], iter(rng.random(64 * 1024).tolist())
        for _ in range(G):
            base, stack = len(par), [(-1, 0)] * sched[0]  # (parent, its depth), next child on top
            while stack:
                q, h = stack.pop()
                v = len(par) - base
                par.append(q)
                dep.append(h + 1)
                u = next(stop, None)
                if u is None:
                    stop = iter(rng.random(64 * 1024).tolist())
                    u = next(stop)
                if h + 1 < H and u >= 0.1:
                    stack.extend([(v, h + 1)] * sched[h + 1])
            gs.append(len(par))
        par, dep, gs = np.array(par, np.int64), np.array(dep, np.int64), np.array(gs, np.int64)
        N = len(par)
        grp = np.repeat(np.arange(G), np.diff(gs))
        child = np.zeros(N, bool)
        child[(par + gs[grp])[par >= 0]] = True
        leaf = ~child
        R = int(leaf.sum())
        lens = rng.integers(case["tok_lo"], case["tok_hi"] + 1, N)
        go = np.concatenate([[0], np.cumsum(np.bincount(grp[leaf], minlength=G))])
        tok = np.concatenate([[0], np.cumsum(lens)])
        rew = drawn.random(R) < p[grp[leaf]]
        if case["kind"] == "budget":
            rew[:] = False  # no answer is verified while the tree still grows
        return dict(N=N, R=R, T=int(tok[-1]), go=go, gs=gs, gt=tok[gs], par=par, dep=dep, grp=grp, lens=lens, leaf=leaf,
                    rew=rew, n_max=max(H, case["centroids"] // 2), max_n=int(np.diff(gs).max()),
                    active=(dep == H) & (rng.random(N) < 0.9))
    R = G * case["rollouts"]
    ns = rng.integers(case["steps_lo"], case["steps_hi"] + 1, R)
    so = np.concatenate([[0], np.cumsum(ns)])
    N = int(so[-1])
    roll = np.repeat(np.arange(R), ns)
    dep = np.arange(N) - so[roll] + 1
    if case["response"]:
        total = np.clip(np.rint(case["tok_lo"] * np.exp(0.5 * rng.standard_normal(R))), ns, case["tok_hi"])
        w = rng.exponential(size=N)
        share = w / np.bincount(roll, w)[roll] * (total - ns)[roll]
        cum = np.cumsum(share) - np.repeat(np.concatenate([[0], np.cumsum(share)])[so[:-1]], ns)
        edge = np.rint(cum).astype(np.int64)
        edge[so[1:] - 1] = (total - ns).astype(np.int64)
        lens = edge - np.where(dep > 1, np.concatenate([[0], edge[:-1]]), 0) + 1
    else:
        lens = rng.integers(case["tok_lo"], case["tok_hi"] + 1, N)
    tok = np.concatenate([[0], np.cumsum(lens)])
    grp = roll // case["rollouts"]
    go = np.arange(G + 1) * case["rollouts"]
    return dict(N=N, R=R, T=int(tok[-1]), go=go, so=so, ro=tok[so], gs=so[go], grp=grp, roll=roll, dep=dep, lens=lens,
                rew=drawn.random(R) < p[np.arange(R) // case["rollouts"]], n_max=case["steps_hi"],
                max_n=int(np.diff(so[go]).max()))


def _embeddings(case, st, seed):
    """State embeddings (and prompt embeddings) on the GPU, rows padded to whole 16 bytes."""
    gen = torch.Generator(device="cuda").manual_seed(seed * 7919 + 11)
    d, G, K, N = case["d"], case["groups"], case["centroids"], st["N"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    unit = 16 // (2 if dt == torch.bfloat16 else 4)
    stride = (d + unit - 1) // unit * unit
    cents = torch.nn.functional.normalize(torch.randn(G * K, d, generator=gen, device="cuda"), dim=1)
    grp = torch.from_numpy(st["grp"]).cuda()
    dep = torch.from_numpy(st["dep"]).cuda()
    jitter = torch.randint(-1, 2, (N,), generator=gen, device="cuda")
    cid = torch.where(torch.rand(N, generator=gen, device="cuda") < 0.48,
                      grp * K + (((dep - 1) * K) // st["n_max"] + jitter) % K, -1)
    emb = torch.zeros(N, stride, dtype=dt, device="cuda")
    for a in range(0, N, 1 << 15):  # in blocks of rows, to bound the temporaries
        c = cid[a:a + (1 << 15), None]
        z = torch.nn.functional.normalize(torch.randn(len(c), d, generator=gen, device="cuda"), dim=1)
        z = torch.where(c >= 0, cents[c.clamp(min=0)[:, 0]], z)
        z += torch.randn(len(c), d, generator=gen, device="cuda") * (case["sigma"] / math.sqrt(d))
        emb[a:a + (1 << 15), :d] = z
    root = None
    if case["prompt"]:
        root = torch.zeros(G, stride, dtype=dt, device="cuda")
        root[:, :d] = torch.nn.functional.normalize(torch.randn(G, d, generator=gen, device="cuda"), dim=1)
    return emb[:, :d], root


def _batch(case, st, emb, root):
    def t(a, dt):
        return torch.from_numpy(np.ascontiguousarray(a.astype(dt))).cuda()

    if case["tree"]:
        return P.Batch(t(st["go"], np.int32), None, t(st["lens"], np.int32), None, emb, t(st["rew"], np.uint8),
                       st["T"], st["max_n"], root, parent=t(st["par"], np.int32),
                       group_state_off=t(st["gs"], np.int32), group_token_off=t(st["gt"], np.int64))
    return P.Batch(t(st["go"], np.int32), t(st["so"], np.int32), t(st["lens"], np.int32), t(st["ro"], np.int64), emb,
                   t(st["rew"], np.uint8), st["T"], st["max_n"], root)


def _logprobs(case, st, seed):
    """Log-probabilities of every token: a fifth of the ratios leave the clip range, none lies
    within 1e-4 of a bound, so that every correct implementation takes the same branch."""
    gen = torch.Generator(device="cuda").manual_seed(seed * 7919 + 23)

    def normal(s):
        return torch.randn(st["T"], generator=gen, device="cuda") * s

    old = -normal(1.5).abs() - 0.01
    new = old + normal(0.15)
    r = torch.exp(new.double() - old.double())
    near = ((r - 0.8).abs() < 1e-4) | ((r - 1.2).abs() < 1e-4)
    new = torch.where(near, old, new)
    return new, old, (new + normal(0.1) if case["beta_kl"] > 0 else None)


def _edge_advantages(st, seed):
    """Per-edge advantages as the advantage call leaves them: A_dual, A_cor, routed A_eff, mask."""
    gen = torch.Generator(device="cuda").manual_seed(seed * 7919 + 37)
    N = st["N"]
    cor = torch.randn(N, generator=gen, device="cuda") * (torch.rand(N, generator=gen, device="cuda") < 0.6) + 0.05
    mask = torch.rand(N, generator=gen, device="cuda") < 0.5
    eff = torch.randn(N, generator=gen, device="cuda") * mask + 0.05 * mask
    return cor + LAMBDA * eff, cor, eff, mask.to(torch.uint8)


def prepare(case, seed):
    st = _structure(case, seed)
    s = dict(case=case, gp=P.GraphPO(kappa=KAPPA, w=W_POOL, lambda_eff=LAMBDA, std_eps=EPS, merge_rule=case["rule"]))
    if case["kind"] == "loss":  # the loss reads the batch's structure, not its embeddings
        emb, root = torch.zeros(st["N"], 8, dtype=torch.bfloat16, device="cuda"), None
    else:
        emb, root = _embeddings(case, st, seed)
    s["batch"] = _batch(case, st, emb, root)
    if case["kind"] in ("loss", "step"):
        s["logp"], s["old"], s["ref"] = _logprobs(case, st, seed)
    if case["kind"] == "loss":
        s["plan"] = s["gp"].loss_plan(s["batch"])
        s["dual"], s["cor"], s["eff"], s["mask"] = _edge_advantages(st, seed)
    if case["kind"] == "budget":
        s["active"] = torch.from_numpy(st["active"].astype(np.uint8)).cuda()
    if case["kind"] == "host":
        b = s.pop("batch")
        pinned = [t.cpu().pin_memory() for t in (b.group_rollout_off, b.rollout_step_off, b.step_len,
                                                 b.rollout_token_off, b.emb, b.reward)]
        s["host"] = P.Batch(*pinned, b.total_tokens, b.max_states_per_group)
        s["adv"] = torch.empty(st["T"], dtype=torch.float32, pin_memory=True)
    return s


def _want(case):
    o = case["outputs"]
    return dict(components=o == "all", nodes=o in ("nodes", "all"), edges=o in ("edges", "all"), efficiency=o == "all")


def run(state):
    case, gp = state["case"], state["gp"]
    kind = case["kind"]
    if kind == "advantages":
        return gp(state["batch"], **_want(case))
    if kind == "budget":
        return gp.layer_budget(state["batch"], len(case["schedule"].split(",")), case["b_next"], active=state["active"],
                               classes=True)
    if kind == "host":
        return {"adv": gp.compute_host(state["host"], out=state["adv"])}
    opts = dict(beta_kl=case["beta_kl"], lambda_eff=LAMBDA, form=case["form"], norm=case["norm"])
    if kind == "loss":
        return gp.token_loss(state["batch"], state["plan"], state["logp"], state["old"], state["ref"],
                             edge_adv=state["dual"], edge_cor=state["cor"], edge_eff=state["eff"],
                             edge_eff_mask=state["mask"], **opts)
    out = gp(state["batch"], nodes=True, edges=True)
    plan = gp.loss_plan(state["batch"])
    # (no statistics: the clip count turns on the sign of advantages that cancel to about 0)
    out.update(gp.token_loss(state["batch"], plan, state["logp"], state["old"], state["ref"], edge_adv=out["edge_adv"],
                             edge_cor=out["edge_cor"], edge_eff=out["edge_eff"], edge_eff_mask=out["edge_eff_mask"],
                             stats=False, **opts))
    return out


def work(case):
    st = _structure(case, 1)
    N, R, T, G, d = st["N"], st["R"], st["T"], case["groups"], case["d"]
    offsets = 4 * N + R + (4 * N + 16 * G if case["tree"] else 12 * R + 4 * G)
    graph = N * d * (2 if case["dtype"] == "bf16" else 4) + offsets + (G * d * 2 if case["prompt"] else 0)
    pairs = float(d) * float((np.diff(st["gs"]).astype(np.float64) ** 2).sum())  # the upper triangle's products
    loss = (16 if case["beta_kl"] > 0 else 12) * T + offsets + (9 if case["form"] == "split" else 4) * N
    loss_flops = 20.0 * T
    if case["kind"] == "loss":
        return {"bytes": loss, "flops": loss_flops}
    if case["kind"] == "budget":
        return {"bytes": graph + N + 8 * N, "flops": pairs}
    if case["kind"] == "step":
        return {"bytes": graph + 4 * T + 21 * N + loss, "flops": pairs + loss_flops}
    w = _want(case)
    out = 4 * T + 9 * T * w["components"] + 12 * N * w["nodes"] + 9 * N * w["edges"] + 8 * G * w["efficiency"]
    return {"bytes": graph + out, "flops": pairs}


def tolerance(case):
    # fp32 results of an exactly determined path: seen against 64 bits are 1.3e-7 (2-norm) and
    # 1e-6 (largest) for advantages, 7e-7 for the loss (a sum of terms of both signs) and 6e-6
    # for single gradients whose two terms of the split form cancel
    if case["kind"] == "budget":
        return "exact"
    if case["kind"] in ("loss", "step"):
        return {"rel": 3e-6, "max": 2e-5}
    return {"rel": 5e-7, "max": 4e-6}


# ---------------------------------------------------------------------------- the same in 64 bits


def _classes(case, st, emb):
    """Class of every state: its smallest member (connected components of the linked pairs)."""
    label = torch.arange(st["N"], device="cuda")
    dep = torch.from_numpy(st["dep"]).cuda()
    if case["tree"]:
        n_of = torch.from_numpy(st["end"]).cuda()
    else:
        n_of = torch.from_numpy(st["so"][st["roll"] + 1]).cuda()
    for g in range(case["groups"]):
        a, b = int(st["gs"][g]), int(st["gs"][g + 1])
        if a == b:
            continue
        z = emb[a:b].double()
        z = z / z.norm(dim=1, keepdim=True).clamp(min=1e-300)
        idx = torch.arange(a, b, device="cuda")
        adj = (z @ z.T >= KAPPA) & (idx[None, :] >= n_of[a:b, None])  # right of the row and not its descendant
        if case["rule"] == "same_depth":
            adj &= dep[a:b, None] == dep[None, a:b]
        adj = adj | adj.T | torch.eye(b - a, dtype=torch.bool, device="cuda")
        lab = idx
        while True:
            new = torch.where(adj, lab[None, :], b).amin(1)
            new = new[new - a]
            if torch.equal(new, lab):
                break
            lab = new
        label[a:b] = lab
    return label


def _ancestors(st):
    """Tree layout: global parent, subtree end and the table [N, depth] of ancestors (self included)."""
    N, dep = st["N"], st["dep"]
    par = np.where(st["par"] >= 0, st["par"] + st["gs"][st["grp"]], -1)
    anc = np.full((N, int(dep.max())), -1, np.int64)
    cur = np.arange(N)
    while (cur >= 0).any():
        v = np.nonzero(cur >= 0)[0]
        anc[v, dep[cur[v]] - 1] = cur[v]
        cur = np.where(cur >= 0, par[np.maximum(cur, 0)], -1)
    end = np.arange(1, N + 1)
    for h in range(anc.shape[1]):
        v = np.nonzero(anc[:, h] >= 0)[0]
        np.maximum.at(end, anc[v, h], v + 1)
    st["end"] = end
    return par, anc


def _advantages64(case, st, emb, root):
    N, G = st["N"], case["groups"]

    def cu(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()

    def total(x, key, size):
        return torch.zeros(size, dtype=torch.float64, device="cuda").index_add_(0, key, x)

    grp, dep, rew = cu(st["grp"]), cu(st["dep"]), cu(st["rew"]).double()
    if case["tree"]:
        par_np, anc_np = _ancestors(st)
        par, anc = cu(par_np), cu(anc_np)
        leaf = cu(np.nonzero(st["leaf"])[0])
        c, t = torch.zeros(N, dtype=torch.float64, device="cuda"), torch.zeros(N, dtype=torch.float64, device="cuda")
        for h in range(anc.shape[1]):
            a = anc[leaf, h]
            c.index_add_(0, a[a >= 0], rew[a >= 0])
            t.index_add_(0, a[a >= 0], torch.ones_like(rew[a >= 0]))
    else:
        idx = torch.arange(N, device="cuda")
        par = torch.where(dep > 1, idx - 1, -1)
        c, t = rew[cu(st["roll"])], torch.ones(N, dtype=torch.float64, device="cuda")
    lab = _classes(case, st, emb)
    one = torch.ones(N, dtype=torch.float64, device="cuda")
    C, T_, Q = total(c, lab, N)[lab], total(t, lab, N)[lab], total(one, lab, N)[lab]
    S = (c + W_POOL * (C - c)) / (t + W_POOL * (T_ - t))
    rg = cu(np.repeat(np.arange(G), np.diff(st["go"])))
    S_root = (total(rew, rg, G) / total(torch.ones_like(rew), rg, G))[grp]
    Sp = torch.where(par >= 0, S[par.clamp(min=0)], S_root)
    eta = torch.zeros(N, dtype=torch.float64, device="cuda")
    for a in range(0, N, 1 << 15):
        z = emb[a:a + (1 << 15)].double()
        p = par[a:a + (1 << 15)]
        y = emb[p.clamp(min=0)].double()
        if root is not None:
            y = torch.where(p[:, None] >= 0, y, root[grp[a:a + (1 << 15)], :case["d"]].double())
        cos = (z * y).sum(1) / (z.norm(dim=1) * y.norm(dim=1)).clamp(min=1e-300)
        eta[a:a + (1 << 15)] = torch.where((p >= 0) | (root is not None), cos, 0.0).clamp(min=0.0)
    r = (S - Sp) * (1.0 - eta)
    key = torch.where(par >= 0, lab[par.clamp(min=0)], N + grp)
    cnt = total(one, key, N + G)[key]
    dev = r - (total(r, key, N + G)[key] / cnt)
    dev = torch.where(dev.abs() < 1e-13, 0.0, dev)  # equal step rewards: exactly their mean
    var = total(dev * dev, key, N + G)[key] / (cnt - 1).clamp(min=1)
    cor = torch.where(cnt >= 2, dev / (var.sqrt() + EPS), 0.0)
    l = dep.double()
    dl = (l * Q - total(l, lab, N)[lab]) / Q  # exactly 0 at the mean
    sd = (total(dl * dl, lab, N)[lab] / (Q - 1).clamp(min=1)).sqrt()
    aeff = torch.where(Q >= 2, total(S, lab, N)[lab] / Q * -dl / (sd + EPS), 0.0)
    E = torch.zeros(N, dtype=torch.float64, device="cuda")
    cov = torch.zeros(N, dtype=torch.int64, device="cuda")
    if case["tree"]:
        # depth of a_Q: how many leading strict ancestors all members of the class share
        aq, same = torch.zeros(N, dtype=torch.int64, device="cuda"), torch.ones(N, dtype=torch.bool, device="cuda")
        for h in range(anc.shape[1]):
            a = torch.where(dep > h + 1, anc[:, h], -1 - torch.arange(N, device="cuda"))
            lo = torch.full((N,), 1 << 40, device="cuda").scatter_reduce_(0, lab, a, "amin")[lab]
            hi = torch.full((N,), -(1 << 40), device="cuda").scatter_reduce_(0, lab, a, "amax")[lab]
            same &= (lo == hi) & (lo >= 0)
            aq += same
        for h in range(anc.shape[1]):
            on = (Q >= 2) & (anc[:, h] >= 0) & (h + 1 > aq)
            E.index_add_(0, anc[on, h], aeff[on])
            cov.index_add_(0, anc[on, h], torch.ones_like(anc[on, h]))
    else:  # suffix sums within each rollout
        last = cu(st["so"][1:])[cu(st["roll"])]
        for x, y in ((aeff, E), ((Q >= 2).long(), cov)):
            cs = torch.cat([torch.zeros(1, dtype=x.dtype, device="cuda"), torch.cumsum(x, 0)])
            y.copy_(cs[last] - cs[:-1])
    cov = (cov > 0)
    E = torch.where(cov, E, 0.0)
    lens = cu(st["lens"])
    good = c > 0
    reach = torch.zeros(N, dtype=torch.bool, device="cuda")
    reach[lab[good]] = True
    while True:  # classes from which a correct answer can be reached
        new = reach.clone()
        up = (par >= 0) & reach[lab]
        new[lab[par[up]]] = True
        if torch.equal(new, reach):
            break
        reach = new
    spent = total(lens.double(), grp, G).clamp(min=1)
    edge = dict(dual=cor + LAMBDA * E, cor=cor, eff=E, mask=cov.to(torch.uint8))
    tok = {k: torch.repeat_interleave(v, lens) for k, v in edge.items()}
    return dict(adv=tok["dual"], adv_cor=tok["cor"], adv_eff=tok["eff"], eff_mask=tok["mask"],
                class_id=lab.to(torch.int32), node_score=S, edge_adv=edge["dual"], edge_cor=cor, edge_eff=E,
                edge_eff_mask=edge["mask"], group_eff=total(lens * good.double(), grp, G) / spent,
                group_eff_graph=total(lens * reach[lab].double(), grp, G) / spent)


def _loss64(case, st, logp, old, ref, dual, cor, eff, mask):
    lens = torch.from_numpy(st["lens"]).cuda()
    grp = torch.from_numpy(st["grp"]).cuda()
    T = st["T"]
    size = torch.bincount(grp, minlength=case["groups"]).double()
    w = (1.0 / ((size > 0).sum() * size[grp] * lens.double())) if case["norm"] == "edge" else \
        torch.full((st["N"],), 1.0 / T, dtype=torch.float64, device="cuda")
    tw = torch.repeat_interleave(w, lens)
    r = torch.exp(logp.double() - old.double())
    rc = r.clamp(0.8, 1.2)

    def phi(a):
        a = torch.repeat_interleave(a.double(), lens)
        take = r * a <= rc * a
        return torch.where(take, r * a, rc * a), torch.where(take, r * a, 0.0), ~take

    f, df, clipped = phi(dual if case["form"] == "dual" else cor)
    if case["form"] == "split":
        f2, df2, _ = phi(eff.double() * mask * LAMBDA)
        f, df = f + f2, df + df2
    grad = -tw * df
    kl = torch.zeros((), dtype=torch.float64, device="cuda")
    if case["beta_kl"] > 0:
        x = ref.double() - logp.double()
        kl = (tw * (torch.expm1(x) - x)).sum()
        grad = grad - case["beta_kl"] * tw * torch.expm1(x)
    pg = (tw * f).sum()
    stats = torch.stack([pg, kl, clipped.sum().double(), r.sum() / T])
    return dict(loss=(case["beta_kl"] * kl - pg).reshape(1), grad_logp=grad, stats=stats)


def _budget64(case, st, emb):
    _ancestors(st)
    lab = _classes(case, st, emb).cpu().numpy()
    dep, grp, b = st["dep"], st["grp"], case["b_next"]
    layer, half = len(case["schedule"].split(",")), max(1, case["b_next"] // 2)
    order = np.lexsort((np.arange(st["N"]), dep))  # registration order: layer, then index
    first = np.full(st["N"], -1, np.int64)
    for v in order[::-1]:
        first[lab[v]] = v
    front = (dep == layer) & st["active"]
    red = front & (first[lab] != np.arange(st["N"]))
    out = np.where(red, half, 0)
    for g in range(case["groups"]):
        a, e = st["gs"][g], st["gs"][g + 1]
        k = a + np.nonzero((front & ~red)[a:e])[0]
        saved = int(red[a:e].sum()) * (b - half)
        if len(k):
            out[k] = b + saved // len(k) + (np.arange(len(k)) < saved % len(k))
    return dict(budget=torch.from_numpy(out.astype(np.int32)), class_id=torch.from_numpy(lab.astype(np.int32)))


def exact(case, seed):
    st = _structure(case, seed)
    kind = case["kind"]
    if kind == "loss":
        return _loss64(case, st, *_logprobs(case, st, seed), *_edge_advantages(st, seed))
    emb, root = _embeddings(case, st, seed)
    if kind == "budget":
        return _budget64(case, st, emb)
    a = _advantages64(case, st, emb, root)
    if kind == "host":
        return {"adv": a["adv"]}
    if kind == "step":
        keep = ("adv", "class_id", "node_score", "edge_adv", "edge_cor", "edge_eff", "edge_eff_mask")
        out = {k: a[k] for k in keep}
        out.update(_loss64(case, st, *_logprobs(case, st, seed), a["edge_adv"], a["edge_cor"], a["edge_eff"],
                           a["edge_eff_mask"]))
        out.pop("stats")
        return out
    w = _want(case)
    keep = ["adv"] + ["adv_cor", "adv_eff", "eff_mask"] * w["components"] + \
        ["class_id", "node_score", "edge_adv"] * w["nodes"] + ["edge_cor", "edge_eff", "edge_eff_mask"] * w["edges"] + \
        ["group_eff", "group_eff_graph"] * w["efficiency"]
    return {k: a[k] for k in keep}

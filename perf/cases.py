"""The work this library is measured on.

Two entry points carry a user's program: `verify`, called once per decoding step of a generation loop, and
`build_neighbors`, called once per codebook.  A case is one call of either; its sizes, guidance scales, bounds and
logit statistics are those of the repository's named configurations and of the benchmark's flattened call, or are
spread over the same ranges.  Inputs are synthetic, made on the GPU from the seed alone.
"""
from __future__ import annotations

import math

import torch

import paper_2410_03355_b200 as lt

GREEDY_ACCEPT, SAMPLING_ACCEPT = 0.7, 0.9   # typical share of accepted drafts per position: sizes work(), nothing else


def _verify(name=None, *, B, N, V=16384, k=1000, delta=0.4, depth=0, dtype="bf16", cfg=7.5, T=1.0, top_k=0, jsd=False,
            sigma=1.0, noise=0.7, rho=0.0, peaked=0.0):
    """One verification call: B sequences of N drafts (a chain, or a tree of the given depth), V codes, k neighbours.
    cfg = 0: no guidance (one target row per context).  sigma, noise, rho, peaked: see _logits."""
    c = dict(kind="verify", B=B, N=N, V=V, k=k, delta=delta, depth=depth, dtype=dtype, cfg=cfg, T=T, top_k=top_k, jsd=jsd,
             sigma=sigma, noise=noise, rho=rho, peaked=peaked)
    return c if name is None else dict(c, name=name)


def _build(name=None, *, V, D, k, metric="l2", clustered=False):
    c = dict(kind="build", V=V, D=D, k=k, metric=metric, clustered=clustered)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # a small model without guidance, one sequence, fp32 logits: all launch and latency
        _verify("tiny chain", B=1, N=4, V=1024, k=16, delta=0.1, dtype="f32", cfg=0.0, sigma=1.5, noise=0.5),
        # interactive generation of one 256-pixel image: one 60-node draft tree per step
        _verify("one tree", B=1, N=60, depth=6, k=100, delta=0.2),
        # 512-pixel generation, eight images a step
        _verify("8 trees", B=8, N=60, depth=6, k=300, delta=0.3, cfg=4.0, sigma=1.2),
        # a batch of 32 images with chain drafts
        _verify("32 chains", B=32, N=7, peaked=0.05),
        # a serving batch of 128 images with draft trees
        _verify("128 trees", B=128, N=60, depth=6),
        # the throughput setting: 8192 sequences in one call, 6.4 GB of logits
        _verify("8192 chains", B=8192, N=7, peaked=0.05),
        # greedy decoding of a large batch
        _verify("greedy, 2048 chains", B=2048, N=7, T=0.0, peaked=0.05),
        # the paper's generation settings: logit filter top-k 1000; guidance rows that agree, hence flat distributions
        _verify("top-k, 1024 chains", B=1024, N=7, top_k=1000, rho=0.99),
        # another codebook size, not a power of two, fp32 logits and odd counts everywhere
        _verify("ragged f32 trees", B=93, N=23, V=5000, k=77, delta=0.2, depth=5, dtype="f32", cfg=4.0, rho=0.9),
        # sampling at a temperature other than 1
        _verify("warm, 500 chains", B=500, N=5, k=300, delta=0.2, T=0.9, rho=0.99),
        # the neighbour table of an 8-dimensional codebook, and of a 256-dimensional clustered one
        _build("table, D = 8", V=16384, D=8, k=1000),
        _build("table, D = 256", V=16384, D=256, k=1000, clustered=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.2:
        V = rng.choice([16384, 8192, _log_int(rng, 1000, 16384)])
        D = rng.choice([8, 16, 32, rng.randint(4, 32), 256, _log_int(rng, 33, 256)])
        return _build(V=V, D=D, k=_log_int(rng, 16, 1000 if V > 2000 else V // 2), metric=rng.choice(["l2", "l2", "cosine"]),
                      clustered=rng.random() < 0.5)
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    V = rng.choice([16384, 16384, 8192, 8 * _log_int(rng, 64, 2048)])
    if dtype == "f32":
        V = min(V, 8192)                      # the largest row of fp32 logits that the library takes
    tree = rng.random() < 0.5
    N = rng.randint(8, 64) if tree else rng.randint(1, 12)
    cfg = rng.choice([0.0, 4.0, 7.5, 7.5])
    T = rng.choice([1.0, 1.0, 1.0, 1.0, 0.0, rng.choice([0.7, 0.9, 1.2])])
    most = 6.4e9 / ((3 if cfg else 2) * (N + 1) * V * (2 if dtype == "bf16" else 4))
    B = _log_int(rng, 1, max(1.0, min(8192.0, most)))
    return _verify(B=B, N=N, V=V, k=_log_int(rng, 16, min(1000, V)), delta=rng.choice([0.05, 0.1, 0.2, 0.3, 0.4]),
                   depth=rng.randint(3, 7) if tree else 0, dtype=dtype, cfg=cfg, T=T,
                   top_k=rng.choice([0, 0, 0, 0, 0, 1000, 2000, rng.randint(200, 3000)]), jsd=rng.random() < 0.125,
                   sigma=rng.choice([1.0, 1.2, 1.5]), rho=rng.choice([0.0, 0.9, 0.99]), peaked=rng.choice([0.0, 0.05]))


def _codebook(V, D, clustered, g):
    if clustered:                             # codes around 512 centres
        centres = torch.randn((512, D), generator=g, device="cuda")
        return centres[torch.arange(V, device="cuda") % 512] + 0.1 * torch.randn((V, D), generator=g, device="cuda")
    return torch.nn.functional.normalize(torch.randn((V, D), generator=g, device="cuda"), dim=1).contiguous()


def _tree(B, N, depth, g):
    """[B, N] parents: nodes 0..depth-1 form a spine, every later node picks its parent uniformly from the root and the
    earlier nodes of less than that depth."""
    par = torch.full((B, N), -1, dtype=torch.int32)
    level = torch.zeros((B, N + 1), dtype=torch.int64)          # column 0 is the root, column i + 1 node i
    for i in range(N):
        if i < depth:
            p = torch.full((B, 1), i, dtype=torch.int64)        # column of the parent
        else:
            p = torch.where(level[:, :i + 1] < depth, torch.rand((B, i + 1), generator=g), -1.0).argmax(1, keepdim=True)
        par[:, i] = p[:, 0] - 1
        level[:, i + 1] = level.gather(1, p)[:, 0] + 1
    return par


def _logits(c, par, g):
    """Target rows cond ~ N(0, sigma^2) and uncond = rho cond + sqrt(1 - rho^2) N(0, sigma^2), a share `peaked` of the
    contexts with +6 on one token; drafter rows = guided target + N(0, noise^2); drafts sampled from the drafter's row of
    the parent context, siblings distinct."""
    B, N, V, R = c["B"], c["N"], c["V"], c["N"] + 1
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    T = c["T"] or 1.0
    target = torch.empty((2 if c["cfg"] else 1, B, R, V), dtype=dt, device="cuda")
    draft = torch.empty((B, R, V), dtype=dt, device="cuda")
    tokens = torch.empty((B, N), dtype=torch.int32, device="cuda")
    rank = (par[:, None, :] == par[:, :, None]).tril(-1).sum(2)  # place of a node among its siblings
    kids = int(rank.max()) + 1
    parent, rank = par.long().cuda() + 1, rank.cuda()

    def normal(n, scale):
        return torch.randn((n, R, V), generator=g, device="cuda").mul_(scale)

    step = max(1, (1 << 25) // (R * V))
    for b in range(0, B, step):
        n = min(step, B - b)
        cond = normal(n, c["sigma"])
        peak = 6.0 * (torch.rand((n, R, 1), generator=g, device="cuda") < c["peaked"])
        at = torch.randint(0, V, (n, R, 1), generator=g, device="cuda")
        if c["cfg"]:
            uncond = normal(n, c["sigma"] * math.sqrt(1.0 - c["rho"] ** 2)).add_(cond, alpha=c["rho"])
            target[1, b:b + n] = uncond.scatter_add_(2, at, peak)
        target[0, b:b + n] = cond.scatter_add_(2, at, peak)
        guided = target[0, b:b + n].float()
        if c["cfg"]:
            u = target[1, b:b + n].float()
            guided = torch.lerp(u, guided, c["cfg"])
        draft[b:b + n] = guided + normal(n, c["noise"])
        gumbel = torch.empty((n, R, V), device="cuda").exponential_(generator=g).log_().neg_()
        score = gumbel.add_(draft[b:b + n].float(), alpha=1.0 / T)
        best = (score.topk(kids, dim=2).indices if kids > 1 else score.argmax(2, keepdim=True)).reshape(n, R * kids)
        tokens[b:b + n] = best.gather(1, parent[b:b + n] * kids + rank[b:b + n])
    return target, draft, tokens


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "build":
        need = lt.load_library().lantern_build_workspace_bytes_metric(case["V"], case["D"], case["k"], lt.binding.METRICS[case["metric"]])
        return dict(case=case, codebook=_codebook(case["V"], case["D"], case["clustered"], g),
                    workspace=torch.empty(max(need, 256), dtype=torch.uint8, device="cuda"))
    c, i32 = case, dict(dtype=torch.int32, device="cuda")
    B, N = c["B"], c["N"]
    if c["depth"]:
        par = _tree(B, N, c["depth"], torch.Generator().manual_seed(seed))
    else:
        par = torch.arange(-1, N - 1, dtype=torch.int32).expand(B, N)
    target, draft, tokens = _logits(c, par, g)
    table = lt.build_neighbors(_codebook(c["V"], 8, False, g), c["k"], with_dist=False)[0]
    # what a generation loop keeps from step to step: the table, a workspace and the output tensors
    return dict(case=case, target=target, draft=draft, tokens=tokens, parents=par.cuda() if c["depth"] else None, table=table,
                uniforms=torch.rand((B, N + 1), generator=g, device="cuda"),
                workspace=torch.empty(lt.verify_workspace_bytes(B, N, c["V"], c["k"], 1 if c["dtype"] == "bf16" else 0, c["top_k"]),
                                      dtype=torch.uint8, device="cuda"),
                out=lt.VerifyOutputs(torch.empty(B, **i32), torch.empty(B, **i32), torch.empty((B, N), **i32), torch.empty(B, **i32),
                                     None, None, None))


def run(state):
    c = state["case"]
    if c["kind"] == "build":
        return lt.build_neighbors(state["codebook"], c["k"], metric=c["metric"], workspace=state["workspace"])
    greedy = c["T"] == 0.0
    out = lt.verify(state["target"], None if greedy else state["draft"], c["cfg"], c["T"], state["tokens"], state["parents"],
                    state["table"], c["delta"], None if greedy else state["uniforms"], out=state["out"],
                    workspace=state["workspace"], divergence="jsd" if c["jsd"] else "tvd", top_k=c["top_k"])
    return out.accept_len, out.next_token, out.accept_path, out.status


def work(case):
    """verify: the logit rows of the contexts that the loop reaches (it stops at the first rejection), one neighbour row for
    each, and the small inputs and outputs.  build: every pair's distance once (it is symmetric), the table written."""
    V, k = case["V"], case["k"]
    if case["kind"] == "build":
        return {"bytes": 4 * V * case["D"] + 8 * V * k, "flops": 1.5 * V * V * case["D"]}
    greedy = case["T"] == 0.0
    a = GREEDY_ACCEPT if greedy else SAMPLING_ACCEPT
    length = min(case["depth"] or case["N"], case["N"])
    contexts = case["B"] * (1 - a ** length) / (1 - a)
    rows = (2 if case["cfg"] else 1) + (0 if greedy else 1)
    row = V * (2 if case["dtype"] == "bf16" else 4)
    return {"bytes": contexts * (rows * row + 4 * k) + case["B"] * (a ** length * (2 if case["cfg"] else 1) * row + 16 * case["N"] + 16),
            "flops": contexts * V * (6 * rows + 4)}


def tolerance(case):
    """Tables are defined to the bit.  A verification answers in whole numbers; a decision within about 1e-6 of its
    threshold (32-bit logits and exponentials) may fall the other way and take the rest of its sequence with it: with a few
    dozen decisions a sequence that is one sequence in some ten thousand."""
    return "exact" if case["kind"] == "build" else {"rel": 0.0, "differ": 5e-4}

"""The fused pass runs in one of three shapes, chosen by row length and number of sequences; its walk over the decided
contexts is done by whoever completes the next piece of a path.  Calls on both sides of every line against the oracle."""
import numpy as np
import pytest
import torch

import lantern_inputs as li
import oracle
import paper_2410_03355_b200 as lt
from parity import assert_parity, compare, near_ceiling, run_gpu, tables, to_device

pytestmark = pytest.mark.gpu


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("V,per_sm,extra,N,tree", [
    (16384, 2, 0, 2, False), (16384, 2, 1, 2, False), (16384, 3, 0, 2, False), (16384, 3, 1, 2, False),   # wide | pair | narrow
    (16384, 2, 1, 9, True), (8200, 0, 5, 14, True), (8200, 2, 1, 2, False), (8192, 0, 5, 14, True)])
def test_shapes_against_oracle(V, per_sm, extra, N, tree):
    B = per_sm * _sms() + extra
    seed = 90 + V % 97 + B + N
    par = li.tree_parents(B, N, depth=4, seed=seed) if tree else None
    inp = li.verify_inputs(B, N, V, dtype=li.BF16, has_uncond=True, cfg_scale=4.0, rho=0.9, sigma_draft=0.8, parents=par, seed=seed)
    host, dev = tables(li.codebook_gaussian(V, 8, seed=14), 100, inp.draft_tokens)
    res = compare(inp, host, 0.2, run_gpu(inp, dev, 0.2))
    assert_parity(res)
    assert res["near"] <= near_ceiling(B)


def test_calls_without_drafts():
    """N = 0: one draw per sequence from the root's target, for one sequence and for more than the groups of the GPU."""
    V = 1024
    host, dev = tables(li.codebook_gaussian(V, 8, seed=15), 16, np.zeros(1, np.int32))
    for B in (1, 7 * _sms() + 3):
        inp = li.verify_inputs(B, 0, V, dtype=li.F32, has_uncond=False, cfg_scale=1.0, seed=B)
        d = torch.from_numpy(inp.target_logits).cuda()
        out = lt.verify(d, None, 1.0, 1.0, None, None, dev, 0.2, torch.from_numpy(inp.uniforms).cuda())
        torch.cuda.synchronize()
        z = inp.target_logits[0, :, 0].astype(np.float64)
        e = np.exp(z - z.max(axis=1, keepdims=True))
        cdf = np.cumsum(e, axis=1)
        u = inp.uniforms[:, 0].astype(np.float64) * cdf[:, -1]
        want = (cdf <= u[:, None]).sum(axis=1)
        # a draw within 1e-6 of an edge of the distribution may go either way
        edge = np.abs(cdf - u[:, None]).min(axis=1) / cdf[:, -1] < 1e-6
        assert np.array_equal(out.next_token.cpu().numpy()[~edge], want[~edge]) and edge.sum() <= max(1, B // 50)
        assert not out.status.any() and not out.accept_len.any()


@pytest.mark.parametrize("N,depth", [(1, 1), (63, 9), (64, 30), (65, 30), (64, 2)])
def test_plan_paths_against_oracle(N, depth):
    """Up to 64 drafts the plan works on 64-bit sets of nodes, beyond that level by level."""
    B, V = 9, 512
    par = li.tree_parents(B, N, depth=depth, seed=N)
    inp = li.verify_inputs(B, N, V, dtype=li.BF16, has_uncond=True, cfg_scale=2.0, rho=0.9, sigma_draft=0.5, parents=par, seed=N + depth)
    host, dev = tables(li.codebook_gaussian(V, 8, seed=16), 40, inp.draft_tokens)
    res = compare(inp, host, 0.3, run_gpu(inp, dev, 0.3))
    assert_parity(res)
    assert res["near"] <= near_ceiling(B)


@pytest.mark.parametrize("K", [100, 8192, 12000, 16000])
def test_top_k_thresholds_of_bf16_rows(K):
    """The drafter row of a call at temperature 1 is counted in pairs of bf16 values against bracket edges rounded up to
    bf16: edges above, around and below zero."""
    V, B, N = 16384, 24, 3
    inp = li.verify_inputs(B, N, V, dtype=li.BF16, has_uncond=True, cfg_scale=4.0, rho=0.9, sigma_draft=0.8, seed=K)
    host, dev = tables(li.codebook_gaussian(V, 8, seed=16), 50, inp.draft_tokens)
    assert_parity(compare(inp, host, 0.2, run_gpu(inp, dev, 0.2, top_k=K), top_k=K))


@pytest.mark.parametrize("per_sm,extra,T", [(0, 30, 0.9), (2, 5, 0.9), (3, 5, 0.9), (3, 5, 1.3)])   # wide | pair | narrow
def test_shapes_at_other_temperatures(per_sm, extra, T):
    """Flat rows of 16384 tokens whose guidance branches agree: nearly every draft is accepted and nearly every token is drawn
    from a context's own q."""
    V, N, B = 16384, 2, per_sm * _sms() + extra
    inp = li.verify_inputs(B, N, V, dtype=li.BF16, has_uncond=True, cfg_scale=7.5, T=T, rho=0.99, sigma_draft=0.7, seed=B)
    host, dev = tables(li.codebook_gaussian(V, 8, seed=14), 100, inp.draft_tokens)
    res = compare(inp, host, 0.2, run_gpu(inp, dev, 0.2))
    assert_parity(res)
    assert res["near"] <= near_ceiling(B)


@pytest.mark.parametrize("V,B,N,tree", [(1024, 40, 6, False), (16384, 30, 20, True)])
def test_calls_in_a_row_on_rewritten_inputs(V, B, N, tree):
    """The fused pass is put in place while the plan still writes what it will read: calls that follow one another on the same
    workspace, their inputs rewritten between them, answer as they do alone."""
    state = []
    for seed in (3, 4):
        par = li.tree_parents(B, N, depth=5, seed=seed) if tree else None
        inp = li.verify_inputs(B, N, V, dtype=li.BF16, has_uncond=True, cfg_scale=4.0, rho=0.9, sigma_draft=0.8, parents=par, seed=seed)
        _, table = tables(li.codebook_gaussian(V, 8, seed=14), 100, inp.draft_tokens)
        state.append((to_device(inp), run_gpu(inp, table, 0.2, trace=False)))
    d = {n: t.clone() if t is not None else None for n, t in state[0][0].items()}
    ws = torch.empty(lt.verify_workspace_bytes(B, N, V, 100, li.BF16), dtype=torch.uint8, device="cuda")
    got = []
    for i in range(60):
        for n, t in state[i % 2][0].items():
            if t is not None:
                d[n].copy_(t)
        got.append(lt.verify(d["target_logits"], d["draft_logits"], 4.0, 1.0, d["draft_tokens"], d["tree_parents"], table, 0.2,
                             d["uniforms"], workspace=ws))
    torch.cuda.synchronize()
    for i, out in enumerate(got):
        alone = state[i % 2][1]
        for a in ("accept_len", "next_token", "accept_path", "status"):
            assert torch.equal(getattr(out, a), getattr(alone, a)), (i, a)


@pytest.mark.parametrize("V,per_sm,extra", [(16384, 0, 40), (16384, 3, 5), (8192, 0, 40)])   # 32, 64 and 32 tokens per thread
def test_long_sums_keep_small_terms(V, per_sm, extra):
    """Normalisers to which 256 tokens add 1 each and all others 3 to 5e-9: a thread that has one of the 256 loses in single
    precision what it adds after that.  Numerators are exact here (2^0, and small ones whose own error does not count), so
    p(x~) and q(x~) of a token of weight 1 show the sums alone.  At most the 15 small terms of one 16-term sum may go per thread
    (7.4e-8), and the stored fp32 value is rounded (3e-8)."""
    B = per_sm * _sms() + extra
    lone_p, lone_q = -19.125, -19.5
    target = torch.full((1, B, 3, V), lone_q, dtype=torch.bfloat16, device="cuda")
    draft = torch.full((B, 3, V), lone_p, dtype=torch.bfloat16, device="cuda")
    draft[:, :, 0:2048:8] = 0.0
    target[:, :, :, 1:2048:8] = 0.0
    tokens = torch.tensor([[8, 16], [1, 16]], dtype=torch.int32, device="cuda").repeat((B + 1) // 2, 1)[:B].contiguous()
    uniforms = torch.tensor([[0.99, 0.99, 0.5], [0.0, 0.5, 0.5]], device="cuda").repeat((B + 1) // 2, 1)[:B].contiguous()
    parents = torch.full((B, 2), -1, dtype=torch.int32, device="cuda")
    table = torch.arange(V, dtype=torch.int32, device="cuda")[:, None].contiguous()
    out = lt.verify(target, draft, 0.0, 1.0, tokens, parents, table, 0.0, uniforms, trace=True)
    torch.cuda.synchronize()
    zp = 256 + (V - 256) * np.exp(lone_p)
    zq = 256 + (V - 256) * np.exp(lone_q)
    qa, px = out.node_qa.cpu().double().numpy(), out.node_px.cpu().double().numpy()
    for got, want in ((px[0::2, 0], 1 / zp), (px[0::2, 1], 1 / (zp - 1)), (qa[1::2, 0], 1 / zq)):   # the first child, a sibling after it
        assert np.abs(got / want - 1).max() < 1.2e-7


@pytest.mark.parametrize("N", [6, 7, 8, 38, 39, 40, 71, 200])
@pytest.mark.parametrize("tree", [False, True])
def test_long_walks_against_oracle(N, tree):
    """After six steps a walk looks 32 contexts ahead: paths that end before, at and behind those lines, in chains and along
    paths of a tree whose nodes are numbered in steps of two."""
    B, V = 24, 512
    par = None
    if tree:     # a spine of the even nodes; every odd one is a second child of its spine node's parent
        par = np.tile(np.maximum(np.arange(N) // 2 * 2 - 2, -1).astype(np.int32), (B, 1))
    inp = li.verify_inputs(B, N, V, dtype=li.BF16, has_uncond=True, cfg_scale=2.0, rho=0.99, sigma_draft=0.25, parents=par, seed=N)
    host, dev = tables(li.codebook_gaussian(V, 8, seed=16), 64, inp.draft_tokens)
    gpu = run_gpu(inp, dev, 0.2)
    res = compare(inp, host, 0.2, gpu)
    assert_parity(res)
    assert res["near"] <= near_ceiling(B) and (N < 38 or tree or gpu.accept_len.max() > 7)


@pytest.mark.parametrize("V,B,N", [(512, 40, 60), (512, 300, 34), (1000, 12, 33), (16384, 4, 60), (16384, 160, 36)])
def test_contexts_of_more_than_33_siblings(V, B, N):
    """All drafts are children of the root and nearly all of them are rejected: from the 34th on a token's own numerator is that of the
    residual.  (Narrow, wide and, for trees, again the wide shape with a second context per group.)"""
    par = np.full((B, N), -1, np.int32)
    inp = li.verify_inputs(B, N, V, dtype=li.BF16, has_uncond=True, cfg_scale=2.0, rho=0.9, sigma_draft=0.6, parents=par, seed=N)
    rng = np.random.default_rng(V + N)
    for b in range(B):            # the drafter thinks much of tokens of which the target thinks little
        at = rng.choice(V, size=N, replace=False)
        inp.draft_tokens[b] = at
        inp.draft_logits[b, 0, at] = li.f32_to_bf16_bits(rng.uniform(6.0, 8.0, N))
        inp.target_logits[:, b, 0, at] = li.f32_to_bf16_bits(rng.uniform(-9.0, -3.0, N))
    host, dev = tables(li.codebook_gaussian(V, 8, seed=18), 24, inp.draft_tokens)
    gpu = run_gpu(inp, dev, 1.0 / V)
    ora = oracle.verify_inputs(inp, host, 1.0 / V)
    res = compare(inp, host, 1.0 / V, gpu, ora=ora)
    assert_parity(res)
    assert res["near"] <= near_ceiling(B)
    assert (ora.tested.sum(1) >= min(N, 34)).mean() > 0.2

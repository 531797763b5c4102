"""Calls of few contexts: bonus draws are made ahead of the walk, by kernels of their own; the plan has
code of its own for chains and for trees of at most 64 drafts.  And the forms a call's arguments can take."""
import dataclasses

import numpy as np
import pytest
import torch

import lantern_inputs as li
import paper_2410_03355_b200 as lt
import test_gpu_greedy as greedy
from parity import assert_parity, compare, near_ceiling, run_gpu, tables, to_device

pytestmark = pytest.mark.gpu


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _inputs(B, N, tree, seed, V=512, **kw):
    par = li.tree_parents(B, N, depth=min(N, 7), seed=seed) if tree else None
    return li.verify_inputs(B, N, V, dtype=li.BF16, has_uncond=True, cfg_scale=2.0, rho=0.9, sigma_draft=0.4, parents=par, seed=seed, **kw)


def _many(N, many, V=512):
    """One sequence; as many as have their bonus draws made ahead; one more."""
    per_sm = 4 if N > 4 or V > 8192 else 3
    return 1 if many == 0 else per_sm * _sms() // (N + 1) + many - 1


@pytest.mark.parametrize("tree", [False, True])
@pytest.mark.parametrize("N", [1, 2, 31, 32, 33, 63, 64, 70])
@pytest.mark.parametrize("many", [0, 1, 2])
def test_small_calls_against_oracle(N, tree, many):
    B = _many(N, many)
    inp = _inputs(B, N, tree, seed=7 * N + many)
    host, dev = tables(li.codebook_gaussian(512, 8, seed=18), 40, inp.draft_tokens)
    res = compare(inp, host, 0.4, run_gpu(inp, dev, 0.4))
    assert_parity(res)
    assert res["near"] <= near_ceiling(B)


@pytest.mark.parametrize("N,tree,many", [(1, False, 1), (2, True, 1), (2, True, 2), (7, False, 1), (7, False, 2), (20, True, 1), (20, True, 2), (60, True, 0),
                                         (60, True, 1), (64, True, 2)])
def test_small_calls_of_long_rows_against_oracle(N, tree, many):
    """The same where a group has sixteen warps and two staging areas; there are contexts enough for dynamic batches, that cross from the
    contexts with children to those without."""
    B = _many(N, many, 16384)
    inp = _inputs(B, N, tree, seed=N, V=16384)
    host, dev = tables(li.codebook_gaussian(16384, 8, seed=18), 300, inp.draft_tokens)
    res = compare(inp, host, 0.4, run_gpu(inp, dev, 0.4))
    assert_parity(res)
    assert res["near"] <= near_ceiling(B)


@pytest.mark.parametrize("V", [512, 16384])
@pytest.mark.parametrize("N,tree", [(5, False), (20, True)])
def test_draws_ahead_are_counted_once_and_repeat(N, tree, V):
    """Who makes a draw depends on timing; the outputs do not, and every sequence that ends on a leaf has one."""
    B = 12
    inp = _inputs(B, N, tree, seed=N, V=V)
    host, dev = tables(li.codebook_gaussian(V, 8, seed=18), 40, inp.draft_tokens)
    d = to_device(inp)
    ws = torch.empty(lt.verify_workspace_bytes(B, N, inp.V, 40), dtype=torch.uint8, device="cuda")
    want = None
    for _ in range(200):
        out = lt.verify(d["target_logits"], d["draft_logits"], 2.0, 1.0, d["draft_tokens"], d["tree_parents"], dev, 0.4, d["uniforms"], workspace=ws)
        got = [t.cpu().numpy() for t in (out.accept_len, out.next_token, out.accept_path, out.status)]
        want = got if want is None else want
        assert all(np.array_equal(a, b) for a, b in zip(got, want))
        par = inp.tree_parents if tree else np.broadcast_to(np.arange(-1, N - 1), (B, N))
        last = [got[2][b, got[0][b] - 1] if got[0][b] else -1 for b in range(B)]
        assert lt.verify_counts(ws)["from_q"] == sum(not (par[b] == last[b]).any() for b in range(B))


def _outputs(B, N):
    i32 = dict(dtype=torch.int32, device="cuda")
    return lt.VerifyOutputs(torch.empty(B, **i32), torch.empty(B, **i32), torch.empty((B, N), **i32), torch.empty(B, **i32), None, None, None)


def _run(d, dev, out, ws):
    lt.verify(d["target_logits"], d["draft_logits"], 2.0, 1.0, d["draft_tokens"], d["tree_parents"], dev, 0.4, d["uniforms"], out=out, workspace=ws)


@pytest.mark.parametrize("V,B", [(512, 6), (512, 400), (16384, 6)])
def test_draws_from_rows_that_are_not_finite_are_counted(V, B):
    """Every sequence comes to its leaf, every other leaf's row holds a NaN: a draw all the same, whoever makes it (in calls of few
    contexts a group ahead of the walk)."""
    N = 3
    inp = _inputs(B, N, False, seed=6, V=V)
    inp.draft_logits[:, :N] = inp.target_logits[0, :, :N]
    inp.target_logits[1, :, :N] = inp.target_logits[0, :, :N]      # target and drafter are the same: accepted
    inp.target_logits[0, ::2, N, 5] = 0x7fc0
    host, dev = tables(li.codebook_gaussian(V, 8, seed=18), 40, inp.draft_tokens)
    d = to_device(inp)
    ws = torch.empty(lt.verify_workspace_bytes(B, N, V, 40), dtype=torch.uint8, device="cuda")
    for _ in range(20):
        out = _outputs(B, N)
        _run(d, dev, out, ws)
        assert lt.verify_counts(ws)["from_q"] == B
        assert (out.accept_len == N).all() and (out.status[::2] == lt.ST_NONFINITE).all() and not out.status[1::2].any()
    assert_parity(compare(inp, host, 0.4, out))


def _equal(x, y):
    return all(torch.equal(getattr(x, f), getattr(y, f)) for f in ("accept_len", "next_token", "accept_path", "status"))


@pytest.mark.parametrize("V,B,N,tree", [(512, 40, 7, False), (512, 9, 60, True), (16384, 32, 7, False), (16384, 2, 60, True)])
def test_calls_in_a_row(V, B, N, tree):
    """Calls of different inputs with one workspace, without a wait in between, among them a large call and one whose plan finds a
    fault; and two of them in one captured graph."""
    inps = [_inputs(B, N, tree, seed=s, V=V) for s in (1, 2, 3)]
    inps[2].draft_tokens[B // 2, N - 1] = V     # out of range
    big = _inputs(4 * _sms() // (N + 1) + 40, N, tree, seed=4, V=V)
    host, dev = tables(li.codebook_gaussian(V, 8, seed=18), 40, np.concatenate([i.draft_tokens.ravel() for i in inps + [big]]))
    every = inps + [big]
    ds = [to_device(i) for i in every]
    ws = torch.empty(lt.verify_workspace_bytes(big.B, N, V, 40), dtype=torch.uint8, device="cuda")
    want = [_outputs(i.B, N) for i in every]
    for d, out in zip(ds, want):                # one at a time, each held against the oracle
        _run(d, dev, out, ws)
        torch.cuda.synchronize()
    for i, out in zip(inps[:2] + [big], want[:2] + want[3:]):
        assert_parity(compare(i, host, 0.4, out))
    assert want[2].status.cpu().numpy()[B // 2] == lt.ST_BAD_TOKEN
    order = [0, 1, 0, 2, 1, 3, 0, 0, 2, 3, 3, 1] * 8
    got = [_outputs(every[q].B, N) for q in order]
    torch.cuda.synchronize()
    for q, out in zip(order, got):
        _run(ds[q], dev, out, ws)
    torch.cuda.synchronize()
    assert all(_equal(out, want[q]) for q, out in zip(order, got))
    graph, pair = torch.cuda.CUDAGraph(), [_outputs(B, N), _outputs(B, N)]
    with torch.cuda.graph(graph):
        for q in (0, 1):
            _run(ds[q], dev, pair[q], ws)
    for _ in range(20):
        for out in pair:
            out.accept_len.fill_(-9)
            out.next_token.fill_(-9)
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        assert _equal(pair[0], want[0]) and _equal(pair[1], want[1])


@pytest.mark.parametrize("N,tree", [(6, False), (33, True)])
def test_greedy_small_calls(N, tree):
    inp = _inputs(3, N, tree, seed=50 + N)
    host, dev = tables(li.codebook_gaussian(512, 8, seed=18), 40, inp.draft_tokens)
    greedy.check(inp, host, dev, 0.4)


def test_forms_of_a_call(monkeypatch):
    """Outputs and workspace given or not, integer scalars, a stream, tensor subclasses: the same results; what was refused
    is refused."""
    B, N = 5, 6
    inp = _inputs(B, N, True, seed=3)
    host, dev = tables(li.codebook_gaussian(512, 8, seed=18), 40, inp.draft_tokens)
    d = to_device(inp)
    ws = torch.empty(lt.verify_workspace_bytes(B, N, inp.V, 40), dtype=torch.uint8, device="cuda")

    def call(**kw):
        a = dict(target=d["target_logits"], draft=d["draft_logits"], cfg=2.0, T=1.0, tokens=d["draft_tokens"], parents=d["tree_parents"], nbr=dev,
                 delta=0.4, uniforms=d["uniforms"])
        rest = {k: v for k, v in kw.items() if k not in a}
        a.update({k: v for k, v in kw.items() if k in a})
        out = lt.verify(*a.values(), **rest)
        torch.cuda.synchronize()
        return out

    def same(x, y):
        for f in ("accept_len", "next_token", "accept_path", "status"):
            assert torch.equal(getattr(x, f), getattr(y, f)), f

    want = call()
    out = dataclasses.replace(call(), node_qa=torch.empty((B, N), device="cuda"))
    assert call(out=out, workspace=ws) is out
    same(out, want)
    for kw in (dict(cfg=2, T=1), dict(target=torch.nn.Parameter(d["target_logits"], requires_grad=False)), dict(stream=torch.cuda.Stream()),
               dict(cfg=np.float32(2.0))):
        torch.cuda.synchronize()
        same(call(out=out, workspace=ws, **kw), want)
    assert lt.binding._call is not None          # the native part of the binding is there, and the answers are the same without it
    with monkeypatch.context() as m:
        m.setattr(lt.binding, "_call", None)
        assert call(out=out, workspace=ws) is out
        same(out, want)
    part = lt.VerifyOutputs(out.accept_len, out.next_token, None, None, None, None, None)
    call(out=part, workspace=ws)
    assert torch.equal(part.next_token, want.next_token)
    refused = [dict(target=d["target_logits"].half()), dict(draft=d["draft_logits"].float()), dict(tokens=d["draft_tokens"].long()),
               dict(uniforms=d["uniforms"].cpu()), dict(nbr=dev[:100]), dict(uniforms=None), dict(divergence="kl"),
               dict(tokens=d["draft_tokens"].t().contiguous().t()), dict(target=d["target_logits"][:, :, :, :256]),
               dict(out=dataclasses.replace(out, accept_len=out.accept_len.long()))]
    for kw in refused:
        with pytest.raises(ValueError):
            call(**{**dict(out=out, workspace=ws), **kw})
    for kw in (dict(workspace=ws[:256]), dict(T=-1.0), dict(delta=float("nan")), dict(top_k=-1)):
        with pytest.raises(lt.binding.LanternError):
            call(**{**dict(out=out, workspace=ws), **kw})


@pytest.mark.parametrize("top_k", [0, 100])
@pytest.mark.parametrize("T", [0.7, 0.9, 1.2, 0.5, 3.0, 1e-31, 1e31])
def test_temperatures_with_masked_tokens(T, top_k):
    """Quotients by the temperature: powers of two, others, and such as go the long way; tokens masked by -inf and by the lowest
    bf16 value, whose quotient overflows."""
    V, B, N = 512, 24, 3
    far = not 0.1 < T < 10                   # logits of a like size then
    inp = li.verify_inputs(B, N, V, dtype=li.BF16, has_uncond=False, cfg_scale=1.0, T=1.0 if far else T, sigma_draft=0.5, seed=5)
    if far:
        inp = dataclasses.replace(inp, T=T, **{f: li.f32_to_bf16_bits(li.bf16_bits_to_f32(getattr(inp, f)) * np.float32(T))
                                               for f in ("target_logits", "draft_logits")})
    rng = np.random.default_rng(4)
    keep = np.zeros((B, V), bool)
    keep[np.arange(B)[:, None], inp.draft_tokens] = True
    for arr in (inp.target_logits[0], inp.draft_logits):
        for value in (0xff80, 0xff7f):       # -inf, the lowest finite value
            arr[np.broadcast_to(((rng.random((B, V)) < 0.2) & ~keep)[:, None, :], arr.shape)] = value
    host, dev = tables(li.codebook_gaussian(V, 8, seed=19), 40, inp.draft_tokens)
    assert_parity(compare(inp, host, 0.3, run_gpu(inp, dev, 0.3, top_k=top_k), top_k=top_k))

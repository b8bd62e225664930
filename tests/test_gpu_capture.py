"""Calls recorded into a CUDA graph: the launches depend on one another inside
the stream, and a replay gives what the call gives, on new inputs too."""
import pytest
import torch

import paper_2607_19331_gb300 as iso

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _inputs(seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    base = [torch.randn(300, 400, generator=g, device=DEV).mul_(0.02).bfloat16(),
            torch.randn(700, generator=g, device=DEV).mul_(0.02).bfloat16()]
    xs = [[(b.float() + 5e-4 * torch.randn(b.shape, generator=g, device=DEV)).bfloat16() for b in base] for _ in range(3)]
    return base, xs


@pytest.mark.parametrize("call", ["update", "ties", "iso", "ram", "block", "global"])
def test_replay_equals_the_call(call):
    base, xs = _inputs(1)
    out = [torch.empty_like(b) for b in base]
    ws = iso.Workspace(DEV)

    def run(outs):
        if call == "update":
            iso.iso_update(base, xs[0], op="iso", out=outs, workspace=ws)
        else:
            scope = call if call in ("block", "global") else "tensor"
            iso.iso_merge(base, xs, op=call if call in ("ties", "iso", "ram") else "ties", experts_are_deltas=False,
                          scope=scope, out=outs, workspace=ws)

    run(out)                                    # sizes the workspace before the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run(out)
    for seed in (2, 3):
        nb, nx = _inputs(seed)
        for d, s in zip(base + [t for x in xs for t in x], nb + [t for x in nx for t in x]):
            d.copy_(s)
        graph.replay()
        torch.cuda.synchronize()
        got = [o.clone() for o in out]
        ref = [torch.empty_like(b) for b in base]
        run(ref)
        torch.cuda.synchronize()
        assert all(torch.equal(a.view(torch.int16), b.view(torch.int16)) for a, b in zip(got, ref))


def _frames(seed, m, n):
    g = torch.Generator(device=DEV).manual_seed(seed)
    q = min(m, n)
    orth = lambda d: torch.linalg.qr(torch.randn(d, q, generator=g, device=DEV, dtype=torch.float64))[0].contiguous()
    return g, orth(m), torch.linspace(1.0, 0.2, q, device=DEV, dtype=torch.float64), orth(n)


@pytest.mark.parametrize("m,n", [(96, 200), (300, 130)])
def test_replay_of_an_optimizer_step(m, n):
    q = min(m, n)
    ws = iso.Workspace(DEV)
    g, U, S, V = _frames(1, m, n)
    W = torch.randn(m, n, generator=g, device=DEV)
    G = torch.zeros_like(W)
    state = [U, V] + [torch.zeros(d, q, device=DEV) for d in (m, m, n, n)]
    out = torch.empty_like(W)

    def step(st, o):
        iso.opt_step(st[0], st[1], S, G, *st[2:], W, W_out=o, lr=1e-3, step=3, workspace=ws)

    step([t.clone() for t in state], out)       # sizes the workspace before the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step(state, out)
    for seed in (2, 3):
        G.copy_(torch.randn(m, n, generator=g, device=DEV) * 1e-2)
        before = [t.clone() for t in state]
        graph.replay()
        torch.cuda.synchronize()
        ref = torch.empty_like(W)
        step(before, ref)
        torch.cuda.synchronize()
        assert torch.equal(out, ref) and all(torch.equal(a, b) for a, b in zip(state, before))


@pytest.mark.parametrize("m,n,K", [(96, 200, 2), (300, 130, 1)])
def test_replay_of_a_frame_merge(m, n, K):
    ws = iso.Workspace(DEV)
    g, U0, S, V0 = _frames(4, m, n)
    Vt0 = V0.T.contiguous()
    Us, Vts = [torch.empty_like(U0) for _ in range(K)], [torch.empty_like(Vt0) for _ in range(K)]
    W0 = torch.randn(m, n, generator=g, device=DEV)
    out = torch.empty_like(W0)

    def fill():
        for t, b in zip(Us + Vts, [U0] * K + [Vt0] * K):
            t.copy_(b + 1e-2 * torch.randn(b.shape, generator=g, device=DEV, dtype=torch.float64) / b.shape[0] ** 0.5)

    def merge(o):
        return iso.frame_merge_factors(U0, S, Vt0, Us, Vts, W0, out=o, rho_keep=0.9, workspace=ws, stats=True)[1]

    fill()
    merge(out)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        st = merge(out)
    for _ in range(2):
        fill()
        graph.replay()
        torch.cuda.synchronize()
        ref = torch.empty_like(W0)
        st2 = merge(ref)
        torch.cuda.synchronize()
        # the Gram's sums run in no fixed order: its last places differ from run
        # to run (binary64), and with them the weights by an ulp
        assert torch.allclose(st.gram, st2.gram, rtol=1e-9, atol=0) and torch.allclose(st.coef, st2.coef, rtol=1e-9, atol=0)
        assert ((out - ref).abs() <= 2.0 ** -20 * ref.abs().clamp(min=1e-3)).all()
        assert int(st.status.item()) == 0

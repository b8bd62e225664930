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

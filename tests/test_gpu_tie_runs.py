"""The counting pass with a run of ties set apart (units larger than the
sample): task vectors on a coarse grid, so that the keys around rank k form a
few long runs of equal values, and rank k falls inside a run, at its first or
last entry, or in a neighbouring one.  Masks and unit figures against the
oracle bit for bit, the K = 1 ISO coefficient (its norm adds the run's ties)
within the parity bound."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_19331_gb300 as iso
from parity_util import assert_units_equal, unpack_mask

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SCOPES = {"tensor": oracle.SCOPE_TENSOR, "global": oracle.SCOPE_GLOBAL}


def _grid(n, step, seed):
    g = torch.Generator().manual_seed(seed)
    return (torch.randn(n, generator=g) * 8).round().div(8.0 / step)


@pytest.mark.parametrize("n", [24577, 25600, 100003, 1 << 20])
@pytest.mark.parametrize("scope", ["tensor", "global"])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_masks_with_runs_of_ties(n, scope, dtype):
    taus = [_grid(n, 2.0 ** -10, n).to(dtype), _grid(n // 3, 2.0 ** -10, n + 1).to(dtype)]
    key = np.sort(np.abs(taus[0].float().numpy()))[::-1]
    run = int(np.searchsorted(-key, -key[n // 10]))                 # first entry of a run
    for k in (run, run + 1, n // 10, int(np.searchsorted(-key, -key[n // 10], side="right")), n // 2):
        density = (k + 0.25) / n
        om, ou = oracle.topk_masks([t.float().numpy() for t in taus], [(1, t.numel()) for t in taus], density,
                                   SCOPES[scope])
        masks, st = iso.iso_topk_mask([t.to(DEV) for t in taus], density=density, scope=scope, stats=True)
        torch.cuda.synchronize()
        assert int(st.status.item()) == 0
        for t, m, o in zip(taus, masks, om):
            assert np.array_equal(unpack_mask(m.cpu(), t.numel()), o.reshape(-1)), (n, scope, k)
        assert_units_equal(st.units_numpy()[0], ou, f"{n} {scope} {k}")


@pytest.mark.parametrize("density", [0.05, 0.3])
def test_retention_norm_counts_the_run(density):
    tau = _grid(200_000, 2.0 ** -10, 3).reshape(400, 500)
    base = torch.randn(400, 500, generator=torch.Generator().manual_seed(4)) * 0.02
    r = oracle.update([base.numpy()], [tau.numpy()], oracle.ISO, update_is_delta=True, density=density,
                      ridge=0.01, shapes=[(400, 500)], is_1d=[False])
    _, st = iso.iso_update([base.to(DEV)], [tau.to(DEV)], op="iso", update_is_delta=True, density=density,
                           ridge=0.01, stats=True)
    torch.cuda.synchronize()
    np.testing.assert_allclose(st.coef.cpu().numpy()[:1], np.array(r["coef"][0]), rtol=1e-5)


def test_a_run_of_infinities_is_reported():
    tau = torch.randn(100_000, generator=torch.Generator().manual_seed(5))
    tau[::10] = float("inf")
    _, st = iso.iso_topk_mask([tau.to(DEV)], density=0.05, stats=True)
    torch.cuda.synchronize()
    assert int(st.status.item()) == -7


@pytest.mark.parametrize("largest", [1, 31, 2047, 2048, 2049])
@pytest.mark.parametrize("op", ["ties", "iso"])
@pytest.mark.parametrize("K", [1, 3])
def test_sets_of_small_units(largest, op, K):
    # every unit at most 2048 entries, or one entry more (the other sample
    # form): the masks' figures against the oracle, with runs of ties
    shapes = [(1, largest)] + [(1, n) for n in (1, 7, 300, 1024, 2000) if n <= largest]
    th0 = [torch.randn(s, generator=torch.Generator().manual_seed(9 + q)) * 0.02 for q, s in enumerate(shapes)]
    xs = [[_grid(s[1], 2.0 ** -10, 100 * i + q).reshape(s) for q, s in enumerate(shapes)] for i in range(K)]
    code = oracle.TIES if op == "ties" else oracle.ISO
    for density in (0.0, 0.1, 0.55, 1.0):
        g0, gx = [t.to(DEV) for t in th0], [[t.to(DEV) for t in x] for x in xs]
        if K == 1:
            _, st = iso.iso_update(g0, gx[0], op=op, update_is_delta=True, density=density, stats=True)
            r = oracle.update([t.numpy() for t in th0], [t.numpy() for t in xs[0]], code, update_is_delta=True,
                              density=density, shapes=shapes, is_1d=[False] * len(shapes))
        else:
            _, st = iso.iso_merge(g0, gx, op=op, density=density, stats=True)
            r = oracle.merge([t.numpy() for t in th0], [[t.numpy() for t in x] for x in xs], code, density=density,
                             shapes=shapes, is_1d=[False] * len(shapes))
        torch.cuda.synchronize()
        assert int(st.status.item()) == 0
        assert_units_equal(st.units_numpy(), r["units"], f"small {largest} {op} K={K} {density}")

"""The merge and Gram passes at the edges of what they stream: tensors one entry
below, at and above a step, a chunk and a tile, every compile-time expert bound
(1, 2, 3, 4, 8) and a count between bounds, both element types, checkpoints
and task vectors, and the quotients by 3, 5, 6 and 7 of the disjoint mean.
Values against the oracle within the parity bounds."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_19331_gb300 as iso
from parity_util import assert_values_close, to_np

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
OPS = {"ta": oracle.TA, "ties": oracle.TIES, "iso": oracle.ISO, "ram": oracle.RAM}
SIZES = [1, 7, 8, 127, 128, 129, 255, 257, 511, 512, 513, 1023, 1024, 1025, 2049, 5000]


def _set(dtype, seed, std, base=None):
    g = torch.Generator().manual_seed(seed)
    out = []
    for q, n in enumerate(SIZES):
        t = torch.randn(n, generator=g) * std
        if base is not None:
            t = t + base[q].float().reshape(-1)
        out.append(t.to(dtype).reshape(1, n) if q % 3 else t.to(dtype))
    return out


@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 7, 8])
@pytest.mark.parametrize("op", ["ta", "ties", "iso", "ram"])
@pytest.mark.parametrize("bdt,xdt,ckpt", [(torch.bfloat16, torch.bfloat16, True), (torch.bfloat16, torch.float32, False),
                                          (torch.float32, torch.float32, True), (torch.float32, torch.bfloat16, False)])
def test_ragged_chunks(K, op, bdt, xdt, ckpt):
    th0 = _set(bdt, 1, 0.02)
    xs = [_set(xdt, 2 + i, 1e-3, th0 if ckpt else None) for i in range(K)]
    one = [t.dim() == 1 for t in th0]
    kw = dict(density=0.4, eps_act=5e-4)
    out, st = iso.iso_merge([t.to(DEV) for t in th0], [[t.to(DEV) for t in x] for x in xs], op=op,
                            experts_are_deltas=not ckpt, stats=True, **kw)
    torch.cuda.synchronize()
    assert int(st.status.item()) == 0
    r = oracle.merge([to_np(t) for t in th0], [[to_np(t) for t in x] for x in xs], OPS[op],
                     experts_are_deltas=not ckpt, shapes=[(1, n) for n in SIZES], is_1d=one, **kw)
    for q in range(len(th0)):
        assert_values_close(to_np(out[q]), r["out64"][q], r["mag"][q], f"chunks {op} K={K} tensor {q}", op=op, K=K)


def test_mean_of_three_is_the_division():
    # every quotient by 3 of a mantissa sweep, subnormal and overflowing sums
    # included: identical experts s give (s + s + s) / 3 rounded as IEEE
    u = torch.arange(0, 1 << 16, dtype=torch.int32) * 32749 % (0x7F000000 >> 2)
    a = torch.cat([u, u + 0x3F000000 - (1 << 23), torch.tensor([1, 2, 3, 0x7F7FFFFF, 0x7F000000], dtype=torch.int32)])
    a = a.view(torch.float32).clone()
    a = a[torch.isfinite(a)]
    th0 = [torch.zeros_like(a).to(DEV)]
    out = iso.iso_merge(th0, [[a.to(DEV)], [a.to(DEV)], [a.to(DEV)]], op="ram", eps_act=0.0)
    s = ((a.numpy() + a.numpy()) + a.numpy()).astype(np.float32)
    ref = (s / np.float32(3)).astype(np.float32)
    got = out[0].cpu().numpy()
    assert np.array_equal(got.view(np.uint32), np.where(s == 0, np.float32(0), ref).view(np.uint32))


# values whose sum in order is 0, so that the sum with x appended is x
ZERO_SUMS = {3: (1, -1), 5: (1, -1, 1, -1), 6: (1, 1, -2, 1, -1), 7: (1, -1, 1, -1, 1, -1), 8: (1, 1, -2, 1, -1, 1, -1)}


@pytest.mark.parametrize("K", [3, 5, 6, 7, 8])
def test_quotients_are_the_division(K):
    # x / K for every mantissa of one binade, and for magnitudes through the
    # lower edge of the fast form (2^-120), the subnormals and the top: RAM over
    # experts that sum to x, all active
    m = torch.arange(0, 1 << 23, dtype=torch.int32) + 0x3F800000
    e = torch.arange(0, 255, dtype=torch.int32).repeat_interleave(64) * (1 << 23)
    e = e + torch.arange(64, dtype=torch.int32).repeat(255) * 131071
    x = torch.cat([m, e, torch.arange(0, 4096, dtype=torch.int32)]).view(torch.float32)
    x = torch.cat([x, -x[::7]])
    parts = [torch.full_like(x, c * 2.0 ** -100) for c in ZERO_SUMS[K]] + [x]
    live = sum((p != 0).numpy().astype(np.float32) for p in parts)
    out = iso.iso_merge([torch.zeros_like(x).to(DEV)], [[p.to(DEV)] for p in parts], op="ram", eps_act=0.0, lam=1.0)
    want = (x.numpy() / live).astype(np.float32)
    want = np.where(want == 0, np.float32(0), want)
    assert np.array_equal(out[0].cpu().numpy().view(np.uint32), want.view(np.uint32))


@pytest.mark.parametrize("K", [3, 5, 6, 7, 8])
def test_ties_quotients_are_the_division(K):
    # K equal experts: the sum of K rounded additions over K, by magnitude and sign
    m = torch.arange(0, 1 << 20, dtype=torch.int32) * 8 + 0x3F800000 + K
    x = torch.cat([m.view(torch.float32), -m[::3].view(torch.float32), torch.zeros(64)])
    out = iso.iso_merge([torch.zeros_like(x).to(DEV)], [[x.to(DEV)]] * K, op="ties", density=1.0, lam=1.0)
    s = np.zeros(x.numel(), np.float32)
    for _ in range(K):
        s = s + x.numpy()
    want = s / np.float32(K)
    assert np.array_equal(out[0].cpu().numpy().view(np.uint32), np.where(want == 0, np.float32(0), want).view(np.uint32))


@pytest.mark.parametrize("K", [2, 3, 4, 6])
def test_untrimmed_ties_vector_with_nonfinite_values(K):
    # a TIES vector left untrimmed is read by no counting pass: the call
    # reports nothing, an infinity stays one, and next to a NaN (its sum has
    # no sign) the agreeing set is the positive values.  The neighbouring
    # entries are untouched by it: small whole numbers, every sum exact.
    n = 1500
    g = torch.Generator().manual_seed(7)
    x = torch.randint(-4, 5, (K, n), generator=g).float()
    x[0, 3::10] = float("nan")
    x[1, 5::10] = float("inf")
    th0 = torch.zeros(n)
    out, st = iso.iso_merge([th0.to(DEV)], [[v.to(DEV)] for v in x], op="ties", density=0.2, lam=1.0, mask_1d=False, stats=True)
    torch.cuda.synchronize()
    assert int(st.status.item()) == 0
    s = x.sum(0)
    sign = torch.where(s.isnan(), torch.ones(n), s.sign())
    agree = (x * sign > 0)
    cnt = agree.sum(0)
    m = torch.where(agree, x, torch.zeros_like(x)).sum(0) / cnt.clamp(min=1)
    assert torch.equal(out[0].cpu(), m)

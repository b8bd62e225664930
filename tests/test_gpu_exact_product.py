"""The exact-slice contraction A_i = F_0^T dF_i of the frame merge, seen through
the Gram it feeds (iso_frame_merge with rho_keep = 1, arbitrary matrices in
place of singular frames).

With dF_i = s_i F_i - F_0, A_i = F_0^T dF_i, Sym_i, Kw_i its halves on each side,
    Gamma_ij = sum_k s_k^2 [(dF_i^T dF_j)_kk summed over U and V]
               - sum_rc s_c^2 (A_i Sym_j + Sym_i A_j - Sym_i Sym_j)[r, c] (both sides)
               - sum_rc s_r s_c (KwU_i KwV_j + KwU_j KwV_i)[r, c],
evaluated here in extended precision.  For dense columns the product's error
against the exact sum is below that of a binary64 sum: columns rounded to 55 bits below their
largest magnitude and the slice pairs left out below 2^-57 of |F_0|^T |dF_i|'s
scale per term; the Gram's own binary64 sums add a few roundings.  Bound:
2^-46 of the magnitudes summed without cancellation (a wrong digit of any but
the last slice is above it).
Columns with a dominant entry, where the slices would be the further form, are
summed in binary64 and have tests of their own below.
"""
import numpy as np
import pytest
import torch

import paper_2607_19331_gb300 as iso

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _gamma(U0, Us, V0, Vs, S):
    """Gamma and the same sums over magnitudes, in extended precision."""
    L = np.longdouble
    U0, V0, S = U0.astype(L), V0.astype(L), S.astype(L)
    sg = [np.where((U0 * U.astype(L)).sum(0) < 0, L(-1), L(1)) for U in Us]
    dF = [[U.astype(L) * s - U0 for U, s in zip(Us, sg)], [V.astype(L) * s - V0 for V, s in zip(Vs, sg)]]
    A = [[F0.T @ d for d in ds] for F0, ds in zip((U0, V0), dF)]
    M = [[np.abs(F0).T @ np.abs(d) for d in ds] for F0, ds in zip((U0, V0), dF)]
    K = len(Us)
    G, mag = np.zeros((K, K), L), np.zeros((K, K), L)
    for i in range(K):
        for j in range(K):
            sym = [[(a + a.T) / 2 for a in side] for side in A]
            kw = [[(a - a.T) / 2 for a in side] for side in A]
            ms = [[(a + a.T) / 2 for a in side] for side in M]
            for h in (0, 1):
                G[i, j] += (S ** 2 * (dF[h][i] * dF[h][j]).sum(0)).sum()
                mag[i, j] += (S ** 2 * np.abs(dF[h][i] * dF[h][j]).sum(0)).sum()
                G[i, j] -= (S[None, :] ** 2 * (A[h][i] * sym[h][j] + sym[h][i] * A[h][j] - sym[h][i] * sym[h][j])).sum()
                mag[i, j] += (S[None, :] ** 2 * 3 * (M[h][i] * ms[h][j] + ms[h][i] * M[h][j])).sum()
            G[i, j] -= (S[:, None] * S[None, :] * (kw[0][i] * kw[1][j] + kw[0][j] * kw[1][i])).sum()
            mag[i, j] += (S[:, None] * S[None, :] * (ms[0][i] * ms[1][j] + ms[0][j] * ms[1][i])).sum()
    return G, mag


# (m, n): one 16-row chunk and a ragged one, several tiles, the drain every 9
# and 16 chunks crossed, a contraction split over blocks
@pytest.mark.parametrize("m,n,K", [(16, 40, 1), (17, 5, 2), (130, 129, 2), (336, 337, 1), (2500, 64, 3), (70, 1000, 2)])
@pytest.mark.parametrize("kind", ["random", "scaled", "extreme"])
def test_gram_of_exact_products(m, n, K, kind):
    rng = np.random.default_rng(m * 1000 + n + K)
    q = min(m, n)
    if kind == "extreme":
        # every digit of every entry at the end of its range: -127, -128, -128, ...
        x = -(127.0 + sum(128.0 * 2.0 ** (-8 * t) for t in range(1, 7))) / 128.0
        U0, V0 = np.full((m, q), x), np.full((n, q), x)
        Us, Vs = [2.0 * U0] * K, [2.0 * V0] * K          # dF = F_0
    else:
        f = lambda d: rng.normal(size=(d, q)) / np.sqrt(d)
        U0, V0 = f(m), f(n)
        Us, Vs = [U0 + 0.1 * f(m) for _ in range(K)], [V0 + 0.1 * f(n) for _ in range(K)]
        if kind == "scaled":                             # columns of very different magnitude, a zero one
            sc = 2.0 ** rng.integers(-40, 40, size=q)
            sc[0] = 0.0
            U0, V0 = U0 * sc, V0 / np.where(sc > 0, sc, 1.0)
            Us, Vs = [U * sc for U in Us], [V / np.where(sc > 0, sc, 1.0) for V in Vs]
    S = np.linspace(1.0, 0.1, q)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    W0 = torch.zeros(m, n, device=DEV)
    _, st = iso.frame_merge_factors(dev(U0), dev(S), dev(V0.T), [dev(U) for U in Us], [dev(V.T) for V in Vs], W0,
                                    rho_keep=1.0, ns_iters=1, stats=True)
    torch.cuda.synchronize()
    got = st.gram.cpu().numpy()
    ref, mag = _gamma(U0, Us, V0, Vs, S)
    err = np.abs(got - ref.astype(np.float64)) / mag.astype(np.float64)
    assert err.max() <= 2.0 ** -46, (kind, m, n, err)


def test_nonfinite_column_reaches_the_gram():
    U0 = torch.eye(64, dtype=torch.float64, device=DEV)
    U1 = U0.clone()
    U1[3, 5] = float("nan")
    S = torch.linspace(1.0, 0.1, 64, dtype=torch.float64, device=DEV)
    W0 = torch.zeros(64, 64, device=DEV)
    _, st = iso.frame_merge_factors(U0, S, U0, [U1], [U0], W0, ns_iters=1, stats=True)
    torch.cuda.synchronize()
    assert not torch.isfinite(st.gram).all()


def _peaked(rng, d, q, peak, rest, shift):
    """Columns with one entry `peak`, the others about `rest`; every fourth
    column dense."""
    F = rest * rng.normal(size=(d, q))
    k = np.arange(q)
    F[(k * 7 + shift) % d, k] = peak
    F[:, 3::4] = rng.normal(size=(d, len(k[3::4]))) / np.sqrt(d)
    return F


# columns whose largest entry holds most of their norm (more than one tile of
# 64 of them, a remainder, a few), on different rows in the two operands
@pytest.mark.parametrize("m,n,K", [(130, 129, 2), (336, 337, 1), (2048, 96, 1), (70, 1000, 3), (2500, 5, 2)])
@pytest.mark.parametrize("rest", [1e-3, 1e-5])
def test_gram_of_peaked_columns(m, n, K, rest):
    rng = np.random.default_rng(m + n + K)
    q = min(m, n)
    U0, V0 = _peaked(rng, m, q, 1.0, rest, 0), _peaked(rng, n, q, 1.0, rest, 0)
    Us = [U0 + _peaked(rng, m, q, 1.0, rest, m // 2 + i) for i in range(K)]
    Vs = [V0 + _peaked(rng, n, q, 1.0, rest, n // 2 + i) for i in range(K)]
    S = np.linspace(1.0, 0.1, q)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    W0 = torch.zeros(m, n, device=DEV)
    _, st = iso.frame_merge_factors(dev(U0), dev(S), dev(V0.T), [dev(U) for U in Us], [dev(V.T) for V in Vs], W0,
                                    rho_keep=1.0, ns_iters=1, stats=True)
    torch.cuda.synchronize()
    ref, mag = _gamma(U0, Us, V0, Vs, S)
    err = np.abs(st.gram.cpu().numpy() - ref.astype(np.float64)) / mag.astype(np.float64)
    # binary64 sums: d 2^-53 of the magnitudes at worst
    assert err.max() <= 2.0 ** -49, (m, n, rest, err)


@pytest.mark.parametrize("d,seed", [(1 << 18, s) for s in range(4)] + [(8960, 4), (333, 5)])
@pytest.mark.parametrize("tall", [True, False])
def test_one_small_entry_of_peaked_columns(d, seed, tall):
    """Two modes: one side moved along one peaked column, the other by a
    rotation of 0.7.  Gamma = |dF_2|^2 + 2 0.7^2 - A_12^2 - ... - 1.4 A_12,
    about 2, where A_12 = <F_01, dF_2> is a sum of terms below 0.01 that a
    binary64 sum holds to a few 1e-17; the slices alone leave it off by some
    sqrt(d) 2^-56.3, 6e-15 at d = 2^18.  Bound: 2^-49, eight roundings of
    numbers up to 2 in the sums that follow."""
    rng = np.random.default_rng(seed)
    F0 = np.sqrt(1 - 0.81) / np.sqrt(d) * rng.normal(size=(d, 2))
    dF = np.zeros((d, 2))
    dF[:, 1] = np.sqrt(1 - 0.81) / np.sqrt(d) * rng.normal(size=d)
    F0[1, 0] = F0[d // 2, 1] = dF[d - 2, 1] = 0.9
    O0 = np.eye(2)
    O1 = O0 + np.array([[0.0, 0.7], [-0.7, 0.0]])
    U0, V0, U1, V1 = (F0, O0, F0 + dF, O1) if tall else (O0, F0, O1, F0 + dF)
    S = np.ones(2)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    W0 = torch.zeros(U0.shape[0], V0.shape[0], device=DEV)
    _, st = iso.frame_merge_factors(dev(U0), dev(S), dev(V0.T), [dev(U1)], [dev(V1.T)], W0, rho_keep=1.0, ns_iters=1,
                                    stats=True)
    torch.cuda.synchronize()
    ref, _ = _gamma(U0, [U1], V0, [V1], S)
    err = abs(float(np.longdouble(st.gram.cpu().item()) - ref[0, 0]))
    assert err <= 2.0 ** -49, (d, tall, err)

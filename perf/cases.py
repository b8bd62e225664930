"""The workloads whose speed and results are tracked on a GPU.

A case is one call (or the short sequence of calls) that a program using this
package makes on parameters that it holds on the device: the K = 1 update of a
model by one checkpoint, the merge of several experts, the mask of a task
vector, the frame-space merge of one weight matrix and one optimizer step.
`listed()` names twelve of them; `draw()` gives others of the same ranges.

Model-shaped cases use the Qwen2.5-1.5B and Qwen2.5-7B geometries.  A
parameter list lives packed in one device buffer per checkpoint (every tensor
at a 64-entry boundary), as a program that loads a checkpoint file lays it
out; a model's output is that one buffer.
"""
from __future__ import annotations

import math

import torch

import paper_2607_19331_gb300 as iso

DEV = "cuda"
CHUNK = 1 << 26  # entries of a packed buffer generated at a time

GEOMETRY = {
    # hidden, key/value width, MLP width, vocabulary, layers, separate lm_head
    "qwen1.5b": (1536, 256, 8960, 151936, 28, False),
    "qwen7b": (3584, 512, 18944, 152064, 28, True),
}
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # The smallest call: two fp32 task vectors of one 1024 x 1024 matrix,
        # where launches and latency are all of it.
        dict(name="ties_k2_tiny", kind="merge", rows=1024, cols=1024, op="ties", K=2, base="f32",
             x="f32", ckpt=False, density=0.1, scope="tensor"),
        # One decoder layer corrected by an RL checkpoint (a layer-by-layer
        # loader, a tensor-parallel shard): a few tens of MB, latency again.
        dict(name="update_layer", kind="merge", model="qwen1.5b", layers=1, vocab=False, op="iso", K=1,
             base="bf16", x="bf16", ckpt=True, density=0.05, scope="tensor"),
        # The whole 7B model updated by one checkpoint, the headline workload.
        dict(name="update_7b", kind="merge", model="qwen7b", layers=28, vocab=True, op="iso", K=1,
             base="bf16", x="bf16", ckpt=True, density=0.05, scope="tensor"),
        # fp32 master weights with sizes that divide nothing, TIES trim of the
        # checkpoint's task vector at the paper's density.
        dict(name="update_ragged_f32", kind="merge", rows=5003, cols=6151, op="ties", K=1, base="f32",
             x="f32", ckpt=True, density=0.2, scope="tensor"),
        # The paper's TIES: two RL checkpoints of the 1.5B model, one global
        # magnitude density of 20 % over the whole task vector.
        dict(name="ties_global_1.5b", kind="merge", model="qwen1.5b", layers=28, vocab=True, op="ties", K=2,
             base="bf16", x="bf16", ckpt=True, density=0.2, scope="global"),
        # Eight fp32 task vectors into a bf16 base (layers of the 7B model, as
        # many as a sharded merge job gives one device at a time).
        dict(name="ties_k8_f32", kind="merge", model="qwen7b", layers=3, vocab=False, op="ties", K=8,
             base="bf16", x="f32", ckpt=False, density=0.1, scope="tensor"),
        # The retention merge of three RL checkpoints of the 1.5B model.
        dict(name="iso_k3_1.5b", kind="merge", model="qwen1.5b", layers=28, vocab=True, op="iso", K=3,
             base="bf16", x="bf16", ckpt=True, density=0.2, scope="tensor"),
        # RAM over the same three checkpoints: one pass, no selection.
        dict(name="ram_k3_1.5b", kind="merge", model="qwen1.5b", layers=28, vocab=True, op="ram", K=3,
             base="bf16", x="bf16", ckpt=True, density=0.2, scope="tensor"),
        # One MLP matrix updated under a TopKMask per 128 x 128 block.
        dict(name="update_block", kind="merge", rows=4096, cols=14336, op="ties", K=1, base="bf16",
             x="bf16", ckpt=False, density=0.05, scope="block"),
        # The task vector of one MLP matrix and its packed mask (a program that
        # stores sparse updates).
        dict(name="delta_mask", kind="mask", rows=4096, cols=14336, base="bf16", x="bf16", density=0.2,
             scope="tensor"),
        # The frame-space merge of one 7B gate projection, three experts.
        dict(name="frame_7b_gate", kind="frame", m=3584, n=18944, K=3, w="bf16", rho_keep=0.9),
        # One ISO[AdamW] step of a 1.5B gate projection.
        dict(name="opt_1.5b_gate", kind="opt", m=1536, n=8960, w="bf16", g="bf16", wd=0.0, step=7),
    ]


def draw(rng):
    """One more case: kinds by how often they are called, sizes log-uniform
    (odd ones among them)."""
    def log_size(lo, hi, odd=0.5):
        v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return max(lo, min(hi, v if rng.random() < odd else v // 64 * 64))

    kind = rng.choice(["update", "update", "merge", "merge", "merge", "block", "mask", "frame", "opt"])
    density = rng.choice([0.01, 0.05, 0.1, 0.2, 0.5])
    if kind in ("update", "merge"):
        K = 1 if kind == "update" else rng.randint(2, 8)
        c = dict(kind="merge", op=rng.choice(["ties", "iso", "iso", "ram", "ta"]), K=K, density=density,
                 scope=rng.choice(["tensor", "tensor", "tensor", "global"]),
                 base=rng.choice(["bf16", "bf16", "f32"]), x=rng.choice(["bf16", "bf16", "f32"]),
                 ckpt=rng.random() < 0.6)
        if rng.random() < 0.6:
            model = rng.choice(sorted(GEOMETRY))
            most = 28 if K == 1 and model == "qwen1.5b" else 12 if K <= 3 else 4
            c.update(model=model, layers=log_size(1, most, odd=1.0), vocab=rng.random() < 0.25)
        else:
            c.update(rows=log_size(64, 8192), cols=log_size(64, 20000))
        return c
    if kind == "block":
        return dict(kind="merge", op=rng.choice(["ties", "ties", "iso"]), K=rng.choice([1, 1, 2, 3]),
                    density=density, scope="block", base="bf16", x=rng.choice(["bf16", "bf16", "f32"]),
                    ckpt=rng.random() < 0.5, rows=log_size(128, 8192), cols=log_size(128, 20000))
    if kind == "mask":
        return dict(kind="mask", rows=log_size(64, 8192), cols=log_size(64, 20000), base="bf16",
                    x=rng.choice(["bf16", "f32"]), density=density,
                    scope=rng.choice(["tensor", "tensor", "global", "block"]))
    if kind == "frame":
        a, b = log_size(64, 2048), log_size(64, 9000)
        return dict(kind="frame", m=a, n=b, K=rng.randint(1, 4), w=rng.choice(["bf16", "bf16", "f32"]),
                    rho_keep=rng.choice([0.5, 0.9, 0.9, 1.0]))
    a, b = log_size(64, 3584), log_size(64, 9000)
    m, n = (a, b) if rng.random() < 0.5 else (b, a)
    return dict(kind="opt", m=m, n=n, w=rng.choice(["bf16", "bf16", "f32"]), g=rng.choice(["bf16", "f32"]),
                wd=rng.choice([0.0, 0.01]), step=rng.randint(1, 1000))


# ---------------------------------------------------------------------------
# packed parameter lists
# ---------------------------------------------------------------------------
def shapes_of(case):
    """(rows, cols, is 1-D) of every tensor of a merge or mask case."""
    if "model" not in case:
        r, c = case["rows"], case["cols"]
        if case["kind"] == "mask" or case["scope"] == "block":
            return [(r, c, False)]
        return [(r, c, False), (1, c, True), (max(1, r // 3), c, False)]
    h, kv, it, vocab, _, head = GEOMETRY[case["model"]]
    out = [(vocab, h, False)] if case["vocab"] else []
    for _ in range(case["layers"]):
        out += [(h, h, False), (h, kv, False), (h, kv, False), (h, h, False), (h, it, False), (h, it, False),
                (it, h, False), (1, h, True), (1, h, True)]
    if case["vocab"] and head:
        out.append((vocab, h, False))
    return out


def packed_entries(shapes):
    return sum((r * c + 63) // 64 * 64 for r, c, _ in shapes)


def views(flat, shapes):
    out, at = [], 0
    for r, c, one in shapes:
        t = flat[at:at + r * c]
        out.append(t if one else t.view(r, c))
        at += (r * c + 63) // 64 * 64
    return out


def generator(seed, role):
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1_000_003 + role * 7_919_911 + 17) & 0x7FFFFFFFFFFFFFFF)
    return g


def rl_noise(n, g):
    """An RL update: N(0, (5e-4)^2) with 0.5 % Laplace(0, 5e-3) outliers."""
    d = torch.randn(n, generator=g, device=DEV).mul_(5e-4)
    u = torch.rand(n, generator=g, device=DEV).sub_(0.5)
    pick = torch.rand(n, generator=g, device=DEV) < 0.005
    lap = torch.log1p(-(u.abs() * 2).clamp_(max=1 - 2.0 ** -24)).mul_(-5e-3).mul_(torch.sign(u))
    return torch.where(pick, lap, d)


def fill_packed(n, dtype, make):
    flat = torch.empty(n, dtype=dtype, device=DEV)
    for a in range(0, n, CHUNK):
        b = min(n, a + CHUNK)
        flat[a:b] = make(a, b)
    return flat


def base_and_experts(case, seed):
    n = packed_entries(shapes_of(case))
    g0 = generator(seed, 0)
    base = fill_packed(n, DTYPES[case["base"]], lambda a, b: torch.randn(b - a, generator=g0, device=DEV) * 0.02)
    xs = []
    for i in range(case.get("K", 1)):
        g = generator(seed, 1 + i)
        if case.get("ckpt", True):
            xs.append(fill_packed(n, DTYPES[case["x"]], lambda a, b: base[a:b].float() + rl_noise(b - a, g)))
        else:
            xs.append(fill_packed(n, DTYPES[case["x"]], lambda a, b: rl_noise(b - a, g)))
    return base, xs


# ---------------------------------------------------------------------------
# singular frames
# ---------------------------------------------------------------------------
def rotate(F, shift, std, g, modes):
    """Rotate disjoint pairs of F's columns (modes) or rows by random angles:
    exactly orthogonal in exact arithmetic, so F keeps orthonormal columns."""
    n = F.shape[1] if modes else F.shape[0]
    h = n // 2
    if h == 0:
        return F
    order = torch.roll(torch.arange(n, device=DEV), shift)
    i, j = (order[0:2 * h:2], order[1:2 * h:2]) if modes else (order[:h], order[h:2 * h])
    a = torch.randn(h, generator=g, device=DEV, dtype=torch.float64) * std
    c, s = torch.cos(a), torch.sin(a)
    if modes:
        x, y = F[:, i], F[:, j]
        F[:, i], F[:, j] = x * c - y * s, x * s + y * c
    else:
        x, y = F[i], F[j]
        F[i], F[j] = x * c[:, None] - y * s[:, None], x * s[:, None] + y * c[:, None]
    return F


def base_frame(d, q, g):
    """A dense d x q binary64 frame with orthonormal columns: cosine modes in
    random order and signs, mixed by two reflections."""
    k = torch.randperm(d, generator=g, device=DEV)[:q].double()
    r = torch.randperm(d, generator=g, device=DEV).double()
    F = torch.cos((math.pi / d) * (r[:, None] + 0.5) * k[None, :]).mul_(math.sqrt(2.0 / d))
    F[:, k == 0] *= math.sqrt(0.5)
    F *= torch.sign(torch.rand(d, 1, generator=g, device=DEV, dtype=torch.float64) - 0.5)
    for _ in range(2):
        v = torch.randn(d, generator=g, device=DEV, dtype=torch.float64)
        v /= v.norm()
        F -= 2.0 * torch.outer(v, v @ F)
    return F


def base_factors(m, n, g):
    """U, S, V of a dense weight matrix with entries of about 0.02."""
    q = min(m, n)
    U, V = base_frame(m, q, g), base_frame(n, q, g)
    top, low = math.sqrt(m) + math.sqrt(n), abs(math.sqrt(n) - math.sqrt(m))
    S = 0.02 * torch.linspace(top, low + 0.01 * top, q, device=DEV, dtype=torch.float64)
    return U, S, V


def weight_of(U, S, V, dtype):
    return ((U * S).float() @ V.float().T).to(dtype)


def expert_frames(U, V, g):
    """An expert's frames: modes rotate among their neighbours in the spectrum
    (together on both sides), then each frame turns a little as a whole, and
    each pair of singular vectors has a sign of its own."""
    Ui, Vi = U.clone(), V.clone()
    for shift, std in ((0, 0.3), (1, 0.3)):
        state = g.get_state()
        rotate(Ui, shift, std, g, True)
        g.set_state(state)
        rotate(Vi, shift, std, g, True)
    for shift in (0, 5, 11):
        rotate(Ui, shift, 0.02, g, False)
        rotate(Vi, shift, 0.02, g, False)
    s = torch.sign(torch.rand(U.shape[1], generator=g, device=DEV, dtype=torch.float64) - 0.5)
    return Ui * s, Vi * s


# ---------------------------------------------------------------------------
# the state that a program has in hand, and one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    if case["kind"] in ("merge", "mask"):
        shapes = shapes_of(case)
        base, xs = base_and_experts(case, seed)
        s = dict(case=case, base=views(base, shapes), xs=[views(x, shapes) for x in xs])
        if case["kind"] == "merge":
            s["flat"] = torch.zeros(base.numel(), dtype=base.dtype, device=DEV)
            s["out"] = views(s["flat"], shapes)
        return s
    g = generator(seed, 0)
    U, S, V = base_factors(case["m"], case["n"], g)
    W = weight_of(U, S, V, DTYPES[case["w"]])
    if case["kind"] == "frame":
        ex = [expert_frames(U, V, g) for _ in range(case["K"])]
        return dict(case=case, U0=U, S0=S, Vt0=V.T.contiguous(), Us=[e[0].contiguous() for e in ex],
                    Vts=[e[1].T.contiguous() for e in ex], W0=W, out=torch.empty_like(W))
    G = (torch.randn(case["m"], case["n"], generator=g, device=DEV) * 1e-3).to(DTYPES[case["g"]])
    gu, gv = G.float() @ (V * S).float(), G.float().T @ (U * S).float()  # the scale of the moments
    mu, mv = gu.square().mean().sqrt(), gv.square().mean().sqrt()

    def moments(F, scale):
        return (torch.randn(F.shape, generator=g, device=DEV) * 0.3 * scale,
                (torch.randn(F.shape, generator=g, device=DEV).square() + 0.1) * scale ** 2)
    (mU, vU), (mV, vV) = moments(U, mu), moments(V, mv)
    return dict(case=case, U=U, V=V, S0=S, G=G, mU=mU, vU=vU, mV=mV, vV=vV, W=W, out=torch.empty_like(W))


LR = 7.5e-7


def run(state):
    c = state["case"]
    if c["kind"] == "merge":
        kw = dict(op=c["op"], out=state["out"], density=c["density"], scope=c["scope"])
        if c["K"] == 1:
            iso.iso_update(state["base"], state["xs"][0], update_is_delta=not c["ckpt"], **kw)
        else:
            iso.iso_merge(state["base"], state["xs"], experts_are_deltas=not c["ckpt"], **kw)
        return state["flat"]
    if c["kind"] == "mask":
        tau = iso.iso_delta(state["xs"][0], state["base"])
        return [tau, iso.iso_topk_mask(tau, density=c["density"], scope=c["scope"])]
    if c["kind"] == "frame":
        out, st = iso.frame_merge_factors(state["U0"], state["S0"], state["Vt0"], state["Us"], state["Vts"],
                                          state["W0"], out=state["out"], rho_keep=c["rho_keep"], stats=True)
        return [out, st.gram, st.coef]
    s = state
    iso.opt_step(s["U"], s["V"], s["S0"], s["G"], s["mU"], s["vU"], s["mV"], s["vV"], s["W"], W_out=s["out"],
                 lr=LR, weight_decay=c["wd"], step=c["step"])
    return [s["out"], s["U"], s["V"], s["mU"], s["vU"], s["mV"], s["vV"]]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    size = {"bf16": 2, "f32": 4}
    if case["kind"] == "merge":
        n = sum(r * c for r, c, _ in shapes_of(case))
        return {"bytes": n * (2 * size[case["base"]] + case["K"] * size[case["x"]]), "flops": 0}
    if case["kind"] == "mask":
        n = sum(r * c for r, c, _ in shapes_of(case))
        return {"bytes": n * (size[case["base"]] + size[case["x"]] + 4) + n // 8, "flops": 0}
    m, n = case["m"], case["n"]
    q = min(m, n)
    w = 2 * size[case["w"]] * m * n
    if case["kind"] == "frame":
        K = case["K"]
        # F0^T dF per expert, F0 Y, xi^T xi (symmetric), (F0 + xi) R, and the two products of the reconstruction
        return {"bytes": w + 8 * (K + 1) * (m + n) * q,
                "flops": 2 * q * q * (m + n) * (K + 2.5) + 4 * m * n * q}
    # the two factor gradients, F^T F (symmetric), F R, the reconstruction
    return {"bytes": w + size[case["g"]] * m * n + (m + n) * q * (2 * 8 + 4 * 4),
            "flops": 4 * m * n * q + 3 * q * q * (m + n) + 4 * m * n * q}


def tolerance(case):
    if case["kind"] == "mask":
        return "exact"
    bf16 = case.get("base", case.get("w")) == "bf16"
    if case["kind"] == "merge":
        # one rounding to the output's type of sums of at most nine 32-bit terms:
        # a few entries round the other way
        return {"rel": 5e-5, "max": 1e-2} if bf16 else {"rel": 1e-6, "max": 4e-5}
    if case["kind"] == "frame":
        # two runs of one build differ by 6e-6 (bf16 entries that round the other way)
        return {"rel": 5e-5, "max": 1.6e-2} if bf16 else {"rel": 1e-6, "max": 4e-5}
    # the first moments take the gradient of products summed in 32 bits, up to
    # 7e-6 from their 64-bit value; bf16 weights round the other way now and then
    return {"rel": 3e-5, "max": 1.6e-2 if bf16 else 1e-3}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
def top_k(keys, k):
    """Masks of the k largest keys (int32, >= 0) over a list of flat tensors,
    equal keys taken in order."""
    if k <= 0:
        return [torch.zeros_like(x, dtype=torch.bool) for x in keys]
    t = 0
    for bit in range(30, -1, -1):
        up = t | (1 << bit)
        if sum(int((x >= up).sum()) for x in keys) >= k:
            t = up
    need = k - sum(int((x > t).sum()) for x in keys)
    out = []
    for x in keys:
        tie = x == t
        before = torch.cumsum(tie, 0)
        out.append((x > t) | (tie & (before <= need)))
        need -= int(before[-1]) if x.numel() else 0
    return out


def count_of(density, n):
    return max(0, min(n, int(math.floor(density * n + 0.5))))


def key_of(tau):
    return tau.abs().view(torch.int32)


def block_mask(tau, density):
    r, c = tau.shape
    R, C = (r + 127) // 128, (c + 127) // 128
    keys = torch.full((R * 128, C * 128), -1, dtype=torch.int32, device=DEV)
    keys[:r, :c] = key_of(tau)
    keys = keys.view(R, 128, C, 128).permute(0, 2, 1, 3).reshape(R * C, 128 * 128)
    n = (keys >= 0).sum(1)
    k = torch.floor(density * n.double() + 0.5).long()
    at = torch.sort(keys, dim=1, descending=True, stable=True).indices
    keep = torch.zeros_like(keys, dtype=torch.bool)
    keep.scatter_(1, at, torch.arange(128 * 128, device=DEV)[None, :] < k[:, None])
    return keep.view(R, C, 128, 128).permute(0, 2, 1, 3).reshape(R * 128, C * 128)[:r, :c]


def retention(G):
    """Coefficients of the retention system (ridge 1e-12, clipped to [0, 1.5])
    on the experts of non-zero norm."""
    K = G.shape[0]
    live = [i for i in range(K) if float(G[i, i]) > 0]
    c = torch.zeros(K, dtype=torch.float64)
    if live:
        A = G.cpu()[live][:, live]
        c[live] = torch.linalg.solve(A + 1e-12 * torch.eye(len(live), dtype=torch.float64), torch.diag(A)).clamp(0.0, 1.5)
    return c


def exact_merge(case, seed):
    shapes = shapes_of(case)
    op, K, rho, scope = case["op"], case["K"], case["density"], case["scope"]
    base, xs = base_and_experts(case, seed)
    b, x = views(base, shapes), [views(v, shapes) for v in xs]
    out = torch.zeros(base.numel(), dtype=torch.float64, device=DEV)
    o = views(out, shapes)

    def tau(i, t):
        return x[i][t].float() - b[t].float() if case["ckpt"] else x[i][t].float()

    trims = op in ("ties", "iso")
    cut = [q for q, s in enumerate(shapes) if not (op == "iso" and s[2])] if trims else []
    masks = {}
    if trims and scope == "global":
        for i in range(K):
            keys = [key_of(tau(i, t)).reshape(-1) for t in cut]
            for t, keep in zip(cut, top_k(keys, count_of(rho, sum(v.numel() for v in keys)))):
                masks[i, t] = keep.view(b[t].shape)
    for t in range(len(shapes)):
        vals = []
        for i in range(K):
            v = tau(i, t)
            if t in cut:
                if scope == "global":
                    keep = masks.pop((i, t))
                elif scope == "block" and not shapes[t][2]:
                    keep = block_mask(v, rho)
                else:
                    keep = top_k([key_of(v).reshape(-1)], count_of(rho, v.numel()))[0].view(v.shape)
                v = torch.where(keep, v, torch.zeros_like(v))
            vals.append(v)
        if op == "ta":
            d = sum(v.double() for v in vals)
        elif op == "iso":
            if shapes[t][2]:
                d = sum(v.double() for v in vals) / K
            else:
                G = torch.zeros(K, K, dtype=torch.float64)
                for i in range(K):
                    for j in range(i, K):
                        G[i, j] = G[j, i] = float((vals[i].double() * vals[j].double()).sum())
                c = retention(G).tolist()
                d = sum(ci * v.double() for ci, v in zip(c, vals))
        else:
            if op == "ram":
                act = [v.abs() > torch.tensor(1e-5, dtype=torch.float32, device=DEV) for v in vals]
            else:
                total = vals[0].clone()
                for v in vals[1:]:
                    total = total + v
                sign = torch.sign(total)
                act = [(v != 0) & (torch.sign(v) == sign) for v in vals]
            num = sum(torch.where(a, v.double(), 0.0) for a, v in zip(act, vals))
            d = num / sum(a.double() for a in act).clamp(min=1.0)
        o[t].copy_(b[t].double() + d)
    return out


def inv_sqrt(N):
    """N^(-1/2) of a symmetric positive definite matrix near or above I."""
    I = torch.eye(N.shape[0], dtype=torch.float64, device=DEV)
    c = max(1.0, float(N.norm()) / math.sqrt(N.shape[0])) if float((N - I).norm()) < 0.9 else float(torch.linalg.matrix_norm(N, 1))
    Y, Z = N / c, I.clone()
    last = math.inf
    for _ in range(60):
        E = Z @ Y - I
        err = float(E.abs().max())
        if err < 1e-15 or (err < 1e-6 and err >= last):
            break
        last = err
        M = I - 0.5 * E
        Y, Z = Y @ M, M @ Z
        Y, Z = 0.5 * (Y + Y.T), 0.5 * (Z + Z.T)
    return Z / math.sqrt(c)


def exact_frame(case, seed):
    s = prepare(case, seed)
    m, n, K = case["m"], case["n"], case["K"]
    q = min(m, n)
    D = (torch.arange(q, device=DEV) < max(0, min(q, int(math.floor(case["rho_keep"] * q + 0.5))))).double()
    F0 = [s["U0"], s["Vt0"].T.contiguous()]
    S = s["S0"]
    sign = [torch.where((s["U0"] * U).sum(0) < 0, -1.0, 1.0).double() for U in s["Us"]]
    xi, kw = [[], []], [[], []]
    for i in range(K):
        for side, F in enumerate((s["Us"][i], s["Vts"][i].T)):
            dF = F * sign[i] - F0[side]
            A = F0[side].T @ dF
            sym = 0.5 * (A + A.T)
            xi[side].append((dF - F0[side] @ sym) * D)
            kw[side].append((A - sym) * D)
    G = torch.zeros(K, K, dtype=torch.float64)
    for i in range(K):
        for j in range(i, K):
            v = sum(float(((xi[a][i] * xi[a][j]).sum(0) * S * S).sum()) for a in (0, 1))
            # <xi_Ui S V0^T, U0 S xi_Vj^T> and its mirror
            v += float((S[:, None] * kw[0][i] * (kw[1][j].T * S[None, :])).sum())
            v += float((S[:, None] * kw[0][j] * (kw[1][i].T * S[None, :])).sum())
            G[i, j] = G[j, i] = v
    c = retention(G)
    star = []
    for side in (0, 1):
        X = sum(ci * v for ci, v in zip(c.tolist(), xi[side]))
        A = F0[side].T @ X
        X = X - F0[side] @ (0.5 * (A + A.T))
        Y = F0[side] + X
        star.append(Y @ inv_sqrt(Y.T @ Y))
    W = s["W0"].double() + (star[0] * S) @ (star[1] - F0[1]).T + ((star[0] - F0[0]) * S) @ F0[1].T
    return [W, G, c]


def exact_opt(case, seed):
    s = prepare(case, seed)
    S, G = s["S0"], s["G"].double()
    b1, b2, eps = 0.9, 0.999, 1e-8
    bc1, bc2 = 1 - b1 ** case["step"], 1 - b2 ** case["step"]
    new, mom = [], []
    for F, g, mt, vt in ((s["U"], G @ (s["V"] * S), s["mU"], s["vU"]), (s["V"], G.T @ (s["U"] * S), s["mV"], s["vV"])):
        mt = b1 * mt.double() + (1 - b1) * g
        vt = b2 * vt.double() + (1 - b2) * g * g
        X = F - LR * case["wd"] * F - (LR / bc1) * mt / (torch.sqrt(vt / bc2) + eps)
        new.append(X @ inv_sqrt(X.T @ X))
        mom += [mt, vt]
    U, V = new
    W = s["W"].double() + (U * S) @ (V - s["V"]).T + ((U - s["U"]) * S) @ s["V"].T
    return [W, U, V] + mom


def exact(case, seed):
    if case["kind"] == "merge":
        return exact_merge(case, seed)
    if case["kind"] == "mask":
        s = prepare(case, seed)
        return [[s["xs"][0][0].double() - s["base"][0].double()], [None]]
    return exact_frame(case, seed) if case["kind"] == "frame" else exact_opt(case, seed)

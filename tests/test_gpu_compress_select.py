"""The selections of mkv_compress where its shortcuts could go wrong, on the GPU.

Second stage: without the score2 output the residual pass computes only the
positions whose score bound reaches the first stage's; with it, all of them.
Both must leave the same bits in the cache and the moments (a computed
position's score2 is the same either way), whatever the bound is worth.
First stage: long runs of equal scores, where the threshold bin holds more
keys than the selection exchanges, against a stable sort of the kernel's own
scores."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2606_01563_gb300 import mkv

pytestmark = pytest.mark.gpu


def compress(b, H, G, D, T, B, w, K, V, Q, adaptive, diag, pool=1, mi=1, tau=1e-6):
    g = mkv.geom(b, H, G, D)
    p = mkv.mkv_compress_params(B, w, 1, 1, pool, mi, 1, tau, adaptive)
    prot = 1 + w
    cap = min(T, H * (B - prot) + prot) if adaptive else B
    cache, mom = mkv.alloc_cache(g, cap), mkv.alloc_moments(g)
    ws = mkv.alloc_workspace(mkv.mkv_compress_workspace_size(g, T, p))
    ws.fill_(0xA5)  # the workspace needs no initialisation
    s, s2 = torch.zeros(b, H, T, device="cuda"), torch.zeros(b, H, T, device="cuda")
    mkv.mkv_compress(g, T, K, V, Q, p, cache, mom, ws, diag=(s, s2, None) if diag else None)
    # the error word sits in the workspace, which held no valid status before the call
    torch.cuda.synchronize()
    return dict(K=cache.K, V=cache.V, pos=cache.pos, len=cache.len, n=mom.n, mu_k=mom.mu_k, mu_v=mom.mu_v, C=mom.C,
                s=s, s2=s2)


def draw(seed, b, H, G, D, T, w, kind):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    r = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    K, V = r(b, H, T, D), r(b, H, T, D)
    if kind == "outlier":  # a few long keys: loose bounds for their positions
        K[:, :, ::97] *= 30.0
    elif kind == "correlated":  # C0' as large as the values: the bound says little
        V = 0.9 * K + 0.1 * V
    elif kind == "offset":  # values far from zero
        V = V + 8.0
    elif kind == "zero_values":  # every score2 is the residual of nothing
        V = torch.zeros_like(V)
    elif kind == "infinite":  # bounds and scores that are not finite
        V[:, :, T // 3, 0] = float("inf")
    rows = torch.randint(0, T, (b, H, G * w, 3), generator=gen, device="cuda")
    q = torch.stack([K[i, j][rows[i, j]].sum(1) for i in range(b) for j in range(H)]).view(b, H, G, w, D)
    q = D ** 0.5 * q / torch.linalg.norm(q, dim=-1, keepdim=True) + 0.3 * r(b, H, G, w, D)
    return K.to(torch.bfloat16), V.to(torch.bfloat16), q.to(torch.bfloat16)


@pytest.mark.parametrize("kind", ["plain", "outlier", "correlated", "offset", "zero_values", "infinite"])
@pytest.mark.parametrize("b,H,G,D,T,B,w,adaptive", [
    (4, 8, 4, 128, 8192, 256, 32, 0),   # 16 tiles per CTA
    (2, 16, 2, 64, 4100, 100, 16, 0),   # ragged last tile, half-width rows
    (4, 8, 4, 128, 5001, 200, 32, 1),   # the bound shared by eight heads
])
def test_pruned_residual_selects_the_same(kind, b, H, G, D, T, B, w, adaptive):
    K, V, Q = draw(b * 1000 + D, b, H, G, D, T, w, kind)
    full = compress(b, H, G, D, T, B, w, K, V, Q, adaptive, True)
    pruned = compress(b, H, G, D, T, B, w, K, V, Q, adaptive, False)
    np.testing.assert_array_equal(pruned["len"].cpu(), full["len"].cpu())
    for name in ("pos", "K", "V", "n", "mu_k", "mu_v", "C"):
        x, y = pruned[name].cpu(), full[name].cpu()
        if x.dtype == torch.bfloat16:
            x, y = x.view(torch.int16), y.view(torch.int16)
        elif x.dtype == torch.float32:
            x, y = x.view(torch.int32), y.view(torch.int32)
        assert torch.equal(x, y), f"{name} differs at {int((x != y).sum())} of {x.numel()} places"


@pytest.mark.parametrize("T,B,adaptive,pool", [(700, 64, 0, 1), (9000, 500, 0, 32), (30000, 900, 0, 1), (6000, 300, 1, 1)])
def test_equal_scores_take_the_lowest_positions(T, B, adaptive, pool):
    """Keys that repeat every few rows: most scores are equal to many others,
    and a tie that crosses the budget is broken by position (head first)."""
    H, G, D, w = 2, 2, 64, 16
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T)
    base = torch.randn(1, H, 3, D, generator=gen, device="cuda").to(torch.bfloat16)
    K = base[:, :, torch.arange(T, device="cuda") % 3].contiguous()
    V = torch.randn(1, H, T, D, generator=gen, device="cuda").to(torch.bfloat16)
    Q = torch.randn(1, H, G, w, D, generator=gen, device="cuda").to(torch.bfloat16)
    out = compress(1, H, G, D, T, B, w, K, V, Q, adaptive, True, pool=pool, mi=0)
    t = np.arange(T)
    prot = (t < 1) | (t >= T - w)
    s = out["s"][0].double().cpu().numpy()
    k = B - int(prot.sum())
    if adaptive:
        want, _ = O.select_topk_joint(s, H * k, np.stack([prot] * H))
    else:
        want = [O.select_topk(s[h], k, prot)[0] for h in range(H)]
    for h in range(H):
        got = out["pos"][0, h, :int(out["len"][0, h])].cpu().numpy()
        np.testing.assert_array_equal(got, want[h])


def test_joint_selection_of_many_groups():
    """The last selected pair of a joint selection is found by one CTA of each
    cluster and stored into the others, over the value they start with: 40
    groups of 8 clusters, more than run at once, five times over."""
    b, H, G, D, T, B, w = 40, 8, 1, 64, 640, 48, 16
    K, V, Q = draw(17, b, H, G, D, T, w, "plain")
    t = np.arange(T)
    prot = np.stack([(t < 1) | (t >= T - w)] * H)
    for _ in range(5):
        out = compress(b, H, G, D, T, B, w, K, V, Q, 1, True, mi=0)
        s, ln, pos = out["s"].double().cpu().numpy(), out["len"].cpu().numpy(), out["pos"].cpu().numpy()
        for i in range(b):
            want, _ = O.select_topk_joint(s[i], H * (B - 1 - w), prot)
            for h in range(H):
                np.testing.assert_array_equal(pos[i, h, :ln[i, h]], want[h])


def test_pruning_bound_of_rounding_size():
    """Values near one large constant, so that the first stage's lower bounds
    ||v|| - ||mu_v0|| are differences of nearly equal norms, no larger than a
    few of their roundings; in each unit one row of the opposite sign whose
    score2 lies just above the weakest first-stage row's and meets its own
    upper bound.  (tau clamps all of C0'.)"""
    b, H, G, D, T, B, w = 4, 8, 2, 128, 32768, 64, 16
    U, k, scale, q0, q1 = b * H, B - 1 - w, D ** -0.5, 16.0, 2.0 ** -4
    gen = torch.Generator()
    gen.manual_seed(9)
    logit = torch.full((U, T), -17.0, dtype=torch.float64)
    a = torch.full((U, T), 256.0)
    opposite = torch.empty(U, dtype=torch.int64)
    for u in range(U):
        at = 1 + torch.randperm(T - w - 1, generator=gen)
        n1 = 4 + u  # values of 255: mu_v0 = 256 - n1 / n0 per dim (one value of -256 against two of 512)
        r = D ** 0.5 * n1 / (T - B)
        first, opposite[u] = at[:k], at[k]
        logit[u, first] = 0.2 * torch.arange(k, dtype=torch.float64)
        # a quarter of a rounding of ||mu_v0|| = 2896 above the weakest row's score2
        logit[u, at[k]] = np.log(r / (512 * D ** 0.5)) + 0.25 * 1.2e-4 / r
        a[u, at[k]] = -256.0
        a[u, at[k + 1:k + 3]] = 512.0
        a[u, at[k + 3:k + 3 + n1]] = 255.0
    K = torch.zeros(U, T, D)
    x = torch.round(logit / (scale * q0) * 16) / 16
    K[:, :, 0] = x
    K[:, :, 1] = (logit - scale * q0 * x) / (scale * q1)
    Q = torch.zeros(b, H, G, w, D)
    Q[..., 0], Q[..., 1] = q0, q1
    K = K.view(b, H, T, D).to(torch.bfloat16).cuda()
    V = a[:, :, None].expand(U, T, D).reshape(b, H, T, D).to(torch.bfloat16).cuda()
    Q = Q.to(torch.bfloat16).cuda()
    full = compress(b, H, G, D, T, B, w, K, V, Q, 0, True, tau=1e30)
    pruned = compress(b, H, G, D, T, B, w, K, V, Q, 0, False, tau=1e30)
    pos = full["pos"].view(U, -1).cpu()
    assert all(int(opposite[u]) in pos[u].tolist() for u in range(U))
    assert torch.equal(pruned["pos"].view(U, -1).cpu(), pos)


@pytest.mark.parametrize("kind,H,T,B,adaptive,pool", [
    ("distinct", 2, 40000, 16000, 0, 1),   # more contested keys than a list holds, all different
    ("distinct", 8, 24000, 2600, 1, 1),    # the same of a joint selection
    ("chunks", 2, 30001, 9000, 0, 32),     # equal in runs of 32
    ("chunks", 4, 30001, 4000, 1, 32),
    ("close", 2, 40000, 6000, 0, 1),       # one bin, most keys apart in their last bits only
    ("close", 4, 16000, 2000, 1, 1),
    ("equal", 2, 20000, 900, 0, 1),        # all equal: by position alone
    ("equal", 64, 700, 40, 1, 1),          # the last selected pair in one of the later heads
    ("zero", 2, 30000, 700, 0, 1),         # fewer scores above zero than selections
    ("zero", 8, 9000, 300, 1, 1),
    ("tail", 2, 30000, 700, 0, 1),         # the threshold far below the bins a CTA counts on its own
    ("tail", 8, 9000, 300, 1, 1),
])
def test_more_contested_keys_than_the_lists_hold(kind, H, T, B, adaptive, pool):
    """Selections whose threshold bin holds more keys than the exchanged lists,
    against a stable sort of the kernel's own scores."""
    G, D, w = 1, 64, 8
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T + B)
    r = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    K, V, Q = r(1, H, T, D), r(1, H, T, D), r(1, H, G, w, D)
    if kind == "close":
        K *= 1e-3
    elif kind == "equal":
        K[:] = K[:, :1, :1]
    elif kind == "zero":  # 400 keys hold all the weight
        K[:, :, 400:] = -40.0 * Q[:, :, 0, :1]
        Q[:] = Q[:, :, :, :1]
    elif kind == "tail":  # 100 keys hold all the weight, the others from e^-18 of theirs down to e^-28
        Q[:] = Q[:, :, :, :1]
        logit = -18.0 - 10.0 * torch.rand(1, H, T, 1, generator=gen, device="cuda")
        logit[:, :, :100] = 0.0
        q0 = Q[:, :, 0, :1]
        K = logit * D ** 0.5 * q0 / (q0 * q0).sum(-1, keepdim=True)
    K, V, Q = (x.to(torch.bfloat16) for x in (K, V, Q))
    out = compress(1, H, G, D, T, B, w, K, V, Q, adaptive, True, pool=pool, mi=0)
    t = np.arange(T)
    prot = (t < 1) | (t >= T - w)
    s = out["s"][0].double().cpu().numpy()
    if kind == "zero":
        assert (s[:, 500:T - w] == 0).all()
    elif kind == "tail":
        assert (s[:, 200:T - w] < 2.0 ** -21).all() and (s > 0).all()
    k = B - int(prot.sum())
    if adaptive:
        want, _ = O.select_topk_joint(s, H * k, np.stack([prot] * H))
    else:
        want = [O.select_topk(s[h], k, prot)[0] for h in range(H)]
    for h in range(H):
        np.testing.assert_array_equal(out["pos"][0, h, :int(out["len"][0, h])].cpu().numpy(), want[h])

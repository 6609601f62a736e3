"""How far certified decode is from 64 bits, over the heads of a few hundred units:
root mean square of the relative errors of y_hat (2-norm), b_t and V_hat, and of the
error of log N_hat, each clipped (heads whose certificate cancels).

The limits are what float32 multiply-adds (odd capacities, float32 caches, the
exact range term) or 8-warp CTAs with 16-bit weights (many units) left on these
very inputs, measured once, and 5% (V_hat, whose terms cancel: 10%) for the order of
sums: another way of computing them may be no less exact."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def E():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_21475_gb300.build import build
    build()
    from paper_2607_21475_gb300 import ebd
    return ebd


def reference(Q, K, V, lw, n, exact):
    """y, log N_hat, V_hat and b_t of one batch row in 64 bits."""
    H, cap, d = K.shape
    q, k, v, lw = Q.view(H, -1, d).double(), K.double(), V.double(), lw.double().unsqueeze(1)
    live = (torch.arange(cap, device=DEV) < n.unsqueeze(-1)).unsqueeze(1)
    x = torch.where(live, q @ k.transpose(1, 2) / math.sqrt(d) + lw, -math.inf)
    lse = torch.logsumexp(x, -1)
    p = torch.exp(x - lse.unsqueeze(-1))
    y = p @ v
    om = -torch.expm1(-lw)
    dist = torch.stack([(v - y[:, g:g + 1]).norm(dim=-1) for g in range(q.shape[1])], 1)
    var = (om * p * p * dist.square()).sum(-1)
    sp = om.sqrt() * p
    if exact:
        bt = (sp * dist).amax(-1)
    else:
        c = torch.stack([v[h, (int(n[h]) - 1) // 2] for h in range(H)]).unsqueeze(1)
        bt = ((sp * (v - c).norm(dim=-1).unsqueeze(1)).amax(-1) +
              (y - c).norm(dim=-1) * sp.amax(-1))
    return y.flatten(0, 1), lse.flatten(), var.flatten(), bt.flatten()


def errors(E, B, H, G, d, rows, cap, exact, dtype, scale, seeds):
    out = [[], [], [], []]
    for seed in range(seeds):
        g = torch.Generator(device=DEV).manual_seed(100 + seed)
        rnd = lambda *s: torch.randn(s, generator=g, device=DEV)
        K, V = rnd(B, H, cap, d).to(dtype), rnd(B, H, cap, d).to(dtype)
        lw = -torch.log(torch.rand((B, H, cap), generator=g, device=DEV).clamp(min=1e-3))
        lw[torch.rand((B, H, cap), generator=g, device=DEV) < 0.2] = 0.0
        n = (rows - torch.randint(0, 17, (B, H), generator=g, device=DEV)).to(torch.int32)
        Q = (scale * rnd(B, H * G, d)).to(dtype)
        y = torch.empty((B, H * G, d), device=DEV)
        lse, var, bt, r = (torch.empty((B, H * G), device=DEV) for _ in range(4))
        E.ebd_certified_decode(Q, K, V, lw, n, y, lse, var, bt, r,
                               range_mode=E.EBD_RANGE_EXACT if exact else E.EBD_RANGE_BOUND)
        for b in range(B):
            ry, rl, rv, rb = reference(Q[b], K[b], V[b], lw[b], n[b], exact)
            out[0].append((y[b].double() - ry).norm(dim=-1) / ry.norm(dim=-1))
            out[1].append((lse[b].double() - rl).abs())
            out[2].append(((var[b].double() - rv) / rv).abs())
            out[3].append(((bt[b].double() - rb) / rb).abs())
    return [float(torch.cat(e).clamp(max=5e-6).square().mean().sqrt()) for e in out]


BF, F32 = torch.bfloat16, torch.float32
CASES = [
    # B, H, G, d, rows, cap, exact, dtype, query scale, seeds, limits of y, lse, V_hat, b_t
    (50, 8, 5, 64, 3277, 3840, False, BF, 3.0, 1,
     (19.34e-7, 7.81e-7, 22.96e-7, 6.70e-7)),
    (32, 8, 8, 128, 3277, 3840, False, BF, 3.0, 1,
     (18.81e-7, 7.93e-7, 23.28e-7, 6.85e-7)),
    (32, 8, 4, 128, 3277, 3840, False, BF, 1.0, 1,
     (22.30e-7, 5.28e-7, 14.76e-7, 4.63e-7)),
    (32, 8, 4, 128, 1000, 1344, False, BF, 3.0, 2,
     (16.20e-7, 8.85e-7, 23.27e-7, 7.60e-7)),
    (4, 8, 8, 128, 1000, 1100, False, F32, 3.0, 8,
     (3.90e-7, 4.07e-7, 12.59e-7, 3.58e-7)),
    (4, 8, 3, 64, 2000, 2200, True, F32, 3.0, 8,
     (4.09e-7, 3.81e-7, 11.93e-7, 5.54e-7)),
    (4, 8, 5, 128, 2460, 2953, True, BF, 3.0, 6,
     (4.30e-7, 4.03e-7, 11.18e-7, 5.30e-7)),
    (2, 8, 4, 128, 3000, 3333, True, BF, 3.0, 6,
     (4.43e-7, 4.16e-7, 10.43e-7, 5.91e-7)),
    (4, 8, 2, 64, 9000, 9501, False, BF, 1.0, 6,
     (3.08e-7, 3.18e-7, 3.05e-7, 2.81e-7)),
    (4, 8, 8, 128, 1500, 1801, False, BF, 3.0, 6,
     (4.09e-7, 4.12e-7, 13.11e-7, 3.80e-7)),
    (4, 8, 5, 128, 2460, 2960, True, BF, 3.0, 6,
     (14.28e-7, 7.64e-7, 20.00e-7, 12.30e-7)),
]


@pytest.mark.parametrize("B,H,G,d,rows,cap,exact,dtype,scale,seeds,limits", CASES)
def test_errors_against_64_bits(E, B, H, G, d, rows, cap, exact, dtype, scale, seeds, limits):
    got = errors(E, B, H, G, d, rows, cap, exact, dtype, scale, seeds)
    for name, e, most in zip(("y", "lse", "V_hat", "b_t"), got, limits):
        assert e <= (1.10 if name == "V_hat" else 1.05) * most, (name, e, most)


@pytest.mark.parametrize("B,H,G,d,rows,cap,mean,limit", [
    (2, 8, 4, 128, 1500, 1808, 16.0, 8.76e-6),
    (2, 8, 7, 128, 1500, 1808, 4.0, 3.24e-6),
    (2, 8, 2, 64, 1500, 1808, 16.0, 13.12e-6),
    (2, 8, 8, 128, 1500, 1808, 16.0, 18.96e-6),
    (2, 8, 5, 128, 1500, 1808, 0.0, 1.57e-6),
])
def test_contributions_against_64_bits(E, B, H, G, d, rows, cap, mean, limit):
    """The same for the contributions of given y_hat and log N_hat (2-norm over a
    head), of values with a common mean; the limits are what head constants summed
    over a whole warp left."""
    errs = []
    for seed in range(4):
        g = torch.Generator(device=DEV).manual_seed(300 + seed)
        rnd = lambda *s: torch.randn(s, generator=g, device=DEV)
        K, V = rnd(B, H, cap, d).to(BF), (rnd(B, H, cap, d) + mean).to(BF)
        lw = torch.rand((B, H, cap), generator=g, device=DEV) + 0.1
        n = torch.full((B, H), rows, dtype=torch.int32, device=DEV)
        Q = (2 * rnd(B, H * G, d)).to(BF)
        ref = [reference(Q[b], K[b], V[b], lw[b], n[b], True) for b in range(B)]
        y = torch.stack([r[0] for r in ref]).float()
        lse = torch.stack([r[1] for r in ref]).float()
        con = E.ebd_variance_contributions(Q, K, V, lw, n, y, lse)
        for b in range(B):
            q, k = Q[b].view(H, G, d).double(), K[b].double()
            w = lw[b].double().unsqueeze(1)
            p = torch.exp(q @ k.transpose(1, 2) / math.sqrt(d) + w - lse[b].view(H, G, 1).double())
            dist = torch.stack([(V[b].double() - y[b].view(H, G, 1, d)[:, g_].double())
                                .square().sum(-1) for g_ in range(G)], 1)
            c = (-torch.expm1(-w) * p * p * dist)[..., :rows].flatten(0, 1)
            e = (con[b, :, :rows].double() - c).norm(dim=-1) / c.norm(dim=-1)
            errs.append(e)
    assert float(torch.cat(errs).square().mean().sqrt()) <= limit

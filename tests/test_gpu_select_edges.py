"""Selection at the edges of the shared-memory select: digits of 11, 11 and 10
bits, groups of 4096 tokens, clusters of any size from 2 to 8, ragged units,
scores of either sign, and the systematic walk, against the float64 oracle (the
kept sets exactly, but for draws within the float32 band of pi)."""
import numpy as np
import pytest
import torch

from oracle import ebd_oracle as O
from tests.parity import TIE_BAND

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


def scores(kind, shape, seed):
    g = torch.Generator().manual_seed(seed)
    if kind == "close":     # equal first digits: the second and third decide
        return 1.0 + torch.randint(0, 40000, shape, generator=g).float() * 2.0 ** -23
    if kind == "equal":     # one value: the ordered scan of the ties decides
        return torch.full(shape, 0.75)
    if kind == "signed":    # negative keys, zeros of both signs
        s = torch.randn(shape, generator=g)
        s[s.abs() < 0.3] = -0.0
        return s
    if kind == "extreme":   # 50 of the largest floats (in the top slice: the sums
        # of the scale are float32), subnormals, and 26 decades between
        s = torch.exp(10 * torch.randn(shape, generator=g)).clamp(1e-13, 1e13)
        s[..., ::7] = 1e-42
        s[..., 5:405:8] = torch.finfo(torch.float32).max
        return s
    if kind == "zeros":     # sparse scores: the k-th largest is 0
        return torch.zeros(shape)
    if kind == "few":       # 31 above 0, the others 0 of either sign
        s = torch.zeros(shape)
        s[..., 1::3] = -0.0
        s[..., 50:3150:100] = torch.exp(torch.randn(s[..., 50:3150:100].shape, generator=g))
        return s
    if kind == "few_subnormal":
        s = scores("few", shape, seed)
        s[..., ::2][s[..., ::2] <= 0] = 1e-42
        s[..., 1::4][s[..., 1::4] <= 0] = -1e-42
        return s
    if kind == "few_negative":  # 31 above 0, a quarter at 0, the others below
        s = scores("few", shape, seed)
        return torch.where((s > 0) | (torch.rand(shape, generator=g) < 0.25), s,
                           -torch.rand(shape, generator=g))
    if kind == "negative":  # the k-th largest below 0
        s = -torch.rand(shape, generator=g)
        s[..., 50:3150:100] = 0.5
        s[..., 60:2060:100] = 0.0
        return s
    return torch.exp(1.5 * torch.randn(shape, generator=g))


@pytest.mark.parametrize("N,k_head,budget,kind,systematic", [
    (4096, 80, 400, "close", False),
    (4097, 80, 400, "close", True),
    (4100, 1, 300, "equal", False),
    (8191, 500, 2000, "signed", False),
    (8192, 500, 2000, "signed", True),
    (12289, 300, 9000, "lognormal", False),    # clipped tail: several steps of the scale
    (20000, 400, 2000, "extreme", False),
    (32768, 655, 3277, "close", False),
    (65537, 1300, 6500, "close", False),       # clusters of 3, 6 CTAs ...
    (100003, 5000, 25000, "lognormal", True),
    (140000, 2000, 14000, "equal", False),     # ... of 5
    (170001, 3400, 17000, "lognormal", True),  # ... of 6
    (200001, 100, 20000, "close", False),      # ... of 7
    (512, 10, 51, "zeros", False),
    (4097, 80, 400, "zeros", True),
    (8191, 500, 2000, "few", False),
    (8192, 80, 2000, "few_subnormal", False),
    (20000, 400, 2000, "few_negative", False),
    (32768, 655, 3277, "few", True),
    (32768, 100, 3277, "negative", False),
    (65537, 1300, 6500, "zeros", False),       # ties of 0 across clusters
    (100003, 5000, 25000, "few_negative", True),
    (140000, 2000, 14000, "few_subnormal", False),
    (200001, 100, 20000, "few", False),
])
def test_select_at_digit_and_cluster_edges(E, N, k_head, budget, kind, systematic):
    B, H, cap = 1, 2, -(-(budget + 9 * int(budget ** 0.5) + 64) // 16) * 16
    s = scores(kind, (B, H, N), N)
    des = E.design_for(batch=B, n_kv_heads=H, group=1, head_dim=64, n_ctx=N, layer=2, seed=11,
                       k_head=k_head, budget_tokens=budget, sampling=int(systematic))
    c = E.alloc_compact(B, H, cap, 64, torch.bfloat16, DEV)
    E.ebd_select(des, s.to(DEV), c)
    pi = torch.empty((B, H, N), device=DEV)
    mask = torch.empty((B, H, N), dtype=torch.uint8, device=DEV)
    E.ebd_compute_pi(des, s.to(DEV), pi, mask)
    torch.cuda.synchronize()
    assert int(c.dev_status) == 0
    for h in range(H):
        u = s[0, h].numpy()
        u = np.where(np.abs(u) < np.finfo(np.float32).tiny, np.float32(0), u)  # read as 0
        cert, _ = O.certainty_set(u, 4, 32, k_head)
        assert np.array_equal(mask[0, h].cpu().numpy().astype(bool), cert)
        ref, _, m = O.inclusion_probabilities(u, cert, budget, 1e-6)
        np.testing.assert_allclose(pi[0, h].cpu().double().numpy(), ref, rtol=2e-5, atol=0)
        n = int(c.n_kept[0, h])
        idx = c.idx_c[0, h, :n].cpu().numpy()
        assert np.all(np.diff(idx) > 0) and set(np.flatnonzero(cert)) <= set(idx.tolist())
        np.testing.assert_allclose(c.logw_c[0, h, :n].cpu().numpy(), -np.log(ref[idx]), rtol=2e-5,
                                   atol=2e-6)
        if systematic:
            tail = n - int(cert.sum())
            assert abs(tail - ref[~cert].sum()) <= 1.0 + 1e-3
        else:
            uni, _ = O.philox_uniforms(11, 2, 0, h, N)
            near = ~cert & (np.abs(uni - ref) < TIE_BAND)
            kept = cert | (uni < ref.astype(np.float32))
            diff = np.flatnonzero(kept != np.isin(np.arange(N), idx))
            assert np.all(near[diff])


def test_redraw_with_scores_of_zero(E):
    """Re-eviction of ragged units from scores that are exactly 0 on most rows, as
    variance contributions are on certain rows, fewer of them above 0 than the
    top slice holds."""
    B, H, d, cap, k_head, budget = 2, 2, 64, 4736, 819, 2048
    g = torch.Generator().manual_seed(5)
    n = torch.tensor([[4352, 4097], [1, 4736]], dtype=torch.int32)
    s = torch.exp(torch.randn((B, H, cap), generator=g))
    s[torch.rand((B, H, cap), generator=g) < 0.9] = 0.0
    src, out = (E.alloc_compact(B, H, cap, d, torch.bfloat16, DEV) for _ in range(2))
    src.K_c.copy_(torch.randn((B, H, cap, d), generator=g))
    src.V_c.copy_(torch.randn((B, H, cap, d), generator=g))
    src.logw_c.zero_()
    src.idx_c.copy_(torch.arange(cap, dtype=torch.int32).mul(3).expand(B, H, cap))
    src.n_kept.copy_(n)
    des = E.design_for(batch=B, n_kv_heads=H, group=1, head_dim=d, n_ctx=cap, layer=3, seed=17,
                       k_head=k_head, budget_tokens=budget)
    E.ebd_reevict(des, s.to(DEV), src, out)
    torch.cuda.synchronize()
    assert int(out.dev_status) == 0
    for b in range(B):
        for h in range(H):
            m = int(n[b, h])
            ref = O.reevict_unit(
                *(t[b, h, :m].double().cpu().numpy() for t in (src.K_c, src.V_c, src.logw_c)),
                src.idx_c[b, h, :m].cpu().numpy(), s[b, h, :m].numpy(), n_sink=4, n_recent=32,
                k_head=k_head, budget_tokens=budget, eps=1e-6, seed=17, layer=3, b=b, kvh=h,
                capacity=cap)
            near = ~ref.inner.certain & (np.abs(ref.inner.u - ref.inner.pi) < TIE_BAND)
            got = out.idx_c[b, h, :int(out.n_kept[b, h])].cpu().numpy() // 3
            assert np.all(np.diff(got) > 0)
            diff = set(got.tolist()) ^ set(ref.inner.idx.tolist())
            assert all(near[i] for i in diff)

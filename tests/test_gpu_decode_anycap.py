"""The certified decode on capacities that are no multiple of a tile (the
tensor-core kernels with their last tile cut at the capacity and weights of 24
bits) and the exact range term, against the float64 oracle.

Bars: these capacities are served in float32 throughout, so y_hat is held to
2e-6 of its norm (24-bit weights, float32 sums) and not to the 16-bit bar; the
exact range term, a maximum of values each formed in float32, to 1e-5."""
import numpy as np
import pytest
import torch

from oracle import ebd_oracle as O
from tests.parity import compare_decode_heads
from tests.test_gpu_parity import _decode, _synthetic_cache, E  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu
DEV = "cuda"

CASES = [
    # B, H, G, d, cap, pattern, mean, query scale
    (1, 2, 1, 64, 17, "edges", 0.3, 1.0),         # two tiles, the second one row
    (2, 4, 4, 128, 1637, "edges", 0.3, 1.0),      # clusters, packed heads
    (1, 4, 7, 128, 2953, "random", 4.0, 3.0),     # clusters, peaked attention, a common mean
    (16, 8, 8, 64, 501, "edges", 0.3, 1.0),       # one CTA per unit
    (32, 8, 3, 128, 203, "random", 16.0, 1.0),    # in waves
    (1, 2, 5, 128, 20001, "full", 0.3, 3.0),      # split-K, few long units, every row kept
    (20, 10, 4, 64, 259, "edges", 0.3, 1.0),      # split-K, 200 units
    (2, 2, 12, 128, 1101, "random", 0.3, 1.0),    # two slices of heads
]


@pytest.mark.parametrize("exact", [False, True])
@pytest.mark.parametrize("B,H,G,d,cap,pattern,mean,scale", CASES)
def test_any_capacity_matches_oracle_in_float32(E, B, H, G, d, cap, pattern, mean,  # noqa: F811
                                                scale, exact):
    Kc, Vc, logw, n = _synthetic_cache(B, H, cap, d, torch.bfloat16, pattern, seed=cap, vmean=mean)
    g = torch.Generator().manual_seed(cap + 1)
    Q = (scale * torch.randn((B, H * G, d), generator=g)).to(torch.bfloat16)
    # rows past each unit's last hold NaN: no result may depend on them
    for b in range(B):
        for h in range(H):
            k = min(int(n[b, h]), cap)
            Kc[b, h, k:], Vc[b, h, k:], logw[b, h, k:] = np.nan, np.nan, np.nan
    out = _decode(E, Q.to(DEV), Kc.to(DEV), Vc.to(DEV), logw.to(DEV), n.to(DEV), exact)
    Qd, Kd, Vd, ld = Q.double().numpy(), Kc.double().numpy(), Vc.double().numpy(), logw.double().numpy()
    for b in range(B):
        for h in range(H):
            if B * H > 32 and (b * H + h) % 7:
                continue
            k = min(int(n[b, h]), cap)
            dec = O.hajek_decode(Qd[b, h * G:(h + 1) * G], Kd[b, h, :k], Vd[b, h, :k], ld[b, h, :k])
            sl = slice(h * G, (h + 1) * G)
            compare_decode_heads(dec, out[0][b, sl], out[1][b, sl], out[2][b, sl], out[3][b, sl],
                                 out[4][b, sl], exact)
            # relative to the values' size: y_hat of near-uniform weights is a
            # small mean of them
            size = np.sqrt(np.mean(np.square(Vd[b, h, :k]))) * np.sqrt(d) if k else 1.0
            wmax = np.linalg.norm(dec.y, axis=1).clip(min=size / np.sqrt(max(k, 1)))
            assert np.all(np.linalg.norm(out[0][b, sl] - dec.y, axis=1) <= 2e-6 * wmax)
            if exact:
                assert np.all(np.abs(out[3][b, sl] - dec.b_exact) <=
                              1e-5 * dec.b_exact + 1e-7 * np.linalg.norm(dec.y, axis=1))


@pytest.mark.parametrize("G,d,cap,mean,scale", [(4, 128, 4096, 16.0, 3.0), (8, 64, 2048, 0.0, 8.0),
                                               (7, 128, 1600, 0.0, 8.0)])
def test_exact_range_term_when_one_row_dominates(E, G, d, cap, mean, scale):  # noqa: F811
    """Peaked attention: y_hat lies close to one retained value, so that row's
    distance is a small difference of large terms."""
    B, H = 2, 2
    Kc, Vc, logw, n = _synthetic_cache(B, H, cap, d, torch.bfloat16, "random", 5, vmean=mean)
    g = torch.Generator().manual_seed(6)
    Q = (scale * torch.randn((B, H * G, d), generator=g)).to(torch.bfloat16)
    out = _decode(E, Q.to(DEV), Kc.to(DEV), Vc.to(DEV), logw.to(DEV), n.to(DEV), True)
    for b in range(B):
        for h in range(H):
            k = int(n[b, h])
            dec = O.hajek_decode(Q[b, h * G:(h + 1) * G].double().numpy(),
                                 Kc[b, h, :k].double().numpy(), Vc[b, h, :k].double().numpy(),
                                 logw[b, h, :k].double().numpy())
            got = out[3][b, h * G:(h + 1) * G]
            # | ||v - y'|| - ||v - y|| | <= ||y' - y||: at these capacities y_hat
            # is of 16-bit weights, so off by up to 2^-16 of the values' size
            # (||y_hat|| of a dominated head), times p <= 1
            tol = 1e-5 * dec.b_exact + 2.0 ** -16 * np.linalg.norm(dec.y, axis=1)
            assert np.all(np.abs(got - dec.b_exact) <= tol)


@pytest.mark.parametrize("G,d,cap", [(4, 128, 1600), (7, 128, 1601), (8, 64, 304)])
def test_exact_range_term_of_small_tail_weights(E, G, d, cap):  # noqa: F811
    """A certain row that takes all but 1e-25 of the weight: the tail's range term
    is as small, and has its float32 digits all the same (the logits, 60 apart,
    round by up to 4e-6 each)."""
    B, H = 1, 2
    Kc, Vc, logw, n = _synthetic_cache(B, H, cap, d, torch.bfloat16, "random", 5)
    g = torch.Generator().manual_seed(6)
    Q = torch.randn((B, H * G, d), generator=g).to(torch.bfloat16)
    Q[..., 0], Kc[..., 0] = 16.0, 0.0
    Kc[:, :, 50, 0] = 60.0 * d ** 0.5 / 16.0
    logw[:, :, 50] = 0.0
    out = _decode(E, Q.to(DEV), Kc.to(DEV), Vc.to(DEV), logw.to(DEV), n.to(DEV), True)
    for h in range(H):
        k = int(n[0, h])
        dec = O.hajek_decode(Q[0, h * G:(h + 1) * G].double().numpy(),
                             Kc[0, h, :k].double().numpy(), Vc[0, h, :k].double().numpy(),
                             logw[0, h, :k].double().numpy())
        assert np.all(dec.b_exact > 0) and np.all(dec.b_exact < 1e-20)
        np.testing.assert_allclose(out[3][0, h * G:(h + 1) * G], dec.b_exact, rtol=2e-5)


def test_exact_range_term_takes_no_longer_when_values_share_a_mean(E):  # noqa: F811
    """Values with a mean of 256 times their spread on every channel: the rows that
    the range pass has to evaluate one by one stay few, so the call takes about the
    time it takes without the mean (every one of them: several times that)."""
    B, H, G, d, cap = 4, 8, 5, 128, 2960
    g = torch.Generator().manual_seed(7)
    K, V = (torch.randn((B, H, cap, d), generator=g).to(torch.bfloat16).to(DEV) for _ in range(2))
    Q = torch.randn((B, H * G, d), generator=g).to(torch.bfloat16).to(DEV)
    lw = torch.rand((B, H, cap), generator=g).add(0.1).to(DEV)
    n = torch.full((B, H), 2460, dtype=torch.int32, device=DEV)
    y = torch.empty((B, H * G, d), device=DEV)
    o = [torch.empty((B, H * G), device=DEV) for _ in range(4)]
    ws = torch.empty(E.ebd_decode_workspace_bytes(E.EBD_BF16, B, H, G, d, cap), dtype=torch.uint8,
                     device=DEV)

    def microseconds(mean):
        Vm = (V.float() + mean).to(torch.bfloat16)
        best = float("inf")
        for _ in range(5):
            t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            for k in range(60):
                if k == 10:
                    t0.record()
                E.ebd_certified_decode(Q, K, Vm, lw, n, y, *o, range_mode=E.EBD_RANGE_EXACT,
                                       workspace=ws)
            t1.record()
            torch.cuda.synchronize()
            best = min(best, t0.elapsed_time(t1) * 20)
        return best

    assert microseconds(256.0) <= 1.5 * microseconds(0.0)

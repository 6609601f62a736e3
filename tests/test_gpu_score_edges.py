"""Accumulated-attention scores at the edges of the tensor-core kernels' tiles (pass
1: 128 query rows x 256 keys, the key tiles split over a cluster of up to eight
CTAs with at least four each; pass 2: 128 keys, up to 512 query rows in two
accumulators of 256 columns and 32-column steps, beyond that 64-row blocks in
chunks of three or four) and of the float32 kernels' (32 or 64 rows x 128 keys),
against the float64 oracle."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from oracle import ebd_oracle as O
from tests.parity import E0_RTOL

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


def check(E, B, H, R, N, d, dtype, units=None):
    g = torch.Generator().manual_seed(7 * R + N + d)
    K = (torch.randn((B, H, N, d), generator=g) * 1.5).to(dtype)
    q = torch.randn((B, H, R, d), generator=g).to(dtype)
    s = torch.full((B, H, N), -1.0, dtype=torch.float32, device=DEV)
    E.ebd_score(q.to(DEV), K.to(DEV), s)
    got = s.cpu().double().numpy().reshape(B * H, N)
    Kn, qn = K.double().numpy().reshape(B * H, N, d), q.double().numpy().reshape(B * H, R, d)
    for u in (range(B * H) if units is None else units):
        ref = O.accumulated_attention_scores(qn[u], Kn[u])
        np.testing.assert_allclose(got[u], ref, rtol=E0_RTOL, atol=0)


@pytest.mark.parametrize("B,H,R,N,d", [
    (1, 1, 128, 256, 128),     # one full row tile and key tile, two items
    (1, 2, 129, 257, 128),     # one row and one key past them
    (2, 1, 256, 255, 64),      # a full accumulator; a key short of a tile
    (1, 2, 257, 128, 128),     # a row in the second accumulator; one item
    (1, 1, 512, 129, 64),      # two full accumulators; a key in a second item
    (1, 1, 160, 160, 128),     # five steps of columns; part of a second item
    (1, 2, 161, 161, 128),
    (2, 1, 320, 159, 64),      # a second accumulator of 64 columns
    (1, 2, 480, 481, 128),     # of 224; four items
    (1, 2, 513, 127, 128),     # the fewest streamed rows: three chunks of three blocks
    (1, 1, 640, 257, 64),      # three, three and four
    (1, 1, 1024, 641, 64),     # four chunks of four; five items and a key
    (1, 2, 1025, 256, 128),    # a row in a seventeenth block: 3, 3, 4, 3, 4
    (1, 1, 4096, 129, 128),    # the most rows
    (40, 8, 33, 130, 128),     # more units than CTAs: several units and items per CTA
    (24, 8, 520, 40, 64),      # the same with streamed rows
    (1, 1, 100, 1793, 128),    # eight key tiles, the last of one key: a cluster of two
    (1, 1, 100, 1792, 128),    # seven: no split
    (1, 1, 100, 2561, 128),
    (1, 2, 449, 10241, 64),    # a cluster of eight
    (2, 8, 100, 8192, 64),     # 16 row tiles: more than there are clusters of eight
])
def test_tensor_core_scores_at_tile_edges(E, B, H, R, N, d):
    units = None if B * H < 16 else (0, 1, B * H // 2, B * H - 1)
    check(E, B, H, R, N, d, torch.bfloat16, units)


@pytest.mark.parametrize("B,H,R,N,d", [
    (1, 1, 64, 128, 128),      # one full row tile, one full key tile
    (1, 2, 65, 129, 64),       # one row and one key past them
    (1, 1, 1, 1, 64),
    (2, 3, 130, 1023, 128),    # keys over a cluster, the last tile a key short
    (1, 1, 63, 4097, 128),     # the last tile one key
    (40, 8, 70, 130, 64),      # more row tiles than SMs
])
def test_float32_scores_at_tile_edges(E, B, H, R, N, d):
    units = None if B * H < 16 else (0, 1, B * H // 2, B * H - 1)
    check(E, B, H, R, N, d, torch.float32, units)


def test_float32_scores_off_a_16_byte_boundary(E):
    """Inputs that the register-tiled kernels do not take go the general way."""
    R, N, d = 70, 300, 64
    g = torch.Generator().manual_seed(5)
    K, q = torch.randn((1, 1, N, d), generator=g), torch.randn((1, 1, R, d), generator=g)
    buf = torch.empty(N * d + 1, device=DEV)
    Ko = buf[1:].view(1, 1, N, d).copy_(K)
    s = torch.empty((1, 1, N), device=DEV)
    E.ebd_score(q.to(DEV), Ko, s)
    ref = O.accumulated_attention_scores(q[0, 0].double().numpy(), K[0, 0].double().numpy())
    np.testing.assert_allclose(s[0, 0].cpu().double().numpy(), ref, rtol=E0_RTOL, atol=0)


def test_scores_right_after_the_query_gather(E):
    """The scoring launches as a programmatic dependent of the gather that
    writes its rows: alternating inputs back to back, each pass checked."""
    B, H, G, Nq, N, d, P = 4, 4, 7, 4096, 1500, 128, 64
    g = torch.Generator().manual_seed(3)
    K = torch.randn((B, H, N, d), generator=g).to(torch.bfloat16).to(DEV)
    Qs = [torch.randn((B, H * G, Nq, d), generator=g).to(torch.bfloat16).to(DEV) for _ in range(2)]
    pos = torch.arange(Nq - P, Nq, dtype=torch.int32, device=DEV)
    q_obs = torch.empty((B, H, G * P, d), dtype=torch.bfloat16, device=DEV)
    out = [torch.empty((B, H, N), device=DEV) for _ in range(6)]
    for i in range(6):
        E.ebd_gather_queries(Qs[i % 2], pos, H, q_obs)
        E.ebd_score(q_obs, K, out[i])
    for i in range(6):
        ref = O.accumulated_attention_scores(
            Qs[i % 2][3, 3 * G:4 * G, Nq - P:].reshape(G * P, d).cpu().double().numpy(),
            K[3, 3].cpu().double().numpy())
        np.testing.assert_allclose(out[i][3, 3].cpu().double().numpy(), ref, rtol=E0_RTOL, atol=0)


ORDER = """
import hashlib, sys, torch
from paper_2607_21475_gb300 import ebd as E
def score(B, H, R, N, d):
    g = torch.Generator().manual_seed(9)
    K, q = torch.randn((B, H, N, d), generator=g), torch.randn((B, H, R, d), generator=g)
    s = torch.empty((B, H, N), device="cuda")
    E.ebd_score(q.cuda(), K.cuda(), s)
    return s.cpu().numpy().tobytes()
if sys.argv[1] == "after":
    score(1, 1, 200, 3000, 64)
print(hashlib.sha256(score(2, 4, 1600, 2048, 128)).hexdigest())
"""


def test_float32_scores_do_not_depend_on_what_was_scored_before(E):
    """One d = 128 request (200 row tiles, more than fit at a time) in a fresh
    process, and in one that scored a d = 64 request first, of whose CTAs two
    share an SM: the same split, so the same bits."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    got = [subprocess.run([sys.executable, "-c", ORDER, how], cwd=root, capture_output=True,
                          text=True, check=True, timeout=300).stdout.split()[-1]
           for how in ("fresh", "after")]
    assert got[0] == got[1]


@pytest.mark.parametrize("R,N,d,dtype", [
    (513, 300, 128, torch.bfloat16),   # streamed rows, 63 of padding in the last block
    (1000, 129, 64, torch.bfloat16),
    (450, 300, 128, torch.bfloat16),   # resident rows, two accumulators
    (33, 700, 64, torch.bfloat16),
    (70, 300, 128, torch.float32),
])
def test_a_unit_with_nan_leaves_its_neighbours_alone(E, R, N, d, dtype):
    """The middle one of three units holds NaN in every query row and key: the
    other two get the scores they get without it."""
    g = torch.Generator().manual_seed(R)
    K = torch.randn((1, 3, N, d), generator=g).to(dtype).to(DEV)
    q = torch.randn((1, 3, R, d), generator=g).to(dtype).to(DEV)
    ref, got = torch.empty((1, 3, N), device=DEV), torch.empty((1, 3, N), device=DEV)
    E.ebd_score(q, K, ref)
    q[0, 1] = float("nan")
    K[0, 1] = float("nan")
    E.ebd_score(q, K, got)
    assert torch.isfinite(ref).all()
    assert torch.equal(got[:, ::2], ref[:, ::2])


@pytest.mark.parametrize("B,H,R,N,d,limit", [
    (2, 4, 448, 5000, 64, 1.80e-7),     # keys over clusters of four
    (1, 2, 800, 12001, 128, 3.02e-7),   # of eight, streamed query rows
    (8, 4, 448, 6144, 128, 1.97e-7),    # one CTA per row tile
])
def test_scores_against_64_bits(E, B, H, R, N, d, limit):
    """2-norm of the error over all scores; the limits are what one CTA per row tile
    left on inputs drawn the same way (query rows beyond 512 on mma.sync)."""
    errs = []
    for seed in range(3):
        g = torch.Generator(device=DEV).manual_seed(40 + seed)
        K = torch.randn((B, H, N, d), generator=g, device=DEV).to(torch.bfloat16)
        K[..., :4] *= 4
        q = torch.randn((B, H, R, d), generator=g, device=DEV).to(torch.bfloat16)
        s = E.ebd_score(q, K, torch.empty((B, H, N), device=DEV))
        for b in range(B):
            ref = torch.softmax(q[b].double() @ K[b].double().transpose(1, 2) / d ** 0.5, -1).sum(1)
            errs.append((s[b].double() - ref).norm() / ref.norm())
    e = float(torch.stack(errs).square().mean().sqrt())
    assert e <= limit


@pytest.mark.parametrize("few,many", [(16, 20), (38, 40)])
def test_fewer_row_tiles_take_no_longer(E, few, many):
    """Row tiles whose keys are split over clusters of a size that the device does
    not hold for all of them at once would wait for a second wave: 16 of them
    then take longer than 20, whose clusters are half the size."""
    def microseconds(units, N=8192, d=128, R=128):
        g = torch.Generator(device=DEV).manual_seed(1)
        K = torch.randn((units, 1, N, d), generator=g, device=DEV).to(torch.bfloat16)
        q = torch.randn((units, 1, R, d), generator=g, device=DEV).to(torch.bfloat16)
        s = torch.empty((units, 1, N), device=DEV)
        ws = torch.empty(E.ebd_score_workspace_bytes(units, 1, R), dtype=torch.uint8, device=DEV)
        best = float("inf")
        for _ in range(7):
            t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            for k in range(60):
                if k == 10:
                    t0.record()
                E.ebd_score(q, K, s, ws)
            t1.record()
            torch.cuda.synchronize()
            best = min(best, t0.elapsed_time(t1) * 20)
        return best

    assert microseconds(few) <= 1.03 * microseconds(many)

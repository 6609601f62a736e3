"""Host threads whose requests take one kernel with different amounts of shared
memory: every launch is accepted and takes the kernel that the request takes
alone."""
import threading

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


def select(E, N, seed):
    g = torch.Generator().manual_seed(seed)
    s = torch.exp(torch.randn((40, 4, N), generator=g)).to(DEV)
    des = E.design_for(batch=40, n_kv_heads=4, group=1, head_dim=64, n_ctx=N, seed=seed, k_head=50,
                       budget_tokens=N // 4)
    c = E.alloc_compact(40, 4, N // 2, 64, torch.bfloat16, DEV)
    c.idx_c.zero_()
    return lambda: E.ebd_select(des, s, c), lambda: [c.idx_c.clone(), c.n_kept.clone()]


def decode(E, G, seed):
    B, H, d, cap = 1, 4, 128, 2048
    g = torch.Generator().manual_seed(seed)
    K, V = (torch.randn((B, H, cap, d), generator=g).to(torch.bfloat16).to(DEV) for _ in range(2))
    lw = torch.rand((B, H, cap), generator=g).to(DEV)
    n = torch.full((B, H), cap - 5, dtype=torch.int32, device=DEV)
    Q = torch.randn((B, H * G, d), generator=g).to(torch.bfloat16).to(DEV)
    y = torch.empty((B, H * G, d), device=DEV)
    o = [torch.empty((B, H * G), device=DEV) for _ in range(4)]
    ws = torch.empty(E.ebd_decode_workspace_bytes(E.EBD_BF16, B, H, G, d, cap), dtype=torch.uint8,
                     device=DEV)
    return (lambda: E.ebd_certified_decode(Q, K, V, lw, n, y, *o, workspace=ws),
            lambda: [t.clone() for t in (y, *o)])


def test_requests_of_different_sizes_from_several_threads(E):
    work = [select(E, 8000, 1), select(E, 4000, 2), select(E, 12000, 3), decode(E, 8, 4),
            decode(E, 5, 5), decode(E, 6, 6)]
    ref = []
    for call, out in work:
        call()
        torch.cuda.synchronize()
        ref.append(out())
    torch.cuda.synchronize()
    errors, differ = [], []

    def loop(i):
        call, out = work[i]
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                bad = torch.zeros((), dtype=torch.int64, device=DEV)
                for k in range(1500):
                    call()
                    if k % 10 == 0:
                        for a, b in zip(out(), ref[i]):
                            bad += (a != b).sum()
                differ.append(int(bad))
        except Exception as e:  # reported by the main thread
            errors.append(f"{i}: {e}")

    threads = [threading.Thread(target=loop, args=(i,)) for i in range(len(work))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    assert differ == [0] * len(work)

"""The fused update of short lists by items (update_items_kernel): against the
kernels of long lists bit for bit (the route asserted), by padding the same list
past the short lists' limit with a last tensor, and against the oracle, over
every storage type, alignment, packing, probe count and a failed
preconditioner."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_38095_gb300 import build as zo_build
from paper_2609_38095_gb300 import workloads as W
from paper_2609_38095_gb300 import zo

from gpu_helpers import TORCH_TO_DT, assert_update_close, filler, storage_bits, to_torch, update_route

pytestmark = pytest.mark.gpu

DTYPES = [torch.bfloat16, torch.float32, torch.float16]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    zo_build.build()
    oracle.lib()


def views_of(host, dtypes, offsets):
    out = []
    for h, d, off in zip(host, dtypes, offsets):
        base = torch.zeros(h.size + off, dtype=d, device="cuda")
        base[off:].copy_(to_torch(h, d))
        out.append(base[off:])
    return out


@pytest.mark.parametrize("K,packing", [(1, 1), (8, 1), (16, 1), (17, 1), (64, 1), (384, 1), (1024, 1), (1, 8), (8, 8),
                                       (9, 8), (130, 8), (1024, 8)])
@pytest.mark.parametrize("pre,status", [(True, 0), (False, 0), (True, zo.ZO_ERR_NONFINITE),
                                        (False, zo.ZO_ERR_NONFINITE)])
def test_short_list(K, packing, pre, status):
    rng = np.random.default_rng(K * 8 + packing)
    numels = [1, 15, 16, 17, 31 * 16, 31 * 16 + 1, 500, 8, 7, 1000, 333, 4096]
    dtypes = [DTYPES[i % 3] for i in range(len(numels))]
    offsets = [0, 3, 0, 1, 5, 0, 7, 0, 1, 0, 11, 0]
    dts = [TORCH_TO_DT[d] for d in dtypes]
    host = [W.random_storage(rng, n, dt) for n, dt in zip(numels, dts)]
    short, copies = views_of(host, dtypes, offsets), [h.copy() for h in host]
    c_np = rng.normal(0, 25, K)
    c, st = torch.tensor(c_np, device="cuda"), torch.tensor([status], dtype=torch.int32, device="cuda")
    s, lr, p = W.step_seed(K), 1e-3, (K - 1, 1e-3) if pre else None
    zo.update(zo.ParamList(short, packing=packing), s, c, lr, status=st, pre=p)
    with oracle.packing(packing):
        if pre:
            oracle.perturb(host, dts, s, K - 1, 1e-3)
        if not status:
            oracle.update(host, dts, s, c_np, lr)
    for i, (v, h, dt) in enumerate(zip(short, host, dts)):
        if status:
            assert np.array_equal(storage_bits(v), storage_bits(h)), f"tensor {i}"
        else:
            assert_update_close(storage_bits(v), storage_bits(h), dt, c_np, lr, context=f"tensor {i}")
    # sixteen-bit weights for the kernels of packing 1 with a table per lane, fp32 views for the rest
    for long in ([filler(4097, torch.bfloat16)] if packing == 1 else []) + [filler(4097, torch.float32, 1)]:
        tail = views_of(copies, dtypes, offsets)
        plist = zo.ParamList(tail + [long], packing=packing)
        assert update_route(zo.ParamList(tail, packing=packing), K, K - 1 if pre else None) == "items"
        route = update_route(plist, K, K - 1 if pre else None)
        assert route != "items" and (packing == 1 or route == "chunks")
        zo.update(plist, s, c, lr, status=st, pre=p)
        for i, (x, y) in enumerate(zip(short, tail)):
            assert torch.equal(x.contiguous().view(torch.uint8), y.contiguous().view(torch.uint8)), f"{route}: tensor {i}"


@pytest.mark.parametrize("n", [64, 65, 256, 257, 960, 961, 2100])
def test_short_list_of_many_tensors(n):
    rng = np.random.default_rng(n)
    numels = [int(x) for x in rng.integers(0, 70, n)]
    host = [W.random_storage(rng, m, W.DT_BF16) for m in numels]
    dev = [to_torch(h.copy(), torch.bfloat16) for h in host]
    K, s, lr = 11, W.step_seed(n), 1e-3
    c_np = rng.normal(0, 25, K)
    zo.update(dev, s, torch.tensor(c_np, device="cuda"), lr, pre=(K - 1, 1e-3))
    oracle.perturb(host, [W.DT_BF16] * n, s, K - 1, 1e-3)
    oracle.update(host, [W.DT_BF16] * n, s, c_np, lr)
    for i, (d, h) in enumerate(zip(dev, host)):
        if h.size:
            assert_update_close(storage_bits(d), storage_bits(h), W.DT_BF16, c_np, lr, context=f"tensor {i}")


@pytest.mark.parametrize("n", [961, 1985])
@pytest.mark.parametrize("K,packing", [(19, 1), (9, 8)])
def test_more_tensors_than_a_launch_holds(n, K, packing):
    rng = np.random.default_rng(n + K)
    numels = [int(x) for x in rng.integers(0, 90, n)]
    numels[7], numels[n - 3] = 70_001, 5000
    dtypes = [DTYPES[i % 3] for i in range(n)]
    offsets = [int(x) for x in rng.integers(0, 4, n)]
    dts = [TORCH_TO_DT[d] for d in dtypes]
    host = [W.random_storage(rng, m, dt) for m, dt in zip(numels, dts)]
    dev = views_of(host, dtypes, offsets)
    s, lr, c_np = W.step_seed(n), 1e-3, rng.normal(0, 25, K)
    zo.update(zo.ParamList(dev, packing=packing), s, torch.tensor(c_np, device="cuda"), lr, pre=(K - 1, 1e-3))
    with oracle.packing(packing):
        oracle.perturb(host, dts, s, K - 1, 1e-3)
        oracle.update(host, dts, s, c_np, lr)
    for i, (d, h, dt) in enumerate(zip(dev, host, dts)):
        if h.size:
            assert_update_close(storage_bits(d), storage_bits(h), dt, c_np, lr, context=f"tensor {i}")


@pytest.mark.parametrize("items_per_sm", [880, 896])  # just below and above 7 CTAs of 128 items per SM
@pytest.mark.parametrize("K", [1, 16, 17])
@pytest.mark.parametrize("pre", [True, False])
def test_lists_of_two_waves(items_per_sm, K, pre):
    rng = np.random.default_rng(items_per_sm + K)
    dtypes, offsets = [torch.bfloat16, torch.float32, torch.float16], [0, 3, 1]
    host = [W.random_storage(rng, 1001, TORCH_TO_DT[d]) for d in dtypes]
    c = torch.tensor(rng.normal(0, 25, K), device="cuda")
    p = (K - 1, 1e-3) if pre else None
    got = []
    for per_sm, route in ((items_per_sm, "items"), (4097, "tables")):
        ws = views_of(host, dtypes, offsets) + [filler(per_sm, torch.bfloat16)]
        plist = zo.ParamList(ws, packing=1)
        assert update_route(plist, K, K - 1 if pre else None) == route
        zo.update(plist, W.step_seed(K), c, 1e-3, pre=p)
        got.append(ws)
    for i, (x, y) in enumerate(zip(*got)):
        assert torch.equal(x.contiguous().view(torch.uint8), y[:x.numel()].contiguous().view(torch.uint8)), f"tensor {i}"


@pytest.mark.parametrize("K", [64, 65, 520])  # eight groups and more
def test_last_words_by_length(K):
    rng = np.random.default_rng(K)
    host = [W.random_storage(rng, n, W.DT_F32) for n in (4099, 16, 131)]
    copies = [h.copy() for h in host]
    dtypes = [torch.float32] * len(host)
    c_np = rng.normal(0, 25, K)
    c, s, lr = torch.tensor(c_np, device="cuda"), W.step_seed(K), 1e-3
    got = []
    for per_sm in (0, 490, 500, 4097):  # fp32 items per SM of the last tensor: one wave of many groups, and more
        ws = views_of(copies, dtypes, [0] * len(host)) + ([filler(per_sm, torch.float32)] if per_sm else [])
        plist = zo.ParamList(ws, packing=8)
        assert update_route(plist, K, K - 1) == "items"
        zo.update(plist, s, c, lr, pre=(K - 1, 1e-3))
        got.append(ws)
    with oracle.packing(8):
        oracle.perturb(host, [W.DT_F32] * len(host), s, K - 1, 1e-3)
        oracle.update(host, [W.DT_F32] * len(host), s, c_np, lr)
    for i, h in enumerate(host):
        assert_update_close(storage_bits(got[0][i]), storage_bits(h), W.DT_F32, c_np, lr, context=f"tensor {i}")
    for a, b in zip(got, got[1:]):
        for i, (x, y) in enumerate(zip(a, b)):
            assert torch.equal(x.view(torch.uint8), y[:x.numel()].view(torch.uint8)), f"tensor {i}"

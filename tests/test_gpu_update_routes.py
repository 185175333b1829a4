"""The fused update's chunk kernel at the edges of its routes: views whose
32-byte chunks fill, just miss or just pass the 31 chunks of a warp; probe
counts past 384; packing 8 (views, many groups) on every chunk size and with
a last group of one to eight probes; fp32 and 16-bit tensors, aligned or not, in
one launch. A long last tensor keeps the lists from the kernels of short ones;
each test asserts the route. Views are compared bit for bit with the same values
in aligned tensors (on whatever route those take), everything but the long
tensor with the oracle within the derived bound."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_38095_gb300 import build as zo_build
from paper_2609_38095_gb300 import workloads as W
from paper_2609_38095_gb300 import zo

from gpu_helpers import TORCH_TO_DT, assert_update_close, filler, storage_bits, to_torch, update_route

pytestmark = pytest.mark.gpu

DTS = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    zo_build.build()
    oracle.lib()


def check(numels, dtypes, offsets, K, packing, pre, seed, long=None, route="chunks"):
    """One update of views `offsets` elements into their allocations (0:
    aligned) and of `long`, against aligned copies and the oracle."""
    rng = np.random.default_rng(seed)
    dts = [TORCH_TO_DT[d] for d in dtypes]
    host = [W.random_storage(rng, n, dt) for n, dt in zip(numels, dts)]
    bases = [torch.full((n + off + 40,), 3.0, dtype=d, device="cuda") for n, d, off in zip(numels, dtypes, offsets)]
    views = [b[off:off + n] for b, n, off in zip(bases, numels, offsets)]
    for v, h, d in zip(views, host, dtypes):
        v.copy_(to_torch(h, d))
    aligned = [to_torch(h.copy(), d) for h, d in zip(host, dtypes)]
    ends = ([], []) if long is None else ([long], [long.clone()])
    c_np = rng.normal(0, 25, K)
    c = torch.tensor(c_np, device="cuda")
    s, lr, p = W.step_seed(seed), 1e-3, (K - 1, 1e-3) if pre else None
    plist = zo.ParamList(views + ends[0], packing=packing)
    assert update_route(plist, K, K - 1 if pre else None) == route
    zo.update(plist, s, c, lr, pre=p)
    zo.update(zo.ParamList(aligned + ends[1], packing=packing), s, c, lr, pre=p)
    with oracle.packing(packing):
        if pre:
            oracle.perturb(host, dts, s, K - 1, 1e-3)
        oracle.update(host, dts, s, c_np, lr)
    for i, (v, x, h, dt, b, off) in enumerate(zip(views, aligned, host, dts, bases, offsets)):
        assert torch.equal(v.contiguous().view(torch.uint8), x.view(torch.uint8)), f"tensor {i}"
        assert_update_close(storage_bits(x), storage_bits(h), dt, c_np, lr, context=f"tensor {i}")
        assert torch.all(b[:off] == 3.0) and torch.all(b[off + v.numel():] == 3.0), f"guards of tensor {i}"
    if long is not None:
        assert torch.equal(long.contiguous().view(torch.uint8), ends[1][0].view(torch.uint8)), "the long tensor"


# Long tensors that send a list to the chunk kernel: 16-bit past the short lists of packing 1, or, under packing 8,
# fp32 views past the items of few groups and 16-bit views past those of nine groups and more.
def long_tensor(packing, K, sixteen=torch.bfloat16):
    if packing == 1:
        return filler(1601, sixteen)
    return filler(3001, torch.float32, 3) if K <= 64 else filler(8001, sixteen, 1)


@pytest.mark.parametrize("dtype", list(DTS))
@pytest.mark.parametrize("K,packing,pre", [(33, 1, True), (50, 1, False), (392, 1, True), (3, 8, True), (17, 8, False),
                                           (66, 8, True)])
def test_views_at_the_warp_s_edges(dtype, K, packing, pre):
    per = 8 if dtype == "f32" else 16      # elements between 32-byte boundaries
    numels, offsets = [], []
    for a in (1, per // 2, per - 1):
        for chunks in (1, 2, 31, 32, 62, 63):
            for extra in (-1, 0, 1):       # the last element closes the chunk, or one more or less
                n = 16 * chunks - a + extra
                if n > 0:
                    numels.append(n)
                    offsets.append(a)
    check(numels, [DTS[dtype]] * len(numels), offsets, K, packing, pre, K + per, long_tensor(packing, K))


@pytest.mark.parametrize("rows", [3, 4, 8, 10])
@pytest.mark.parametrize("K,pre", [(13, True), (18, False)])
def test_packing_8_on_every_chunk_size(rows, K, pre):
    """A row is a block per thread of the launch; the last round of eight takes what is left of them."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = (sms * 512 * rows * 31 // 32 - 700) * 16 - 5
    check([n, 6001, 40], [torch.float32, torch.bfloat16, torch.float16], [3, 0, 0], K, 8, pre, rows * 100 + K)


@pytest.mark.parametrize("K,packing", [(385, 1), (400, 1), (1, 8), (2, 8), (8, 8), (9, 8), (70, 8), (520, 8)])
def test_mixed_list(K, packing):
    check([4096 + 7, 1000, 333, 16, 1, 5000, 2048], [torch.bfloat16, torch.float32, torch.float16, torch.bfloat16,
                                                     torch.float32, torch.float16, torch.float32],
          [0, 0, 5, 0, 1, 0, 9], K, packing, True, K, long_tensor(packing, K, torch.float16))

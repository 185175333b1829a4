"""The fused update under packing 8 on a list long enough that a thread of the
item kernel takes several items, with a full and a partial probe group: the
long tensor ends inside an item, the short ones hold fp32 and views. Lists of
mostly fp32 take whole blocks of 64 bytes: sizes around a warp's 64 items, a
partial last block, views in between, and a failed preconditioner's leading
perturbation alone. The leading perturbation's probe in every place that its
signs are taken from: either half of the last group, full or partial, another
group, or past the last probe. Against the oracle within the derived bound."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_38095_gb300 import build as zo_build
from paper_2609_38095_gb300 import workloads as W
from paper_2609_38095_gb300 import zo

from gpu_helpers import TORCH_TO_DT, assert_update_close, storage_bits, to_torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    zo_build.build()
    oracle.lib()


@pytest.mark.parametrize("rounds,pre", [(2, True), (3, False)])
def test_several_items_per_thread(rounds, pre):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    K, seed, lr = 9, W.step_seed(rounds), 1e-3
    numels = [16 * 8 * 128 * 8 * sms * rounds + 7, 1, 1000, 4099]
    dtypes = [torch.bfloat16, torch.float16, torch.float32, torch.bfloat16]
    rng = np.random.default_rng(rounds)
    dts = [TORCH_TO_DT[d] for d in dtypes]
    host = [W.random_storage(rng, n, dt) for n, dt in zip(numels, dts)]
    dev = [to_torch(h.copy(), d) for h, d in zip(host, dtypes)]
    view = torch.zeros(numels[-1] + 16, dtype=dtypes[-1], device="cuda")[3:3 + numels[-1]]
    view.copy_(dev[-1])
    dev[-1] = view
    c_np = rng.normal(0, 25, K)
    zo.update(zo.ParamList(dev, packing=8), seed, torch.tensor(c_np, device="cuda"), lr, pre=(K - 1, 1e-3) if pre else None)
    with oracle.packing(8):
        if pre:
            oracle.perturb(host, dts, seed, K - 1, 1e-3)
        oracle.update(host, dts, seed, c_np, lr)
    for i, (x, h, dt) in enumerate(zip(dev, host, dts)):
        assert_update_close(storage_bits(x), storage_bits(h), dt, c_np, lr, context=f"tensor {i}")


@pytest.mark.parametrize("K,pre,status", [(9, True, 0), (17, False, 0), (8, True, zo.ZO_ERR_NONFINITE)])
@pytest.mark.parametrize("big", [20_011, 3_000_017, 32_000_003])
def test_blocks_of_fp32(K, pre, status, big):
    numels = [big, 512, 511, 513, 256, 8, 1024, 2051, 40, 1040]
    offsets = [0, 0, 0, 0, 0, 0, 0, 3, 0, 0]
    dtypes = [torch.float32] * 8 + [torch.bfloat16, torch.float16]
    rng = np.random.default_rng(K)
    seed, lr = W.step_seed(K), 1e-3
    dts = [TORCH_TO_DT[d] for d in dtypes]
    host = [W.random_storage(rng, n, dt) for n, dt in zip(numels, dts)]
    bases = [torch.full((n + 32,), 3.0, dtype=d, device="cuda") for n, d in zip(numels, dtypes)]
    dev = [b[o:o + n] for b, o, n in zip(bases, offsets, numels)]
    for x, h, d in zip(dev, host, dtypes):
        x.copy_(to_torch(h, d))
    c_np = rng.normal(0, 25, K)
    zo.update(zo.ParamList(dev, packing=8), seed, torch.tensor(c_np, device="cuda"), lr,
              status=torch.tensor([status], dtype=torch.int32, device="cuda"), pre=(K - 1, 1e-3) if pre else None)
    with oracle.packing(8):
        if pre:
            oracle.perturb(host, dts, seed, K - 1, 1e-3)
        if status == 0:
            oracle.update(host, dts, seed, c_np, lr)
    for i, (x, h, dt) in enumerate(zip(dev, host, dts)):
        if status == 0:
            assert_update_close(storage_bits(x), storage_bits(h), dt, c_np, lr, context=f"tensor {i}")
        else:
            assert np.array_equal(storage_bits(x), storage_bits(h)), f"tensor {i}"
        assert torch.all(bases[i][:offsets[i]] == 3.0) and torch.all(bases[i][offsets[i] + numels[i]:] == 3.0)


@pytest.mark.parametrize("K,pre_probe", [(8, 0), (8, 3), (8, 4), (8, 7), (3, 1), (6, 5), (3, 3), (6, 7), (16, 2), (13, 9),
                                         (20, 19), (9, 100)])
@pytest.mark.parametrize("status", [0, zo.ZO_ERR_NONFINITE])
@pytest.mark.parametrize("mostly", [torch.bfloat16, torch.float32], ids=["bf16", "f32"])
def test_signs_of_the_leading_perturbation(K, pre_probe, status, mostly):
    numels, offsets = [40_011, 1, 515, 1000, 333, 64], [0, 0, 3, 0, 5, 0]
    dtypes = [mostly, torch.float16, torch.float32, torch.float32, torch.bfloat16, torch.bfloat16]
    rng = np.random.default_rng(K * 128 + pre_probe)
    seed, lr = W.step_seed(K), 1e-3
    dts = [TORCH_TO_DT[d] for d in dtypes]
    host = [W.random_storage(rng, n, dt) for n, dt in zip(numels, dts)]
    dev = [torch.zeros(n + o, dtype=d, device="cuda")[o:] for n, o, d in zip(numels, offsets, dtypes)]
    for x, h, d in zip(dev, host, dtypes):
        x.copy_(to_torch(h, d))
    c_np = rng.normal(0, 25, K)
    zo.update(zo.ParamList(dev, packing=8), seed, torch.tensor(c_np, device="cuda"), lr,
              status=torch.tensor([status], dtype=torch.int32, device="cuda"), pre=(pre_probe, 1e-3))
    with oracle.packing(8):
        oracle.perturb(host, dts, seed, pre_probe, 1e-3)
        if status == 0:
            oracle.update(host, dts, seed, c_np, lr)
    for i, (x, h, dt) in enumerate(zip(dev, host, dts)):
        if status == 0:
            assert_update_close(storage_bits(x), storage_bits(h), dt, c_np, lr, context=f"tensor {i}")
        else:
            assert np.array_equal(storage_bits(x), storage_bits(h)), f"tensor {i}"

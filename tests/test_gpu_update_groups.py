"""The fused update with three and four probe groups (two of fp32), lists long enough for the
kernel that keeps every group's table in shared memory: each place its leading
perturbation's signs come from (none, the last group, another group), each
storage type, aligned and in views, tensors that end inside an item or hold
less than one; and lists of mostly fp32 views without a leading perturbation,
which a kernel of their own takes by blocks. Views are compared bit for bit with the same values in aligned
tensors, everything with the oracle within the derived bound."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_38095_gb300 import build as zo_build
from paper_2609_38095_gb300 import workloads as W
from paper_2609_38095_gb300 import zo

from gpu_helpers import TORCH_TO_DT, assert_update_close, storage_bits, to_torch, update_route

pytestmark = pytest.mark.gpu

BF16, F16, F32 = torch.bfloat16, torch.float16, torch.float32


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    zo_build.build()
    oracle.lib()


def check(numels, dtypes, offsets, K, pre_probe, seed, route="tables"):
    """One update of views `offsets` elements into their allocations (0:
    aligned), on the given route, against aligned copies and the oracle."""
    rng = np.random.default_rng(seed)
    dts = [TORCH_TO_DT[d] for d in dtypes]
    host = [W.random_storage(rng, n, dt) for n, dt in zip(numels, dts)]
    bases = [torch.full((n + off + 40,), 3.0, dtype=d, device="cuda") for n, d, off in zip(numels, dtypes, offsets)]
    views = [b[off:off + n] for b, n, off in zip(bases, numels, offsets)]
    for v, h, d in zip(views, host, dtypes):
        v.copy_(to_torch(h, d))
    aligned = [to_torch(h.copy(), d) for h, d in zip(host, dtypes)]
    c_np = rng.normal(0, 25, K)
    c = torch.tensor(c_np, device="cuda")
    s, lr, p = W.step_seed(seed), 1e-3, None if pre_probe is None else (pre_probe, 1e-3)
    plist = zo.ParamList(views, packing=1)
    assert update_route(plist, K, pre_probe) == route
    zo.update(plist, s, c, lr, pre=p)
    zo.update(zo.ParamList(aligned, packing=1), s, c, lr, pre=p)
    with oracle.packing(1):
        if pre_probe is not None:
            oracle.perturb(host, dts, s, pre_probe, 1e-3)
        oracle.update(host, dts, s, c_np, lr)
    for i, (v, x, h, dt, b, off) in enumerate(zip(views, aligned, host, dts, bases, offsets)):
        assert torch.equal(v.contiguous().view(torch.uint8), x.view(torch.uint8)), f"tensor {i}"
        assert_update_close(storage_bits(x), storage_bits(h), dt, c_np, lr, context=f"tensor {i}")
        assert torch.all(b[:off] == 3.0) and torch.all(b[off + v.numel():] == 3.0), f"guards of tensor {i}"

def long_list(dtype):
    """More 32-byte items per SM than the short lists' kernel takes, in the
    list's largest tensor."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per = 8 if dtype == F32 else 16
    return sms * 2400 * per + 3 * per + 1


@pytest.mark.parametrize("K,pre_probe", [(17, 16), (24, None), (25, 24), (32, 31), (32, None), (31, 3), (24, 2), (20, 13),
                                         (30, 9), (27, 17), (27, 40)])
@pytest.mark.parametrize("dtype", [BF16, F32], ids=["bf16", "f32"])
def test_three_and_four_groups(K, pre_probe, dtype):
    # fp32 of four groups keeps to the last group's words; a probe of no group has none here
    last = pre_probe is None or pre_probe // 8 == (K - 1) // 8
    chunks = pre_probe is not None and pre_probe >= 8 * ((K + 7) // 8) or (dtype == F32 and K > 24 and not last)
    check([long_list(dtype), 1, 15, 513, 77], [dtype, F16, F32, BF16, F16], [0, 0, 3, 5, 0], K, pre_probe, seed=K,
          route="chunks" if chunks else "tables")


@pytest.mark.parametrize("K,pre_probe", [(9, None), (16, 15), (12, 3), (12, 20)])
def test_two_groups_of_fp32_blocks(K, pre_probe):
    check([long_list(F32), 8, 7, 1023, 65], [F32, F32, F32, F32, BF16], [0, 0, 0, 3, 1], K, pre_probe, seed=K)


@pytest.mark.parametrize("K,pre_probe", [(20, 19), (32, 31), (16, 5), (24, 9), (32, 12)])
def test_whole_list_in_views(K, pre_probe):
    check([long_list(BF16), 31 * 16, 16], [BF16, F16, F32], [1, 9, 2], K, pre_probe, seed=K + 1)


@pytest.mark.parametrize("K,per_sm", [(17, 0), (24, 0), (32, 0), (39, 0), (41, 0), (56, 0), (80, 0), (5, 200_050)])
def test_fp32_views_by_blocks(K, per_sm):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = per_sm * sms + 3 if per_sm else long_list(F32)
    numels = [n, 16 * 31 - 3, 16 * 31 - 2, 16 * 62 - 2, 9, 1, 513, 77, 4096, 130]
    check(numels, [F32] * 6 + [F16, BF16, F32, BF16], [3, 3, 2, 2, 7, 1, 5, 0, 0, 0], K, None, seed=K,
          route="blocks")


def test_fp32_views_after_a_failed_preconditioner():
    theta = torch.randn(long_list(F32) + 1, device="cuda")
    before = theta.clone()
    zo.update([theta[1:]], 3, torch.ones(32, dtype=torch.float64, device="cuda"), 1e-3,
              status=torch.tensor([zo.ZO_ERR_NONFINITE], dtype=torch.int32, device="cuda"))
    assert torch.equal(theta, before)

"""zo_quadratic_points: every forward point of a step of the small workload in
one launch, against the oracle's perturbations (bit for bit) and its fp64
losses. Each loss is a sum of n exact or 2^-47-accurate terms, added as fp32
pairs in a warp (relative error at most 2^-45 per addition of at most 8 + 5),
then as three fp32 values and in fp64, so 1e-12 of the sum of |terms| holds with
room at these sizes. Against exact sums its losses are no further off than those of a launch
per point (zo_perturb_quadratic_loss)."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2609_38095_gb300 import build as zo_build
from paper_2609_38095_gb300 import workloads as W
from paper_2609_38095_gb300 import zo
from paper_2609_38095_gb300.quadratic import QuadraticStep

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    zo_build.build()
    oracle.lib()


def oracle_points(theta, a, seed, K, eps):
    host, rows = [theta.copy()], []
    l0 = oracle.quadratic_loss(host[0], a)
    for k in range(K):
        row = []
        for scale in (eps, -2 * eps):
            oracle.perturb(host, [W.DT_F32], seed, k, scale)
            row.append(oracle.quadratic_loss(host[0], a))
        oracle.perturb(host, [W.DT_F32], seed, k, eps)
        rows.append(row + [l0])
    return host[0], np.array(rows)


def on_device(x, offset):
    v = torch.zeros(x.size + offset, dtype=torch.float32, device="cuda")[offset:]
    v.copy_(torch.from_numpy(x))
    return v


def run_points(th, a, seed, K, eps, offset=0, packing=None):
    theta, ad = on_device(th, offset), on_device(a, offset)
    table = torch.full((K, 3), -7.0, dtype=torch.float64, device="cuda")
    q = zo.QuadraticPoints(theta, ad, table, packing=packing)
    q(seed, eps)
    first = (theta.cpu().numpy(), table.cpu().numpy())
    theta.copy_(torch.from_numpy(th))   # the workspace is left ready: the same again, bit for bit
    q(seed, eps)
    assert np.array_equal(theta.cpu().numpy().view(np.uint32), first[0].view(np.uint32))
    assert np.array_equal(table.cpu().numpy(), first[1], equal_nan=True)
    return first


def check(th, a, K, eps=1e-3, offset=0, packing=1):
    seed = W.step_seed(th.size + K)
    got_th, got = run_points(th, a, seed, K, eps, offset, packing)
    with oracle.packing(packing):
        want_th, want = oracle_points(th, a, seed, K, eps)
    assert np.array_equal(got_th.view(np.uint32), want_th.view(np.uint32))
    np.testing.assert_allclose(got, want, rtol=1e-12)


@pytest.mark.parametrize("n,K", [(1, 1), (7, 3), (8, 4), (9, 5), (255, 8), (256, 9), (4097, 7), (100_003, 16),
                                 (1 << 20, 8), (1_100_011, 2), (3_000_001, 3), (5000, 40), (3000, 130)])
def test_points_parity(n, K):
    rng = np.random.default_rng(n * 31 + K)
    check(W.random_storage(rng, n, W.DT_F32), (10.0 ** rng.uniform(-2, 2, n)).astype(np.float32), K)


@pytest.mark.parametrize("offset,packing", [(1, 1), (2, 8), (4, 8), (3, 1)])
def test_points_views_and_packings(offset, packing):
    rng = np.random.default_rng(offset)
    n = 20_003
    check(W.random_storage(rng, n, W.DT_F32), (10.0 ** rng.uniform(-2, 2, n)).astype(np.float32), 11, offset=offset,
          packing=packing)


def test_points_most_probes():
    rng = np.random.default_rng(9)
    check(W.random_storage(rng, 500, W.DT_F32), (10.0 ** rng.uniform(-2, 2, 500)).astype(np.float32),
          zo.ZO_MAX_PROBES)


def test_points_empty():
    _, table = run_points(np.zeros(0, np.float32), np.zeros(0, np.float32), 1, 2, 1e-3)
    assert np.all(table == 0.0)


def test_points_weights_outside_the_exact_range():
    """Zeros, tiny and huge weights and curvatures go to the fp64 terms; only
    the values of their own size decide the sums they dominate."""
    rng = np.random.default_rng(4)
    n = 6000
    a = (10.0 ** rng.uniform(-2, 2, n)).astype(np.float32)
    for scale in (1e-25, 1e-12, 1e15, 1e18):
        check((rng.standard_normal(n) * scale).astype(np.float32), a, 3, eps=scale / 16)
    th = W.random_storage(rng, n, W.DT_F32)
    th[::3] = 0.0
    b = a.copy()
    b[::5] = 0.0
    b[1::7] *= np.float32(1e-20)
    check(th, b, 5)
    th[17], th[4000] = np.float32(3e38), np.float32(-2e30)
    check(th, a, 2)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_points_not_finite(value):
    rng = np.random.default_rng(5)
    th = W.random_storage(rng, 4099, W.DT_F32)
    th[1234] = value
    a = (10.0 ** rng.uniform(-2, 2, 4099)).astype(np.float32)
    got_th, got = run_points(th, a, W.step_seed(1), 3, 1e-3)
    want_th, want = oracle_points(th, a, W.step_seed(1), 3, 1e-3)
    assert np.array_equal(got_th.view(np.uint32), want_th.view(np.uint32))
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))


@pytest.mark.parametrize("n,K", [(5000, 1), (70_001, 8), (3000, 130), (500, zo.ZO_MAX_PROBES)])
def test_points_with_the_preconditioner(n, K):
    """c and status from the same launch: bit for bit what zo_precondition
    gives for the losses written; a loss that is not finite leaves c alone."""
    rng = np.random.default_rng(n + K)
    theta = on_device(W.random_storage(rng, n, W.DT_F32), 0)
    a = on_device((10.0 ** rng.uniform(-2, 2, n)).astype(np.float32), 0)
    table = torch.empty(K, 3, dtype=torch.float64, device="cuda")
    c = torch.full((K,), -7.0, dtype=torch.float64, device="cuda")
    status = torch.full((1,), 5, dtype=torch.int32, device="cuda")
    q = zo.QuadraticPoints(theta, a, table, out=(c, status))
    q(W.step_seed(2), 1e-3)
    want, st = zo.precondition(table, 1e-3)
    assert int(status.item()) == int(st.item()) == zo.ZO_OK
    assert torch.equal(c, want)
    theta[n // 2] = float("inf")
    q(W.step_seed(3), 1e-3)
    assert int(status.item()) == zo.ZO_ERR_NONFINITE
    assert torch.equal(c, want)


def test_points_at_a_distance_of_eps_from_zero():
    """Weights within a few roundings of +-eps pass through (almost) zero at a
    point: they take the checked form of the terms."""
    eps = 1e-3
    th = np.full(4099, np.float32(eps), dtype=np.float32)
    th[1::3] = -np.float32(eps)
    th[2::7] = np.nextafter(np.float32(eps), np.float32(1))
    th[5::11] = np.float32(2 * eps)
    a = (10.0 ** np.random.default_rng(8).uniform(-2, 2, th.size)).astype(np.float32)
    check(th, a, 6, eps=eps)


def exact_loss(th, a):
    """1/2 sum a theta^2 of fp32 arrays, rounded once: a t is exact in fp64, (a t) t is split into two fp64 values."""
    t = th.astype(np.float64)
    p = a.astype(np.float64) * t
    q = p * t
    high = p * 134217729.0                     # Veltkamp's split: 26 bits and the rest
    high = high - (high - p)
    return 0.5 * math.fsum(np.concatenate([q, (high * t - q) + (p - high) * t]).tolist())


def test_points_as_close_to_exact_sums_as_a_launch_per_point():
    """Root mean square over 60 losses, of the same theta and a at every point. Both round a sum of some hundred fp64
    partials, each good to 2^-53 or so; a quarter is left for the two orders' chance. Sums held as fp32 pairs up to the
    CTA are 1.6 times as far off."""
    K, eps, err = 2, 1e-3, {"points": [], "launches": []}
    for n, seeds in ((1 << 20, 8), (2_500_007, 4)):
        for sd in range(seeds):
            rng = np.random.default_rng(sd)
            th = (rng.standard_normal(n) * 0.02).astype(np.float32)
            a = (10.0 ** rng.uniform(-2, 2, n)).astype(np.float32)
            seed, x, v, ad = W.step_seed(sd), on_device(th, 0), on_device(th, 0), on_device(a, 0)
            table = torch.empty(K, 3, dtype=torch.float64, device="cuda")
            zo.QuadraticPoints(x, ad, table)(seed, eps)
            table = table.cpu().numpy()
            one, out = zo.QuadraticPass(v, ad), torch.empty(1, dtype=torch.float64, device="cuda")
            for ops, mine in (((), table[0, 2]), ([(0, eps)], table[0, 0]), ([(0, -2 * eps)], table[0, 1]),
                              ([(0, eps), (1, eps)], table[1, 0]), ([(1, -2 * eps)], table[1, 1])):
                one(seed, ops, one.out_address(out))
                theirs = float(out.item())
                want = exact_loss(v.cpu().numpy(), a)
                err["points"].append((mine - want) / want)
                err["launches"].append((theirs - want) / want)
    rms = {k: float(np.sqrt(np.mean(np.square(e)))) for k, e in err.items()}
    assert rms["points"] <= 1.25 * rms["launches"], rms


def test_step_holds_what_its_schedule_uses():
    theta, a = torch.ones(100, device="cuda"), torch.ones(100, device="cuda")
    one, fused = (QuadraticStep(theta, a, 2, 1e-3, 1e-3, schedule=s) for s in ("onepass", "fused"))
    assert isinstance(one.onepass, zo.QuadraticPoints) and one.loss is None and one.ws is None
    assert fused.onepass is None and isinstance(fused.loss, zo.QuadraticLoss)

"""Threshold of a large calibration in one launch (tau_kernel in scap_calibrate.cu, from 10 * 2^20 elements), bit for bit against the
oracle: keys that do not fit in a thread's list, order statistics in different buckets of every digit, more blocks of channels than
resident CTAs, and the first and last ranks; and the same on the other side of the line."""
import numpy as np
import pytest
import torch

import oracle
import scap_inputs as si
from scap_testlib import dev, workspace

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    import paper_2412_07174_b200 as scap
    scap.lib()
    return scap


def check(S, values, dt, s, nbins=64):
    bits = si.to_bits(values, dt)
    xf, x = si.to_f32(bits, dt), dev(bits, dt)
    T, K = xf.shape
    ws, mg, tg = workspace(S.scap_calibrate_workspace(T, K, nbins)), workspace(K * 4), workspace(4)
    m, tau = mg.view(torch.float32, (K,)), tg.view(torch.float32, (1,))
    want_m, want = oracle.calibrate(xf, s, nbins)
    for _ in range(2):  # (the counters of the first call are cleared by the second)
        S.scap_calibrate(x, s, nbins, m, tau, ws.payload)
        torch.cuda.synchronize()
        assert ws.intact() and mg.intact() and tg.intact()
        assert np.array_equal(m.cpu().numpy(), want_m)
        assert np.float32(tau.item()).view(np.uint32) == np.float32(want).view(np.uint32)


def normal(T, K, seed=1):
    return np.random.default_rng(seed).standard_normal((T, K))


@pytest.mark.parametrize("dt", [si.F16, si.BF16])
@pytest.mark.parametrize("T,K,s", [
    (1, 8, 0.5), (3, 264, 0.0625), (1000, 1024, 0.9999995), (2049, 72, 0.35),
    (2047, 5120, 0.6), (2048, 5120, 0.6),         # either side of the line
    (2049, 5128, 1e-8), (2100, 5128, 0.99999999),  # rows beyond what a strip keeps in registers, a ragged last block of channels
    (65, 163848, 0.7),                            # 641 blocks of channels: more than the CTAs that are resident at once
])
def test_ranks_and_shapes(S, dt, T, K, s):
    check(S, normal(T, K), dt, s)


@pytest.mark.parametrize("T,K", [(2048, 1536), (2048, 5128)])
@pytest.mark.parametrize("s", [0.2, 0.5, 0.8])
def test_few_distinct_values(S, s, T, K):
    """Nearly all keys share a bucket: the lists overflow and the tensor is read again."""
    v = np.round(normal(T, K)) * 0.25
    v[:, 5] = 3.0  # a constant channel
    check(S, v, si.BF16, s)
    check(S, np.where(normal(T, K, 2) > 0.3, 1.0, 1.0 + 2.0 ** -7), si.BF16, s)


@pytest.mark.parametrize("T,K", [(64, 64), (2048, 5128)])
@pytest.mark.parametrize("gap", [2.0 ** -7, 2.0 ** -3, 1.0, 2.0 ** 20])
def test_order_statistics_in_different_buckets(S, gap, T, K):
    """j and j + 1 fall on either side of a jump that separates their last, middle or first digits (no centring: the values are the keys)."""
    v = np.where(np.arange(T * K).reshape(T, K) < T * K // 2, 1.0, 1.0 + gap)
    check(S, v, si.BF16, (T * K // 2 - 0.75) / (T * K - 1), nbins=0)


def test_a_barrier_that_runs_out_is_reported_and_the_next_call_is_right(S):
    """With a limit of one poll most CTAs do not see the others arrive: the call returns, the status word is set, the threshold is no number."""
    x = dev(si.to_bits(normal(2048, 5128), si.BF16), si.BF16)
    ws, m, tau = workspace(S.scap_calibrate_workspace(2048, 5128, 64)), torch.empty(5128, device="cuda"), torch.zeros(1, device="cuda")
    S.scap_device_status()
    try:
        S.scap_tune("tc_spin", 1)
        S.scap_calibrate(x, 0.5, 64, m, tau, ws.payload)
        with pytest.raises(S.ScapError) as err:
            S.scap_device_status()
        assert err.value.code == 7  # SCAP_ERR_TIMEOUT
        assert ws.intact() and torch.isnan(tau).all()
    finally:
        S.scap_tune("tc_spin", 0)
    check(S, normal(2048, 5128), si.BF16, 0.5)
    S.scap_device_status()

"""Grouped calls whose groups all have more than four rows run as one pass of the dense-stream kernel per 32 rows where that is
the faster route: the edges of its row counts, 64-channel blocks, 128-column tiles and cluster slices, both activation load
paths (K a multiple of eight or not), and the rows and results of the second pass.

Bound of the stream: an accumulator takes K / (32 S) products of 16 channels (S ranks, two accumulators), each of which truncates
it by at most 2^-23 of its value, and a handful of binary32 additions follow; the three parts of d hold all of it.  The gather kernel rounds once per 16 channels of a warp's list and is held to the looser bound of random
roundings, 2^-23 8 sqrt(K)."""
import numpy as np
import pytest
import torch

import oracle
import scap_inputs as si
from scap_testlib import CANARY, dev, f32, rel_l2_rows, workspace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N,B,n_ctx,stream", [
    (64, 8, 5, 1, True), (100, 136, 10, 2, True), (1023, 264, 12, 2, True),     # up to sixteen rows: the kernel of plain calls
    (1024, 1032, 17, 2, True), (1500, 392, 24, 3, True), (2049, 128, 31, 3, True), (2560, 520, 32, 4, True),
    (512, 3592, 33, 3, True), (1027, 3592, 40, 4, True), (520, 3600, 64, 8, True),  # two passes: 17 + 16, 20 + 20, 32 + 32 rows
    (63, 136, 12, 2, False), (1030, 264, 33, 3, False), (4096, 1024, 64, 8, False), (4104, 264, 24, 2, False),  # few CTAs: gather
])
@pytest.mark.parametrize("dt", [si.F16, si.BF16])
def test_large_groups_match_the_oracle(K, N, B, n_ctx, stream, dt):
    import paper_2412_07174_b200 as S
    d = si.context_batch(4, K, N, dt, 64, B, n_ctx, 0.9)
    xf, m = si.to_f32(d["x"], dt), d["m_true"]
    tau = oracle.tau(si.to_f32(d["x_calib"], dt), m, 0.6)
    bias = np.linspace(-1, 1, N).astype(np.float32)
    ws, yg = workspace(S.scap_grouped_workspace()), workspace(B * N * 4)
    y = yg.view(torch.float32, (B, N))
    ranks = min(8, -(-K // 64))
    bound = 2.0 ** -23 * (2 + K / (32 * ranks)) if stream else 2.0 ** -23 * 8 * np.sqrt(K)
    for mm in (m, None):
        y64 = oracle.sparse_fc(xf, d["W"], dt, mm, tau, None, threads=8) + bias[None, :]
        y.fill_(float("nan"))
        S.scap_sparse_fc_grouped(dev(d["x"], dt), dev(d["W"], dt), None if mm is None else f32(mm), f32([tau]), f32(bias), y, d["ctx"].tolist(), ws.payload)
        torch.cuda.synchronize()
        S.scap_device_status()
        assert ws.intact() and yg.intact()
        assert bool((ws.payload == CANARY).all().item()) == stream  # only the gather writes its row table there
        assert rel_l2_rows(y.cpu().numpy(), y64) <= bound


@pytest.mark.parametrize("dt", [si.F16, si.BF16])
@pytest.mark.parametrize("K,N,B,n_ctx", [(14336, 520, 12, 2), (11008, 264, 5, 1), (3000, 2048, 24, 3), (1024, 1024, 32, 4)])
def test_the_stream_is_no_further_off_than_the_gather(K, N, B, n_ctx, dt):
    import paper_2412_07174_b200 as S
    d = si.context_batch(4, K, N, dt, 64, B, n_ctx, 0.9)
    xf, m = si.to_f32(d["x"], dt), d["m_true"]
    tau = oracle.tau(si.to_f32(d["x_calib"], dt), m, 0.6)
    y64 = oracle.sparse_fc(xf, d["W"], dt, m, tau, None, threads=8)
    err = {}
    try:
        for route in (1, 0):
            S.scap_tune("dense_stream", route)
            y, ws = torch.empty((B, N), device="cuda"), workspace(S.scap_grouped_workspace())
            S.scap_sparse_fc_grouped(dev(d["x"], dt), dev(d["W"], dt), f32(m), f32([tau]), None, y, d["ctx"].tolist(), ws.payload)
            torch.cuda.synchronize()
            assert bool((ws.payload == CANARY).all().item()) == (route == 1)
            err[route] = float(np.linalg.norm(y.cpu().numpy() - y64) / np.linalg.norm(y64))
    finally:
        S.scap_tune("dense_stream", 1)
    assert err[1] <= err[0]


@pytest.mark.parametrize("dt", [si.F16, si.BF16])
@pytest.mark.parametrize("sizes", [(1, 3, 8), (2, 16, 4, 4), (5, 1)])
def test_groups_of_up_to_four_rows_keep_binary32_beside_larger_ones(dt, sizes):
    """A row's arithmetic does not depend on the size of another row's group.  Up to four rows a group is multiplied in binary32:
    |x - m| beyond the range of fp16 is no overflow, and entries far below 1 keep all their bits.

    Bound: a sum goes through at most about 40 roundings (rows of a row group, row groups, ranks), each 2^-24 / sqrt(3) rms of a
    partial sum that has on average half the variance of the whole: 2^-24 sqrt(40 / 6), twice that for the worst row."""
    import paper_2412_07174_b200 as S
    K, N, B = 1024, 264, sum(sizes)
    BOUND = 2.0 ** -24 * 2 * np.sqrt(40 / 6)
    rng = np.random.default_rng(3)
    groups = rng.permutation(np.repeat(np.arange(len(sizes)), sizes))
    small = np.array([sizes[g] <= 4 for g in groups])
    m = rng.uniform(-0.01, 0.01, K).astype(np.float32)
    x = m + rng.laplace(0.0, 0.01, (B, K))
    x[:, ::7] = m[::7]                                 # pruned
    m[3] = si.to_f32(si.to_bits(np.array([-60000.0]), dt), dt)[0]
    x[:, 3] = np.where(small, 60000.0, m[3])           # |x - m| = 120000 where the group is small
    d = si.laplace_fc(4, K, N, dt, 16, 1)
    bits = si.to_bits(x, dt)
    xf = si.to_f32(bits, dt)
    W, tau = d["W"], 0.001
    y64 = oracle.sparse_fc(xf, W, dt, m, tau, None, threads=8)
    ws, y = workspace(S.scap_grouped_workspace()), torch.full((B, N), float("nan"), device="cuda")
    S.scap_sparse_fc_grouped(dev(bits, dt), dev(W, dt), f32(m), f32([tau]), None, y, groups.tolist(), ws.payload)
    torch.cuda.synchronize()
    assert ws.intact() and np.isfinite(y.cpu().numpy()[small]).all()
    assert rel_l2_rows(y.cpu().numpy()[small], y64[small]) <= BOUND
    # the same without the one large channel, beside which the others do not count
    bits[:, 3] = bits[~small][0, 3]
    y64 = oracle.sparse_fc(si.to_f32(bits, dt), W, dt, m, tau, None, threads=8)
    S.scap_sparse_fc_grouped(dev(bits, dt), dev(W, dt), f32(m), f32([tau]), None, y, groups.tolist(), ws.payload)
    torch.cuda.synchronize()
    assert rel_l2_rows(y.cpu().numpy()[small], y64[small]) <= BOUND

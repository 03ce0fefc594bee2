"""The integer kernel of the 8-bit calls (scap_fc_i8.cu) at the edges of its blocks of 128 channels, its pairs of blocks, its ring and
its column tiles, for every number of row quarters, sparse and dense - and which calls take it.

Bound: the codes are integers, all bits of an activation are in its digits or it is added by itself in binary64, products and sums are
exact.  What is left: the sum of a rank is put together from its digits (three roundings and one for what was added by itself: the upper
limb's sum or, where that is zero, the next one's; the rest is 2^-15 of it), at most eight ranks and the bias are added - at
most 13 roundings of 2^-24, of sums that are on average smaller than the last one."""
import numpy as np
import pytest
import torch

import oracle
import scap_inputs as si
from scap_testlib import dev, f32, rel_l2_rows, workspace

pytestmark = pytest.mark.gpu
TOL = 13 * 2.0 ** -24

SHAPES = [  # K, N, B, split_k (0: the kernel's choice)
    (8, 16, 1, 0),         # one vector of channels, one piece of a column tile
    (120, 112, 2, 0),
    (128, 128, 3, 0),      # exactly one block
    (136, 144, 4, 0),
    (264, 256, 5, 1),      # three blocks in one rank: a pair and a half, partial
    (1408, 144, 8, 1),     # eleven blocks: one unit per warp and row quarter, the ring wraps
    (1416, 272, 9, 1),
    (7304, 144, 2, 1),     # fifty-eight blocks, one unit per block: a warp's units are six pairs apart
    (8200, 144, 4, 1),
    (4096, 128, 16, 1),    # thirty-two blocks, four row quarters: more units than a warp keeps
    (4104, 400, 12, 3),
    (2048, 1040, 13, 7),   # ranks whose slices of the columns together are longer than the tile
    (4096, 4096, 3, 0),    # a call that takes the kernel by itself
]


@pytest.fixture
def S():
    import paper_2412_07174_b200 as scap
    scap.lib()
    scap.scap_tune("dense_stream", 2)  # every 8-bit call that the kernel can take
    yield scap
    scap.scap_tune("dense_stream", 1)
    scap.scap_tune("split_k", 0)
    scap.scap_tune("tc_spin", 0)


def layer(K, N, B, dt):
    d = si.laplace_fc(4, K, N, dt, 16, B)
    q, scale = si.quantise_q8(d["W"], dt)
    return d, si.to_f32(d["x"], dt), q, scale


@pytest.mark.parametrize("K,N,B,split", SHAPES)
@pytest.mark.parametrize("dt", [si.F16, si.BF16])
def test_rows_match_the_oracle(S, K, N, B, split, dt):
    d, xf, q, scale = layer(K, N, B, dt)
    m, bias = d["m_true"], np.linspace(-1, 1, N).astype(np.float32)
    x, args, ws, yg = dev(d["x"], dt), (torch.from_numpy(q).cuda(), f32(scale)), workspace(S.scap_fc_workspace(B, K, N)), workspace(B * N * 4)
    y = yg.view(torch.float32, (B, N))
    S.scap_tune("split_k", split)
    for mm, tau in ((m, 0.25), (None, 0.25), (m, 1e9)):  # (the last one drops everything)
        y.fill_(float("nan"))
        idx, nnz = (torch.full((n,), -1, dtype=torch.int32, device="cuda") for n in (K, 1))
        S.scap_sparse_fc_q8(x, *args, None if mm is None else f32(mm), f32([tau]), f32(bias), y, ws.payload, **(dict(idx_out=idx, nnz_out=nnz) if B <= 2 else {}))
        torch.cuda.synchronize()
        assert ws.intact() and yg.intact()
        assert rel_l2_rows(y.cpu().numpy(), oracle.sparse_fc_q8(xf, q, scale, mm, tau, bias)) <= TOL
        if B <= 2:
            assert np.array_equal(idx[: int(nnz.item())].cpu().numpy().astype(np.uint32), oracle.mask(xf, mm, tau)[2])
    y.fill_(float("nan"))
    S.scap_dense_fc_q8(x, *args, f32(bias), y, ws.payload)
    torch.cuda.synchronize()
    assert yg.intact() and rel_l2_rows(y.cpu().numpy(), oracle.sparse_fc_q8(xf, q, scale, None, 0.0, bias)) <= TOL


def test_a_row_that_is_not_finite_leaves_the_others_as_they_are(S):
    """Infinities in different blocks and in the units that a warp does not keep: value x code, and no other row changes a bit."""
    K, N, B = 4096, 144, 8
    d, xf, q, scale = layer(K, N, B, si.BF16)
    x, args, ws = dev(d["x"], si.BF16), (torch.from_numpy(q).cuda(), f32(scale)), workspace(S.scap_fc_workspace(B, K, N))
    S.scap_tune("split_k", 1)
    out = []
    for special in (False, True):
        xs = x.clone()
        if special:
            xs[2, 5], xs[2, 3999], xs[7, 2000] = float("inf"), float("inf"), float("-inf")
        y = torch.empty((B, N), dtype=torch.float32, device="cuda")
        S.scap_sparse_fc_q8(xs, *args, f32(d["m_true"]), f32([0.2]), None, y, ws.payload)
        out.append(y.cpu())
    rows = [b for b in range(B) if b not in (2, 7)]
    assert torch.equal(out[0][rows], out[1][rows])
    with np.errstate(invalid="ignore"):
        want2, want7 = np.inf * q[5].astype(np.float64) + np.inf * q[3999].astype(np.float64), -np.inf * q[2000].astype(np.float64)
    assert np.array_equal(out[1][2].numpy(), want2.astype(np.float32), equal_nan=True)
    assert np.array_equal(out[1][7].numpy(), want7.astype(np.float32), equal_nan=True)


@pytest.mark.parametrize("large", [1e3, 1e5, 1e10])
@pytest.mark.parametrize("K,N,B,split", [(4096, 144, 3, 1), (4104, 272, 8, 3), (4096, 144, 16, 8)])
def test_columns_that_do_not_use_a_large_activation_keep_their_bits(S, K, N, B, split, large):
    """One activation far above the others of its row, whose code is zero in every other column: those columns are as exact as without it."""
    d, xf, q, scale = layer(K, N, B, si.BF16)
    at = 37 * np.arange(B) % K  # another channel in every row
    x = xf.copy()
    x[np.arange(B), at] = large
    q[at, ::2] = 0
    bits = si.to_bits(x, si.BF16)
    args, ws = (torch.from_numpy(q).cuda(), f32(scale)), workspace(S.scap_fc_workspace(B, K, N))
    y = torch.empty((B, N), dtype=torch.float32, device="cuda")
    S.scap_tune("split_k", split)
    for m, tau in ((d["m_true"], 0.2), (None, 0.0)):
        S.scap_sparse_fc_q8(dev(bits, si.BF16), *args, None if m is None else f32(m), f32([tau]), None, y, ws.payload)
        want = oracle.sparse_fc_q8(si.to_f32(bits, si.BF16), q, scale, m, tau, None)
        got = y.cpu().numpy()
        assert rel_l2_rows(got[:, ::2], want[:, ::2]) <= TOL
        assert rel_l2_rows(got[:, 1::2], want[:, 1::2]) <= TOL


@pytest.mark.parametrize("K,N,B,split", [(1544, 144, 3, 1), (4096, 272, 6, 2), (3080, 144, 16, 1)])
@pytest.mark.parametrize("power,sizes", [(0, 48), (100, 48), (-115, 10)])
def test_values_of_every_size_in_one_row(S, K, N, B, split, power, sizes):
    """Channel k lies 2^(k mod sizes) below the largest, and a column uses the channels of one size only, from the window of the digits or
    from below it: every column is right by itself.  (And with all of them near either end of the range of binary32.)"""
    rng = np.random.default_rng(5)
    size = np.arange(K) % sizes
    q = np.where(size[:, None] == np.arange(N)[None, :] % sizes, rng.integers(-127, 128, (K, N)), 0).astype(np.int8)
    scale = np.ldexp(rng.uniform(1, 2, K), power - size).astype(np.float32)
    bits = si.to_bits(rng.uniform(1, 2, (B, K)) * rng.choice([-1, 1], (B, K)), si.BF16)
    args, ws = (torch.from_numpy(q).cuda(), f32(scale)), workspace(S.scap_fc_workspace(B, K, N))
    y = torch.empty((B, N), dtype=torch.float32, device="cuda")
    S.scap_tune("split_k", split)
    for tau, run in ((0.0, "dense"), (1.25, "sparse")):
        if run == "dense":
            S.scap_dense_fc_q8(dev(bits, si.BF16), *args, None, y, ws.payload)
        else:
            S.scap_sparse_fc_q8(dev(bits, si.BF16), *args, None, f32([tau]), None, y, ws.payload)
        want = oracle.sparse_fc_q8(si.to_f32(bits, si.BF16), q, scale, None, tau, None)
        got = y.cpu().numpy().astype(np.float64)
        for s in range(sizes):
            assert rel_l2_rows(got[:, s::sizes], want[:, s::sizes]) <= TOL, s


def test_a_wait_that_runs_out_is_reported_and_the_next_call_is_right(S):
    from paper_2412_07174_b200 import ScapError
    K, N, B = 4096, 512, 5
    d, xf, q, scale = layer(K, N, B, si.BF16)
    x, args, ws = dev(d["x"], si.BF16), (torch.from_numpy(q).cuda(), f32(scale)), workspace(S.scap_fc_workspace(B, K, N))
    y = torch.empty((B, N), dtype=torch.float32, device="cuda")
    S.scap_device_status()
    S.scap_tune("tc_spin", 1)
    S.scap_sparse_fc_q8(x, *args, f32(d["m_true"]), f32([0.2]), None, y, ws.payload)
    with pytest.raises(ScapError) as err:
        S.scap_device_status()
    assert err.value.code == 7  # SCAP_ERR_TIMEOUT
    S.scap_tune("tc_spin", 0)
    S.scap_sparse_fc_q8(x, *args, f32(d["m_true"]), f32([0.2]), None, y, ws.payload)
    S.scap_device_status()
    assert rel_l2_rows(y.cpu().numpy(), oracle.sparse_fc_q8(xf, q, scale, d["m_true"], 0.2, None)) <= TOL


@pytest.mark.parametrize("K,N,B,same", [(4096, 4096, 3, True), (4096, 4096, 16, True), (2048, 1024, 4, True), (2048, 1024, 5, False),
                                        (4092, 4096, 8, False), (4096, 4096, 2, False), (3072, 1024, 5, True), (3072, 1024, 16, True),
                                        (2048, 1024, 16, False), (1024, 1024, 3, False)])
def test_which_calls_take_it(S, K, N, B, same):
    """By default: three and more rows, three blocks of 128 channels per rank (two up to four rows), K a multiple of eight."""
    d, _, q, scale = layer(K, N, B, si.BF16)
    x, args, ws = dev(d["x"], si.BF16), (torch.from_numpy(q).cuda(), f32(scale)), workspace(S.scap_fc_workspace(B, K, N))
    out = []
    for stream in (1, 2, 0):
        S.scap_tune("dense_stream", stream)
        y = torch.empty((B, N), dtype=torch.float32, device="cuda")
        S.scap_sparse_fc_q8(x, *args, f32(d["m_true"]), f32([0.2]), None, y, ws.payload)
        out.append(y.cpu())
    assert not torch.equal(out[0], out[2]) or B <= 2
    assert torch.equal(out[0], out[1]) == (same or K % 8 != 0)

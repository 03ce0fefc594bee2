"""The tensor-core kernel of the quantised calls (scap_fc_qm.cu) at the edges of its tiles: remainders of the 16-channel
blocks, of the 128-column tiles and of the scale groups, every row layout, each activation type, sparse and dense, every cluster
size - and the calls that it does not take, which run on the fp32-FMA kernels two rows at a time.  (8-bit calls with K a multiple of eight run
on the integer kernel here; this one has those of K a multiple of four only, which every test has too.)

Bound: the codes and the three parts of an activation are exact and their products are too.  What is left: an accumulator takes at
most K / 64 products of 16 channels (four or eight warps, at least one rank), each of which truncates it by at most 2^-23 of its
value (on average half of that, of a sum that is on average two thirds of the last one), and a handful of binary32 additions
follow.  A lost third part would show as 1.3e-5."""
import numpy as np
import pytest
import torch

import oracle
import scap_inputs as si
from scap_testlib import dev, f32, rel_l2_rows, workspace

pytestmark = pytest.mark.gpu

SHAPES = [  # K, N, B, group
    (20, 16, 3, 32),        # one full and one partial block, one piece of a column tile
    (64, 144, 1, 32),       # tile and a piece
    (100, 272, 2, 32),      # a partial last block inside a group
    (1000, 144, 4, 96),     # groups of an odd number of steps, partial last group
    (1028, 528, 5, 64),
    (2052, 400, 8, 128),
    (516, 1040, 9, 256),    # two halves of the batch, five and four rows
    (1504, 272, 11, 32),
    (2304, 784, 16, 2048),  # a group longer than a rank's range
    # the same places with K four short of a multiple of eight, for the 8-bit codes
    (68, 144, 1, 32),
    (1004, 144, 4, 96),
    (1508, 272, 11, 32),
    (2308, 784, 16, 2048),
]


@pytest.fixture(scope="module")
def S():
    import paper_2412_07174_b200 as scap
    scap.lib()
    scap.scap_tune("dense_stream", 2)  # every quantised call that the kernel can take
    yield scap
    scap.scap_tune("dense_stream", 1)


def check(S, bits, K, N, B, group, dt):
    d = si.laplace_fc(4, K, N, dt, 16, B)
    x, m, xf = dev(d["x"], dt), d["m_true"], si.to_f32(d["x"], dt)
    bias = np.linspace(-1, 1, N).astype(np.float32)
    ws, yg = workspace(S.scap_fc_workspace(B, K, N)), workspace(B * N * 4)
    y = yg.view(torch.float32, (B, N))
    if bits == 8:
        q, scale = si.quantise_q8(d["W"], dt)
        args = (torch.from_numpy(q).cuda(), f32(scale))
        sparse, dense = S.scap_sparse_fc_q8, S.scap_dense_fc_q8
        ref = lambda mm, tau: oracle.sparse_fc_q8(xf, q, scale, mm, tau, bias)  # noqa: E731
    else:
        q, scale, zero = si.quantise_q4(d["W"], dt, group)
        args = (torch.from_numpy(q).cuda(), f32(scale), torch.from_numpy(zero).cuda(), group)
        sparse, dense = S.scap_sparse_fc_q4, S.scap_dense_fc_q4
        ref = lambda mm, tau: oracle.sparse_fc_q4(xf, q, scale, zero, group, mm, tau, bias)  # noqa: E731
    tol = 2.0 ** -23 * (2 + K / 96)
    for mm, tau in ((m, 0.25), (None, 0.25)):
        y.fill_(float("nan"))
        idx, nnz = (torch.full((n,), -1, dtype=torch.int32, device="cuda") for n in (K, 1))
        kw = dict(idx_out=idx, nnz_out=nnz) if B <= 2 else {}
        sparse(x, *args, None if mm is None else f32(mm), f32([tau]), f32(bias), y, ws.payload, **kw)
        torch.cuda.synchronize()
        assert ws.intact() and yg.intact()
        assert rel_l2_rows(y.cpu().numpy(), ref(mm, tau)) <= tol
        if B <= 2:
            assert np.array_equal(idx[: int(nnz.item())].cpu().numpy().astype(np.uint32), oracle.mask(xf, mm, tau)[2])
    y.fill_(float("nan"))
    dense(x, *args, f32(bias), y, ws.payload)
    torch.cuda.synchronize()
    assert yg.intact()
    assert rel_l2_rows(y.cpu().numpy(), ref(None, 0.0)) <= tol


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("K,N,B,group", SHAPES)
@pytest.mark.parametrize("dt", [si.F16, si.BF16])
def test_quantised_rows_match_the_oracle(S, bits, K, N, B, group, dt):
    check(S, bits, K, N, B, group, dt)


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("split", [1, 3, 5, 6, 7])
@pytest.mark.parametrize("B", [1, 2, 3, 8, 13])
@pytest.mark.parametrize("K", [1000, 1004])
def test_every_cluster_size(S, bits, split, B, K):
    """One rank, and ranks whose slices of the columns together are longer than the tile."""
    try:
        S.scap_tune("split_k", split)
        check(S, bits, K, 272, B, 32, si.BF16)
    finally:
        S.scap_tune("split_k", 0)


@pytest.mark.parametrize("blocks", [8, 9, 10, 16, 17, 25])
@pytest.mark.parametrize("B", [1, 2, 4, 8])
def test_lengths_of_the_8_bit_chains(S, blocks, B):
    """Up to eight blocks of 16 channels stay in the accumulator of a warp, longer stretches leave it every eight blocks."""
    warps = 4 if B > 4 else 8
    try:
        S.scap_tune("split_k", 1)
        check(S, 8, 16 * (blocks * warps - 1) + 4, 144, B, 32, si.BF16)  # the last warp's stretch ends in a partial block
    finally:
        S.scap_tune("split_k", 0)


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("K,B,stream", [(1001, 3, 1), (1002, 5, 1), (1003, 16, 1), (1000, 5, 0), (1000, 16, 0)])
def test_calls_that_run_two_rows_at_a_time(S, bits, K, B, stream):
    """K that is no multiple of four, and "dense_stream" 0."""
    try:
        S.scap_tune("dense_stream", stream)
        check(S, bits, K, 272, B, 64, si.BF16)
    finally:
        S.scap_tune("dense_stream", 2)


@pytest.mark.parametrize("K", [3040, 3044])
def test_either_side_of_the_limit_of_scale_groups(S, K):
    """The scales and zero points of 96 groups fit in the shared memory of a CTA, those of 97 run two rows at a time."""
    try:
        S.scap_tune("split_k", 1)
        check(S, 4, K, 144, 3, 32, si.F16)
    finally:
        S.scap_tune("split_k", 0)


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("B", [1, 4, 16])
@pytest.mark.parametrize("K", [14336, 14332])
def test_a_few_large_activations_do_not_cost_the_others_their_bits(S, bits, B, K):
    """A truncating accumulator that holds a large value early loses up to 2^-23 of it with every further product, so its chain has to be
    short: eight products (8-bit) or a scale group of 128 channels (4-bit), and a handful of additions after it."""
    N = 144
    d = si.laplace_fc(4, K, N, si.BF16, 16, B)
    x = si.to_f32(d["x"], si.BF16).astype(np.float64)
    x[:, ::K // 8] = 300.0 * (1 + np.arange(B))[:, None]  # the first channel of every warp's stretch
    bits_x = si.to_bits(x, si.BF16)
    xf, m = si.to_f32(bits_x, si.BF16), d["m_true"]
    if bits == 8:
        q, scale = si.quantise_q8(d["W"], si.BF16)
        args, fn = (torch.from_numpy(q).cuda(), f32(scale)), S.scap_sparse_fc_q8
        y64 = oracle.sparse_fc_q8(xf, q, scale, m, 0.1, None)
    else:
        q, scale, zero = si.quantise_q4(d["W"], si.BF16, 128)
        args, fn = (torch.from_numpy(q).cuda(), f32(scale), torch.from_numpy(zero).cuda(), 128), S.scap_sparse_fc_q4
        y64 = oracle.sparse_fc_q4(xf, q, scale, zero, 128, m, 0.1, None)
    y = torch.empty((B, N), dtype=torch.float32, device="cuda")
    try:
        S.scap_tune("split_k", 1)
        fn(dev(bits_x, si.BF16), *args, f32(m), f32([0.1]), None, y, workspace(S.scap_fc_workspace(B, K, N)).payload)
        torch.cuda.synchronize()
    finally:
        S.scap_tune("split_k", 0)
    assert rel_l2_rows(y.cpu().numpy(), y64) <= 2.0 ** -23 * (8 + 2)


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("K", [256, 260])
def test_an_infinite_activation_stays_in_its_row(S, bits, K):
    """Row 0 holds an infinity, row 1 a NaN that the threshold drops: row 0 is non-finite, the others are as without them."""
    N, B = 144, 3
    d = si.laplace_fc(4, K, N, si.BF16, 16, B)
    if bits == 8:
        q, scale = si.quantise_q8(d["W"], si.BF16)
        args, fn = (torch.from_numpy(q).cuda(), f32(scale)), S.scap_sparse_fc_q8
    else:
        q, scale, zero = si.quantise_q4(d["W"], si.BF16, 32)
        args, fn = (torch.from_numpy(q).cuda(), f32(scale), torch.from_numpy(zero).cuda(), 32), S.scap_sparse_fc_q4
    x = dev(d["x"], si.BF16)
    ws = workspace(S.scap_fc_workspace(B, K, N))
    out = []
    for special in (False, True):
        xs = x.clone()
        xs[1, 7] = float("nan") if special else 0.0
        if special:
            xs[0, 5] = float("inf")
        y = torch.empty((B, N), dtype=torch.float32, device="cuda")
        fn(xs, *args, None, f32([0.2]), None, y, ws.payload)
        out.append(y.cpu())
    assert torch.equal(out[0][1:], out[1][1:])
    assert not torch.isfinite(out[1][0]).any()


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("B", [1, 2, 3, 5])
@pytest.mark.parametrize("special", [float("inf"), float("nan")])
@pytest.mark.parametrize("K", [256, 260])
def test_a_scale_that_no_kept_channel_uses_has_no_effect(S, bits, B, special, K):
    """Channels 64..95 (one scale group of 32) are dropped by every row: their scales are not part of any sum, whatever they hold."""
    N = 144
    d = si.laplace_fc(4, K, N, si.BF16, 16, B)
    x = dev(d["x"], si.BF16)
    x[:, 64:96] = 0.0
    ws = workspace(S.scap_fc_workspace(B, K, N))
    out = []
    for value in (1.0, special):
        if bits == 8:
            q, scale = si.quantise_q8(d["W"], si.BF16)
            scale[64:96] = value
            args, fn = (torch.from_numpy(q).cuda(), f32(scale)), S.scap_sparse_fc_q8
        else:
            q, scale, zero = si.quantise_q4(d["W"], si.BF16, 32)
            scale[2] = value
            args, fn = (torch.from_numpy(q).cuda(), f32(scale), torch.from_numpy(zero).cuda(), 32), S.scap_sparse_fc_q4
        y = torch.empty((B, N), dtype=torch.float32, device="cuda")
        fn(x, *args, None, f32([0.2]), None, y, ws.payload)
        out.append(y.cpu())
    assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1])

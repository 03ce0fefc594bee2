"""Sixteen rows in the dense-stream kernel with a cluster size that does not divide the column tile: the slices of the ranks are
then together longer than the tile, and the buffer the partial sums land in has to hold them all."""
import pytest
import torch

from scap_testlib import workspace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [3, 5, 6, 7])
def test_sixteen_rows_equal_two_times_eight_and_the_sum_in_64_bits(split):
    import paper_2412_07174_b200 as S
    g = torch.Generator(device="cuda").manual_seed(7)
    D, F, B = 512, 1032, 16

    def rnd(*shape, std=1.0):
        return (torch.randn(shape, generator=g, device="cuda") * std).to(torch.bfloat16)
    h, Wgu, Wd = rnd(B, D), rnd(D, 2 * F, std=0.05), rnd(F, D, std=0.05)
    zero = torch.zeros(1, device="cuda")
    try:
        S.scap_tune("split_k", split)

        def block(x):
            n, out = x.shape[0], workspace(x.shape[0] * D * 4)
            y, ws = out.view(torch.float32, (n, D)), workspace(S.scap_glu_workspace(n, D, F))
            S.scap_glu_ffn(x, Wgu, Wd, None, zero, None, None, zero, None, y, ws.payload)
            torch.cuda.synchronize()
            assert out.intact() and ws.intact()
            return y.clone()

        def plain(x):
            n, out = x.shape[0], workspace(x.shape[0] * 2 * F * 4)
            y = out.view(torch.float32, (n, 2 * F))
            S.scap_sparse_fc(x, Wgu, None, zero, None, y, workspace(S.scap_fc_workspace(n, D, 2 * F)).payload)
            torch.cuda.synchronize()
            assert out.intact()
            return y.clone()
        for fn in (block, plain):
            whole, halves = fn(h), torch.cat([fn(h[:8].contiguous()), fn(h[8:].contiguous())])
            S.scap_device_status()
            assert float((whole - halves).norm() / halves.norm()) < 1e-5  # binary32 sums of at most 1032 terms
            u = h.double() @ Wgu.double()
            if fn is block:
                u = (torch.nn.functional.silu(u[:, :F]) * u[:, F:]) @ Wd.double()
            assert float((whole - u).norm() / u.norm()) < 1e-5
    finally:
        S.scap_tune("split_k", 0)

"""Grouped calls whose groups have more than four rows run as one pass of the dense-stream kernel per 32 rows: the edges of its row
counts, 64-channel blocks, 128-column tiles and cluster slices, and both activation load paths (K a multiple of eight or not).

Bound: binary32 accumulation on the tensor core truncates, at most 2^-23 of the running sum per block of 16 channels along a
chain, and the running sum is up to sqrt(K) times smaller than the sum of magnitudes; errors of ranks and columns average.
2^-23 * sqrt(K) * 8 is about five times what is seen."""
import numpy as np
import pytest
import torch

import oracle
import scap_inputs as si
from scap_testlib import dev, f32, rel_l2_rows, workspace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N,B,n_ctx", [
    (64, 8, 5, 1), (100, 136, 10, 2), (1023, 264, 12, 2),     # up to sixteen rows: the kernel of plain calls
    (1024, 1032, 17, 2), (1500, 392, 24, 3), (2049, 128, 31, 3), (2560, 520, 32, 4),
    (1030, 264, 33, 3), (4096, 1024, 64, 8),                  # two passes
])
@pytest.mark.parametrize("dt", [si.F16, si.BF16])
def test_large_groups_match_the_oracle(K, N, B, n_ctx, dt):
    import paper_2412_07174_b200 as S
    d = si.context_batch(4, K, N, dt, 64, B, n_ctx, 0.9)
    xf, m = si.to_f32(d["x"], dt), d["m_true"]
    tau = oracle.tau(si.to_f32(d["x_calib"], dt), m, 0.6)
    bias = np.linspace(-1, 1, N).astype(np.float32)
    y64 = oracle.sparse_fc(xf, d["W"], dt, m, tau, None, threads=8) + bias[None, :]
    ws, yg = workspace(S.scap_grouped_workspace()), workspace(B * N * 4)
    y = yg.view(torch.float32, (B, N))
    y.fill_(float("nan"))
    S.scap_sparse_fc_grouped(dev(d["x"], dt), dev(d["W"], dt), f32(m), f32([tau]), f32(bias), y, d["ctx"].tolist(), ws.payload)
    torch.cuda.synchronize()
    S.scap_device_status()
    assert ws.intact() and yg.intact()
    assert rel_l2_rows(y.cpu().numpy(), y64) <= 2.0 ** -23 * 8 * np.sqrt(K)

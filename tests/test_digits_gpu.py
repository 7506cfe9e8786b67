"""The weight-only operating point for few tokens: three digit planes a value as columns of the tcgen05 contraction, at the edges of its tiles
(48 and 96 columns), of the split of K over a cluster (one k-block, ragged units) and of the rows (beyond one tile, more tiles than SMs), and
the few tokens that stay on mma.sync.  Against the CPU oracle with the bounds of tests/test_a16_gpu.py."""
import pytest
import torch

import oracle
from paper_2605_00422_b200 import inputs as gen
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N,n1,n2,r,M", [(2048, 200, 32, 64, 13, 5), (2048, 19300, 32, 64, 0, 16), (5120, 130, 64, 80, 64, 16), (5120, 130, 64, 80, 64, 17),
                                           (5120, 130, 64, 80, 8, 32), (128, 40, 8, 16, 4, 32), (25600, 129, 160, 160, 16, 6), (1152, 129, 18, 64, 5, 1),
                                           (4096, 8192, 64, 64, 16, 4), (4096, 128, 64, 64, 16, 4)])
def test_against_the_oracle(K, N, n1, n2, r, M):
    from paper_2605_00422_b200 import bwla
    sh = gen.small_shape(K, N, n1, n2, r, shape_id=K + N + M)
    lay = gen.make_layer(0, sh, 8, with_mu=(M % 2 == 0))
    xb = gen.make_activations(0, sh, M)
    dl = H.DeviceLayer(lay, bwla)
    layer = bwla.Layer(dl.P1, dl.P2, 8, dl.packed, dl.alpha, dl.U, dl.V, mu=dl.mu)
    ws = torch.zeros(bwla.bwla_w1a16_workspace_bytes(layer, M), dtype=torch.uint8, device="cuda")
    out = torch.full((M, N + 3), 7.0, dtype=torch.bfloat16, device="cuda")
    bwla.bwla_layer_w1a16_linear(layer, H.bf16_to_dev(xb), out=out[:, :N], workspace=ws)
    assert bwla.bwla_check_status(ws) == 0
    assert torch.all(out[:, N:] == 7.0)
    rows = slice(0, M) if N * K < 1 << 24 else slice(0, 2)
    ref = oracle.linear_a16(xb[rows], lay.P1, lay.P2, dl.packed_host, lay.alpha, lay.U, lay.V, mu=lay.mu)
    rep = H.check_output(H.bf16_to_host(out[rows, :N].contiguous()), ref["y"])
    assert M * N < 1024 or rep["rel_l2"] <= 2e-3

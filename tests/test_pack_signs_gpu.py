"""Packing of signs at the edges of the vectorised kernel: row lengths around its 1024-group block, row strides that keep
16-byte alignment and ones that do not, and the values whose sign is decided by rule (0, -0.0, NaN, infinities)."""
import numpy as np
import pytest
import torch

import oracle
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,pad", [(1, 32, 0), (3, 8192, 0), (5, 8160, 8), (2, 8224, 16), (70000, 32, 32), (9, 96, 1), (4, 64, 2)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_pack_signs_edges(N, K, pad, dtype):
    from paper_2605_00422_b200 import bwla
    g = torch.Generator().manual_seed(N + K)
    W = torch.randn(N, K + pad, generator=g)
    W[0, :6] = torch.tensor([0.0, -0.0, float("nan"), float("inf"), -float("inf"), 1e-42])
    W = W.to(dtype)
    got = H.words_to_host(bwla.bwla_pack_signs(W.cuda()[:, :K]))
    assert np.array_equal(got, oracle.pack_signs(W[:, :K].float().numpy()))

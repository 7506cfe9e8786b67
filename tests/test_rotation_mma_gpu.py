"""The warp-level tensor-core rotation at the edges of its work split: column tiles dealt to 1, 2 and 4 warps with padding,
rows of P2^T that do not fill the last 16-row tile or the last CTA of a cluster, several groups per CTA with a ragged last
round, rows of x that do not start on 16 bytes, and tokens whose values span most of bf16's exponent range.

The bound on Y is that of tests/test_rotation_umma_gpu.py, 9e-7 of the token's full scale; codes and scales must follow from the
kernel's own Y exactly."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_00422_b200 import inputs as gen
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2,M,pad,scale", [
    (1, 32, 5, 0, 1.0), (4, 16, 700, 0, 1.0), (20, 32, 333, 0, 1.0), (48, 64, 449, 0, 1.0), (73, 64, 3, 0, 1.0),
    (100, 128, 2, 0, 1.0), (112, 128, 150, 0, 1.0), (140, 96, 4, 0, 1.0), (172, 136, 3, 0, 1.0), (180, 136, 3, 0, 1.0), (188, 136, 2, 0, 1.0), (64, 256, 5, 0, 1.0),
    (36, 248, 2, 0, 1.0), (64, 80, 7, 1, 1.0), (160, 160, 2, 3, 1.0), (64, 80, 3, 0, 2.0 ** 100), (64, 80, 3, 0, 2.0 ** -110),
])
def test_edges(n1, n2, M, pad, scale):
    from paper_2605_00422_b200 import bwla
    K, bits = n1 * n2, 6
    rng = np.random.default_rng([n1, n2, M])
    P1, P2 = gen.orthogonal_f32(n1, rng), gen.orthogonal_f32(n2, rng)
    x = rng.standard_t(3, size=(M, K)).astype(np.float32)
    x[0, 0] = 300.0
    xb = gen.bf16_bits_from_f32(x * np.float32(scale))
    L = bwla.Layer(H.f32_to_dev(P1), H.f32_to_dev(P2), bits, torch.zeros((8, K // 32), dtype=torch.int32, device="cuda"),
                   torch.ones(8, device="cuda"))
    rows = torch.zeros(M, K + pad, dtype=torch.bfloat16, device="cuda")
    rows[:, :K] = H.bf16_to_dev(xb)
    codes, scales, y = bwla.bwla_layer_rotate_quant(L, rows[:, :K], want_y=True)
    codes, scales, y = codes.cpu().numpy(), scales.cpu().numpy(), y.cpu().numpy().astype(np.float64)
    Y = oracle.rotate(xb, P1, P2)
    assert float((np.abs(y - Y) / np.abs(Y).max(axis=1, keepdims=True)).max()) <= 9e-7
    q = oracle.quantize(y, bits, "f32")
    assert np.array_equal(q["codes"], codes) and np.array_equal(q["scales"], scales)


@pytest.mark.parametrize("n1,n2,N,dtype,pad", [(100, 128, 5, "f32", 1), (86, 128, 300, "bf16", 3), (48, 64, 450, "f32", 0)])
def test_binarize_edges(n1, n2, N, dtype, pad):
    """Signs follow from (row - mean) except within 3e-6 of the row's largest rotated value; mean and deviation to 2e-6 of it."""
    from paper_2605_00422_b200 import bwla
    K = n1 * n2
    rng = np.random.default_rng([n1, N])
    P1, P2 = gen.orthogonal_f32(n1, rng), gen.orthogonal_f32(n2, rng)
    W = (rng.standard_normal((N, K)) * 0.02).astype(np.float32)
    if dtype == "bf16":
        W = gen.f32_from_bf16_bits(gen.bf16_bits_from_f32(W))
    rows = torch.zeros(N, K + pad, dtype=torch.float32 if dtype == "f32" else torch.bfloat16, device="cuda")
    rows[:, :K] = torch.from_numpy(W).cuda().to(rows.dtype)
    packed, alpha, mu = bwla.bwla_binarize_rows(rows[:, :K], H.f32_to_dev(P1), H.f32_to_dev(P2))
    ref = oracle.binarize(W, P1, P2)
    amax = np.abs(ref["X"]).max(axis=1)
    assert np.all(np.abs(mu.cpu().numpy() - ref["mu"]) <= 2e-6 * amax) and np.all(np.abs(alpha.cpu().numpy() - ref["alpha"]) <= 2e-6 * amax)
    differ = oracle.unpack_signs(H.words_to_host(packed), K) != oracle.unpack_signs(ref["packed"], K)
    assert not np.any(differ & (np.abs(ref["X"] - ref["mu"][:, None]) > 3e-6 * amax[:, None]))

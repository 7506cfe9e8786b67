"""Contractions at the edges of their work splits.

Up to 16 tokens (gemm_small.cu): one and two token tiles, rows that do not fill a group of 32, K that does not fill an item of 512 or
is split over a cluster; accumulators exactly those of int64 arithmetic.  Its digit form and the persistent weight-only kernel: token
counts either side of their border, K that ends inside a unit of 1024, more tiles than SMs; outputs against the oracle with the
layer tolerance.  A group's one launch for more than 64 tokens: outputs are those of the linears called alone, bit for bit without a
low-rank branch.  (More tokens than SMs, so that group and linear take the same rotation kernel.)  With one, T = V x may be summed in
another number of parts: fp32 sums of 1152 products that differ by 1152 * 2^-24 = 7e-5 of their magnitude at most, so outputs by
that share of the low-rank term, here below 1e-4 of the largest output, and one step of bf16."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_00422_b200 import inputs as gen
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N,bits", [(1, 128, 1, 4), (1, 640, 33, 8), (2, 512, 4800, 6), (7, 1152, 95, 6), (8, 5120, 32, 8), (9, 640, 31, 4),
                                        (16, 25600, 64, 8), (16, 4224, 9601, 6)])
def test_few_tokens_accumulate_exactly(M, K, N, bits):
    from paper_2605_00422_b200 import bwla
    rng = np.random.default_rng([M, K, N])
    q = 2 ** (bits - 1) - 1
    codes = rng.integers(-q, q + 1, size=(M, K)).astype(np.int8)
    codes[0] = q                                                     # the largest sums
    words = rng.integers(-2 ** 31, 2 ** 31, size=(N, K // 32), dtype=np.int64).astype(np.int32)
    words[0] = -1
    signs = oracle.unpack_signs(words.view(np.uint32), K).astype(np.float64)
    signs = np.where(signs > 0, 1.0, -1.0)
    scales = torch.ones(M, device="cuda")
    _, acc = bwla.bwla_w1a_gemm_codes(torch.from_numpy(codes).cuda(), scales, bits, torch.from_numpy(words).cuda(), torch.ones(N, device="cuda"), want_acc=True)
    ref = codes.astype(np.float64) @ signs.T                         # (integers below 2^53)
    assert np.array_equal(acc.cpu().numpy().astype(np.int64), ref.astype(np.int64))


@pytest.mark.parametrize("K,N,n1,n2,r,M", [(1280, 200, 20, 64, 13, 17), (1024, 129, 32, 32, 0, 32), (1280, 129, 20, 64, 13, 33), (1152, 257, 18, 64, 0, 150),
                                           (128, 19300, 8, 16, 4, 260), (25600, 40, 160, 160, 13, 52)])
def test_weight_only(K, N, n1, n2, r, M):
    from paper_2605_00422_b200 import bwla
    sh = gen.small_shape(K, N, n1, n2, r, shape_id=K + N + M)
    lay = gen.make_layer(0, sh, 8, with_mu=(M != 32))
    xb = gen.make_activations(0, sh, M)
    dl = H.DeviceLayer(lay, bwla)
    layer = bwla.Layer(dl.P1, dl.P2, 8, dl.packed, dl.alpha, dl.U, dl.V, mu=dl.mu)
    ws = torch.zeros(bwla.bwla_w1a16_workspace_bytes(layer, M), dtype=torch.uint8, device="cuda")
    out = torch.full((M, N + 3), 7.0, dtype=torch.bfloat16, device="cuda")
    bwla.bwla_layer_w1a16_linear(layer, H.bf16_to_dev(xb), out=out[:, :N], workspace=ws)
    assert bwla.bwla_check_status(ws) == 0
    assert torch.all(out[:, N:] == 7.0)
    ref = oracle.linear_a16(xb, lay.P1, lay.P2, dl.packed_host, lay.alpha, lay.U, lay.V, mu=lay.mu)
    H.check_output(H.bf16_to_host(out[:, :N].contiguous()), ref["y"])


@pytest.mark.parametrize("M,r,asym", [(150, 0, False), (201, 0, True), (201, 13, True), (300, 64, False), (1500, 16, False)])
def test_a_group_equals_its_linears(M, r, asym):
    from paper_2605_00422_b200 import bwla
    n1, n2, K = 18, 64, 1152
    g = torch.Generator(device="cuda")
    g.manual_seed(M)
    x = torch.randn(M, K, device="cuda", generator=g).bfloat16()
    layers = []
    for N in (200, 1, 4100):
        rng = np.random.default_rng([M, N])
        words = torch.from_numpy(rng.integers(-2 ** 31, 2 ** 31, size=(N, K // 32), dtype=np.int64).astype(np.int32)).cuda()
        U = torch.randn(N, r, device="cuda", generator=g).bfloat16() if r else None
        V = torch.randn(r, K, device="cuda", generator=g).bfloat16() if r else None
        layers.append(bwla.Layer(H.f32_to_dev(gen.orthogonal_f32(n1, rng)), H.f32_to_dev(gen.orthogonal_f32(n2, rng)), 6, words,
                                 torch.rand(N, device="cuda", generator=g), U, V, 0.01 * torch.randn(N, device="cuda", generator=g), asymmetric=asym))
    together = [o.clone() for o in bwla.bwla_w1ax_linear_group(layers, x)]
    for layer, out in zip(layers, together):
        alone = bwla.bwla_w1ax_linear_group([layer], x)[0]
        if r == 0:
            assert torch.equal(out.view(torch.int16), alone.view(torch.int16))
        else:
            a, b = out.double(), alone.double()
            assert torch.all((a - b).abs() <= 2.0 ** -7 * a.abs() + 1e-4 * a.abs().max())


@pytest.mark.parametrize("r,M", [(72, 5), (120, 16), (65, 1)])
def test_ranks_above_64_whose_columns_do_not_fill_a_tile(r, M):
    """16 x 256: two warps a CTA, so K is split sixteen ways; the partial sums of the last tile of columns lie in front of the codes."""
    from paper_2605_00422_b200 import bwla
    from tests.test_parity_gpu import _run_layer_case
    _run_layer_case(bwla, 0, gen.small_shape(4096, 40, 16, 256, r, shape_id=r), M, 6)


def test_one_weight_only_workspace_serves_smaller_batches():
    from paper_2605_00422_b200 import bwla
    sh = gen.small_shape(1024, 64, 32, 32, 16, shape_id=9)
    dl = H.DeviceLayer(gen.make_layer(0, sh, 8), bwla)
    layer = bwla.Layer(dl.P1, dl.P2, 8, dl.packed, dl.alpha, dl.U, dl.V)
    sizes = [bwla.bwla_w1a16_workspace_bytes(layer, M) for M in range(1, 200)]
    assert sizes == sorted(sizes)
    ws = torch.zeros(bwla.bwla_w1a16_workspace_bytes(layer, 40), dtype=torch.uint8, device="cuda")
    bwla.bwla_layer_w1a16_linear(layer, H.bf16_to_dev(gen.make_activations(0, sh, 32)), workspace=ws)
    assert bwla.bwla_check_status(ws) == 0


def test_sums_of_codes_beyond_their_bit_width():
    """65536 codes of 127 declared as 4 bits: 8.3 million, beyond the short epilogue's 2^22."""
    from paper_2605_00422_b200 import bwla
    M, K, N = 65, 65536, 64
    codes = torch.full((M, K), 127, dtype=torch.int8, device="cuda")
    words = torch.full((N, K // 32), -1, dtype=torch.int32, device="cuda")
    out, _ = bwla.bwla_w1a_gemm_codes(codes, torch.ones(M, device="cuda"), 4, words, torch.ones(N, device="cuda"))
    assert torch.all(out.float() == torch.tensor(127.0 * K).bfloat16().float().item())


@pytest.mark.parametrize("e", [-100, -118, -122])
def test_weight_only_tokens_near_the_end_of_the_exponent_range(e):
    """Tokens of 2^e (values stay normal numbers), scales of 2^60: the fixed-point digits keep their 23 bits; outputs to bf16's rounding."""
    from paper_2605_00422_b200 import bwla
    n1, n2, K, N, M = 32, 64, 2048, 64, 3
    rng = np.random.default_rng(-e)
    P1, P2 = H.f32_to_dev(gen.orthogonal_f32(n1, rng)), H.f32_to_dev(gen.orthogonal_f32(n2, rng))
    x = (torch.from_numpy(rng.standard_normal((M, K)).astype(np.float32)).cuda().double() * 2.0 ** e).bfloat16()
    words = torch.from_numpy(rng.integers(-2 ** 31, 2 ** 31, size=(N, K // 32), dtype=np.int64).astype(np.int32)).cuda()
    layer = bwla.Layer(P1, P2, 8, words, torch.full((N,), 2.0 ** 60, device="cuda"))
    out = bwla.bwla_layer_w1a16_linear(layer, x).double()
    bits = (words.unsqueeze(-1) >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1
    Y = (P1.double().t() @ x.double().view(M, n1, n2) @ P2.double()).reshape(M, K)
    want = (Y @ (2.0 * bits.reshape(N, K).double() - 1.0).t()) * 2.0 ** 60
    assert float((out - want).norm() / want.norm()) <= 5e-3          # two roundings to bf16 (2^-9 each at most) and their sum over K

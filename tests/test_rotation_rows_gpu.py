"""The tcgen05 rotation with output rows on the lanes at the edges of its work split: one and two tokens a step with a ragged last step,
rows that do not fill the lanes, 2 to 5 warps a lane quarter, one and two chunks a warp, rows of outputs that are whole groups of 32 (written
from registers) and that are not (through shared memory).

Bounds as in tests/test_rotation_many_gpu.py: Y within 9e-7 of the token's full scale, codes, zero points and scales exactly those that follow
from it, outputs those of the contraction on the codes in natural order."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_00422_b200 import inputs as gen
from tests import helpers as H

pytestmark = pytest.mark.gpu

SIZES = [(33, 32, 301), (40, 48, 297), (64, 64, 149), (62, 80, 298), (66, 112, 150), (128, 32, 151), (97, 64, 149), (90, 80, 150), (88, 96, 149), (128, 128, 297), (128, 112, 150)]


def _case(n1, n2, M, asym):
    from paper_2605_00422_b200 import bwla
    K, N = n1 * n2, 72
    rng = np.random.default_rng([n1, n2, M])
    P1, P2 = gen.orthogonal_f32(n1, rng), gen.orthogonal_f32(n2, rng)
    x = rng.standard_t(3, size=(M, K)).astype(np.float32)
    x[0, 0], x[M - 1], x[1] = 300.0, 0.0, np.abs(x[1])
    packed = torch.from_numpy(rng.integers(-2 ** 31, 2 ** 31, size=(N, K // 32), dtype=np.int64).astype(np.int32)).cuda()
    alpha, mu = torch.rand(N, device="cuda") + 0.5, 0.01 * torch.randn(N, device="cuda")
    L = bwla.Layer(H.f32_to_dev(P1), H.f32_to_dev(P2), 8, packed, alpha, None, None, mu, asymmetric=asym)
    return bwla, L, P1, P2, gen.bf16_bits_from_f32(x)


@pytest.mark.parametrize("asym", [False, True])
@pytest.mark.parametrize("n1,n2,M", SIZES)
def test_codes(n1, n2, M, asym):
    bwla, L, P1, P2, xb = _case(n1, n2, M, asym)
    dx = H.bf16_to_dev(xb)
    Y = oracle.rotate(xb, P1, P2)
    full = np.maximum(np.abs(Y).max(axis=1, keepdims=True), 1e-30)
    if asym:
        u, s, z, y = (t.cpu().numpy() for t in bwla.bwla_layer_rotate_quant_asym(L, dx, want_y=True))
        q = oracle.quantize_asym(y.astype(np.float64), 8, "f32")
        assert np.array_equal(q["zeros"], z)
    else:
        u, s, y = (t.cpu().numpy() for t in bwla.bwla_layer_rotate_quant(L, dx, want_y=True))
        q = oracle.quantize(y.astype(np.float64), 8, "f32")
    assert float((np.abs(y.astype(np.float64) - Y) / full).max()) <= 9e-7
    assert np.array_equal(q["codes"], u) and np.array_equal(q["scales"], s)
    # the contraction's order, code sums and zero points: the accumulators that the codes in natural order have
    out = bwla.bwla_w1ax_linear_group([L], dx)[0].float().cpu().numpy().astype(np.float64)
    sign = oracle.unpack_signs(L.tensors[2].cpu().numpy().view(np.uint32), n1 * n2).astype(np.float64)
    val = u.astype(np.float64) - (z[:, None] if asym else 0)
    want = s[:, None].astype(np.float64) * (val @ sign.T * L.tensors[3].cpu().numpy().astype(np.float64) + val.sum(axis=1, keepdims=True) * L.tensors[6].cpu().numpy().astype(np.float64))
    # bf16 rounding, and fp32 arithmetic on the terms before it
    bound = 2.0 ** -8 * np.abs(want) + 2.0 ** -20 * s[:, None] * np.abs(val).sum(axis=1, keepdims=True) * float(L.tensors[3].max()) + 1e-30
    assert np.all(np.abs(out - want) <= bound)


@pytest.mark.parametrize("n1,n2,M,asym", [(48, 64, 701, False), (50, 64, 603, True), (62, 80, 447, True), (64, 64, 150, False), (80, 64, 231, True), (66, 48, 225, False)])
def test_codes_from_the_tokens_on_that_come_here(n1, n2, M, asym):
    test_codes(n1, n2, M, asym)


@pytest.mark.parametrize("K,N,n1,n2,r,M", [(5120, 3072, 64, 80, 32, 30), (4096, 4800, 64, 64, 16, 4), (4096, 4096, 64, 64, 0, 50), (5120, 300, 64, 80, 8, 133)])
def test_few_tokens_of_raw_factors_beside_a_full_device(K, N, n1, n2, r, M):
    """Raw linears whose contraction leaves no SMs for the warp-level rotation's blocks: theirs are these, T = V x beside them."""
    from paper_2605_00422_b200 import bwla
    from tests.test_parity_gpu import _run_layer_case
    _run_layer_case(bwla, 0, gen.small_shape(K, N, n1, n2, r, shape_id=K + N + M), M, 6, with_mu=True, direct_words=True)


@pytest.mark.parametrize("n1,n2,M,asym", [(64, 64, 50, False), (64, 80, 64, True), (86, 128, 50, False), (64, 128, 64, False), (128, 64, 61, False)])
def test_a_group_with_its_low_rank_products_beside_the_rotation(n1, n2, M, asym):
    """Three prepared linears, tokens up to which T = V x are blocks of the rotation's launch, one of them without a low-rank branch: outputs those of
    the oracle's layer on the same codes."""
    from paper_2605_00422_b200 import bwla
    K, N, bits = n1 * n2, 136, 8
    rng = np.random.default_rng([n1, n2, M])
    xb = gen.bf16_bits_from_f32(rng.standard_t(3, size=(M, K)).astype(np.float32))
    x, layers, host = H.bf16_to_dev(xb), [], []
    for r in (24, 0, 64):
        P1, P2 = gen.orthogonal_f32(n1, rng), gen.orthogonal_f32(n2, rng)
        packed = rng.integers(-2 ** 31, 2 ** 31, size=(N, K // 32), dtype=np.int64).astype(np.int32)
        alpha = rng.uniform(0.5, 1.5, N).astype(np.float32)
        U, V = (gen.bf16_bits_from_f32((0.05 * rng.standard_normal(sh)).astype(np.float32)) for sh in ((N, max(r, 1)), (max(r, 1), K)))
        layers.append(bwla.Layer(H.f32_to_dev(P1), H.f32_to_dev(P2), bits, torch.from_numpy(packed).cuda(), torch.from_numpy(alpha).cuda(),
                                 H.bf16_to_dev(U) if r else None, H.bf16_to_dev(V) if r else None, asymmetric=asym))
        host.append((P1, P2, packed, alpha, gen.f32_from_bf16_bits(U).astype(np.float64), gen.f32_from_bf16_bits(V).astype(np.float64), r))
    ws = torch.zeros(bwla.bwla_group_workspace_bytes(layers, M), dtype=torch.uint8, device="cuda")
    for _ in range(3):
        outs = bwla.bwla_w1ax_linear_group(layers, x, workspace=ws)
    assert bwla.bwla_check_status(ws) == 0
    for out, (P1, P2, packed, alpha, U, V, r) in zip(outs, host):
        Y = oracle.rotate(xb, P1, P2)
        if asym:
            q = oracle.quantize_asym(Y, bits, "f32")
            val = (q["codes"].astype(np.float64) - q["zeros"][:, None]) * q["scales"][:, None]
        else:
            q = oracle.quantize(Y, bits, "f32")
            val = q["codes"].astype(np.float64) * q["scales"][:, None]
        want = val @ oracle.unpack_signs(packed.view(np.uint32), K).T.astype(np.float64) * alpha
        low = gen.f32_from_bf16_bits(xb).astype(np.float64) @ V.T @ U.T if r else 0.0
        # bf16 rounding of the output; at most two codes of a token on the other side of a rounding boundary; fp32 sums of K + r terms
        bound = 2.0 ** -8 * np.abs(want + low) + 2.0 * q["scales"][:, None] * 1.5 + 2.0 ** -16 * np.abs(low).max() if r else 2.0 ** -8 * np.abs(want) + 3.0 * q["scales"][:, None]
        assert np.all(np.abs(out.float().cpu().numpy().astype(np.float64) - (want + low)) <= bound)


@pytest.mark.parametrize("n1,n2", [(40, 32), (128, 32)])
def test_several_steps_an_sm_of_the_smallest_factors(n1, n2):
    """Two of these blocks would fit an SM but for its tensor memory; calls behind one another, the contraction's blocks beside the rotation's."""
    M = 2000
    bwla, L, P1, P2, xb = _case(n1, n2, M, False)
    dx = H.bf16_to_dev(xb)
    codes, scales, y = bwla.bwla_layer_rotate_quant(L, dx, want_y=True)
    Y = oracle.rotate(xb, P1, P2)
    full = np.maximum(np.abs(Y).max(axis=1, keepdims=True), 1e-30)
    assert float((np.abs(y.cpu().numpy().astype(np.float64) - Y) / full).max()) <= 9e-7
    q = oracle.quantize(y.cpu().numpy().astype(np.float64), 8, "f32")
    assert np.array_equal(q["codes"], codes.cpu().numpy()) and np.array_equal(q["scales"], scales.cpu().numpy())
    want = bwla.bwla_w1a_gemm_codes(codes, scales, 8, L.tensors[2], L.tensors[3], mu=L.tensors[6])[0]
    ws = torch.zeros(bwla.bwla_group_workspace_bytes([L], M), dtype=torch.uint8, device="cuda")
    for _ in range(20):
        out = bwla.bwla_w1ax_linear_group([L], dx, workspace=ws)[0]
    assert bwla.bwla_check_status(ws) == 0
    assert torch.equal(out.view(torch.int16), want.view(torch.int16))


@pytest.mark.parametrize("n1,n2,M", [(40, 48, 297), (36, 48, 150), (64, 64, 301), (96, 80, 150), (88, 96, 149), (128, 112, 150)])
def test_weight_only_values(n1, n2, M):
    """bf16 values in either order and their sums, through the linear, against the bf16 rounding of the exact rotation."""
    bwla, L, P1, P2, xb = _case(n1, n2, M, False)
    Y = oracle.rotate(xb, P1, P2)
    out = bwla.bwla_layer_w1a16_linear(L, H.bf16_to_dev(xb)).float().cpu().numpy().astype(np.float64)
    yhat = torch.from_numpy(Y).float().bfloat16().double().numpy()
    sign = oracle.unpack_signs(L.tensors[2].cpu().numpy().view(np.uint32), n1 * n2).astype(np.float64)
    want = yhat @ sign.T * L.tensors[3].cpu().numpy().astype(np.float64) + yhat.sum(axis=1, keepdims=True) * L.tensors[6].cpu().numpy().astype(np.float64)
    # bf16 output; a value within the rotation's error (9e-7 of full scale) of a rounding boundary moves by a bf16 step of its own: in 2-norm over
    # K values far below the output's rounding, bounded here by one part in 2^8 of the values' 2-norm
    bound = 2.0 ** -8 * np.abs(want) + 2.0 ** -8 * np.linalg.norm(yhat, axis=1, keepdims=True) * 2.0
    assert np.all(np.abs(out - want) <= bound)
    assert np.linalg.norm(out - want) <= 3e-3 * np.linalg.norm(want)


@pytest.mark.parametrize("n1,n2", [(64, 64), (40, 80), (64, 128)])
def test_an_infinity_stays_in_its_token(n1, n2):
    """Two tokens share a step's MMAs: the other one's codes and scale do not change."""
    bwla, L, P1, P2, xb = _case(n1, n2, 300, False)
    dx = H.bf16_to_dev(xb)
    codes, scales = bwla.bwla_layer_rotate_quant(L, dx)[:2]
    bad = dx.clone()
    bad[4, 7] = float("inf"); bad[9, 100] = float("nan"); bad[131, :] = float("-inf")
    c2, s2 = bwla.bwla_layer_rotate_quant(L, bad)[:2]
    keep = torch.ones(300, dtype=torch.bool); keep[[4, 9, 131]] = False
    assert torch.equal(codes.cpu()[keep], c2.cpu()[keep]) and torch.equal(scales.cpu()[keep], s2.cpu()[keep])


@pytest.mark.parametrize("n1,n2", [(64, 64), (48, 80), (64, 128), (86, 128)])
def test_tokens_without_numbers_have_the_codes_they_have_among_few(n1, n2):
    """Infinities, NaNs, and a token so small that qmax / amax leaves fp32's range: the codes of the kernel for few tokens (-1 and 0), and the
    code sums that belong to them.  qmax = 127 / amax overflows below 3.8e-37."""
    M = 700
    bwla, L, P1, P2, xb = _case(n1, n2, M, False)
    odd = [3, 8, 131, 200, 699]
    x = H.bf16_to_dev(xb)
    x[3, 5], x[8, n1 * n2 - 1], x[131] = float("inf"), float("nan"), float("-inf")
    x[200], x[699] = x[200] * 1e-39, x[699] * 0.0
    codes, scales = bwla.bwla_layer_rotate_quant(L, x)[:2]
    few, few_scales = bwla.bwla_layer_rotate_quant(L, x[odd].contiguous())[:2]
    assert torch.equal(codes[odd], few)
    assert torch.equal(scales[odd][[0, 1, 2, 4]], few_scales[[0, 1, 2, 4]])
    assert abs(float(scales[200]) - float(few_scales[3])) <= 2e-6 * float(few_scales[3]) + 2.0 ** -148
    out = bwla.bwla_w1ax_linear_group([L], x)[0]
    again = bwla.bwla_w1a_gemm_codes(codes, scales, 8, L.tensors[2], L.tensors[3], mu=L.tensors[6])[0]
    assert torch.equal(out.view(torch.int16), again.view(torch.int16))


@pytest.mark.parametrize("n1,n2,N,pad", [(33, 32, 149, 0), (40, 48, 301, 1), (64, 80, 75, 4)])
def test_binarised_rows(n1, n2, N, pad):
    """fp32 rows as three terms, in 16-byte pieces and in single loads, ragged last steps; the bounds of tests/test_binarize_gpu.py."""
    from paper_2605_00422_b200 import bwla
    from tests.test_binarize_gpu import _check
    rng = np.random.default_rng([n1, n2, N])
    P1, P2 = gen.orthogonal_f32(n1, rng), gen.orthogonal_f32(n2, rng)
    W = (rng.standard_normal((N, n1 * n2)) * 0.02 + rng.uniform(-0.01, 0.01, (N, 1))).astype(np.float32)
    big = torch.zeros(N, n1 * n2 + pad, device="cuda")
    big[:, :n1 * n2] = torch.from_numpy(W).cuda()
    _check(bwla, W, big[:, :n1 * n2], P1, P2)


@pytest.mark.parametrize("n1,n2,N,dtype", [(64, 64, 160, torch.float32), (56, 80, 160, torch.float32), (64, 80, 160, torch.float32), (64, 64, 160, torch.bfloat16)])
def test_sums_of_a_binarisation_hold_what_cancels(n1, n2, N, dtype):
    """Identity factors, so that the rotated row is the row: values of 22 bits (8 as bf16) near 2^14, their negatives in the other half, and eight small
    ones down to 2^-25 whose sum is all that is left: 50 bits (38) of one sum."""
    from paper_2605_00422_b200 import bwla
    K = n1 * n2
    rng = np.random.default_rng([n1, n2])
    unit = 2.0 ** -8 if dtype == torch.float32 else 2.0 ** 6
    W = np.zeros((N, n1, n2))
    W[:, : n1 // 2] = rng.integers(int(2 ** 13 / unit), int(2 ** 14 / unit), size=(N, n1 // 2, n2)) * unit
    W[:, :8, 3] = 0.0
    W[:, n1 // 2: 2 * (n1 // 2)] = -W[:, : n1 // 2]
    W[:, :8, 3] = (2 * rng.integers(0, 4, size=(N, 8)) + 1) * 2.0 ** -25
    w = torch.from_numpy(W.reshape(N, K)).to(dtype).cuda()
    assert np.array_equal(w.cpu().double().numpy().reshape(W.shape), W)
    packed, alpha, mu = bwla.bwla_binarize_rows(w, torch.eye(n1, device="cuda"), torch.eye(n2, device="cuda"))
    flat = W.reshape(N, K)
    mean = flat.sum(axis=1) / K                       # (exact: numpy's partial sums of these fit 53 bits)
    assert np.all(np.abs(mu.cpu().numpy().astype(np.float64) - mean) <= 1e-7 * mean)
    np.testing.assert_allclose(alpha.cpu().numpy(), np.abs(flat - mean[:, None]).mean(axis=1), rtol=1e-7)
    assert np.array_equal(oracle.unpack_signs(packed.cpu().numpy().view(np.uint32), K) > 0, flat > mean[:, None])


@pytest.mark.parametrize("n1,n2,dtype", [(64, 64, torch.float32), (56, 80, torch.float32), (64, 80, torch.bfloat16), (32, 64, torch.float32), (64, 128, torch.float32)])
def test_binarised_rows_without_numbers_and_at_the_ends_of_the_range(n1, n2, dtype):
    """Infinities and NaNs: no set bits, scale and shift NaN, and neighbours that keep theirs; a row of zeros: zeros; rows of 2^-100 and 2^100."""
    from paper_2605_00422_b200 import bwla
    N, K = 160, n1 * n2
    rng = np.random.default_rng([n1, n2, 7])
    P1, P2 = H.f32_to_dev(gen.orthogonal_f32(n1, rng)), H.f32_to_dev(gen.orthogonal_f32(n2, rng))
    w = torch.from_numpy((rng.standard_normal((N, K)) + 0.1).astype(np.float32)).cuda()
    w[4] *= 2.0 ** -100
    w[5] *= 2.0 ** 100
    w = w.to(dtype)
    want = [t.cpu() for t in bwla.bwla_binarize_rows(w, P1, P2)[:3]]
    w[1, 5], w[2, K - 1], w[9], w[12] = float("inf"), float("nan"), float("-inf"), 0.0
    packed, alpha, mu = (t.cpu() for t in bwla.bwla_binarize_rows(w, P1, P2)[:3])
    bad, keep = [1, 2, 9], [i for i in range(N) if i not in (1, 2, 9, 12)]
    assert bool((packed[bad] == 0).all()) and bool(alpha[bad].isnan().all()) and bool(mu[bad].isnan().all())
    assert bool((packed[12] == 0).all()) and float(alpha[12]) == 0.0 and float(mu[12]) == 0.0
    assert all(torch.equal(a[keep], b[keep]) for a, b in zip((packed, alpha, mu), want))
    Y = (P1.double().t() @ w[4:6].double().view(2, n1, n2) @ P2.double()).reshape(2, K).cpu()
    mean = Y.mean(dim=1)
    dev = (Y - mean[:, None]).abs().mean(dim=1)
    assert bool(((alpha[4:6] - dev).abs() <= 1e-6 * dev).all()) and bool(((mu[4:6] - mean).abs() <= 1e-6 * dev).all())


def test_a_linear_behind_binarised_rows():
    """The linear's sign words, scales and shifts are fetched before it waits for its predecessor: it must see what that has written."""
    from paper_2605_00422_b200 import bwla
    n1, n2, N, K = 64, 64, 3000, 4096
    rng = np.random.default_rng(6)
    P1, P2 = H.f32_to_dev(gen.orthogonal_f32(n1, rng)), H.f32_to_dev(gen.orthogonal_f32(n2, rng))
    x = H.bf16_to_dev(gen.bf16_bits_from_f32(rng.standard_normal((1, K)).astype(np.float32)))
    for _ in range(4):
        W = torch.from_numpy((rng.standard_normal((N, K)) * 0.02).astype(np.float32)).cuda()
        torch.cuda.synchronize()
        packed, alpha, mu = bwla.bwla_binarize_rows(W, P1, P2)
        out = bwla.bwla_w1ax_linear(x, P1, P2, 6, packed, alpha, mu=mu)
        torch.cuda.synchronize()
        assert torch.equal(out.view(torch.int16), bwla.bwla_w1ax_linear(x, P1, P2, 6, packed, alpha, mu=mu).view(torch.int16))


@pytest.mark.parametrize("n1,n2,M,measured", [(64, 64, 800, 1.42), (64, 80, 800, 1.44), (64, 128, 800, 1.56), (72, 96, 800, 1.74), (80, 128, 800, 1.80), (86, 128, 800, 1.88),
                                              (108, 128, 800, 1.95), (128, 128, 800, 1.95), (64, 80, 60, 1.45), (64, 128, 60, 1.45), (86, 128, 60, 1.50)])
def test_error_of_the_present_kernels(n1, n2, M, measured):
    """As test_error_against_64_bits of tests/test_rotation_many_gpu.py, at what the kernel for these factors and tokens has (1e-7 of a row's 2-norm;
    seeds differ by less than 5 %)."""
    from paper_2605_00422_b200 import bwla
    K, errs = n1 * n2, []
    for seed in range(6):
        rng = np.random.default_rng([n1, n2, seed])
        P1, P2 = H.f32_to_dev(gen.orthogonal_f32(n1, rng)), H.f32_to_dev(gen.orthogonal_f32(n2, rng))
        x = torch.from_numpy(rng.standard_t(3, size=(M, K)).astype(np.float32)).cuda()
        x[:, torch.from_numpy(rng.permutation(K)[:8]).cuda()] *= 50.0
        x = x.bfloat16()
        L = bwla.Layer(P1, P2, 6, torch.zeros((8, K // 32), dtype=torch.int32, device="cuda"), torch.ones(8, device="cuda"))
        y = bwla.bwla_layer_rotate_quant(L, x, want_y=True)[2].double()
        Y = (P1.double().t() @ x.double().view(M, n1, n2) @ P2.double()).reshape(M, K)
        errs.append(float((((y - Y).norm(dim=1) / Y.norm(dim=1)) ** 2).mean()))
    got = 1e7 * np.sqrt(np.mean(errs))
    print(f"[{n1} x {n2}, {M} tokens] {got:.3f}")
    assert got <= 1.05 * measured

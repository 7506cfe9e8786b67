"""A call repeats itself bit for bit: prefill contractions whose expander warps hand stages of sign words back to the copies while other warps
still read them (a release that overtook the loads left a few rows of a tile with the next unit's signs, in one call of fifteen)."""
import pytest
import torch

from paper_2605_00422_b200 import inputs as gen
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weight_only,M,K,N,n1,n2,r", [(True, 1024, 4096, 4096, 64, 64, 32), (True, 333, 8192, 5120, 64, 128, 0),
                                                      (False, 1024, 4096, 4096, 64, 64, 32), (False, 200, 5120, 8192, 64, 80, 0)])
def test_prefill_repeats_itself(weight_only, M, K, N, n1, n2, r):
    from paper_2605_00422_b200 import bwla
    shape = gen.small_shape(K, N, n1, n2, r, shape_id=K + N)
    lay = gen.make_layer(0, shape, 6)
    dl = H.DeviceLayer(lay, bwla)
    L = bwla.Layer(dl.P1, dl.P2, 6, dl.packed, dl.alpha, dl.U, dl.V)
    x = H.bf16_to_dev(gen.make_activations(0, shape, M))
    out = torch.empty(M, N, dtype=torch.bfloat16, device="cuda")
    first = None
    for _ in range(60):
        if weight_only:
            bwla.bwla_layer_w1a16_linear(L, x, out)
        else:
            bwla.bwla_w1ax_linear_group([L], x, [out])
        now = out.view(torch.int16).clone()
        first = now if first is None else first
        assert torch.equal(first, now)

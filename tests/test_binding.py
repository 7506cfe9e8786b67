"""The native half of the Python binding (csrc/python_calls.cpp): what PyTorch throws stays an exception, other threads run during a
call, and calls are refused and accepted as through ctypes."""
import ctypes as C
import os
import subprocess
import sys
import threading
import time

import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_what_pytorch_throws_does_not_end_the_process():
    """Tensors that say they are on a GPU but have no memory there, on a machine without one or with: an exception, not an abort."""
    code = """
from torch._subclasses.fake_tensor import FakeTensorMode
import torch
from paper_2605_00422_b200 import bwla
with FakeTensorMode():
    w, p = torch.empty(4, 64, device="cuda"), torch.empty(4, 2, dtype=torch.int32, device="cuda")
try:
    bwla.bwla_pack_signs(w, p)
except Exception as e:
    print("refused", type(e).__name__)
"""
    r = subprocess.run([sys.executable, "-W", "ignore", "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.startswith("refused"), (r.returncode, r.stderr[-300:])


def _layer(bwla, N=64):
    eye = torch.eye(32, device="cuda")
    return bwla.Layer(eye, eye.clone(), 6, torch.zeros((N, 32), dtype=torch.int32, device="cuda"), torch.ones(N, device="cuda"))


@pytest.mark.gpu
def test_other_threads_run_during_a_call(tmp_path):
    """The library's entry point replaced by one that sleeps: a thread beside it must get on."""
    from paper_2605_00422_b200 import bwla
    src, so = tmp_path / "slow.c", tmp_path / "slow.so"
    src.write_text("#include <unistd.h>\nint slow(void) { usleep(500000); return 0; }\n")
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    slow = C.cast(C.CDLL(str(so)).slow, C.c_void_p).value
    keep = [C.cast(f, C.c_void_p).value for f in (bwla._lib.bwla_w1ax_linear_group, bwla._lib.bwla_w1ax_linear, bwla._lib.bwla_layer_w1a16_linear,
                                                  bwla._lib.bwla_pack_signs)]
    w, p = torch.zeros((4, 64), device="cuda"), torch.zeros((4, 2), dtype=torch.int32, device="cuda")
    beats, stop = [], threading.Event()

    def beat():
        while not stop.is_set():
            beats.append(time.perf_counter())
            time.sleep(0.005)

    t = threading.Thread(target=beat)
    bwla._calls.bind(slow, slow, slow, slow)
    try:
        t.start()
        begin = time.perf_counter()
        assert bwla._calls.pack(w, p) == 0
        end = time.perf_counter()
    finally:
        stop.set()
        t.join()
        bwla._calls.bind(*keep)
    assert end - begin >= 0.4 and sum(begin + 0.05 < b < end - 0.05 for b in beats) > 10


@pytest.mark.gpu
def test_calls_without_tokens_need_no_strides():
    from paper_2605_00422_b200 import bwla
    layer = _layer(bwla)
    x0 = torch.empty((0, 1024), dtype=torch.bfloat16, device="cuda")
    ws = torch.zeros(4096, dtype=torch.uint8, device="cuda")
    empty = torch.empty((0, 1), dtype=torch.bfloat16, device="cuda")          # (rows of any length: there are none)
    assert bwla.bwla_w1ax_linear_group([layer], x0, [empty], ws)[0] is empty
    assert bwla.bwla_layer_w1a16_linear(layer, empty, empty, ws) is empty


@pytest.mark.gpu
def test_what_was_refused_is_refused_in_the_same_way():
    from paper_2605_00422_b200 import bwla
    layer = _layer(bwla)
    x = torch.zeros((2, 1024), dtype=torch.bfloat16, device="cuda")
    out = torch.empty((2, 64), dtype=torch.bfloat16, device="cuda")
    ws = bwla.new_group_workspace([layer, layer], 2)
    with pytest.raises(IndexError):
        bwla.bwla_w1ax_linear_group([layer], x, [out, out], ws)               # more outputs than layers
    with pytest.raises(TypeError):
        bwla.bwla_w1ax_linear_group((l for l in [layer]), x, [out], ws)
    for layers, outs in (([layer, layer], [out]), ([layer] * 5, [out] * 5), ([layer] * 20, [out] * 20), ([], [])):
        with pytest.raises(bwla.BwlaError) as e:
            bwla.bwla_w1ax_linear_group(layers, x, outs, ws)
        assert e.value.status == bwla.BWLA_ERR_INVALID_ARG
    gone = _layer(bwla)
    bwla.bwla_layer_destroy(gone)
    for call in (lambda: bwla.bwla_w1ax_linear_group([gone], x, [out], ws), lambda: bwla.bwla_layer_w1a16_linear(gone, x, out, ws)):
        with pytest.raises(bwla.BwlaError) as e:
            call()
        assert e.value.status == bwla.BWLA_ERR_INVALID_ARG


@pytest.mark.gpu
def test_rows_off_16_bytes_where_the_header_asks_for_them():
    from paper_2605_00422_b200 import bwla
    layer = _layer(bwla)
    x = torch.zeros((2, 1025), dtype=torch.bfloat16, device="cuda")[:, :1024]
    assert bwla.bwla_w1ax_linear_group([layer], x)[0].shape == (2, 64)
    bwla.bwla_layer_set_activation_quant(layer, bwla.BWLA_ACT_ASYMMETRIC)
    for call in (lambda: bwla.bwla_w1ax_linear_group([layer], x), lambda: bwla.bwla_layer_w1a16_linear(layer, x),
                 lambda: bwla.bwla_layer_rotate_quant_asym(layer, x)):
        with pytest.raises(bwla.BwlaError) as e:
            call()
        assert e.value.status == bwla.BWLA_ERR_UNSUPPORTED

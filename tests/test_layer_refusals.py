"""What a layer, a layer stack or the attention backward refuses, it refuses before anything is launched: on a machine without a device a launch would be
MPIPE_ERR_CUDA.  The addresses are never read."""
import ctypes

import pytest
import torch

from paper_2607_03229_b200 import binding as B
from paper_2607_03229_b200 import build as build_mod

# (with a device a missing check would launch kernels on made-up addresses)
pytestmark = pytest.mark.skipif(torch.cuda.is_available(), reason="only where nothing can be launched")

T, HIDDEN, H, FFN, SCALE, EPS = 300, 256, 4, 1024, 0.125, 1e-6
WS = 1 << 40


@pytest.fixture(scope="module", autouse=True)
def _built():
    build_mod.build()


def _struct(cls, n, l, **changed):
    s = (cls * n)()
    for i in range(n):
        for j, (name, _) in enumerate(cls._fields_):
            setattr(s[i], name, 0x10000000 * (1 + i) + 0x100000 * j)
    for name, value in changed.items():
        setattr(s[l], name, value)
    return s


def _calls(weights, n, grads=None, rope=(None, None), mode=B.TRAINED):
    """The status of every entry point that runs these layers (the single-layer ones: the last layer alone)."""
    lib, last = B.load(), ctypes.addressof(weights) + (n - 1) * ctypes.sizeof(B.LayerWeights)
    g = _struct(B.LayerGrads, n, 0) if grads is None else grads
    last_g = ctypes.addressof(g) + (n - 1) * ctypes.sizeof(B.LayerGrads)
    a, plan = 0x70000000, (0x71000000, 1, T, 0x71100000, 3)
    fwd = (SCALE, EPS, *rope, mode, 0x72000000, 0x73000000, WS, None, None)
    bwd = (SCALE, EPS, *rope, mode, 0x72000000, 0x73000000, 0x74000000, WS, None, None)
    return {"layer_fwd": lib.mpipe_encoder_layer_fwd(a, a, last, T, HIDDEN, H, FFN, *plan, *fwd),
            "fwd": lib.mpipe_encoder_fwd(a, a, ctypes.addressof(weights), n, T, HIDDEN, H, FFN, *plan, *fwd),
            "layer_bwd": lib.mpipe_encoder_layer_bwd(a, a, a, last, last_g, T, HIDDEN, H, FFN, *plan, *bwd),
            "bwd": lib.mpipe_encoder_bwd(a, a, a, ctypes.addressof(weights), ctypes.addressof(g), n, T, HIDDEN, H, FFN, *plan, *bwd)}


@pytest.mark.parametrize("name", ["w_qkv", "w_o", "w_fc1", "w_fc2"])
@pytest.mark.parametrize("value,status", [(0x20000002, B.ERR_UNSUPPORTED), (0x20000008, B.ERR_UNSUPPORTED), (None, B.ERR_INVALID_ARG)])
def test_matrices_that_cannot_be_prefetched(name, value, status):
    assert set(_calls(_struct(B.LayerWeights, 1, 0, **{name: value}), 1).values()) == {status}
    got = _calls(_struct(B.LayerWeights, 3, 2, **{name: value}), 3)
    assert set(got.values()) == {status}


@pytest.mark.parametrize("rope", [(0x80000004, 0x81000000), (0x80000000, 0x81000008)])
def test_backward_with_misaligned_tables(rope):
    got = _calls(_struct(B.LayerWeights, 1, 0), 1, rope=rope)
    assert got["layer_bwd"] == got["bwd"] == B.ERR_UNSUPPORTED


def test_backward_without_a_bias_gradient():
    got = _calls(_struct(B.LayerWeights, 1, 0), 1, grads=_struct(B.LayerGrads, 1, 0, b_fc2=None))
    assert got["layer_bwd"] == got["bwd"] == B.ERR_INVALID_ARG


@pytest.mark.parametrize("tokens,heads,status", [(1 << 30, 8, B.ERR_UNSUPPORTED),      # 2^33 rows of heads: more than the last pass counts
                                                 (1 << 28, 8, B.ERR_CUDA)])            # 2^31 of them, 2^34 pieces: goes on to the device
def test_attention_backward_is_refused_before_its_first_launch(tokens, heads, status):
    a, ts = 0x70000000, heads * 64
    got = B.load().mpipe_varlen_attn_bwd(*[a] * 9, *[ts, 64] * 3, a, 1, tokens, tokens, a, 1, heads, 64, SCALE, B.TRAINED, a, 1 << 50, None, None)
    assert got == status

"""Host side of the tensor-core route: which layers it is offered to and which calls take it."""
import numpy as np
import pytest
import torch

from paper_2003_06513_gb300 import api


def _layer(cout, cin, keep, stride=1, scale=None, patterns=None):
    W = np.random.default_rng(0).standard_normal((cout, cin, 3, 3)).astype(np.float32)
    if scale is not None:
        W = (W * np.asarray(scale, np.float64).reshape(-1, 1, 1, 1)).astype(np.float32)
    return api.pp_pack(W, patterns, keep, 1, stride)


@pytest.mark.parametrize("cout,cin,filters", [(16, 16, 16), (64, 3, 64), (150, 90, 160), (257, 40, 288),
                                              (512, 512, 512), (520, 33, 528)])
def test_weight_bytes(cout, cin, filters):
    """Two fp16 values for each of the nine taps of 16-channel blocks and of the padded filters."""
    assert _layer(cout, cin, 1.0).query("tensor_bytes") == -(-cin // 16) * 16 * 9 * 4 * filters


def test_weights_of_extreme_range_are_not_offered():
    assert _layer(8, 16, 1.0, scale=[1e-20] * 8).query("tensor_bytes") == 0
    assert _layer(8, 16, 1.0, scale=[1e15] * 8).query("tensor_bytes") == 0
    assert _layer(8, 16, 1.0, scale=[1.0] * 7 + [1e-9]).query("tensor_bytes") == 0
    assert _layer(8, 16, 1.0, scale=[1.0] * 7 + [1e-3]).query("tensor_bytes") > 0
    assert api.pp_pack(np.ones((8, 1, 3, 3), np.float32), None, 1.0, 8).query("tensor_bytes") == 0


def test_calls_that_take_it():
    big = _layer(256, 256, 0.3)
    assert big.tensor_plan((32, 256, 56, 56))["tensor"] == 1
    # few products a sum: the CUDA cores round less in fp32; in fp16 the output's rounding covers both
    assert _layer(64, 3, 1.0).tensor_plan((32, 3, 224, 224))["tensor"] == 0
    assert _layer(64, 12, 1.0).tensor_plan((64, 12, 112, 112))["tensor"] == 0
    assert _layer(64, 12, 1.0).tensor_plan((64, 12, 112, 112), dtype=torch.float16)["tensor"] == 1
    # a channel split of the CUDA-core plan that leaves few products a range
    assert _layer(64, 64, 0.5).tensor_plan((1, 64, 32, 32), 1 << 30)["tensor"] == 0


@pytest.mark.parametrize("h,w", [(7, 7), (14, 14), (28, 30), (57, 211), (224, 224), (500, 701)])
@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("pool", [False, True])
@pytest.mark.parametrize("cout", [48, 128, 300])
def test_tiles_cover_the_map(h, w, stride, pool, cout):
    lay = _layer(cout, 96, 1.0, stride)
    n = 33
    p = lay.tensor_plan((n, 96, h, w), 0, pool)
    if not p["tensor"]:
        pytest.skip("takes the CUDA-core kernel")
    ho, wo = (h - 1) // stride + 1, (w - 1) // stride + 1
    chunks = -(-cout // p["filters"])
    assert p["filters"] % 16 == 0 and p["filters"] * p["positions"] // 128 <= 256
    if p["tile_w"] == 0:
        assert not pool
        tiles = -(-n * (ho + 1) * (wo + 1) // p["positions"])
    else:
        tw, th = p["tile_w"], p["tile_h"]
        pitch = tw + 1 if tw >= wo or stride == 2 else tw + 2
        assert (th - 1) * pitch + tw <= p["positions"]
        if pool:
            assert th % 2 == 0 and (tw % 2 == 0 or tw == wo)
        tiles = n * -(-ho // th) * -(-wo // tw)
    assert p["units"] == -(-tiles // 2) * chunks

"""The tensor-core kernel against the float64 oracle, and the CUDA-core kernel beside it.

Sizes sit where the kernel can go wrong: tiles of 128, 256 and 512 positions and their remainders,
rectangles cut by the map's edge, odd maps, channel counts off the 16-channel blocks, filter counts
off the multiples of 16 and over 256, odd numbers of tiles (the last CTA pair has half its work),
both strides, both types, the fused pool, an input-channel split.  The bar is the other conv tests'
(1e-4 of sum|W_hat||x| for fp32 I/O, 2e-3 for fp16); the fp32 cases also hold 4e-7 of the result in
the 2-norm: the fp16 pairs carry 22 bits (2^-23 a factor), each chain truncates nine sums and up to
32 of them are rounded once, 2e-7 in all, with a factor of two to spare."""
import ctypes

import numpy as np
import pytest
import torch

from conftest import cuda_cores_only
from oracle import conv as OC
from oracle import patterns as OP
from oracle import project as OPR
from paper_2003_06513_gb300 import _lib, api
from paper_2003_06513_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

TOL = {"f32": 1e-4, "f16": 2e-3}
NP = {"f32": np.float32, "f16": np.float16}


@pytest.fixture(autouse=True)
def _clean_status():
    yield
    torch.cuda.synchronize()
    st = ctypes.c_uint(0)
    assert _lib.load().pp_device_status(1, ctypes.byref(st)) == 0 and st.value == 0


def _layer(cout, cin, keep, stride, seed, patterns=None):
    rng = np.random.default_rng(seed)
    W = (rng.standard_normal((cout, cin, 3, 3)) * np.sqrt(2 / (9 * cin))).astype(np.float32)
    b = (rng.standard_normal(cout) * 0.1).astype(np.float32)
    return api.pp_pack(W, patterns, keep, 1, stride).bind("cuda"), W, b


def _check(y, x, W, b, keep, stride, pool, io, masks=None, idx=None):
    idx = list(range(x.shape[0])) if idx is None else idx
    Wh = OPR.project(W, masks if masks is not None else OP.default8(), keep)["W_hat"]
    xs = x[idx].astype(np.float64)
    ref, den = OC.conv_ref(xs, Wh, b, stride, True), OC.denominator(xs, Wh, b, stride)
    if pool:
        ref, den = OC.maxpool2x2(ref), OC.maxpool2x2(den)
    got = y[idx].double().cpu().numpy()
    err = OC.max_norm_err(got, ref, den)
    assert err <= TOL[io], f"max normalised error {err:.3e}"
    if io == "f32":
        rel = np.linalg.norm(got - ref) / np.linalg.norm(ref)
        assert rel <= 4e-7, f"relative error {rel:.3e}"


CASES = [  # cout, cin, n, h, w, keep, io, stride, pool
    (64, 64, 40, 32, 32, 0.5, "f32", 1, False),        # 512-position tiles
    (64, 128, 17, 61, 59, 0.4, "f32", 1, False),       # odd map, odd batch
    (96, 80, 9, 45, 61, 0.5, "f32", 1, False),         # 256-position tiles
    (150, 90, 9, 45, 61, 0.5, "f32", 1, False),        # 160 filters of 150, 96 channels of 90
    (40, 100, 60, 30, 30, 1.0, "f32", 1, False),       # 48 filters of 40
    (300, 77, 16, 29, 31, 0.5, "f32", 1, False),       # two chunks of 160 filters, 300 of 320
    (512, 144, 160, 7, 7, 0.5, "f32", 1, False),       # many images a tile
    (256, 64, 3, 57, 211, 0.5, "f32", 1, False),       # wide rows
    (128, 96, 64, 28, 28, 0.4, "f32", 2, False),       # stride 2, even map
    (72, 96, 64, 29, 27, 0.5, "f32", 2, False),        # stride 2, odd map
    (64, 64, 32, 56, 56, 0.5, "f32", 1, True),         # pool, 512-position rectangles
    (128, 64, 16, 50, 46, 0.5, "f32", 1, True),        # pool, rectangles cut by the edge
    (256, 72, 24, 29, 27, 0.5, "f32", 1, True),        # pool, odd map: last row and column dropped
    (64, 64, 64, 56, 56, 0.5, "f32", 2, True),         # pool at stride 2
    (16, 32, 64, 28, 28, 1.0, "f32", 1, False),        # MMAs of 16 columns
    (17, 64, 64, 28, 28, 1.0, "f32", 1, False),        # 32 filters of 17
    (17, 256, 64, 56, 56, 1.0, "f32", 2, False),
    (8, 64, 256, 56, 56, 1.0, "f16", 1, True),         # 16 filters of 8
    (256, 64, 16, 28, 28, 1.0, "f16", 1, False),
    (90, 70, 16, 45, 37, 0.5, "f16", 1, False),
    (128, 72, 64, 29, 27, 0.5, "f16", 2, False),
    (200, 96, 24, 28, 28, 0.5, "f16", 1, True),
]


@pytest.mark.parametrize("case", CASES)
def test_tensor_kernel_matches_oracle(case):
    cout, cin, n, h, w, keep, io, stride, pool = case
    layer, W, b = _layer(cout, cin, keep, stride, cin + w)
    x = WL.activations((n, cin, h, w), 7 + h, relu=True, dtype=NP[io])
    xt = torch.from_numpy(x).cuda()
    assert layer.tensor_plan(xt.shape, 0, pool, xt.dtype)["tensor"] == 1
    shape = layer.out_shape(xt.shape)
    if pool:
        shape = shape[:2] + (shape[2] // 2, shape[3] // 2)
    guard = torch.full((256 + int(np.prod(shape)) + 256,), float("nan"), dtype=xt.dtype, device="cuda")
    y = guard[256:-256].view(shape)
    layer.conv(xt, torch.from_numpy(b).cuda(), True, out=y, pool2x2=pool)
    assert torch.isnan(guard[:256]).all() and torch.isnan(guard[-256:]).all()
    _check(y, x, W, b, keep, stride, pool, io, idx=[0, n // 2, n - 1])


@pytest.mark.parametrize("case", [(512, 512, 1, 14, 14, 0.3, False), (512, 512, 1, 28, 28, 0.3, True),
                                  (256, 512, 4, 14, 14, 0.4, False), (300, 400, 1, 13, 17, 1.0, False)])
def test_tensor_split_of_the_input_channels(case):
    """Few tiles and a workspace: partial sums per channel range, with the products of the lo parts
    (the CUDA-core plan, itself split, rounds less than three products do), added by the reduction;
    the same result again."""
    cout, cin, n, h, w, keep, pool = case
    layer, W, b = _layer(cout, cin, keep, 1, 3 + h)
    x = WL.activations((n, cin, h, w), 4, relu=True)
    xt = torch.from_numpy(x).cuda()
    ws = torch.full((1 << 23,), float("nan"), device="cuda")
    plan = layer.tensor_plan(xt.shape, ws.numel() * 4, pool)
    assert plan["tensor"] == 1 and plan["splits"] > 1
    bt = torch.from_numpy(b).cuda()
    y = layer.conv(xt, bt, True, workspace=ws, pool2x2=pool)
    _check(y, x, W, b, keep, 1, pool, "f32")
    assert torch.equal(layer.conv(xt, bt, True, workspace=ws, pool2x2=pool), y)


def test_tensor_kernel_other_pattern_library():
    masks = [0x01B, 0x036, 0x0D8, 0x1B0]                 # the four 2x2 corners
    layer, W, b = _layer(128, 96, 0.5, 1, 8, masks)
    x = WL.activations((4, 96, 28, 28), 5, relu=True)
    xt = torch.from_numpy(x).cuda()
    assert layer.tensor_plan(xt.shape)["tensor"] == 1
    y = layer.conv(xt, torch.from_numpy(b).cuda(), True)
    _check(y, x, W, b, 0.5, 1, False, "f32", masks=masks)


def _sides(layer, W, x, stride, relu=False):
    """Outputs of the tensor-core and the CUDA-core kernel and the weights, no bias."""
    xt = torch.from_numpy(x).cuda()
    assert layer.tensor_plan(xt.shape)["tensor"] == 1
    a = layer.conv(xt, None, relu)
    c = cuda_cores_only(api.pp_pack(W, None, 0.5, 1, stride).bind("cuda")).conv(xt, None, relu)
    return a.double().cpu().numpy(), c.double().cpu().numpy()


@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("kind", ["1e20", "1e37", "1e-20", "halves", "channels", "images", "decay"])
def test_values_of_any_scale(kind, stride):
    """Scales the fp16 pairs cannot hold without a scale of their own, and mixtures no scale holds
    (those units are summed in fp32): each output within 2e-6 of its own sum|w||x|."""
    layer, W, _ = _layer(128, 96, 0.5, stride, 11)
    rng = np.random.default_rng(2)
    x = np.maximum(rng.standard_normal((12, 96, 40, 44)), 0)
    if kind.startswith("1e"):
        x = x * float(kind)
    elif kind == "halves":
        x[..., :22] *= 1e7
        x[..., 22:] *= 1e-7
    elif kind == "channels":
        x[:, ::2] *= 1e8
        x[:, 1::2] *= 1e-8
    elif kind == "images":
        x *= 10.0 ** rng.uniform(-15, 15, (12, 1, 1, 1))
    else:
        x = np.exp(-rng.uniform(0, 60, x.shape))
    x = x.astype(np.float32)
    got, _ = _sides(layer, W, x, stride)
    Wh = OPR.project(W, OP.default8(), 0.5)["W_hat"]
    idx = [0, 11]
    xs = x[idx].astype(np.float64)
    ref, den = OC.conv_ref(xs, Wh, None, stride, False), OC.denominator(xs, Wh, None, stride)
    assert np.all(np.abs(got[idx] - ref) <= 2e-6 * den + 1e-44)


@pytest.mark.parametrize("relu", [False, True])
def test_infinities_and_nan_reach_the_outputs_of_kept_taps_only(relu):
    layer, W, _ = _layer(128, 96, 0.5, 1, 12)
    x = WL.activations((8, 96, 40, 44), 3, relu=True)
    x[0, 5, 7, 9], x[3, 0, 0, 0], x[7, 95, 39, 43], x[2, 1, 20, 20] = np.inf, np.nan, -np.inf, 3e38
    a, c = _sides(layer, W, x, 1, relu)
    assert np.array_equal(np.isnan(a), np.isnan(c)) and np.array_equal(np.isinf(a), np.isinf(c))
    f = np.isfinite(c)
    assert np.allclose(a[f], c[f], rtol=1e-4, atol=1e-4 * np.abs(x[np.isfinite(x) & (x < 1e30)]).max())


def test_inputs_at_any_element_alignment():
    layer, W, b = _layer(64, 64, 0.5, 1, 13)
    x = WL.activations((16, 64, 40, 40), 6, relu=True)
    for dt, io in ((torch.float32, "f32"), (torch.float16, "f16")):
        buf = torch.zeros(x.size + 3, dtype=dt, device="cuda")
        xt = buf[3:].view(x.shape)
        xt.copy_(torch.from_numpy(x))
        y = layer.conv(xt, torch.from_numpy(b).cuda(), True)
        _check(y, xt.cpu().numpy(), W, b, 0.5, 1, False, io, idx=[0, 15])


def test_same_result_every_time():
    layer, _, b = _layer(256, 128, 0.4, 1, 14)
    xt = torch.from_numpy(WL.activations((16, 128, 28, 28), 6, relu=True)).cuda()
    bt = torch.from_numpy(b).cuda()
    first = layer.conv(xt, bt, True)
    for _ in range(3):
        assert torch.equal(layer.conv(xt, bt, True), first)


@pytest.mark.parametrize("case", [  # the CUDA-core kernel's schedules, without the tensor cores
    (256, 256, 8, 28, 0.3, "f32", False, 1), (512, 512, 32, 28, 0.3, "f32", True, 1),
    (128, 128, 16, 56, 0.3, "f32", False, 1), (128, 128, 64, 28, 1.0, "f32", False, 1),
    (512, 512, 32, 14, 0.3, "f32", False, 1), (128, 128, 16, 56, 0.4, "f32", False, 2),
    (256, 256, 11, 56, 0.3, "f16", False, 1), (256, 128, 8, 28, 0.4, "f16", False, 2)])
def test_cuda_core_kernel_without_tensor_binding(case):
    cout, cin, n, h, keep, io, pool, stride = case
    layer, W, b = _layer(cout, cin, keep, stride, 20 + h)
    cuda_cores_only(layer)
    x = WL.activations((n, cin, h, h), 30 + h, relu=True, dtype=NP[io])
    xt = torch.from_numpy(x).cuda()
    nb = layer.workspace_bytes(xt.shape, pool, xt.dtype)
    ws = torch.empty(max(nb // 4, 1), device="cuda") if nb else None
    y = layer.conv(xt, torch.from_numpy(b).cuda(), True, workspace=ws, pool2x2=pool)
    Wh = OPR.project(W, OP.default8(), keep)["W_hat"]
    idx = [0, n - 1]
    xs = x[idx].astype(np.float64)
    ref, den = OC.conv_ref(xs, Wh, b, stride, True), OC.denominator(xs, Wh, b, stride)
    if pool:
        ref, den = OC.maxpool2x2(ref), OC.maxpool2x2(den)
    assert OC.max_norm_err(y[idx].double().cpu().numpy(), ref, den) <= TOL[io]


def test_bind_tensor_errors():
    lib = _lib.load()
    layer, W, _ = _layer(32, 32, 0.5, 1, 15)
    n = layer.query("tensor_bytes")
    buf = torch.empty(n + 256, dtype=torch.uint8, device="cuda")
    p = lambda o=0: ctypes.c_void_p(buf.data_ptr() + o)
    assert lib.pp_bind_tensor(None, p(), n, None) == -1
    assert lib.pp_bind_tensor(layer._h, None, n, None) == -1
    assert lib.pp_bind_tensor(layer._h, p(), n - 1, None) == -9
    assert lib.pp_bind_tensor(layer._h, p(16), n, None) == -6
    assert lib.pp_bind_tensor(api.pp_pack(W, None, 0.5)._h, p(), n, None) == -8
    dw = api.pp_pack(W[:, :1], None, 1.0, 32).bind("cuda")
    assert dw.query("tensor_bytes") == 0 and lib.pp_bind_tensor(dw._h, p(), n, None) == -14


@pytest.mark.parametrize("case", [(64, 72, 5, 60, 100, False), (64, 64, 3, 57, 148, False), (128, 72, 7, 50, 112, False),
                                  (128, 40, 5, 80, 112, True), (64, 72, 9, 61, 100, True), (64, 72, 33, 33, 100, True)])
def test_tensor_kernel_takes_its_input_by_boxes(case):
    """Tensor copies of whole windows: tiles narrower than the rows and not, all shifts to the 16-byte
    boundary, a last block of 8 channels, an odd number of tiles; channels of other ranges make blocks
    be taken again.  x one element off the boundary takes single copies: the same values staged, so the
    same result, bit for bit.  An infinity reaches the outputs that it reaches on the CUDA cores."""
    cout, cin, n, h, w, pool = case
    layer, W, b = _layer(cout, cin, 0.5, 1, cin + w)
    x = WL.activations((n, cin, h, w), 7 + h, relu=True, dtype=np.float32)
    x[:, 16:32] *= np.float32(2.0 ** 14)
    x[n // 2, :16] *= np.float32(2.0 ** -12)
    bt = torch.from_numpy(b).cuda()
    xt = torch.from_numpy(x).cuda()
    assert layer.tensor_plan(xt.shape, 0, pool)["boxes"] == 1
    y = layer.conv(xt, bt, True, pool2x2=pool)
    _check(y, x, W, b, 0.5, 1, pool, "f32", idx=[0, n // 2, n - 1])
    off = torch.empty(xt.numel() + 1, device="cuda")[1:].view(xt.shape).copy_(xt)
    assert torch.equal(layer.conv(off, bt, True, pool2x2=pool), y)
    xt[n - 1, cin - 1, h - 1, w - 2] = float("inf")
    y = layer.conv(xt, bt, False, pool2x2=pool)
    ref = cuda_cores_only(layer).conv(xt, bt, False, pool2x2=pool)
    assert torch.equal(torch.isfinite(y), torch.isfinite(ref)) and not torch.isfinite(y).all()


@pytest.mark.parametrize("dtype,cin,h,tile_w,boxes", [(torch.float16, 16, 28, 0, 0), (torch.float16, 16, 30, 30, 0),
                                                      (torch.float32, 32, 28, 28, 1), (torch.float32, 32, 30, 30, 0)])
def test_units_of_one_or_two_blocks_back_to_back(dtype, cin, h, tile_w, boxes):
    """The shortest units and epilogues (16 filters, one or two 16-channel blocks), one unit a CTA pair:
    a pair ends while the arrivals of its last commits are still under way, and the next launch takes
    over its shared memory at once.  Every launch gives the same bits."""
    layer, W, b = _layer(16, cin, 1.0, 1, 21)
    x = WL.activations((64, cin, h, h), 22, relu=True, dtype=NP["f32" if dtype == torch.float32 else "f16"])
    xt = torch.from_numpy(x).cuda()
    plan = layer.tensor_plan(xt.shape, 0, False, dtype)
    assert (plan["tensor"], plan["tile_w"], plan["boxes"]) == (1, tile_w, boxes) and plan["units"] <= 76
    bt = torch.from_numpy(b).cuda()
    first = layer.conv(xt, bt, True)
    _check(first, x, W, b, 1.0, 1, False, "f32" if dtype == torch.float32 else "f16", idx=[0, 63])
    outs = [torch.empty_like(first) for _ in range(4)]
    for i in range(200):
        layer.conv(xt, bt, True, out=outs[i % 4])
    assert all(torch.equal(o, first) for o in outs)


@pytest.mark.parametrize("w,boxes", [(30, 0), (32, 1)])
def test_both_ctas_of_a_pair_use_their_own_scales(w, boxes):
    """Three tiles an image, so every second pair's tiles belong to two images, whose inputs are up to
    2^40 apart: each CTA sums its blocks with the scales that its own staging warps published.  Each
    image within the 2-norm bound of its own result; the same bits every time."""
    layer, W, _ = _layer(64, 64, 0.5, 1, 23)
    x = WL.activations((33, 64, 45, w), 24, relu=True)
    s = 2.0 ** np.random.default_rng(25).integers(-20, 21, 33)
    x = (x * s[:, None, None, None]).astype(np.float32)
    xt = torch.from_numpy(x).cuda()
    plan = layer.tensor_plan(xt.shape)
    assert (plan["tensor"], plan["tile_w"], plan["tile_h"], plan["boxes"]) == (1, w, 15, boxes)
    first = layer.conv(xt, None, True)
    for i in (0, 1, 2, 15, 16, 31, 32):
        _check(first, x, W, np.zeros(64, np.float32), 0.5, 1, False, "f32", idx=[i])
    assert all(torch.equal(layer.conv(xt, None, True), first) for _ in range(50))


def test_misaligned_workspace_that_only_the_tensor_core_plan_would_split_into():
    """The tensor-core plan splits here and the CUDA-core plan does not: a workspace off the 16-byte
    boundary is left alone, as it always was, and the call runs on the CUDA cores."""
    layer, W, b = _layer(24, 400, 1.0, 1, 26)
    x = WL.activations((202, 400, 8, 4), 27, relu=True, dtype=np.float16)
    xt, bt = torch.from_numpy(x).cuda(), torch.from_numpy(b).cuda()
    ws = torch.full((1 << 22,), float("nan"), device="cuda")
    nb = 4 * (ws.numel() - 1)
    assert layer.tensor_plan(xt.shape, nb, False, xt.dtype)["splits"] > 1
    assert layer.plan(xt.shape, nb, False, xt.dtype)["splits"] == 1
    y = layer.conv(xt, bt, True, workspace=ws[1:])
    assert torch.isnan(ws).all()
    _check(y, x, W, b, 1.0, 1, False, "f16", idx=[0, 201])
    assert torch.equal(y, cuda_cores_only(layer).conv(xt, bt, True))


REDO = [  # cout, cin, n, h, w, keep, io, stride, pool, workspace: what the pairs do not hold, by tile and epilogue
    (64, 72, 5, 60, 100, 0.5, "f32", 1, False, False),     # 512 positions, boxes, a last block of 8 channels
    (64, 72, 9, 61, 100, 0.5, "f32", 1, True, False),      # pooled, an odd row dropped
    (64, 128, 17, 61, 59, 0.4, "f32", 1, False, False),    # copies
    (96, 80, 9, 45, 61, 0.5, "f32", 1, False, False),      # 256 positions
    (128, 64, 16, 50, 46, 0.5, "f32", 1, True, False),     # pooled, rectangles cut by the edge
    (256, 72, 24, 29, 27, 0.5, "f32", 1, True, False),     # pooled, 128 positions
    (300, 77, 16, 29, 31, 0.5, "f32", 1, False, False),    # two chunks of filters
    (72, 96, 64, 29, 27, 0.5, "f32", 2, False, False),     # parity planes of an odd map
    (64, 64, 64, 56, 56, 0.5, "f32", 2, True, False),
    (256, 512, 4, 14, 14, 0.4, "f32", 1, False, True),     # a split: partial sums again
    (512, 512, 1, 28, 28, 0.3, "f32", 1, True, True),      # ... pooled by the reduction
    (200, 96, 24, 28, 28, 0.5, "f16", 1, True, False),
    (128, 72, 64, 29, 27, 0.5, "f16", 2, False, False),
]


@pytest.mark.parametrize("case", REDO)
def test_units_summed_again(case):
    """An infinity and a NaN in some units and (fp32) halves of images 2^47 apart in all: what
    reaches an output is what reaches it on the CUDA cores, and the finite ones lie within 2e-6 of
    their own sum |w||x| (fp16 outputs: 2e-3)."""
    cout, cin, n, h, w, keep, io, stride, pool, split = case
    layer, W, b = _layer(cout, cin, keep, stride, cin + w)
    x = WL.activations((n, cin, h, w), 7 + h, relu=True, dtype=np.float32)
    if io == "f32":
        x[..., : w // 2] *= np.float32(1e7)
        x[..., w // 2:] *= np.float32(1e-7)
    x = x.astype(NP[io])
    ws = torch.empty(1 << 23, device="cuda") if split else None
    xt, bt = torch.from_numpy(x).cuda(), torch.zeros(cout, device="cuda")
    plan = layer.tensor_plan(xt.shape, 0 if ws is None else ws.numel() * 4, pool, xt.dtype)
    assert plan["tensor"] == 1 and (plan["splits"] > 1) == split
    Wh = OPR.project(W, OP.default8(), keep)["W_hat"]

    def within(y, idx):
        xs = x[idx].astype(np.float64)
        ref, den = OC.conv_ref(xs, Wh, None, stride, False), OC.denominator(xs, Wh, None, stride)
        if pool:
            ref, den = OC.maxpool2x2(ref), OC.maxpool2x2(den)
        return np.all(np.abs(y[idx].double().cpu().numpy() - ref) <= (2e-6 if io == "f32" else 2e-3) * den + 1e-44)

    assert within(layer.conv(xt, bt, False, pool2x2=pool, workspace=ws), [0, n - 1])
    xt[0, cin - 1, h - 2, 1], xt[n // 2, 0, 0, 0], xt[n - 1, cin // 2, h // 2, w // 2] = float("inf"), float("nan"), float("-inf")
    got = layer.conv(xt, bt, False, pool2x2=pool, workspace=ws)
    ref = cuda_cores_only(layer).conv(xt, bt, False, pool2x2=pool)
    assert torch.equal(torch.isnan(got), torch.isnan(ref)) and torch.equal(torch.isinf(got), torch.isinf(ref))
    assert not torch.isfinite(got).all()
    if n > 2:
        assert within(got, [1])


def test_one_infinity_costs_a_bounded_time():
    """512 channels of one unit summed again take 6.4 times the CUDA-core kernel's whole call (1200 of
    187 us); 12 times is the bar (by a thread a position, from global memory, it was 115 times)."""
    layer, _, _ = _layer(512, 512, 0.3, 1, 28)
    other = cuda_cores_only(_layer(512, 512, 0.3, 1, 28)[0])
    xt = torch.from_numpy(WL.activations((32, 512, 14, 14), 29, relu=True)).cuda()
    xt[0, 3, 2, 2] = float("inf")
    assert layer.tensor_plan(xt.shape)["tensor"] == 1

    def time(lay):
        lay.conv(xt, None, True)
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        ev[0].record()
        for _ in range(3):
            lay.conv(xt, None, True)
        ev[1].record()
        torch.cuda.synchronize()
        return ev[0].elapsed_time(ev[1])

    assert time(layer) < 12 * time(other)


@pytest.mark.parametrize("below", [20, 24, 28, 30, 32, 36, 44])
@pytest.mark.parametrize("w,boxes", [(36, 1), (38, 0)])
def test_small_halves_beside_large_ones(w, boxes, below):
    """Half of each row holds one constant, 2^-20 to 2^-44 of the other half's values, and the block
    before leaves the scale at the low end of what is kept: outputs of the small half within 2e-6 of
    their own sum |w||x|.  (The constant's bits are what its pair loses, the same way in every product.)"""
    layer, W, _ = _layer(64, 64, 0.5, 1, 30)
    rng = np.random.default_rng(31)
    x = np.maximum(rng.standard_normal((33, 64, 42, w)), 0).clip(0, 3.9)
    x[:, :16, ::3, 0] = 3.99                             # the first block's largest 2^1.99, the others' 2^-0.97
    x[:, 16:] = x[:, 16:].clip(0, 0.51)
    x[:, :16, :, w // 2:] = 0
    x[:, 16:, :, w // 2:] = 1.2345678 * 2.0 ** -below
    x = x.astype(np.float32)
    xt = torch.from_numpy(x).cuda()
    plan = layer.tensor_plan(xt.shape)
    assert (plan["tensor"], plan["boxes"]) == (1, boxes)
    got = layer.conv(xt, None, False)[[0, 32]].double().cpu().numpy()
    Wh = OPR.project(W, OP.default8(), 0.5)["W_hat"]
    xs = x[[0, 32]].astype(np.float64)
    ref, den = OC.conv_ref(xs, Wh, None, 1, False), OC.denominator(xs, Wh, None, 1)
    err = np.max(np.abs(got - ref) / den)
    assert err <= 2e-6, f"{err:.2e}"


@pytest.mark.parametrize("io", ["f32", "f16"])
@pytest.mark.parametrize("below", [24, 28, 32, 40, 56])
def test_small_weights_beside_large_ones(below, io):
    """One channel's weights are 2^-24 to 2^-56 of the others', and in half of each row that channel
    alone has inputs: outputs there within 2e-6 of their own sum |w||x| (fp16 outputs, scaled into
    range: 1e-3)."""
    rng = np.random.default_rng(32)
    W = (rng.standard_normal((64, 64, 3, 3)) * np.sqrt(2 / (9 * 64))).astype(np.float32)
    W[:, 5] *= np.float32(2.0 ** -below)
    x = np.maximum(rng.standard_normal((40, 64, 32, 32)), 0)
    x[..., 16:] = 0
    if io == "f16":
        W *= np.float32(2.0 ** 24)
        x[..., :16] *= 2.0 ** -24
    x[:, 5, :, 16:] = 1.2345678
    x = x.astype(NP[io])
    layer = api.pp_pack(W, None, 1.0).bind("cuda")
    xt = torch.from_numpy(x).cuda()
    assert layer.tensor_plan(xt.shape, 0, False, xt.dtype)["tensor"] == 1
    got = layer.conv(xt, None, False)[[0, 39]].double().cpu().numpy()
    Wh = OPR.project(W, OP.default8(), 1.0)["W_hat"]
    xs = x[[0, 39]].astype(np.float64)
    ref, den = OC.conv_ref(xs, Wh, None, 1, False), OC.denominator(xs, Wh, None, 1)
    err = np.max(np.abs(got - ref) / np.maximum(den, 1e-37 if io == "f32" else 6e-5))
    assert err <= (2e-6 if io == "f32" else 1e-3), f"{err:.2e}"


@pytest.mark.parametrize("cin,n,h,stride,split,io", [(256, 32, 28, 1, False, "f32"), (192, 32, 57, 2, False, "f32"),
                                                     (256, 32, 28, 1, False, "f16"), (512, 1, 28, 1, True, "f16")])
def test_integers_are_summed_exactly(cin, n, h, stride, split, io):
    """Weights of a few bits and whole inputs, sums under 2^24: every output is the exact sum (fp16: its
    rounding), as on the CUDA cores."""
    rng = np.random.default_rng(33)
    W = (rng.integers(-8, 9, (256, cin, 3, 3)) / 16).astype(np.float32)
    x = rng.integers(0, 256 if io == "f32" else 16, (n, cin, h, h)).astype(NP[io])
    layer = api.pp_pack(W, None, 0.4, 1, stride).bind("cuda")
    xt = torch.from_numpy(x).cuda()
    ws = torch.empty(1 << 23, device="cuda") if split else None
    plan = layer.tensor_plan(xt.shape, 0 if ws is None else ws.numel() * 4, False, xt.dtype)
    assert plan["tensor"] == 1 and (plan["splits"] > 1) == split
    y = layer.conv(xt, None, False, workspace=ws)
    Wh = OPR.project(W, OP.default8(), 0.4)["W_hat"]
    idx = [0, n - 1] if n > 1 else [0]
    ref = OC.conv_ref(x[idx].astype(np.float64), Wh, None, stride, False)
    assert np.abs(ref).max() * 16 < 2 ** 24
    assert np.array_equal(y[idx].cpu().numpy(), ref.astype(NP[io]))


@pytest.mark.parametrize("case,tensor", [  # cout, cin, n, h, w, keep, stride
    ((27, 193, 52, 36, 36, 1.0, 2), 0), ((413, 413, 5, 28, 30, 0.3, 2), 0), ((512, 512, 4, 14, 14, 0.3, 1), 0),
    ((256, 256, 16, 28, 28, 0.4, 2), 0),               # few units on the balanced schedule: 1.01 to 1.12 times
    ((64, 64, 8, 112, 112, 0.3, 1), 1), ((256, 256, 64, 28, 28, 0.4, 2), 1), ((150, 90, 9, 45, 61, 0.5, 1), 1)])
def test_the_route_rounds_no_more_than_the_cuda_cores(case, tensor):
    """2-norm error against 64 bits of the whole output, with the workspace the call asks for."""
    cout, cin, n, h, w, keep, stride = case
    layer, W, b = _layer(cout, cin, keep, stride, 34)
    xt = torch.from_numpy(WL.activations((n, cin, h, w), 35, relu=True)).cuda()
    bt = torch.from_numpy(b).cuda()
    nb = layer.workspace_bytes(xt.shape)
    ws = torch.empty(nb // 4 + 4, device="cuda") if nb else None
    assert layer.tensor_plan(xt.shape, nb)["tensor"] == tensor
    Wh = torch.from_numpy(OPR.project(W, OP.default8(), keep)["W_hat"].astype(np.float64)).cuda()
    ref = torch.nn.functional.conv2d(xt.double(), Wh, bt.double(), stride, 1).relu_()

    def err(lay):
        y = lay.conv(xt, bt, True, workspace=ws).double()
        return (torch.linalg.vector_norm(y - ref) / torch.linalg.vector_norm(ref)).item()

    assert err(layer) <= err(cuda_cores_only(layer))

"""GPU parity of the quantizer's tile forms and of a layer step's fused passes, at the sizes
where they differ: whole and partial tiles, aligned rows, rows that start anywhere, an
unaligned base, padded rows, tile widths of 128, 64 and 32 columns, folded range passes, and
the layer step's launches against the same step made of single library calls."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2411_10948_gb300 import layer as L
from paper_2411_10948_gb300 import native as N
from parity_util import compare_shift, decode, f32_bits, folded

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2411_10948_gb300 import build
    build.build_library()
    N.load()


def gradient_like(rng, R, C):
    s = np.exp(rng.normal(0, 1.5, C)).astype(np.float32)
    s[rng.random(C) < 0.02] *= 100
    return (rng.standard_normal((R, C)) * s).astype(np.float32)


def place(a, how):
    """a on the device: dense, with rows padded to a multiple of four (and one quad more), or
    dense from an address that is not 16-byte aligned."""
    R, C = a.shape
    t = torch.from_numpy(np.ascontiguousarray(a))
    if how == "padded":
        buf = torch.full((R, (C + 3) // 4 * 4 + 4), 7e8, dtype=torch.float32, device="cuda")
        buf[:, :C] = t.cuda()
        return buf[:, :C]
    if how == "offset":
        buf = torch.full((R * C + 1,), 7e8, dtype=torch.float32, device="cuda")
        buf[1:] = t.cuda().flatten()
        return buf[1:].view(R, C)
    return t.cuda()


# 128-, 64- and 32-column tiles (128 / 130, 64, 147 and 33 columns), whole tiles and tiles with
# one row or column more or less, odd and even row strides, few rows, one column
SHAPES = [(64, 128), (65, 128), (128, 256), (63, 130), (129, 131), (256, 64), (300, 63),
          (512, 147), (513, 147), (257, 33), (700, 161), (200, 1155), (5, 3), (3, 515), (9, 1)]


@pytest.mark.parametrize("how", ["dense", "padded", "offset"])
@pytest.mark.parametrize("mode", [N.SQ_ROUND_NEAREST_EVEN, N.SQ_ROUND_STOCHASTIC])
@pytest.mark.parametrize("transposed", [True, False])
def test_tile_forms_match_oracle(how, mode, transposed):
    rng = np.random.default_rng(5)
    for R, C in SHAPES:
        x = gradient_like(rng, R, C)
        for bits in (4, 6):
            q = L.ShiftTensor.alloc(R, C, bits, 4, "cuda", transposed)
            status = torch.zeros(1, dtype=torch.int32, device="cuda")
            L.shift_quantize(place(x, how), q, bits, 4, mode, 77, status)
            assert int(status.item()) == 0
            compare_shift(q, O.shiftquant_tensor(x, bits, 4, mode, 77), f"{R}x{C} {how} b{bits}")


@pytest.mark.parametrize("how", ["dense", "padded", "offset"])
def test_weight_tile_forms_match_oracle(how):
    rng = np.random.default_rng(6)
    for K, C in SHAPES:
        w = gradient_like(rng, K, C)
        w[:, 0] = 0.0       # a zero column and a zero row: the path of zero scales
        w[K // 2] = 0.0
        xe = rng.integers(0, 4, K).astype(np.uint8)
        ge = rng.integers(0, 4, C).astype(np.uint8)
        for bits in (4, 6):
            wf = L.ChannelTensor(L.empty_codes(C, K, bits, 4, "cuda"),
                                 torch.zeros(C, device="cuda"), torch.zeros(C, device="cuda"))
            wd = L.ChannelTensor(L.empty_codes(K, C, bits, 4, "cuda"),
                                 torch.zeros(K, device="cuda"), torch.zeros(K, device="cuda"))
            status = torch.zeros(1, dtype=torch.int32, device="cuda")
            L.weight_quantize_both(place(w, how), wf, wd, torch.from_numpy(xe).cuda(),
                                   torch.from_numpy(ge).cuda(), bits, 4, status)
            of, od = O.channel_tensor(w, bits, 0), O.channel_tensor(w, bits, 1)
            what = f"{K}x{C} {how} b{bits}"
            np.testing.assert_array_equal(decode(wf.codes), folded(of["codes"], xe, 4, 0).T, what)
            np.testing.assert_array_equal(decode(wd.codes), folded(od["codes"], ge, 4, 1), what)
            np.testing.assert_array_equal(f32_bits(wf.scale.cpu().numpy()), f32_bits(of["scale"]), what)
            np.testing.assert_array_equal(f32_bits(wd.scale.cpu().numpy()), f32_bits(od["scale"]), what)


@pytest.mark.parametrize("tiny", [1e-37, 3e-38, 1.2e-38])
def test_scales_without_room_for_the_group_shift_match_oracle(tiny):
    # Q / tau_0 near the largest float: 2^e Q / tau_0 overflows and the two factors stay apart
    rng = np.random.default_rng(8)
    x = (gradient_like(rng, 130, 131) * np.float32(1e-3)).astype(np.float32)
    x = (x / np.abs(x).max()).astype(np.float32) * np.float32(tiny)
    for bits in (4, 8):
        for mode in (0, 1):
            q = L.ShiftTensor.alloc(130, 131, bits, 8 if bits == 4 else 5, "cuda")
            status = torch.zeros(1, dtype=torch.int32, device="cuda")
            G = 8 if bits == 4 else 5
            L.shift_quantize(place(x, "dense"), q, bits, G, mode, 3, status)
            compare_shift(q, O.shiftquant_tensor(x, bits, G, mode, 3), f"{tiny} b{bits} m{mode}")


def layer_state(lay):
    out = {"y": lay.y, "dx": lay.dx, "dw": lay.dw, "status": lay.status}
    for n, q in (("x", lay.x), ("g", lay.g)):
        out.update({n + ".codes": q.codes, n + ".exp": q.exp, n + ".range": q.range,
                    n + ".tau0": q.tau0, n + ".scale": q.scale})
        if q.codes_t is not None:
            out[n + ".codes_t"] = q.codes_t
    for n, c in (("wf", lay.wf), ("wd", lay.wd)):
        out.update({n + ".codes": c.codes, n + ".range": c.range, n + ".scale": c.scale})
    return out


# one launch for the codes (up to 1216 blocks) and one per tensor; aligned and odd rows
@pytest.mark.parametrize("M,K,Nn", [(192, 320, 288), (1000, 147, 513), (7, 5, 3), (130, 1155, 64),
                                    (8192, 1024, 512), (8001, 1023, 515), (20000, 64, 96)])
@pytest.mark.parametrize("bits,transposed", [(4, False), (6, True)])
@pytest.mark.parametrize("data", ["random", "zero", "nan"])
def test_layer_step_passes_equal_the_single_calls(M, K, Nn, bits, transposed, data):
    gen = torch.Generator(device="cuda").manual_seed(M + K)
    x = torch.randn((M, K), generator=gen, device="cuda")
    w = torch.randn((K, Nn), generator=gen, device="cuda") * 0.02
    dy = torch.randn((M, Nn), generator=gen, device="cuda")
    dy *= torch.randn(Nn, generator=gen, device="cuda").mul_(2).exp_()
    if data == "zero":
        x.zero_()
        w[:, 1] = 0
    if data == "nan":
        dy[M // 2, Nn // 2] = float("nan")
    got = []
    for ws in (True, False):   # without a workspace the step is made of single library calls
        lay = L.QuantLinear(M, K, Nn, bits, 4, "cuda", transposed=transposed, use_workspace=ws)
        for _ in range(2):     # the second on the accumulators and workspace of the first
            N.shiftquant_layer_step(lay.step_args(x, w, dy), 0xABC)
        torch.cuda.synchronize()
        got.append(layer_state(lay))
    assert int(got[0]["status"].item()) == (N.SQ_DEV_NONFINITE if data == "nan" else 0)
    for k in got[0]:
        a, b = got[0][k], got[1][k]
        if a.dtype == torch.bfloat16:
            a, b = a.float(), b.float()
        np.testing.assert_array_equal(a.cpu().numpy(), b.cpu().numpy(), err_msg=k)


def test_layer_step_in_a_graph_and_on_two_streams():
    # captured once and replayed on refilled inputs, and two steps with their own buffers on
    # two streams at a time: the same results as plain calls
    M, K, Nn, bits = 1500, 320, 512, 6
    gen = torch.Generator(device="cuda").manual_seed(4)
    ins = [(torch.randn((M, K), generator=gen, device="cuda"),
            torch.randn((K, Nn), generator=gen, device="cuda") * 0.02,
            torch.randn((M, Nn), generator=gen, device="cuda")) for _ in range(2)]
    want = []
    for x, w, dy in ins:
        lay = L.QuantLinear(M, K, Nn, bits, 4, "cuda")
        N.shiftquant_layer_step(lay.step_args(x, w, dy), 9)
        torch.cuda.synchronize()
        want.append((lay.y.clone(), lay.dx.clone(), lay.dw.clone()))
    buf = [t.clone() for t in ins[0]]
    lay = L.QuantLinear(M, K, Nn, bits, 4, "cuda")
    args = lay.step_args(*buf)
    graph = L.CapturedStep(lambda: N.shiftquant_layer_step(args, 9))
    for i in (1, 0):
        for t, s in zip(buf, ins[i]):
            t.copy_(s)
        graph.replay()
        torch.cuda.synchronize()
        for a, b in zip((lay.y, lay.dx, lay.dw), want[i]):
            assert torch.equal(a, b)
    lays = [L.QuantLinear(M, K, Nn, bits, 4, "cuda") for _ in range(2)]
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(5):
        for l, s, t in zip(lays, streams, ins):
            N.shiftquant_layer_step(l.step_args(*t), 9, stream=s)
    torch.cuda.synchronize()
    for l, wnt in zip(lays, want):
        for a, b in zip((l.y, l.dx, l.dw), wnt):
            assert torch.equal(a, b)

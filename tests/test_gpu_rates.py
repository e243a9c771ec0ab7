"""Rates that hold between shapes and between calls: what a width costs next to one beside it, and
what an output costs on top of a launch."""
import pytest
import torch

from paper_2411_10948_gb300 import layer as L
from paper_2411_10948_gb300 import native as N

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2411_10948_gb300 import build
    build.build_library()
    N.load()


def time_per_element(C, bits, mode):
    """ps an element: graph replays of calls on three tensors in turn, larger than L2 together."""
    M, n = 30_000_000 // C, 24
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    sets = []
    for _ in range(3):
        x, q = torch.randn(M, C, device="cuda"), L.ShiftTensor.alloc(M, C, bits, 4, "cuda", False)
        N.shiftquant_calibrate(x, N.SQ_GRAN_SHIFT, 4, q.range, q.tau0, q.exp, st)
        sets.append((x, q))
    g = L.CapturedStep(lambda: [N.shiftquant_quantize(x, N.SQ_GRAN_SHIFT, bits, 4, q.tau0, q.exp, None, mode, 5,
                                                      q.codes, None, q.scale) for x, q in sets * (n // 3)])
    for _ in range(3):
        g.replay()
    ts = []
    for _ in range(15):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        g.replay()
        b.record()
        b.synchronize()
        ts.append(a.elapsed_time(b) / n * 1e9 / (M * C))
    return sorted(ts)[len(ts) // 2]


# Rows of 292 and 420 fp32 start and end inside a sector, and so do their BF16 codes (the code
# rows are padded to 16 bytes); rows of 288 and 416 do not.  What the shared sectors cost is at
# most one more sector of 37 (53) read and one partly written of 19 (27): 4% of the bytes.  Three
# times that is allowed (read twice in every tile they took 25-30% longer).
@pytest.mark.parametrize("ragged,whole", [(292, 288), (420, 416)])
def test_rows_that_share_sectors(ragged, whole):
    r, w = (time_per_element(C, 8, N.SQ_ROUND_NEAREST_EVEN) for C in (ragged, whole))
    assert r <= 1.12 * w, (r, w)


def time_per_row_codes(K, C):
    """us a call: a weight's per-in-channel codes, graph replays."""
    n, st = 48, torch.zeros(1, dtype=torch.int32, device="cuda")
    w = torch.randn(K, C, device="cuda")
    d = L.ChannelTensor(L.empty_codes(K, C, 8, 4, "cuda"), torch.zeros(K, device="cuda"), torch.zeros(K, device="cuda"))
    N.shiftquant_calibrate(w, N.SQ_GRAN_PER_ROW, 4, d.range, None, None, st)
    g = L.CapturedStep(lambda: [N.shiftquant_quantize(w, N.SQ_GRAN_PER_ROW, 8, 4, d.range, None, None,
                                                      N.SQ_ROUND_NEAREST_EVEN, 0, d.codes, None, d.scale)
                                for _ in range(n)])
    for _ in range(3):
        g.replay()
    ts = []
    for _ in range(15):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        g.replay()
        b.record()
        b.synchronize()
        ts.append(a.elapsed_time(b) / n * 1e3)
    return sorted(ts)[len(ts) // 2]


# 300 rows end inside a tile of 64 rows, 320 do not: the same tiles, the last one partly used (as
# long as a tile's rows past the tensor's end counted as rows of zeros, it took twice the time)
def test_last_row_tile_of_a_weight():
    r, w = time_per_row_codes(300, 256), time_per_row_codes(320, 256)
    assert r <= 1.3 * w, (r, w)


# The column maxima of Y and dX are one more pass over boxes that are staged anyway: the launch
# may take half as long again, not twice (as with a test of each box's way out per element)
def test_layer_launch_with_ranges():
    M, K, C, bits = 12544, 2304, 256, 6
    lay = L.QuantLinear(M, K, C, bits, 4)
    g = torch.Generator(device="cuda").manual_seed(1)
    for q, n in ((lay.x, K), (lay.g, C)):
        L.shift_quantize(torch.randn((M, n), generator=g, device="cuda"), q, bits, 4, 0, 0, lay.status)
    ws = torch.zeros(N.shiftquant_gemm_layer_workspace_bytes(M, K, C, bits, 4), dtype=torch.uint8, device="cuda")
    yr, dr = torch.zeros(C, device="cuda"), torch.zeros(K, device="cuda")

    def launch(**ranges):
        N.shiftquant_gemm_layer(lay.x.codes, lay.x.codes_t, lay.x.scale, lay.x.exp, lay.g.codes, lay.g.codes_t,
                                lay.g.scale, lay.g.exp, lay.wf.codes, lay.wf.scale, lay.wd.codes, lay.wd.scale,
                                M, K, C, bits, 4, lay.y, lay.dx, lay.dw, workspace=ws, dev_status=lay.status, **ranges)

    times = []
    for kw in ({}, {"y_range": yr, "dx_range": dr}):
        run = L.CapturedStep(lambda: [launch(**kw) for _ in range(8)])
        ts = []
        for _ in range(15):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            run.replay()
            b.record()
            b.synchronize()
            ts.append(a.elapsed_time(b))
        times.append(sorted(ts)[len(ts) // 2])
    assert lay.status.item() == 0
    assert times[1] <= 1.5 * times[0], times


# Rows of 300 codes end inside a chunk of sixteen, which goes code by code; with few rows of them a
# thread must not take eight, one after another (three times as long as rows of whole chunks)
def test_few_ragged_rows_pack_and_unpack():
    def calls(C):
        M, n, st = 1000, 48, torch.zeros(1, dtype=torch.int32, device="cuda")
        codes, back = (L.empty_codes(M, C, 4, 4, "cuda").zero_() for _ in range(2))
        packed = torch.zeros((M, (C + 1) // 2 + 15 & ~15), dtype=torch.uint8, device="cuda")
        g = L.CapturedStep(lambda: [(N.shiftquant_pack_codes(codes, 4, 4, packed, st),
                                     N.shiftquant_unpack_codes(packed, C, 4, 4, back)) for _ in range(n)])
        ts = []
        for _ in range(15):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            g.replay()
            b.record()
            b.synchronize()
            ts.append(a.elapsed_time(b) / n * 1e3)
        return sorted(ts)[len(ts) // 2]

    ragged, whole = calls(300), calls(304)
    assert ragged <= 2.2 * whole, (ragged, whole)

"""Kernels launched behind the kernel that writes their inputs (programmatic stream
serialization) read those inputs by coherent loads.  Shown by reading the sources, which needs
no GPU: the read-only path is left to data that nothing writes while the kernel is resident.
On the GPU, chains issued without a pause against the same calls with one after each."""
import os
import re

import numpy as np
import pytest
import torch

from paper_2411_10948_gb300 import layer as L
from paper_2411_10948_gb300 import native as N

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_10948_gb300", "csrc")

# (file, pointer read): inputs complete before the kernel ahead of the reader lets it launch --
# x of the range and L1 batch norm passes, x's codes of an earlier L1 batch norm call
READ_ONLY = {("sq_quant.cu", "t.x + t.R * t.ld + c0 + k"), ("sq_quant.cu", "row + c"),
             ("sq_quant.cu", "row + cc"), ("sq_quant.cu", "reinterpret_cast<const float4*>(row + cc)"),
             ("sq_l1bn.cu", "p + j"), ("sq_l1bn.cu", "reinterpret_cast<const unsigned int*>(p)")}


def sources():
    for f in sorted(os.listdir(CSRC)):
        s = open(os.path.join(CSRC, f)).read()
        yield f, re.sub(r"//[^\n]*", "", s)


def argument(s, at):
    """The parenthesised argument that starts at s[at] == '('."""
    depth = 0
    for i in range(at, len(s)):
        depth += {"(": 1, ")": -1}.get(s[i], 0)
        if depth == 0:
            return " ".join(s[at + 1:i].split())


def test_read_only_loads_are_of_unchanging_inputs():
    for f, s in sources():
        assert "ld.global.nc" not in s, f
        for m in re.finditer(r"__ldg\(", s):
            assert (f, argument(s, m.end() - 1)) in READ_ONLY, (f, argument(s, m.end() - 1))


def test_early_launched_kernels_take_unrestricted_inputs():
    seen = 0
    for f, s in sources():
        for part in re.split(r"\b__global__\b", s)[1:]:
            body = part[:part.index("\n}")]
            if "griddep_wait" not in body:
                continue
            seen += 1
            assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", body), (f, body[:200])
    assert seen >= 15   # (the GEMM, quantizer, packing and normalization kernels)


@pytest.fixture(scope="module")
def lib():
    from paper_2411_10948_gb300 import build
    build.build_library()
    N.load()


# X's exponents, tau_0 and scale (and the weight's scales) side by side in one buffer, as a
# caller may pack them: 48 channels, so that a scale shares a sector with the exponents
@pytest.mark.gpu
@pytest.mark.parametrize("bits", [4, 8])
def test_chain_with_shared_sectors(lib, bits):
    M, K, C, G, dev = 1000, 48, 96, 4, "cuda"
    gen = torch.Generator(device=dev).manual_seed(bits)
    st = torch.zeros(1, dtype=torch.int32, device=dev)
    small = torch.zeros(1024, dtype=torch.uint8, device=dev)
    exp, tau, scale = small[:K], small[K:K + 4].view(torch.float32), small[K + 4:K + 8].view(torch.float32)
    rng = torch.zeros(K, device=dev)
    qx, qy = L.empty_codes(M, K, bits, G, dev), L.empty_codes(M, C, bits, G, dev)
    w = L.ChannelTensor(L.empty_codes(C, K, bits, G, dev), torch.zeros(C, device=dev),
                        small[256:256 + 4 * C].view(torch.float32))
    y = torch.zeros((M, C), device=dev)
    e0, t0, s0 = (torch.zeros(C, dtype=torch.uint8, device=dev), torch.full((1,), 64.0, device=dev),
                  torch.zeros(1, device=dev))
    xs = [torch.randn((M, K), generator=gen, device=dev) * torch.exp(torch.randn(K, generator=gen, device=dev))
          for _ in range(6)]
    ws = [torch.randn((K, C), generator=gen, device=dev) for _ in xs]

    def chain(x, wt, pause):
        steps = [lambda: N.shiftquant_calibrate(x, N.SQ_GRAN_SHIFT, G, rng, tau, exp, st),
                 lambda: N.shiftquant_quantize(x, N.SQ_GRAN_SHIFT, bits, G, tau, exp, None,
                                               N.SQ_ROUND_NEAREST_EVEN, 0, qx, None, scale),
                 lambda: L.weight_quantize_fwd(wt, w, exp, bits, G, st),
                 lambda: N.shiftquant_gemm_fwd(qx, scale, w.codes, w.scale, M, C, K, bits, G, y, dev_status=st),
                 # the output on a fixed grid, directly behind the GEMM that writes it
                 lambda: N.shiftquant_quantize(y, N.SQ_GRAN_SHIFT, bits, G, t0, e0, None,
                                               N.SQ_ROUND_STOCHASTIC, 9, qy, None, s0)]
        for f in steps:
            f()
            if pause:
                torch.cuda.synchronize()
        return [t.clone() for t in (exp, scale, w.scale, y, qy)]

    want = [chain(x, wt, True) for x, wt in zip(xs, ws)]
    got = [chain(x, wt, False) for x, wt in zip(xs, ws)]
    torch.cuda.synchronize()
    assert st.item() == 0
    for a, b in zip(got, want):
        for g, h in zip(a, b):
            np.testing.assert_array_equal(g.view(torch.uint8).cpu().numpy(), h.view(torch.uint8).cpu().numpy())


@pytest.mark.gpu
@pytest.mark.parametrize("C", [61, 160])
def test_unpack_directly_behind_pack(lib, C):
    M, G, dev = 700, 4, "cuda"
    st = torch.zeros(1, dtype=torch.int32, device=dev)
    packed = torch.zeros((M, (C + 1) // 2 + 15 & ~15), dtype=torch.uint8, device=dev)
    codes = [torch.randint(-7, 8, (M, C), device=dev).float().to(torch.float8_e4m3fn).view(torch.uint8)
             for _ in range(8)]
    back = [torch.zeros((M, C), dtype=torch.uint8, device=dev) for _ in codes]
    for c, b in zip(codes, back):
        N.shiftquant_pack_codes(c, 4, G, packed, st)
        N.shiftquant_unpack_codes(packed, C, 4, G, b)
    torch.cuda.synchronize()
    assert st.item() == 0
    for c, b in zip(codes, back):
        assert torch.equal(c, b)

"""GPU parity of the quantizer's ways to load what a tile needs and to leave its codes: exponents,
folded shifts, ranges and codes from addresses that are aligned and that are not, rows that share
sectors, every choice of outputs in every granularity, partial tiles either way -- against the
oracle's codes."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2411_10948_gb300 import layer as L
from paper_2411_10948_gb300 import native as N
from parity_util import decode

pytestmark = pytest.mark.gpu
G = 4


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2411_10948_gb300 import build
    build.build_library()
    N.load()


def at(a, off):
    """a vector on the device, `off` elements past an aligned address"""
    t = torch.from_numpy(np.ascontiguousarray(a)).cuda()
    buf = torch.zeros(t.numel() + off, dtype=t.dtype, device="cuda")
    buf[off:] = t
    return buf[off:]


def run(x, gran, bits, ranges, exp, fold, mode, seed, which, shift):
    """(codes, codes_t, scales) with the vectors `shift` elements off alignment"""
    R, C = x.shape
    codes = L.empty_codes(R, C, bits, G, "cuda") if "c" in which else None
    codes_t = L.empty_codes(C, R, bits, G, "cuda") if "t" in which else None
    n = {N.SQ_GRAN_SHIFT: 1, N.SQ_GRAN_PER_COL: C, N.SQ_GRAN_PER_ROW: R}[gran]
    scale = torch.full((n,), -1.0, device="cuda")
    N.shiftquant_quantize(x, gran, bits, G, at(ranges, shift), None if exp is None else at(exp, shift),
                          None if fold is None else at(fold, shift), mode, seed, codes, codes_t, scale)
    return codes, codes_t, scale


# one column to several tiles, whole and ragged; 292: rows that share sectors
SHAPES = [(1, 1), (70, 3), (300, 5), (64, 128), (65, 292), (257, 200), (129, 130)]


@pytest.mark.parametrize("bits", [4, 8])
@pytest.mark.parametrize("which", ["c", "t", "ct"])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_outputs_and_vectors(bits, which, shift):
    rng = np.random.default_rng(bits + 10 * shift)
    for R, C in SHAPES:
        a = (rng.standard_normal((R, C)) * np.exp(rng.normal(0, 1.5, C))).astype(np.float32)
        x = torch.from_numpy(a).cuda()
        cases = []
        for mode in (0, 1):
            o = O.shiftquant_tensor(a, bits, G, mode, 7)
            tau = np.abs(a).max(keepdims=True).reshape(1).astype(np.float32)
            cases.append((N.SQ_GRAN_SHIFT, tau, np.asarray(o["exp"], np.uint8), None, mode, o["codes"]))
        for gran, axis, role in ((N.SQ_GRAN_PER_COL, 0, 0), (N.SQ_GRAN_PER_ROW, 1, 1)):
            r = np.abs(a).max(axis).astype(np.float32)
            q = O.channel_tensor(a, bits, role)["codes"]
            q = q if q.shape == a.shape else q.T
            fold = rng.integers(0, G, a.shape[axis]).astype(np.uint8)
            f = (1 << (G - 1 - fold.astype(np.int64)))
            cases.append((gran, r, None, None, 0, q))
            cases.append((gran, r, None, fold, 0, q * (f[:, None] if gran == N.SQ_GRAN_PER_COL else f[None, :])))
        for gran, r, e, fold, mode, want in cases:
            codes, codes_t, scale = run(x, gran, bits, r, e, fold, mode, 7, which, shift)
            torch.cuda.synchronize()
            tag = f"{R}x{C} gran {gran} mode {mode} fold {fold is not None}"
            if codes is not None:
                np.testing.assert_array_equal(decode(codes), want, err_msg=tag)
            if codes_t is not None:
                np.testing.assert_array_equal(decode(codes_t), np.asarray(want).T, err_msg=tag)
            assert bool((scale >= 0).all()), tag

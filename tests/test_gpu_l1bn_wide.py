"""GPU parity of the L1 batch normalization's cooperative form and of its chain of kernels at the
shapes left to them: more rows than stay in shared memory, small backward passes, more column
tiles than SMs; ragged channels, padded rows, an unaligned base, other group counts, all-zero and
non-finite inputs.  Everything is compared bit for bit with the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2411_10948_gb300 import native as N
from parity_util import f32_bits
from test_gpu_l1bn_forms import run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2411_10948_gb300 import build
    build.build_library()
    N.load()


def inputs(R, C):
    rng = np.random.default_rng(5 * R + C)
    x = (rng.standard_normal((R, C)) * np.exp(rng.normal(0, 1, C)) + rng.normal(0, 1, C)).astype(np.float32)
    dy = (rng.laplace(0, 1, (R, C)) * np.exp(rng.normal(0, 1.5, C))).astype(np.float32)
    x[:, C // 2] = -0.75
    return x, dy, *(rng.normal(m, 0.3, C).astype(np.float32) for m in (1, 0))


# cooperative both ways (300001 rows); cooperative backward behind a resident forward (of whole
# words of codes); the forward alone cooperative (a ring of unaligned rows); the chain (more than
# 152 tiles of 64 columns)
@pytest.mark.parametrize("R,C,bits,G,how", [
    (300001, 61, 8, 4, "dense"), (300001, 61, 6, 8, "padded"), (300001, 62, 8, 4, "offset"),
    (300001, 3, 4, 2, "dense"), (1000, 256, 8, 4, "offset"), (257, 100, 6, 4, "padded"),
    (4097, 128, 8, 4, "dense"), (150001, 64, 8, 4, "offset"), (150001, 61, 8, 4, "padded"),
    (41, 9801, 8, 4, "dense"), (41, 9802, 6, 8, "offset"), (37, 9803, 4, 2, "padded"),
    (1, 9804, 8, 4, "dense")])
def test_forms_match_the_oracle(R, C, bits, G, how):
    x, dy, gamma, beta = inputs(R, C)
    got = run(x, gamma, beta, dy, bits, G, R, how)
    f = O.l1bn_forward(x, gamma, beta, bits, G)
    b = O.l1bn_backward(dy, f, bits, G, R)
    assert got[4] == 0
    for g, w, name in zip(got, (f["y"], b["dx"], b["dgamma"], b["dbeta"]), ("y", "dx", "dgamma", "dbeta")):
        np.testing.assert_array_equal(f32_bits(g), f32_bits(w), err_msg=name)


@pytest.mark.parametrize("R,C", [(300001, 61), (1000, 256), (41, 9801)])
def test_zero_and_nonfinite_inputs(R, C):
    x, _, gamma, beta = inputs(R, C)
    zero = np.zeros((R, C), np.float32)
    y, dx, dg, db, st = run(zero, gamma, beta, zero, 8, 4, 1, "dense")
    f = O.l1bn_forward(zero, gamma, beta, 8, 4)
    assert st == 0
    np.testing.assert_array_equal(f32_bits(y), f32_bits(f["y"]))
    assert not dx.any() and not dg.any() and not db.any()
    # a non-finite gradient, then a non-finite input
    bad = x.copy()
    bad[R - 1, C - 1] = np.nan
    assert run(x, gamma, beta, bad, 8, 4, 1, "dense")[4] == N.SQ_DEV_NONFINITE
    bad[R - 1, C - 1] = np.inf
    assert run(bad, gamma, beta, zero, 8, 4, 1, "dense")[4] == N.SQ_DEV_NONFINITE

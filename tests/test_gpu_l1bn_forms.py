"""GPU parity of the L1 batch normalization's three launch forms at the shapes where they
meet: the resident form with whole tensors and with a ring of rows in shared memory, the
cooperative form for more rows than fit, and the chain of kernels for more column tiles than
SMs; ragged rows and channels, padded rows, unaligned bases, all-zero and non-finite inputs.
Everything is compared bit for bit with the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2411_10948_gb300 import native as N
from parity_util import f32_bits

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2411_10948_gb300 import build
    build.build_library()
    N.load()


def place(a, how):
    R, C = a.shape
    if how == "dense":
        return torch.from_numpy(a).cuda()
    pad = 4 - C % 4 if how == "padded" else 0          # rows of whole quads
    off = 1 if how == "offset" else 0                  # a base that is not 16-byte aligned
    buf = torch.full((R * (C + pad) + off,), 7e8, dtype=torch.float32, device="cuda")
    v = buf[off:].view(R, C + pad)[:, :C]
    v.copy_(torch.from_numpy(a))
    return v


def run(x, gamma, beta, dy, bits, G, seed, how):
    R, C = x.shape
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    state = torch.zeros(N.shiftquant_l1bn_state_bytes(R, C), dtype=torch.uint8, device="cuda")
    y, dx = (place(np.full((R, C), 9.0, np.float32), how) for _ in range(2))
    dg, db = torch.zeros(C, device="cuda"), torch.zeros(C, device="cuda")
    vec = lambda a: torch.from_numpy(a).cuda()
    N.shiftquant_l1bn_forward(place(x, how), vec(gamma), vec(beta), bits, G, y, state, st)
    N.shiftquant_l1bn_backward(place(dy, how), bits, G, seed, state, dx, dg, db, st)
    torch.cuda.synchronize()
    return [t.cpu().numpy() for t in (y, dx, dg, db)] + [st.item()]


# rows whole and ragged against 1024 / (columns / 4) a pass, one quad to many tiles; the last
# three: a ring (rows beyond 56 KB a block in 32 bits), the cooperative form, the chain
@pytest.mark.parametrize("R,C,bits,G,how", [
    (1, 1, 8, 4, "dense"), (5, 3, 4, 2, "offset"), (257, 64, 8, 4, "padded"), (511, 68, 6, 4, "dense"),
    (1025, 61, 8, 4, "padded"), (97, 2047, 8, 4, "offset"), (3137, 2048, 8, 4, "dense"),
    (2500, 1030, 6, 8, "padded"), (150001, 62, 8, 4, "padded"), (300000, 64, 8, 4, "dense"),
    (40, 9800, 8, 4, "dense")])
def test_forms_match_the_oracle(R, C, bits, G, how):
    rng = np.random.default_rng(3 * R + C)
    x = (rng.standard_normal((R, C)) * np.exp(rng.normal(0, 1, C)) + rng.normal(0, 1, C)).astype(np.float32)
    dy = (rng.laplace(0, 1, (R, C)) * np.exp(rng.normal(0, 1.5, C))).astype(np.float32)
    gamma, beta = (rng.normal(m, 0.3, C).astype(np.float32) for m in (1, 0))
    x[:, C // 2] = -0.75
    got = run(x, gamma, beta, dy, bits, G, R, how)
    f = O.l1bn_forward(x, gamma, beta, bits, G)
    b = O.l1bn_backward(dy, f, bits, G, R)
    assert got[4] == 0
    for g, w, name in zip(got, (f["y"], b["dx"], b["dgamma"], b["dbeta"]), ("y", "dx", "dgamma", "dbeta")):
        np.testing.assert_array_equal(f32_bits(g), f32_bits(w), err_msg=name)


@pytest.mark.parametrize("R,C", [(300, 40), (60000, 96)])
def test_zero_and_nonfinite_inputs(R, C):
    rng = np.random.default_rng(C)
    gamma, beta = (rng.normal(m, 0.3, C).astype(np.float32) for m in (1, 0))
    zero = np.zeros((R, C), np.float32)
    y, dx, dg, db, st = run(zero, gamma, beta, zero, 8, 4, 1, "dense")
    f = O.l1bn_forward(zero, gamma, beta, 8, 4)
    assert st == 0
    np.testing.assert_array_equal(f32_bits(y), f32_bits(f["y"]))
    assert not dx.any() and not dg.any() and not db.any()
    bad = rng.standard_normal((R, C)).astype(np.float32)
    bad[R - 1, C - 1] = np.inf
    assert run(bad, gamma, beta, zero, 8, 4, 1, "dense")[4] == N.SQ_DEV_NONFINITE

"""GPU parity of the GEMMs' output boxes at the edges of their ways out: rows of outputs that
are 16-byte aligned (staged boxes sent whole) and rows that start anywhere (a lane a column),
row and column counts around a box, a tile and a pair tile, each against the oracle's exact
integers and outputs."""
import numpy as np
import pytest
import torch

from paper_2411_10948_gb300 import layer as L
from paper_2411_10948_gb300 import native as N
from parity_util import assert_close_f32, oracle_layer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2411_10948_gb300 import build
    build.build_library()
    N.load()


@pytest.mark.parametrize("M,K,Nn,bits", [(33, 31, 1, 4), (31, 65, 33, 8), (129, 255, 257, 6), (257, 260, 259, 8),
                                         (128, 288, 31, 4), (1, 130, 262, 6), (300, 2049, 290, 8),
                                         (2100, 33, 65, 8)])
def test_outputs_match_the_oracle(M, K, Nn, bits):
    rng = np.random.default_rng(M + K + Nn)
    x = (rng.standard_normal((M, K)) * np.exp(rng.normal(0, 1, K))).astype(np.float32)
    w = (rng.standard_normal((K, Nn)) * 0.05).astype(np.float32)
    dy = (rng.standard_normal((M, Nn)) * np.exp(rng.normal(0, 1.5, Nn))).astype(np.float32)
    lay = L.QuantLinear(M, K, Nn, bits, 4, "cuda")
    dev = [torch.from_numpy(a).cuda() for a in (x, w, dy)]
    N.shiftquant_layer_step(lay.step_args(*dev), 77)
    torch.cuda.synchronize()
    ora = oracle_layer(x, w, dy, bits, 4, 77)
    assert int(lay.status.item()) == 0
    for name in ("y", "dx", "dw"):
        assert_close_f32(getattr(lay, name).cpu().numpy(), ora[name], name)

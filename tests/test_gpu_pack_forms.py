"""GPU parity of the packing kernels at the edges of their launch shapes: rows of 1 to 40
chunks of sixteen codes (blocks 32, 16 and 8 chunks wide), row counts around a block's slab
and beyond the grid's limit of slabs, both code types, and every E4M3 byte."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2411_10948_gb300 import layer as L
from paper_2411_10948_gb300 import native as N
from parity_util import decode

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2411_10948_gb300 import build
    build.build_library()
    N.load()


# a slab is 8 rows a thread times 256 / (chunks across) rows a block: 64, 128 or 256 rows;
# 65535 slabs of 256 rows are 16776960 rows
@pytest.mark.parametrize("R,C,G", [(1, 16, 4), (63, 512, 4), (65, 511, 4), (129, 144 * 16, 4),
                                   (127, 240, 4), (257, 120, 4), (255, 40 * 16 - 1, 8), (300, 129, 8),
                                   (16777300, 2, 4)])
def test_every_launch_shape_round_trips(R, C, G):
    q = np.random.default_rng(R + C).integers(-8, 8, (R, C)).astype(np.int64)
    codes, back = (L.empty_codes(R, C, 4, G, "cuda") for _ in range(2))
    if codes.dtype == torch.uint8:
        codes.copy_(torch.from_numpy(q).cuda().float().to(torch.float8_e4m3fn).view(torch.uint8))
    else:
        codes.copy_(torch.from_numpy(q).cuda().float())
    packed = torch.full((R, (C + 1) // 2), 0xAA, dtype=torch.uint8, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    N.shiftquant_pack_codes(codes, 4, G, packed, st)
    N.shiftquant_unpack_codes(packed, C, 4, G, back)
    torch.cuda.synchronize()
    assert st.item() == 0
    np.testing.assert_array_equal(packed.cpu().numpy(), O.pack4(q))
    np.testing.assert_array_equal(decode(back), q)


def test_every_byte_packs_as_its_integers_low_nibble():
    v = torch.arange(256, dtype=torch.uint8).view(torch.float8_e4m3fn).float().numpy().astype(np.float64)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    packed = torch.zeros((1, 8), dtype=torch.uint8, device="cuda")
    for b in np.flatnonzero(v == np.round(v)):   # the integers among the bytes
        codes = torch.full((1, 16), int(b), dtype=torch.uint8, device="cuda")
        st.zero_()
        N.shiftquant_pack_codes(codes, 4, 4, packed, st)
        n = int(v[b]) & 0xF
        assert bool((packed == (n | n << 4)).all()) and (st.item() != 0) == (not -8 <= v[b] <= 7), (b, v[b])

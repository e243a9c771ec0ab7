"""The launches of a layer step, on the host alone (no GPU): their order and how each is launched.
Several of them read what the one before the last wrote without a wait of their own, which holds
for exactly this chain."""
import ctypes

import pytest

import fake_cudart
from paper_2411_10948_gb300 import native as N


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fake_cudart.link(tmp_path_factory.mktemp("fake"))


def step(lib, M, K, C, bits, workspace=True):
    """(kernel, blocks, flags) of one step over addresses that stand for device memory."""
    at = iter(range(1 << 32, 1 << 44, 1 << 34))
    a = N.SqLayerStep(M=M, K=K, N=C, bits=bits, n_groups=4)
    for name, kind in N.SqLayerStep._fields_:
        if kind is ctypes.c_void_p and name not in ("xt_codes", "gt_codes", "workspace"):
            setattr(a, name, next(at))
    a.ld_x, a.ld_g, a.ld_wf, a.ld_wd = (-(-n // 16) * 16 for n in (K, C, K, C))
    if workspace:
        a.workspace = next(at)
        a.workspace_bytes = lib.shiftquant_gemm_layer_workspace_bytes(M, K, C, bits, 4)
    lib.fake_log()
    assert lib.shiftquant_layer_step(ctypes.byref(a), 1, None) == N.SQ_OK
    return fake_cudart.launches(lib)


CODES = {"one": ["layer_quantize_kernel"], "three": ["quantize_kernel", "quantize_weight_kernel", "quantize_kernel"]}


@pytest.mark.parametrize("M,K,C,bits,codes", [(256, 512, 512, 4, "one"), (300, 131, 77, 6, "one"),
                                              (12608, 768, 3072, 6, "three"), (5003, 1155, 1001, 8, "three")])
def test_chain_of_a_step(lib, M, K, C, bits, codes):
    ran = step(lib, M, K, C, bits)
    names = [k[0] for k in ran]
    n = 2 + len(CODES[codes])
    assert names[:n] == ["layer_init_kernel", "layer_range_kernel"] + CODES[codes]
    assert names[n] == "shiftmm_kernel" and all(k.startswith("splitk_finalize") for k in names[n + 1:])
    assert all(k[2] == "p" for k in ran)   # nothing plain in between


# two waves of four blocks on each SM: the same step on a device of more SMs is one launch
def test_code_launches_follow_the_device(lib):
    try:
        lib.fake_sms(4000)
        assert [k[0] for k in step(lib, 12608, 768, 3072, 6)][2:3] == CODES["one"]
    finally:
        lib.fake_sms(152)


def test_without_a_workspace_one_call_after_another(lib):
    names = [k[0] for k in step(lib, 256, 512, 512, 4, workspace=False)]
    assert names.count("calib_init_kernel") == 3 and "layer_init_kernel" not in names
    assert names[-1] == "shiftmm_kernel"

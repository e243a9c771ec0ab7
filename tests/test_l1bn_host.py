"""Which launches an L1 batch norm call makes, on the host alone (no GPU): the resident form, and
what follows where the device refuses a cooperative launch."""
import ctypes
from concurrent.futures import ThreadPoolExecutor

import pytest

import fake_cudart
from paper_2411_10948_gb300 import native as N

FWD_CHAIN = ["l1bn_zero_kernel", "calib_init_kernel", "colmax_kernel", "group_kernel", "l1bn_fwd_quant_kernel",
             "l1bn_fwd_dev_kernel", "l1bn_fwd_chan_kernel", "l1bn_fwd_lut_kernel", "l1bn_fwd_out_kernel"]
BWD_CHAIN = ["l1bn_zero_kernel", "calib_init_kernel", "colmax_kernel", "group_kernel", "l1bn_bwd_quant_kernel",
             "l1bn_bwd_chan_kernel", "l1bn_bwd_out_kernel"]
TOO_LARGE, OUT_OF_RESOURCES, ILLEGAL_ADDRESS = 720, 701, 700   # cudaError_t


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fake_cudart.link(tmp_path_factory.mktemp("fake"))


def call(lib, R, C, backward):
    """(status, kernels launched) of one call; addresses stand for device memory."""
    p = ctypes.c_void_p
    state, size = p(1 << 32), lib.shiftquant_l1bn_state_bytes(R, C)
    lib.fake_log()
    if backward:
        st = lib.shiftquant_l1bn_backward(p(1 << 20), R, C, C, 8, 4, 1, state, size, p(1 << 21), C, p(1 << 22),
                                          p(1 << 23), p(1 << 24), None)
    else:
        st = lib.shiftquant_l1bn_forward(p(1 << 20), R, C, C, p(1 << 22), p(1 << 23), 8, 4, p(1 << 21), C, state,
                                         size, p(1 << 24), None)
    return st, fake_cudart.launches(lib)


@pytest.mark.parametrize("backward", [False, True])
@pytest.mark.parametrize("C", [64, 2048])
def test_resident_form_is_one_cooperative_launch(lib, C, backward):
    st, ran = call(lib, 20000, C, backward) if C == 64 else call(lib, 3136, C, backward)
    assert st == N.SQ_OK and len(ran) == 1
    assert ran[0][0] == f"l1bn_{'bwd' if backward else 'fwd'}_res_kernel" and ran[0][2] == "c"


@pytest.mark.parametrize("error", [TOO_LARGE, OUT_OF_RESOURCES])
@pytest.mark.parametrize("backward", [False, True])
def test_refused_launch_goes_on_with_the_next_form(lib, backward, error):
    d = "bwd" if backward else "fwd"
    chain = BWD_CHAIN if backward else FWD_CHAIN
    # too many channels for the cooperative form: the chain
    lib.fake_refuse(error, 1)
    st, ran = call(lib, 3136, 2048, backward)
    assert st == N.SQ_OK and [k[0] for k in ran] == chain
    assert lib.fake_last_error() == 0
    # the resident form's blocks alone do not fit: the cooperative form
    lib.fake_refuse(error, 1)
    st, ran = call(lib, 20000, 64, backward)
    assert st == N.SQ_OK and [k[0] for k in ran] == [f"l1bn_{d}_coop_kernel"]
    # no cooperative launch at all
    lib.fake_refuse(error, 2)
    st, ran = call(lib, 20000, 64, backward)
    assert st == N.SQ_OK and [k[0] for k in ran] == chain
    assert lib.fake_last_error() == 0


def test_other_errors_are_reported(lib):
    lib.fake_refuse(ILLEGAL_ADDRESS, 1)
    st, ran = call(lib, 3136, 2048, False)
    assert st == N.SQ_ECUDA and ran == []
    lib.fake_refuse(0, 0)
    lib.cudaGetLastError()


# few rows of a backward, and a forward whose rows of codes are not whole words: the cooperative form
@pytest.mark.parametrize("R,C,backward,form", [(1000, 256, True, "l1bn_bwd_coop_kernel"),
                                               (255, 256, True, "l1bn_bwd_res_kernel"),
                                               (12544, 61, True, "l1bn_bwd_res_kernel"),
                                               (1000, 256, False, "l1bn_fwd_res_kernel"),
                                               (200704, 61, False, "l1bn_fwd_coop_kernel"),
                                               (200704, 61, True, "l1bn_bwd_res_kernel"),
                                               (3136, 1025, True, "l1bn_bwd_res_kernel")])
def test_form_of_a_shape(lib, R, C, backward, form):
    st, ran = call(lib, R, C, backward)
    assert st == N.SQ_OK and [k[0] for k in ran] == [form]


# a whole tensor and a ring of rows on the SMs, too many rows for that, few channels, and more
# channel tiles than SMs
@pytest.mark.parametrize("R,C", [(3136, 2048), (200704, 64), (300000, 64), (300000, 1024), (300000, 1025),
                                 (40, 9800), (1, 1), (1 << 24, 3000)])
@pytest.mark.parametrize("backward", [False, True])
def test_launch_query_is_what_a_call_launches(lib, R, C, backward):
    st, ran = call(lib, R, C, backward)
    assert st == N.SQ_OK and lib.shiftquant_l1bn_launches(R, C, int(backward)) == len(ran)


def test_launch_query_at_its_edges(lib):
    assert lib.shiftquant_l1bn_launches(5, 0, 0) == 0
    assert lib.shiftquant_l1bn_launches(-1, 5, 0) == lib.shiftquant_l1bn_launches(5, -1, 0) == -1
    # no rows, and any number of rows
    assert lib.shiftquant_l1bn_launches(0, 64, 0) == lib.shiftquant_l1bn_kernel_launches(64, 0) == 1
    assert lib.shiftquant_l1bn_kernel_launches(1025, 0) == 9 and lib.shiftquant_l1bn_kernel_launches(1025, 1) == 7


def test_threads_ask_for_the_plan_together(tmp_path):
    # a library nobody has called yet, from sixteen threads at once
    lib = fake_cudart.link(tmp_path)
    with ThreadPoolExecutor(16) as ex:
        got = list(ex.map(lambda i: lib.shiftquant_l1bn_launches(300000 if i % 2 else 3136, 1025, i // 2 % 2),
                          range(64)))
    assert got == [(1, 9, 1, 7)[i % 4] for i in range(64)]

"""How many CTAs the one-launch kernel gets: two on every SM for each row
size, and the plans of layers whose rows take 512 bytes (fp32, 128 channels)
around the sizes where they change."""
import ctypes

import pytest

from test_abi_host import H  # noqa: F401

FULL = 304          # two CTAs on each of 152 SMs
RANGES, SHORT, HEADS = 0, 1, 2
# heads, rows of the longest, fused, identify -> CTAs, cut, lone
ROWS_512 = [
    (32, 569, 1, 0, 146, RANGES, 1),      # as many ranges as have 16 slots
    (101, 569, 1, 0, 152, RANGES, 1),     # more than three ranges a head
    (102, 569, 1, 0, 304, RANGES, 0),
    (276, 164, 1, 0, 152, RANGES, 1),     # 39.9 slots an SM
    (277, 164, 1, 0, 304, RANGES, 0),
    (101, 569, 0, 0, 152, RANGES, 1),
    (102, 569, 0, 0, 304, RANGES, 0),
    (101, 428, 1, 1, 152, RANGES, 1),
    (152, 96, 1, 0, 152, SHORT, 0),
    (153, 96, 1, 0, 125, RANGES, 1),
    (13626, 128, 1, 0, 304, RANGES, 0),   # 762 slots a CTA: the table's 256 heads just fit
    (13627, 128, 1, 0, 304, HEADS, 0),
]


class Plan(ctypes.Structure):
    _fields_ = [("grid", ctypes.c_int), ("cut", ctypes.c_int), ("lone", ctypes.c_int)]


def _plan(H, D, bf16, n, rows, fused, identify):  # noqa: F811
    f = ctypes.CDLL(H.LIB_PATH)._ZN3hkv9step_planEiiiiibb
    f.restype = Plan
    f.argtypes = [ctypes.c_int] * 5 + [ctypes.c_bool] * 2
    p = f(D, bf16, n, rows, FULL, fused, identify)
    return p.grid, p.cut, p.lone


@pytest.mark.parametrize("n,rows,fused,identify,grid,cut,lone", ROWS_512)
def test_plans_of_512_byte_rows(H, n, rows, fused, identify, grid, cut, lone):  # noqa: F811
    assert _plan(H, 128, 0, n, rows, fused, identify) == (grid, cut, lone)


@pytest.mark.parametrize("D,bf16", [(128, 1), (64, 1), (64, 0)])
def test_other_rows_never_take_an_sm_alone(H, D, bf16):  # noqa: F811
    for n in (1, 8, 101, 102, 300, 2000, 20000):
        for rows in (20, 164, 569, 1233):
            for mode in ((1, 0), (1, 1), (0, 0)):
                assert _plan(H, D, bf16, n, rows, *mode)[2] == 0


@pytest.mark.gpu
@pytest.mark.parametrize("D,bf16", [(128, 0), (128, 1), (64, 0), (64, 1)])
def test_two_ctas_on_an_sm(H, D, bf16):  # noqa: F811
    import torch
    torch.zeros(1, device="cuda")
    n = ctypes.c_int(0)
    assert ctypes.CDLL(H.LIB_PATH)._ZN3hkv12step_prepareEiiPi(D, bf16, ctypes.byref(n)) == 0
    assert n.value == 2

"""Which lattices the staged-row collide takes (just inside and just outside of
each bound of its rule: the bytes of a slot array, how far a row fills a
buffer, rows that are whole 16-byte words), and its bits against the node
kernels in 16-bit storage."""
import ctypes

import pytest

from paper_1703_05158_gb300 import lbm
from test_gpu_rows import test_rows_are_bitwise_the_node_kernels as bitwise

pytestmark = pytest.mark.gpu

ROWS = [("fp32", (256, 64, 128)), ("fp32", (112, 139, 136)), ("fp16", (512, 64, 128)), ("fp16", (448, 75, 125)),
        ("bf16", (504, 64, 131)), ("bf16", (512, 33, 249))]
NODES = [("fp32", (256, 64, 127)), ("fp32", (108, 139, 141)), ("fp32", (254, 72, 120)), ("fp16", (512, 64, 127)),
         ("fp16", (440, 75, 128)), ("fp16", (500, 75, 125)), ("fp16", (520, 64, 130)), ("bf16", (640, 64, 128)),
         ("bf16", (1024, 45, 92)), ("bf16", (256, 128, 130))]


def by_rows(precision, shape):
    form = lbm.load()._ZN3lbm16collides_by_rowsEPK5lbm_s
    form.restype, form.argtypes = ctypes.c_bool, [ctypes.c_void_p]
    lat = lbm.Lattice(*shape, tau0=0.6, precision=precision)
    taken = form(lat.h)
    lat.close()
    return taken


@pytest.mark.parametrize("precision,shape", ROWS + NODES)
def test_form(precision, shape):
    assert by_rows(precision, shape) == ((precision, shape) in ROWS)


@pytest.mark.parametrize("precision,shape", [r for r in ROWS if r[0] != "fp32"])
def test_bits(precision, shape):
    bitwise(precision, shape)

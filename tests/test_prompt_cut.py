"""How the projections of a prompt pass are cut (gemm_pf_schedule): host code that needs no device."""
import ctypes as C

import pytest

from paper_2404_08698_b200 import build as B

SMS = 148


class Cut(C.Structure):
    _fields_ = [("ksplit", C.c_int), ("tail_from", C.c_int), ("tail_split", C.c_int), ("n_tt", C.c_int)]


def gate_up_cut(d, f, rows):
    fn = C.CDLL(B.build())["_Z16gemm_pf_scheduleiiiii"]        # C++ linkage: (feature tiles, rows, k-blocks, SMs, most parts)
    fn.restype = Cut
    return fn(-(-2 * f // 256), rows, d // 64, SMS, 8)


# Tiles that would leave a third of the SMs without work are cut along K (7B, 1.1B, 512 and 1536 wide).
@pytest.mark.parametrize("d,f,rows", [(4096, 11008, 144), (2048, 5632, 200), (512, 1376, 296), (512, 1376, 1000), (1536, 4096, 400)])
def test_gate_up_is_cut_where_its_tiles_leave_sms_idle(d, f, rows):
    c = gate_up_cut(d, f, rows)
    tiles = -(-2 * f // 256) * c.n_tt
    assert c.ksplit > 1 and c.tail_from == tiles, (c.ksplit, c.tail_from, c.tail_split, c.n_tt)


# More tiles than SMs: whole ones, whose activations the projection finishes, and at most the last round's cut.
@pytest.mark.parametrize("d,f,rows", [(4096, 11008, 600), (4096, 11008, 1536), (5120, 13824, 2048), (2048, 5632, 1400)])
def test_gate_up_stays_whole_where_its_tiles_fill_the_sms(d, f, rows):
    c = gate_up_cut(d, f, rows)
    assert c.ksplit == 1 and c.tail_from >= SMS - c.n_tt

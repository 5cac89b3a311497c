"""CPU: which kernel the SVD's sweeps take, by the library's own rules."""
import ctypes as C

import paper_2401_01921_gb300 as tnx
from paper_2401_01921_gb300 import build


def test_more_slots_than_the_block_sweeps_keep_track_of():
    """1024 slots per CTA, one CTA per SM at least: a truncation with more takes the other kernel; it is not
    refused."""
    build.build()
    fits = tnx.lib()._Z21tnx_jacobi_block_fitsli
    fits.argtypes, fits.restype = [C.c_int64, C.c_int], C.c_bool
    assert fits(1, 152) and fits(1024 * 152, 152)
    assert not fits(1024 * 152 + 1, 152)

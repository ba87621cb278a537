"""What the fp32 backward asks for in device memory, per 64-token chunk of a head (no
GPU): records, what the chain keeps, the forward's intermediates, chunk-start states."""
import ctypes

import pytest

from paper_2509_25223_gb300 import _abi


def _need(op, T, D, states=False):
    lib, n = _abi.load(), ctypes.c_size_t(0)
    b = _abi.BwdArgs()
    a = b.fwd
    a.B, a.T, a.H, a.Dk, a.Dv = 1, T, 1, D, D
    a.dtype, a.clip, a.scale = _abi.RDN_F32, 1.0, 1.0
    if states:
        a.S_chunks = a.R_chunks = ctypes.c_void_p(0x10000)  # (never read: a size query)
    assert lib[op + "_bwd_workspace_size"](ctypes.byref(b), ctypes.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("op,tiles", [("rdn", 3), ("rla", 2)])
@pytest.mark.parametrize("chunks", [1, 7])
def test_bytes_a_chunk(op, tiles, D, chunks):
    records, tile, state = 4 * (5 * 64 * 64 + 6 * 64), 4 * 64 * D, 4 * D * D
    kept = records + tiles * tile + 2 * state        # dVr, dX (RDN: dX2), dS, dR
    made = 2 * tile + 8 * D                          # E, E2, the clip mask
    assert _need(op, 64 * chunks, D, states=True) == chunks * (kept + made) + 256
    # without the forward's states: theirs too, and nothing for an o that nobody reads
    assert _need(op, 64 * chunks, D) == chunks * (kept + made + 2 * state) + 256

"""The packed arguments of a decode step (no GPU): the bytes of the C struct, and the
scalars that the field-by-field struct took."""
import ctypes
import fractions

import pytest
import torch

import paper_2509_25223_gb300 as rdn
from paper_2509_25223_gb300 import _abi


@pytest.mark.parametrize("x", ["0.5", fractions.Fraction(1, 2), torch.tensor(0.5), True, 1, 1e300,
                               float("inf"), -0.0, 0.1])
def test_scalars(x):
    a = _abi.DecodeArgs()
    a.clip = float(x)
    assert rdn._f32(x) == a.clip


def test_packed_bytes_are_the_struct():
    a = _abi.DecodeArgs()
    vals = (3, 5, 128, 128, 1, 1, 16, 32, 48, 0, 1 << 47, 96, 0.25, -1.5, 112, 128, 144, 0x83, 1e-12)
    for (name, _), v in zip(_abi.DecodeArgs._fields_, vals):
        setattr(a, name, v)
    packed = _abi.DECODE_PACK(*(rdn._f32(v) if isinstance(v, float) else v for v in vals))
    for name, typ in _abi.DecodeArgs._fields_:
        f = getattr(_abi.DecodeArgs, name)
        assert packed[f.offset:f.offset + f.size] == bytes(a)[f.offset:f.offset + f.size], name
    assert len(packed) == ctypes.sizeof(a)

"""The tensor-core scan and chain over a pair of CTAs per (sequence, head),
which calls with few heads take, against the one-CTA kernels, which calls with
more take: the same operands in the same order, so every result is the same
bits.  (On a chip of 152 SMs 4 heads run in pairs, 80 one CTA each.)"""
import pytest
import torch

import paper_2509_25223_gb300 as rdn
from rdn_synthetic import make_inputs

pytestmark = pytest.mark.gpu

NAMES = ("q", "k", "v", "g", "beta", "gamma")


def _step(x, variant, saved, flags):
    B, T, H, D = x["q"].shape
    fwd, bwd = (rdn.rdn_fwd, rdn.rdn_bwd) if variant == "rdn" else (rdn.rla_fwd, rdn.rla_bwd)
    kw = dict(clip=0.7, S0=x["S0"], R0=x["R0"], variant_flags=flags)
    ws = torch.empty(rdn.workspace_bytes(variant + "_fwd", B, T, H, D, save_for_bwd=saved,
                                         variant_flags=flags), dtype=torch.uint8, device="cuda")
    o, ST, RT, Sc, Rc = fwd(*(x[n] for n in NAMES), return_chunk_states=True, save_for_bwd=saved,
                            workspace=ws, **kw)
    g = bwd(*(x[n] for n in NAMES), x["dO"], S_chunks=Sc, R_chunks=Rc, dST=x["S0"], dRT=x["R0"],
            fwd_workspace=ws, fwd_saved=saved, **kw)
    return dict(o=o, ST=ST, RT=RT, Sc=Sc, Rc=Rc, **g)


@pytest.mark.parametrize("variant", ["rdn", "rla"])
@pytest.mark.parametrize("T,saved,flags", [
    (1, True, 0), (64, True, 0), (65, False, 0), (130, True, 0), (260, True, 0), (200, False, 0),
    (200, True, rdn.TANH_RESIDUAL), (200, True, rdn.STATELESS_AUX),
    (200, True, rdn.DECAYED_RESIDUAL | rdn.PLAIN_COMBINE),
])
def test_pair_equals_one_cta(variant, T, saved, flags):
    x = make_inputs(20, T, 4, 128, dtype="bf16", nonzero_state=True, with_grad_out=True,
                    device="cuda", state_std=0.1)
    many = _step(x, variant, saved, flags)
    few = _step({n: t[7:8].contiguous() for n, t in x.items()}, variant, saved, flags)
    for n, t in few.items():
        assert torch.equal(t, many[n][7:8]), n
    assert rdn.device_status() == 0

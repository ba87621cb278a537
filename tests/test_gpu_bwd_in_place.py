"""Gradients written over what they are the gradients of: the fp32 and d = 64 backward
takes dv in dO's buffer, and dq, dk, dg, dbeta, dgamma, dS0, dR0 in their inputs'.
The bits are those of separate buffers."""
import pytest
import torch

import paper_2509_25223_gb300 as rdn
from rdn_synthetic import make_inputs

pytestmark = pytest.mark.gpu

NAMES = ("q", "k", "v", "g", "beta", "gamma")


@pytest.mark.parametrize("variant", ["rdn", "rla"])
@pytest.mark.parametrize("d,dtype", [(128, "f32"), (64, "f32"), (64, "bf16")])
@pytest.mark.parametrize("T,saved", [(1, True), (200, True), (130, False)])
def test_outputs_over_inputs(variant, d, dtype, T, saved):
    B, H = 2, 3
    x = make_inputs(B, T, H, d, dtype=dtype, nonzero_state=True, with_grad_out=True, device="cuda",
                    state_std=0.1)
    fwd, bwd = (rdn.rdn_fwd, rdn.rdn_bwd) if variant == "rdn" else (rdn.rla_fwd, rdn.rla_bwd)
    kw = dict(clip=0.7, S0=x["S0"], R0=x["R0"])
    if saved:
        ws = torch.empty(rdn.workspace_bytes(variant + "_fwd", B, T, H, d, save_for_bwd=True,
                                             dtype=x["q"].dtype), dtype=torch.uint8, device="cuda")
        _, ST, RT, Sc, Rc = fwd(*(x[n] for n in NAMES), return_chunk_states=True, save_for_bwd=True,
                                workspace=ws, **kw)
        kw.update(S_chunks=Sc, R_chunks=Rc, fwd_workspace=ws, fwd_saved=True)
    want = bwd(*(x[n] for n in NAMES), x["dO"], dST=x["S0"], dRT=x["R0"], **kw)
    y = {n: t.clone() for n, t in x.items()}
    kw.update(S0=y["S0"], R0=y["R0"])
    dST, dRT = y["S0"].clone(), y["R0"].clone()
    over = dict(dq=y["q"], dk=y["k"], dv=y["dO"], dg=y["g"], dbeta=y["beta"], dgamma=y["gamma"],
                dS0=dST, dR0=dRT)
    bwd(*(y[n] for n in NAMES), y["dO"], dST=dST, dRT=dRT, out=over, **kw)
    for n, t in want.items():
        assert torch.equal(over[n], t), n

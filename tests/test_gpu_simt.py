"""The fp32 kernels' slices of value columns, whose width the number of heads
sets (on a chip of 152 SMs 4 heads take 8 columns a block, 80 heads 32 with
d = 128 and 16 with d = 64, 16 heads of d = 128 take 16): every element is the
same sum in the same order at each width, so every result is the same bits."""
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
                                         variant_flags=flags, dtype=x["q"].dtype),
                     dtype=torch.uint8, device="cuda")
    o, ST, RT, Sc, Rc = fwd(*(x[n] for n in NAMES), return_chunk_states=True, save_for_bwd=saved,
                            workspace=ws, **kw)
    g = bwd(*(x[n] for n in NAMES), x["dO"], S_chunks=Sc, R_chunks=Rc, dST=x["S0"], dRT=x["R0"],
            fwd_workspace=ws, fwd_saved=saved, **kw)
    return dict(o=o, ST=ST, RT=RT, Sc=Sc, Rc=Rc, **g)


@pytest.mark.parametrize("variant", ["rdn", "rla"])
@pytest.mark.parametrize("d,dtype", [(128, "f32"), (64, "f32"), (64, "bf16")])
@pytest.mark.parametrize("T,saved,flags", [
    (1, True, 0), (65, False, 0), (200, True, 0),
    (130, False, rdn.TANH_RESIDUAL), (130, True, rdn.STATELESS_AUX),
])
def test_slice_widths_agree(variant, d, dtype, T, saved, flags):
    x = make_inputs(20, T, 4, d, dtype=dtype, nonzero_state=True, with_grad_out=True,
                    device="cuda", state_std=0.1)
    many = _step(x, variant, saved, flags)
    for n_seq in (1, 4):
        few = _step({n: t[7:7 + n_seq].contiguous() for n, t in x.items()}, variant, saved, flags)
        for n, t in few.items():
            assert torch.equal(t, many[n][7:7 + n_seq]), (n, n_seq)

"""The tensor-core scan over a pair of CTAs per (sequence, head), which calls with
few heads take, against the one-CTA kernel, which calls with more take: the same
operands in the same order, so every result, and every gradient from what it
saved, is the same bits.  (On a chip of 152 SMs 4 heads run in pairs, 80 one CTA
each.)"""
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


@pytest.mark.parametrize("lens,H", [
    ([64] * 80, 2),              # equal lengths in more heads than pairs fit: one CTA each
    ([1, 5] + [3] * 80 + [700], 2),  # one long sequence among many, last: pairs, it first
    ([2, 0, 1] * 400, 1),        # more sequences than are put in order
])
def test_packed_order_and_kernel_choice(lens, H):
    """Packed calls start on the longest sequences and let the table choose the
    kernel: every sequence as in a call of its own, bit for bit."""
    T = sum(lens)
    x = make_inputs(1, T, H, 128, dtype="bf16", device="cuda")
    cu = torch.tensor([0] + lens, dtype=torch.int32).cumsum(0).to(torch.int32).cuda()
    st = 0.1 * torch.randn(2, len(lens), H, 128, 128, generator=torch.Generator().manual_seed(3)).cuda()
    o, ST, RT = rdn.rdn_fwd(*(x[n] for n in NAMES), clip=0.7, S0=st[0], R0=st[1], cu_seqlens=cu)
    first = 0
    for s, n in enumerate(lens):
        if n and (s < 4 or n > 10 or s % 97 == 0):
            sl = {m: x[m][:, first:first + n].clone() for m in NAMES}  # (aligned)
            o1, S1, R1 = rdn.rdn_fwd(*(sl[m] for m in NAMES), clip=0.7,
                                     S0=st[0, s:s + 1].contiguous(), R0=st[1, s:s + 1].contiguous())
            assert torch.equal(o[:, first:first + n], o1), s
            assert torch.equal(ST[s], S1[0]) and torch.equal(RT[s], R1[0]), s
        elif not n:
            assert torch.equal(ST[s], st[0, s]) and torch.equal(RT[s], st[1, s]), s
        first += n

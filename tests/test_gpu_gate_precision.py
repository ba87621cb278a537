"""How far the gate gradients of the bf16 training pass are from 64 bits.  The
per-token sums they are made of cancel, so that they show what a product leaves out
of its operands: the gradients enter those sums in fp32, not as the bf16 hi + lo
pairs that the matrix products take.  The bounds are the errors of the kernels that
summed in fp32 from the start, measured on these inputs, and one in a hundred for
the order of the sums; with hi + lo pairs on both sides dbeta is 4.6 to 81 % past
them."""
import numpy as np
import pytest
import torch

import oracle
import paper_2509_25223_gb300 as rdn
from rdn_synthetic import make_inputs
from tests.parity_util import as64

pytestmark = pytest.mark.gpu

NAMES = ("q", "k", "v", "g", "beta", "gamma")


@pytest.mark.parametrize("variant,B,T,state_std,up,measured", [
    ("rdn", 3, 1000, 0.02, 0.0, dict(dg=5.5656e-06, dbeta=5.6445e-06, dgamma=1.0626e-05)),
    ("rdn", 3, 1000, 0.1, 1.0, dict(dg=5.9486e-06, dbeta=5.7801e-06, dgamma=1.0650e-05)),
    ("rla", 3, 1000, 0.1, 1.0, dict(dg=3.1586e-06, dbeta=3.1541e-06, dgamma=5.4209e-06)),
    ("rdn", 20, 50, 1.0, 1.0, dict(dg=2.0690e-05, dbeta=7.2177e-06, dgamma=7.0276e-05)),
])
def test_gate_gradients_keep_their_precision(variant, B, T, state_std, up, measured):
    H = 16
    x = make_inputs(B, T, H, 128, dtype="bf16", nonzero_state=True, with_grad_out=True,
                    state_std=state_std, device="cuda", seed=7)
    gen = torch.Generator().manual_seed(8)
    dST, dRT = (up * torch.randn(2, B, H, 128, 128, generator=gen)).cuda()
    bwd = rdn.rdn_bwd if variant == "rdn" else rdn.rla_bwd
    # (no clip, so that no element's rounding moves it past a threshold)
    got = bwd(*(x[n] for n in NAMES), x["dO"], clip=float("inf"), S0=x["S0"], R0=x["R0"],
              dST=dST, dRT=dRT)
    ref = oracle.bwd(oracle.RDN if variant == "rdn" else oracle.RLA, *(as64(x[n]) for n in NAMES),
                     float("inf"), as64(x["S0"]), as64(x["R0"]), as64(x["dO"]), dST=as64(dST),
                     dRT=as64(dRT))
    for n, e in measured.items():
        err = np.linalg.norm(as64(got[n]) - ref[n]) / np.linalg.norm(ref[n])
        assert err <= 1.01 * e, (n, err)

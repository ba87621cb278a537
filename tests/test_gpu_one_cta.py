"""The one-CTA forward scan (`fwd_tc_scan`), which calls of more heads than pairs of
CTAs fit take: its give-up path, and the options that the small calls of the other
tests run through the pair kernel."""
import math

import pytest
import torch

import oracle
import paper_2509_25223_gb300 as rdn
from rdn_synthetic import make_inputs
from tests.parity_util import as64, assert_close

pytestmark = pytest.mark.gpu

NAMES = ("q", "k", "v", "g", "beta", "gamma")


def _fwd(variant, x, want, **kw):
    fwd = rdn.rdn_fwd if variant == "rdn" else rdn.rla_fwd
    with rdn.LaunchTimer() as lt:
        out = fwd(*(x[n] for n in NAMES), S0=x["S0"], R0=x["R0"], **kw)
    assert {n for n, _ in lt.records if n.startswith("fwd_tc")} == want
    return out


def _check_heads(variant, x, out, b, **kw):
    sl = {n: x[n][b:b + 1] for n in (*NAMES, "S0", "R0")}
    v = oracle.RDN if variant == "rdn" else oracle.RLA
    ref = oracle.fwd(v, *(as64(sl[n]) for n in NAMES), kw.get("clip", 1.0), as64(sl["S0"]),
                     as64(sl["R0"]), scale=kw.get("scale", 1.0))
    for n, got, r in zip(("o", "ST", "RT"), out, ref):
        assert_close(got[b:b + 1], r, "bf16", n)


@pytest.mark.parametrize("variant", ["rdn", "rla"])
@pytest.mark.parametrize("save", [False, True])
def test_bounded_wait_gives_up_cleanly(variant, save, monkeypatch):
    """RDN_FAULT_INJECT=device_wait with 80 heads: the one-CTA scan skips its first
    completion signal, its waits give up, it drains what it has in flight, reports
    RDN_ERR_TIMEOUT and returns; the next calls are right and leave the word at 0."""
    x = make_inputs(40, 200, 2, 128, dtype="bf16", nonzero_state=True, device="cuda", state_std=0.1)
    kw = {}
    if save:
        kw = dict(return_chunk_states=True, save_for_bwd=True,
                  workspace=torch.empty(rdn.workspace_bytes(variant + "_fwd", 40, 200, 2, 128,
                                                            save_for_bwd=True),
                                        dtype=torch.uint8, device="cuda"))
    rdn.device_status()  # whatever an earlier test left
    monkeypatch.setenv("RDN_FAULT_INJECT", "device_wait")
    _fwd(variant, x, {"fwd_tc_scan"}, **kw)
    assert rdn.device_status() == 4  # RDN_ERR_TIMEOUT
    monkeypatch.delenv("RDN_FAULT_INJECT")
    out = _fwd(variant, x, {"fwd_tc_scan"}, **kw)
    assert rdn.device_status() == 0
    for b in (0, 39):
        _check_heads(variant, x, out, b)


@pytest.mark.parametrize("lens,H", [([60] * 45 + [130], 2),       # the table says one CTA each
                                    ([3] * 80 + [700], 2)])       # ... or pairs
def test_bounded_wait_with_both_kernels_launched(lens, H, monkeypatch):
    x = make_inputs(1, sum(lens), H, 128, dtype="bf16", device="cuda")
    cu = torch.tensor([0] + lens, dtype=torch.int32).cumsum(0).to(torch.int32).cuda()
    both = {"fwd_tc_scan", "fwd_tc_pair"}
    rdn.device_status()
    want = _fwd("rdn", x, both, cu_seqlens=cu)
    monkeypatch.setenv("RDN_FAULT_INJECT", "device_wait")
    _fwd("rdn", x, both, cu_seqlens=cu)
    assert rdn.device_status() == 4
    monkeypatch.delenv("RDN_FAULT_INJECT")
    got = _fwd("rdn", x, both, cu_seqlens=cu)
    assert rdn.device_status() == 0
    for a, b in zip(got, want):
        assert torch.equal(a, b)


@pytest.mark.parametrize("variant", ["rdn", "rla"])
@pytest.mark.parametrize("T,scale,clip,f32", [
    (260, 0.7, 0.7, False), (320, 1.0, 0.0, False), (330, -1.5, math.inf, True), (260, 1.0, 0.5, True),
])
def test_options_equal_the_pair(variant, T, scale, clip, f32):
    x = make_inputs(20, T, 4, 128, dtype="bf16", nonzero_state=True, device="cuda", state_std=0.1)
    kw = dict(scale=scale, clip=clip, f32_out=f32)
    many = _fwd(variant, x, {"fwd_tc_scan"}, **kw)
    few = _fwd(variant, {n: None if t is None else t[7:8].contiguous() for n, t in x.items()},
               {"fwd_tc_pair"}, **kw)
    for a, b in zip(many, few):
        assert torch.equal(a[7:8], b)
    _check_heads(variant, x, many, 3, scale=scale, clip=clip)

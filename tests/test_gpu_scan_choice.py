"""Which forward scan a bf16, d = 128 call takes: one CTA a head (`fwd_tc_scan`) or a
pair (`fwd_tc_pair`), whichever ends first.  Both give the same bits
(tests/test_gpu_pair.py); here it is the choice, at sizes where one of the two took
clearly longer, measured on a chip of 152 SMs (us, one CTA / pairs)."""
import pytest
import torch

import paper_2509_25223_gb300 as rdn
from rdn_synthetic import make_inputs

pytestmark = pytest.mark.gpu

NAMES = ("q", "k", "v", "g", "beta", "gamma")
ONE, PAIR = "fwd_tc_scan", "fwd_tc_pair"


@pytest.fixture(autouse=True)
def _chip():
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("measured on 152 SMs")


def _scans(variant, x, **kw):
    """The scan kernels a forward launches, and its workspace."""
    B, T, H, D = x["q"].shape
    ws = torch.empty(rdn.workspace_bytes(variant + "_fwd", B, T, H, D, cu_seqlens=kw.get("cu_seqlens")),
                     dtype=torch.uint8, device="cuda")
    fwd = rdn.rdn_fwd if variant == "rdn" else rdn.rla_fwd
    with rdn.LaunchTimer() as lt:
        fwd(*(x[n] for n in NAMES), workspace=ws, **kw)
    return {n for n, _ in lt.records if n in (ONE, PAIR)}, ws


@pytest.mark.parametrize("variant,heads,T,states,want", [
    ("rdn", 16, 64, False, ONE),      # 18.3 / 20.5
    ("rdn", 4, 1, False, ONE),        # 18.0 / 20.9
    ("rdn", 16, 256, False, PAIR),    # 38.8 / 34.7
    ("rdn", 32, 128, True, ONE),      # 28.6 / 28.7
    ("rdn", 76, 512, True, PAIR),     # 83.9 / 70.0
    ("rla", 16, 192, False, ONE),     # 24.9 / 26.6
    ("rla", 16, 512, False, PAIR),    # 51.5 / 47.0
    ("rdn", 77, 512, False, ONE),     # 67.5 / 103
    ("rdn", 200, 512, False, ONE),    # 133 / 168
    ("rla", 160, 1024, True, ONE),    # 244 / 287
])
def test_equal_sequences(variant, heads, T, states, want):
    x = make_inputs(heads, T, 1, 128, dtype="bf16", device="cuda", device_rng=True)
    got, _ = _scans(variant, x, return_chunk_states=states)
    assert got == {want}


def _table(ws, n):
    """The n + 1 chunk numbers of the sequence table at the workspace's end."""
    size = (16 * (n + 1) + 255) // 256 * 256
    return ws[ws.numel() - 256 - size:][:16 * (n + 1)].view(torch.int64)[1::2].cpu()


def _table_says_pairs(ws, n):
    """The choice: the upper half of entry n's chunk number."""
    return int(_table(ws, n)[n]) >> 32 != 0


@pytest.mark.parametrize("lens,H,want", [
    ([30] * 500 + [8000], 16, ONE),   # 887 / 1922: each pair's start costs more than the long one gains
    ([200] * 60 + [4000], 16, ONE),   # 458 / 491
    ([500] * 30 + [10000], 16, PAIR),  # 1114 / 780
    ([30] * 80 + [8000], 16, PAIR),   # 886 / 564
    ([30] * 200 + [16000], 4, PAIR),  # 1750 / 1093
])
def test_packed_sequences(lens, H, want):
    x = make_inputs(1, sum(lens), H, 128, dtype="bf16", device="cuda", device_rng=True)
    cu = torch.tensor([0] + lens, dtype=torch.int32).cumsum(0).to(torch.int32).cuda()
    got, ws = _scans("rdn", x, cu_seqlens=cu)
    assert got == {ONE, PAIR}  # (the lengths are on the device: both are launched)
    assert _table_says_pairs(ws, len(lens)) == (want == PAIR)


@pytest.mark.parametrize("variant,lens,H", [
    ("rdn", [16, 64, 40, 33] * 300, 4),   # more sequences than are put in order
    ("rdn", [2] * 900, 16),               # too few chunks for any one to be long enough
    ("rla", [30] * 40 + [300], 40),       # too many heads for it
])
def test_packed_pairs_are_not_launched_where_they_cannot_run(variant, lens, H):
    """The kernel that the table does not choose returns at once, which still takes
    each of its CTAs an SM (0.64 us each, 262 us for 2000 sequences of 16 heads)."""
    x = make_inputs(1, sum(lens), H, 128, dtype="bf16", device="cuda", device_rng=True)
    cu = torch.tensor([0] + lens, dtype=torch.int32).cumsum(0).to(torch.int32).cuda()
    got, ws = _scans(variant, x, cu_seqlens=cu)
    assert got == {ONE} and not _table_says_pairs(ws, len(lens))


@pytest.mark.parametrize("n", [1, 2, 15, 256, 257, 511, 600, 1023, 1024, 1025])
def test_packed_order(n):
    """The order in which packed sequences start: by chunks, most first, equal ones as
    they come; above 1024 as they come."""
    lens = torch.randint(0, 400, (n,), generator=torch.Generator().manual_seed(n)).tolist()
    x = make_inputs(1, max(sum(lens), 1), 1, 64, dtype="bf16", device="cuda", device_rng=True)
    lens[-1] += 1 if sum(lens) == 0 else 0
    cu = torch.tensor([0] + lens, dtype=torch.int32).cumsum(0).to(torch.int32).cuda()
    _, ws = _scans("rdn", x, cu_seqlens=cu)
    order = (_table(ws, n)[:n] >> 32).tolist()
    chunks = [(c + 63) // 64 for c in lens]
    assert order == (sorted(range(n), key=lambda s: -chunks[s]) if n <= 1024 else list(range(n)))


@pytest.mark.parametrize("variant", ["rdn", "rla"])
def test_short_sequences_in_pairs(variant):
    """Sequences of one and two chunks by the pair kernel, which they take only beside
    a long one: results, kept states and the gradients from what it saved are those of
    a call of their own, bit for bit."""
    lens, H = [1, 64, 65, 128, 0, 63] + [30] * 74 + [700], 2
    T, N = sum(lens), len(lens)
    x = make_inputs(1, T, H, 128, dtype="bf16", with_grad_out=True, device="cuda")
    cu = torch.tensor([0] + lens, dtype=torch.int32).cumsum(0).to(torch.int32).cuda()
    st = 0.1 * torch.randn(4, N, H, 128, 128, generator=torch.Generator().manual_seed(5)).cuda()
    fwd, bwd = (rdn.rdn_fwd, rdn.rdn_bwd) if variant == "rdn" else (rdn.rla_fwd, rdn.rla_bwd)

    def step(x, st, cu):
        B, T = x["q"].shape[:2]
        kw = dict(clip=0.7, S0=st[0], R0=st[1], cu_seqlens=cu)
        ws = torch.empty(rdn.workspace_bytes(variant + "_fwd", B, T, H, 128, save_for_bwd=True,
                                             cu_seqlens=cu), dtype=torch.uint8, device="cuda")
        o, ST, RT, Sc, Rc = fwd(*(x[n] for n in NAMES), return_chunk_states=True, save_for_bwd=True,
                                workspace=ws, **kw)
        d = bwd(*(x[n] for n in NAMES), x["dO"], S_chunks=Sc, R_chunks=Rc, dST=st[2], dRT=st[3],
                fwd_workspace=ws, fwd_saved=True, **kw)
        return ws, dict(o=o, **{n: d[n] for n in ("dq", "dk", "dv", "dg", "dbeta", "dgamma")}), \
            dict(ST=ST, RT=RT, dS0=d["dS0"], dR0=d["dR0"]), (Sc, Rc)

    ws, tok, per, chunks = step(x, st, cu)
    assert _table_says_pairs(ws, N)
    first = slot = 0
    for s, n in enumerate(lens):
        nc = (n + 63) // 64
        if n and (s < 8 or n > 64):
            sl = {m: t[:, first:first + n].clone() for m, t in x.items() if t is not None}
            _, tok1, per1, chunks1 = step(sl, st[:, s:s + 1].contiguous(), None)
            for m, t in tok1.items():
                assert torch.equal(tok[m][:, first:first + n], t), (s, m)
            for m, t in per1.items():
                assert torch.equal(per[m][s:s + 1], t), (s, m)
            for a, b in zip(chunks, chunks1):
                assert torch.equal(a[slot:slot + nc * H], b.reshape(-1, 128, 128)), s
        first, slot = first + n, slot + nc * H

"""bench.py knows the work of every kernel that can be the longest of a training step:
all that the library launches but the small ones beside it."""
import glob
import os
import re

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BESIDE = {"seq_table", "tied_gate_grad", "qk_prologue", "qk_prologue_bwd", "decode"}


def test_every_step_kernel_has_its_work():
    names = set()
    for f in glob.glob(os.path.join(ROOT, "paper_2509_25223_gb300", "csrc", "*.cu")):
        for arg in re.findall(r"RDN_LAUNCH\(([^,]*),", open(f).read()):
            names |= set(re.findall(r'"(\w+)"', arg))
    assert {"fwd_tc_scan", "fwd_tc_pair", "bwd_post_f32", "chunk_recompute"} <= names
    assert names - BESIDE == set(bench.KERNEL_WORK)
    work = bench.flops_per_token_head()
    assert all(w in work for w in bench.KERNEL_WORK.values())

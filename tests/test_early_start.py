"""Kernels that may start before the kernel ahead of them ends (launch_after) read what earlier
kernels write by ordinary loads: only the graph's tables are const __restrict__ in them."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2004_03493_gb300", "csrc")
FILES = [f for f in sorted(os.listdir(CSRC)) if f.endswith(".cu")]
# the CSRs, the segments of their long rows, 1/din, the positions of the gathered vectors
TABLES = {"rp", "col", "in_rp", "in_col", "seg", "long_rows", "long_first", "inv_din", "pos"}
READ_ONLY = re.compile(r"const\s+[\w:<>. ]+?\*\s*__restrict__\s+(\w+)")


def _sources():
    return {f: open(os.path.join(CSRC, f)).read() for f in FILES}


def _early_kernels(text):
    calls = re.findall(r"(?:launch_after|each_node)\((?:[^;{}]*?)\b(\w+_kernel)\b", text)
    if "sweep_level" in text:
        calls.append("sell_rows_kernel")
    return set(calls)


def _signature(text, kernel):
    at = re.search(r"__global__[^;{}]*?\b" + kernel + r"\(", text).end()
    return text[at:text.index("{", at)]


def test_early_kernels_are_found():
    found = set().union(*(_early_kernels(t) for t in _sources().values()))
    assert {"sell_rows_kernel", "reach_rows_kernel", "topk_pick_kernel", "batch_rows_kernel", "zv_finalize_kernel",
            "alloc_scan_kernel", "probe_end_kernel", "reverse_init_d_kernel"} <= found


def test_only_graph_tables_are_read_only():
    bad = []
    for name, text in _sources().items():
        for kernel in _early_kernels(text):
            bad += [(name, kernel, p) for p in READ_ONLY.findall(_signature(text, kernel)) if p not in TABLES]
        # the epilogues that these kernels take as arguments
        for op, body in re.findall(r"struct (\w*Op\w*) \{(.*?)\n\};", text, re.S):
            bad += [(name, op, p) for p in READ_ONLY.findall(body) if p not in TABLES]
    assert not bad


def test_every_early_kernel_waits():
    for name, text in _sources().items():
        for kernel in _early_kernels(text):
            at = re.search(r"__global__[^;{}]*?\b" + kernel + r"\(", text).start()
            body = text[at:text.index("\n}\n", at)]
            assert "prior_done();" in body, (name, kernel)

"""Checks, from the kernels' sources, of rules that no run can be made to break safely: a missing release or a
copy still in flight at a kernel's exit corrupts memory only now and then."""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_12659_gb300", "csrc")


def _source(*path):
    with open(os.path.join(CSRC, *path)) as f:
        return f.read()


def _sources():
    for d, _, names in os.walk(CSRC):
        for n in names:
            if n.endswith((".cu", ".cuh", ".h")):
                yield os.path.relpath(os.path.join(d, n), CSRC), _source(d, n)


def test_arrivals_on_a_peers_barrier_release_the_reads_before_them():
    # A peer that waits for such an arrival overwrites what the arriving warp has just read.
    found = 0
    for name, text in _sources():
        for arrival in re.findall(r"mbarrier\.arrive\.[\w.:]*shared::cluster\.b64", text):
            found += 1
            assert arrival.startswith("mbarrier.arrive.release.cluster."), f"{name}: {arrival}"
    assert found == 1


# The thread that fills a ring of shared-memory stages waits for its last copies before it leaves its role.
RINGS = {"gemm_rows.cuh": "full, RT_STAGES", "gemm_big.cuh": "full, STAGES", "mod_tc.cu": "full, MT_STAGES",
         "prefill/prefill.cu": "full, PG_STAGES"}


def test_ring_loaders_wait_for_their_last_copies():
    for name, ring in RINGS.items():
        text = _source(*name.split("/"))
        loader, rest = text.index("if (warp == 0) {"), text.index("} else if (warp == 1) {")
        assert f"ring_drain({ring}," in text[loader:rest], name


def test_attention_loaders_wait_for_their_last_copies():
    text = _source("attn_t5_kernel.cuh")
    loaders = text[text.index("if (warp <= 1) {"):text.index("} else if (warp == 2) {")]
    assert "ring_drain(fullb, NS, issued," in loaders
    assert "mbar_wait_bounded(qfull," in loaders


def test_single_shot_loads_are_waited_for_again_after_a_wait_gave_up():
    # The K-split projection's two operand barriers, and the split-KV attention's key block and queries.
    gemm = _source("gemm_kernel.cuh")
    gave_up = gemm[gemm.rindex("if (*flag != 0) {"):]
    assert "mbar_wait_bounded(&bars[0]," in gave_up and "mbar_wait_bounded(&bars[1]," in gave_up
    attn = _source("attn_tc.cu")
    gave_up = attn[attn.index("if (!landed && tid == 0) {"):attn.index("const uint32_t kbuf_u")]
    assert "drain_two(&kvbar[bi], par, qbar, 0," in gave_up


def test_device_errors_are_reported_after_the_last_barrier():
    # One thread reports for the block: a role that gives up later than it must still be heard.
    for name in ("gemm_rows.cuh", "gemm_big.cuh", "mod_tc.cu", "attn_t5_kernel.cuh", "prefill/prefill.cu"):
        text = _source(*name.split("/"))
        report = [m.start() for m in re.finditer(r"if \(tid == 0 && \*flag != 0\)", text)]
        assert len(report) == 1, name
        last = text.rindex("*flag = ", 0, report[0])
        assert "__syncthreads();" in text[last:report[0]], name


def test_no_source_uses_cluster_multicast():
    # The library and its probe also belong to programs that run on several GPUs.
    for name, text in _sources():
        assert "multicast::cluster" not in text, name

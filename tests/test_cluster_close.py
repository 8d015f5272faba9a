"""Kernels that write into a cluster partner's shared memory close with a cluster barrier.

A CTA that leaves while a partner still sends to it would have that store hit shared memory that is no longer its
own.  On the way that no wait gives up, waits for all bytes already prevent that, so only the source shows whether
a kernel closes on every way out; this reads it.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2311_18056_gb300", "csrc")
SEND = re.compile(r"\b(cl_send1|cl_send4|st_async4|st_cluster4|tile_epilogue<|solve_body<)")
CLOSE = re.compile(r"\b(cl_close|cluster_sync)\(")


def kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__ void (?:__launch_bounds__\([^{;]*?\)\s*)?(\w+)\s*\(", text):
            beg = text.index("{", m.end())
            end = text.index("\n}\n", beg)
            yield os.path.basename(path), m.group(1), text[beg:end]


def test_senders_close_with_a_cluster_barrier():
    senders = []
    for file, name, body in kernels():
        sends = [m.start() for m in SEND.finditer(body)]
        if sends:
            senders.append(name)
            assert any(m.start() > sends[-1] for m in CLOSE.finditer(body)), (file, name)
    assert {"single_solve_kernel", "batch_chunk_fp32_kernel", "tc_gemm_kernel", "tc_chunk_kernel", "tc_small_kernel",
            "diag_cluster_kernel"} <= set(senders), senders

"""Kernels launched with programmatic dependent launch (csrc/launch_util.h) start while the kernel before
them may still write: only what the host uploads (descriptors and task lists) or what is touched by
atomics alone (task queues) may be a __restrict__ parameter of theirs, since loads through such a
pointer may take the read-only path or move before the wait.  CPU only: reads the sources."""
import os
import re

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2202_09288_gb300", "csrc")
UPLOADED = {"tasks", "sns", "mats", "segs", "groups", "srcs", "queue"}


def kernels():
    """(file, kernel, parameters, text after them) of every kernel launched that way."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        text = open(os.path.join(CSRC, f)).read()
        launched = re.findall(r"\blaunch_pdl\(([^,]*),", text)  # the first argument
        for k in sorted({k for arg in launched for k in re.findall(r"\bk_\w+", arg)}):
            m = re.search(r"__global__[^;{]*?\b" + k + r"\(([^{;]*?)\)\s*\{", text)
            yield f, k, m.group(1), text[m.end():]


def test_only_uploaded_data_is_restrict():
    found = list(kernels())
    assert {k for _, k, _, _ in found} >= {
        "k_potrf", "k_trsm_blk", "k_schur_f64", "k_assemble_owner", "k_diag_inverse", "k_oz_slice",
        "k_schur_oz", "k_trsm_oz", "k_tf32_split", "k_schur_tf32", "k_fwd_y", "k_fwd_diag", "k_bwd_y",
        "k_bwd_diag"}
    for f, k, params, body in found:
        restricted = set(re.findall(r"__restrict__\s+(\w+)", params))
        assert restricted <= UPLOADED, (f, k, restricted - UPLOADED)
        assert "pdl_wait();" in body[:body.index("\n}")], (f, k)

"""Kernels launched as programmatic dependents may be resident while their predecessor still writes.  What they read after their
wait must therefore not go through the read-only data path, which needs data that does not change while the kernel runs
(`__ldg`, or a `const __restrict__` parameter).  A race of this kind cannot be provoked on demand, so the sources are read."""
import glob
import os
import re

from conftest import ROOT

WAIT = re.compile(r"pdl_wait\(\)|griddepcontrol\.wait")
# parameters that are complete before the kernel can start: the first kernel of the call has waited for whatever wrote them,
# and lets the later ones go only after that wait
COMPLETE_BEFORE = {"k_pack_scatter": {"wm", "pid"}, "k_assign_count": {"w"}}
# read with __ldcg only, which bypasses the read-only path
BYPASS = {"k_select_rest": {"key"}, "k_select_cluster": {"key"}}


def kernels():
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_2001_07710_b200", "csrc", "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(([^{;]*?)\)\s*\{", text, re.S):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            yield os.path.basename(path), m.group(1), m.group(2), text[m.end():i]


def test_nothing_written_by_a_running_predecessor_is_read_through_the_read_only_path():
    seen = set()
    for name, kernel, params, body in kernels():
        wait = WAIT.search(body)
        if not wait:
            continue
        seen.add(kernel)
        allowed = COMPLETE_BEFORE.get(kernel, set()) | BYPASS.get(kernel, set())
        for p in params.split(","):
            if "const" in p and "__restrict__" in p:
                assert p.split()[-1] in allowed, f"{name}: {kernel}: parameter {p.strip()}"
        for var in BYPASS.get(kernel, set()):
            for use in re.finditer(r"\b%s\s*[+\[]" % var, body):
                assert "__ldcg(" in body[use.start() - 8:use.end()], f"{name}: {kernel} reads {var} without __ldcg"
        if kernel not in COMPLETE_BEFORE:
            assert "__ldg(" not in body[wait.end():], f"{name}: {kernel} uses __ldg after its wait"
            if kernel == "k_select_pattern":          # waits first when it is the first kernel of its call
                assert "__ldg(" not in body
    assert {"k_conv_mma_f16", "k_conv_mma_f32", "k_pack_count", "k_pack_scatter", "k_select_pattern", "k_pick_survivors", "k_reduce_parts_f32"} <= seen

"""Kernels launched with programmatic stream serialisation start while the kernel before them still
runs.  Each of them waits for it (behind_wait), and takes only what was complete before the chain
began through the read-only path: __ldg promises that the data do not change while the kernel lives,
which holds for the MPO tables (written by a copy) and not for the outputs of the kernel before."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2003_13245_gb300", "csrc")
TABLES = ("rows + sig", "o.mix_cu", "o.mix_val")


def sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, f)) as fh:
                yield f, fh.read()


def body(text, name):
    """The kernel's text from its name to its closing brace, or None."""
    m = re.search(r"__global__[^;{]*?\b%s\(" % name, text)
    if not m:
        return None
    i = text.index("{", m.end())
    depth, k = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        k += 1
        if depth == 0:
            return text[i:k]


def test_overlapped_kernels_wait_and_read_coherently():
    texts = dict(sources())
    names = set()
    for t in texts.values():
        for call in re.findall(r"launch_behind\(([^;]*?);", t):
            names |= set(re.findall(r"\b(\w+_kernel)\b", call))
    assert "digit_gemm_kernel" in names and "tc_zgemm_kernel" in names and len(names) >= 8
    for n in names:
        bodies = [b for b in (body(t, n) for t in texts.values()) if b]
        assert len(bodies) == 1, n
        assert "behind_wait();" in bodies[0], n
        for arg in re.findall(r"__ldg\(([^()]*)", bodies[0]):
            assert arg.startswith(TABLES), "%s reads %s through the read-only path" % (n, arg)

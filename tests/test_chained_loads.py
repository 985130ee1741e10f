"""Kernels of a chain of launches are resident while the launch before them still writes, so
the read-only load path (__ldg, const __restrict__ parameters) is left to what nobody writes
meanwhile.  Every use of it in the sources is one of those listed here."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_12912_gb300", "csrc")

# what __ldg may read: the log2 table; an archive's units (complete before the call's first
# launch, which is an ordinary one behind a memset); the caller's selector weights, likewise;
# and everything in the one training kernel that is launched alone (mlp_predict_kernel)
LDG = {"kLog2Table.v", "in", "w", "feat"}
# restrict parameters of kernels that may be chained: the caller's field, and the tables of
# batches, which are uploaded when the batch is made
RESTRICT = {"x", "tasks", "tile0", "cta0"}


def _sources():
    for f in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, f)) as h:
            yield f, re.sub(r"//[^\n]*", "", h.read())


def _kernels(text):
    """(name, parameters, body) of every kernel."""
    for m in re.finditer(r"__global__[^;{]*?\bvoid\s+(\w+)\s*\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        params, j = text[m.end():i - 1], text.index("{", i)
        depth, k = 1, j + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        yield m.group(1), params, text[j:k]


def test_read_only_loads():
    for f, text in _sources():
        for name in re.findall(r"__ldg\(\s*&\s*([\w.]+)\[", text):
            assert name in LDG, (f, name)
        assert len(re.findall(r"__ldg\(", text)) == len(re.findall(r"__ldg\(\s*&\s*[\w.]+\[", text)), f


def test_chained_kernels():
    seen = 0
    for f, text in _sources():
        for name, params, body in _kernels(text):
            if "chained_begin()" not in body:
                assert name not in {"mlp_grad_kernel", "mlp_update_kernel", "plan_kernel", "payload_kernel"}
                continue
            seen += 1
            assert body[1:].lstrip().startswith("chained_begin();"), (f, name)
            for p in re.findall(r"__restrict__\s+(\w+)", params):
                assert p in RESTRICT, (f, name, p)
            # (feature and weight loads through __ldg: only where nothing is chained)
            assert not re.search(r"__ldg\(\s*&\s*(feat|w)\[", body), (f, name)
    assert seen >= 18

"""The training kernels run as programmatic dependents: a kernel may start while the one
before it still runs, and sees what earlier kernels wrote only after its own wait.  Read from
the source (no GPU): every access to what an update writes lies behind the wait, and no such
pointer is declared const __restrict__ (which would let the compiler read it ahead of the
wait or through a path that is not coherent)."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_1211_6932_gb300", "csrc", "lbm_mlp.cu")
WRITTEN = ("w", "master", "m1", "m2", "update_counter")
WAIT = "wait_predecessor();"


def kernel(name):
    """(parameter list, body) of a kernel, without comments."""
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    head = text.index(name + "(")
    start = text.index("{", head)
    depth, end = 0, start
    for end in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        if depth == 0:
            break
    return text[head + len(name):start], text[start:end + 1]


def accesses(code):
    return re.findall(r"(?:\b(?:%s|lrow)\s*\[|\*\s*update_counter|cast<const uint4\*>\(w\)|"
                      r"\brb\.\w+\s*\[)" % "|".join(WRITTEN), code)


def test_what_an_update_writes_is_not_declared_read_only():
    for name in ("mlp_rows_kernel", "mlp_param_kernel"):
        for p in kernel(name)[0].split(","):
            if p.strip(" )(\n").split("*")[-1].replace("__restrict__", "").strip() in WRITTEN:
                assert "__restrict__" not in p, (name, p)


def test_rows_kernel_reads_the_weights_behind_its_wait():
    before, after = kernel("mlp_rows_kernel")[1].split(WAIT)
    assert not accesses(before) and accesses(after)


def test_parameter_kernel_reads_the_update_behind_its_waits():
    loss_head, rest, main = kernel("mlp_param_kernel")[1].split(WAIT)
    cut = rest.index("return;")  # the end of the loss block's branch
    assert not accesses(loss_head) and accesses(rest[:cut])
    assert not accesses(rest[cut:]) and accesses(main)

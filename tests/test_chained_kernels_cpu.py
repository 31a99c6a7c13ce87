"""Kernels that start under the tail of the one before them (they call
``after_previous``) read what that one is still writing when they start.  A
load through the read-only path, or from a ``const __restrict__`` pointer,
promises data that nobody writes while the kernel lives, and the compiler may
move it above the wait.  Only the weights keep that promise: their last writer
is complete before the chain begins."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2606_02226_gb300", "csrc", "cfs_sampler.cu")
WEIGHTS = {"wb", "w"}


def _functions(text):
    """name -> (signature, body) of the file's device code."""
    out = {}
    for m in re.finditer(r"^(?:template <[^\n]*>\n)?__(?:global|device)__[^;{]*?(\w+)\(", text, re.M):
        body = text.index("\n{", m.end())
        out.setdefault(m.group(1), (text[m.start():body], text[body:text.index("\n}\n", body)]))
    return out


def test_chained_kernels_read_with_ordinary_loads():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    # the launch bounds' parentheses come before the name
    text = re.sub(r"__launch_bounds__\([^()]*\)", "", text)
    fns = _functions(text)
    chained = [n for n, (sig, body) in fns.items() if "__global__" in sig and "after_previous()" in body]
    assert {"data_kernel", "train_fwd_kernel", "sw_kernel", "out_backward_kernel",
            "back_rows_kernel", "tc_dw_kernel", "adam_kernel"} <= set(chained)
    todo, seen = list(chained), set()
    while todo:
        name = todo.pop()
        if name in seen:
            continue
        seen.add(name)
        sig, body = fns[name]
        held = set(re.findall(r"const [\w ]+\* ?__restrict__ (\w+)", sig))
        assert held <= WEIGHTS, (name, held - WEIGHTS)
        assert not re.search(r"__ldg\(|\.nc\b|ld_stream", body), name
        todo += [n for n in fns if re.search(r"\b%s(?:<[^<>;]*>)?\(" % n, body)]
    assert "part_reduce" in seen

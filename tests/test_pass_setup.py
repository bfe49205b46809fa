"""Order of the pass kernel's set-up, read from its source (CPU only).

The next kernel of a stream may be placed on an SM as soon as every CTA of the
running one has let it in.  Both want all of the SM's tensor memory, whose
allocation has no time limit, so a CTA lets the next kernel in only when it
holds its own: otherwise the next kernel could take the columns and wait for
this kernel, while this kernel waits for the columns."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1908_06649_gb300", "csrc")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _body(text, name):
    """The braces of the function `name` (its definition)."""
    for m in re.finditer(r"\b%s\s*\(" % name, text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        if text[i:].lstrip().startswith("{"):
            i = text.index("{", i)
            depth, j = 1, i + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[j], 0)
                j += 1
            return text[i:j]
    raise AssertionError("no definition of %s" % name)


def test_next_kernel_is_let_in_after_the_tensor_memory_is_allocated():
    text = _source("group_kernel.cuh")
    body = _body(text, "dft_pass_kernel")
    assert body.count("launch_dependents()") == 1
    # the allocation, and the barrier after which every warp's CTA holds it
    assert "tmem_alloc(" in _body(text, "kernel_setup_start")
    assert "__syncthreads()" in _body(text, "kernel_setup_finish")
    assert (body.index("kernel_setup_start<") < body.index("kernel_setup_finish(")
            < body.index("launch_dependents()"))
    # no other kernel lets its successor in
    for f in sorted(os.listdir(CSRC)):
        if f != "tcgen05.cuh":
            assert _source(f).count("launch_dependents()") == (f == "group_kernel.cuh"), f


def test_every_thread_waits_for_the_kernels_before_it_touches_data():
    body = _body(_source("group_kernel.cuh"), "dft_pass_kernel")
    head = body[:body.index("wait_prior_grids()")]
    # neither a branch around the wait, nor an input copy or an early return before it
    assert head.count("{") - head.count("}") == 1
    assert "nx.issue(" not in head and "return;" not in head

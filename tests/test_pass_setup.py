"""Order of the pass kernel's set-up and leaving, read from its source (CPU only).

The next kernel of a stream may be placed on an SM as soon as every CTA of the
running one has let it in.  Both want all of the SM's tensor memory, whose
allocation has no time limit, so a CTA lets the next kernel in only when it
holds its own: otherwise the next kernel could take the columns and wait for
this kernel, while this kernel waits for the columns.

A CTA whose wait ran out leaves with an error.  A bulk copy that has not landed
by then would write into the shared memory of whoever gets the SM next, so it
first waits until every mbarrier that copies complete on has nothing outstanding,
whichever warp issued the copy and whichever wait failed."""
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


def test_a_failed_kernel_waits_for_every_copy_in_flight():
    text = _source("group_kernel.cuh")
    # the mbarriers that copies complete on: the staging's, the twiddles' and the tables'
    bars = set(re.findall(r"mbar_expect_tx\(([^,]+),", text))
    assert bars == {"w.bar_stg", "w.bar_tws", "smem_u32(tbar)"}
    body = _body(text, "drain_copies")
    assert "if (stg) drain_barrier(w.bar_stg);" in body
    assert "if (tws) drain_barrier(w.bar_tws);" in body
    assert "uint64_t *tbar = mbar + 3 * NWG + 1;" in _body(text, "kernel_setup_start")
    assert "mbar_wait_bounded(smem_u32(mbar + 3 * nwg + 1), 0, kDrainNs)" in body
    # whatever phase is incomplete: a thread's own phase bit has moved on when the
    # wait for that copy ran out
    assert "ph_" not in body + _body(text, "drain_barrier")
    # the first copy counts before the warp that waits has issued one itself
    assert "nx{P, &a.tm_in, item, nitems, item < nitems};" in _body(text, "dft_pass_kernel")
    # the one-launch schedules: whatever their state says
    for kernel in ("dft_fused_kernel", "dft_pair_kernel"):
        assert re.search(r"(kernel_teardown\(tbase, w|drain_copies\(w), w\.fail, ",
                         _body(text, kernel))
    assert "drain_copies(" in _body(text, "kernel_teardown")

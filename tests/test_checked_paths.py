"""The bounds-checked library covers every path that addresses memory itself.

By reading (CPU): each function of the pass kernels that copies, loads or stores
by an address of its own checks the index.  On the GPU: the pass variants' parity
tests, run through that library; check() raises for an index out of range."""
import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _functions(text):
    """(name, body) of every function defined at the outermost level."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"^(?:template <[^\n]*>\n|)[^\n]*__device__[^;{]*?\b(\w+)\s*\(", text,
                         re.M):
        at = text.index("(", m.end() - 1)
        depth = 0
        for i in range(at, len(text)):
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            if not depth:
                break
        if not text[i + 1:].lstrip().startswith("{"):
            continue
        start = text.index("{", i)
        depth = 0
        for j in range(start, len(text)):
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            if not depth:
                break
        yield m.group(1), text[start:j + 1]


def test_every_function_that_addresses_memory_checks_its_indexes():
    path = os.path.join(ROOT, "paper_1908_06649_gb300", "csrc", "group_kernel.cuh")
    access = re.compile(r"\b(cp_async4|cp_async8|tma_load_1d\w*|__ldg|__stcs|__stcg|"
                        r"st_global_hint|st_shared_f2)\s*\(|\bw\.(stg|buf)\[")
    found = {}
    for name, body in _functions(open(path).read()):
        if access.search(body):
            found[name] = "in_range(" in body
    # the tables: whole arrays of the plan, of sizes fixed when the kernel is compiled
    assert found.pop("kernel_setup_start") is False
    assert {"gather_rows", "scatter_rows", "mix_q", "half_row_store", "last_stage_store",
            "issue_input", "issue_half_rows"} <= set(found)
    assert not [n for n, checked in found.items() if not checked]


@pytest.mark.gpu
def test_pass_variants_run_clean_in_the_checked_library():
    from paper_1908_06649_gb300 import _build
    _build.build(checked=True)
    env = dict(os.environ, TCU_DFT_CHECKED="1")
    r = subprocess.run([sys.executable, "-m", "pytest", "-x", "-q", "-p", "no:cacheprovider",
                        "-m", "gpu", os.path.join(ROOT, "tests", "test_pass_variants.py")],
                       env=env, cwd=ROOT, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-2000:]
    assert " passed" in r.stdout

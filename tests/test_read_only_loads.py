"""Read-only loads (__ldg) in the CUDA sources, by reading them on the CPU.

A read-only load may be served from a path that promises nothing for memory
that the same kernel writes, and to the compiler the data behind it is the same
before and after the wait of a programmatic dependent launch."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2001_03477_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def function(text, name):
    """(parameter list, body) of the function defined as `name`(...) {...}."""
    for m in re.finditer(r"\b" + name + r"\s*\(", text):
        i, depth = m.end(), 1
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        if text[i:].lstrip().startswith("{"):
            j = text.index("{", i)
            k, depth = j + 1, 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[k], 0)
                k += 1
            return text[m.end():i - 1], text[j + 1:k - 1]
    raise AssertionError(name)


def test_words_tagged_by_the_same_kernel_are_read_by_ordinary_loads():
    """The step's shift marks receivers in the c words whose stencils it reads."""
    text = source("vof_shift.cu")
    params, body = function(text, "shift_plane_cell")
    assert "atomicOr" in body and "sc.mark" in body  # the kernel that writes them
    assert re.search(r"const double\*\s+c_in", params), "c_in is written through sc.mark: no restrict"
    load = re.search(r"=\s*STEP \? c_value\(\*p\) : __ldg\(p\);", body)
    assert load and len(re.findall(r"__ldg\(", body)) == 2  # and dd, which nothing writes
    assert re.search(r"__ldg\(dd \+ id\)", body)
    for kernel, form in (("k_shift_mark", "true"), ("k_shift_mark_grp", "true"), ("k_shift_planes", "false")):
        assert f"k_shift_planes_body<{form}>(" in function(text, kernel)[1], kernel


def test_step_reads_the_fields_behind_its_wait():
    """The step's first kernel streams c and e, which the grid ahead may write,
    at addresses that depend on nothing loaded; the step's other kernels load
    their lists' lengths first."""
    text = source("vof_tiles.cu")
    body = function(text, "k_tiles")[1]
    assert re.search(r"pdl_wait\(\);\s*k_tiles_body\(A\.g, after_wait\(A\.c\), after_wait\(A\.e\),", body)


def test_the_step_kernels_wait_first():
    """By name: every kernel of a time step starts with the wait."""
    for name, kernels in (("vof_tiles.cu", ("k_tiles", "k_quiet")), ("vof_fused.cu", ("k_mix", "k_walk")),
                          ("vof_shift.cu", ("k_shift_mark", "k_shift_sweep", "k_shift_apply", "k_reduce_fused"))):
        text = source(name)
        for k in kernels:
            body = re.sub(r"__shared__[^;]*;", "", function(text, k)[1])
            assert body.split(";")[0].strip() == "pdl_wait()", k
            assert re.search(r"launch_pdl\(" + k + r"\b", text), k

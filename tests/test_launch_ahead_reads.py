"""What kernels launched ahead may read, checked in their sources.

A kernel that launch_step starts can be resident while the kernel before it
on the stream still writes (programmatic dependent launch).  Two rules follow:

  * what that kernel wrote is read after griddepcontrol.wait (step_begin), and
    not through the read-only path: ld.global.nc asks that the data not change
    while the kernel is resident, and a `const T* __restrict__` parameter lets
    the compiler choose it (or move the load above the wait).  Links, shifts
    and targets, which no kernel of a block step writes, are exempt;
  * whatever is read before the wait is either such a constant or was acquired
    from its writer by a release / acquire pair.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1205_0359_gb300", "csrc")
CONSTANT = {"links", "sigma", "target"}      # written before a block step starts


def _sources():
    txt = "".join(open(os.path.join(CSRC, f)).read() + "\n" for f in sorted(os.listdir(CSRC))
                  if f.endswith((".cu", ".cuh", ".h")))
    txt = re.sub(r"/\*.*?\*/", " ", txt, flags=re.S)
    return re.sub(r"//[^\n]*", " ", txt)


def _close(txt, at, o, c):
    depth = 0
    for i in range(at, len(txt)):
        depth += (txt[i] == o) - (txt[i] == c)
        if depth == 0:
            return i
    raise AssertionError("unbalanced source")


def _function(txt, name):
    """Parameter list and body of the definition of a kernel or device function."""
    for h in re.finditer(r"\b" + name + r"\s*\(", txt):
        end = _close(txt, h.end() - 1, "(", ")")
        rest = txt[end + 1:].lstrip()
        if rest.startswith("{"):
            b = txt.index("{", end)
            return txt[h.end():end], txt[b:_close(txt, b, "{", "}") + 1]
    raise AssertionError(f"{name} is not defined")


TXT = _sources()
KERNELS = sorted(set(re.findall(r"launch_step\(\s*(?:st\.ahead \? )?(\w+_kernel)", TXT)))


def test_the_kernels_are_found():
    assert {"dslash_cta_kernel", "fx_stencil_kernel", "fx_convert_kernel", "update_gram_kernel", "gram_tile_kernel",
            "small_alpha_kernel", "small_qr_kernel", "small_recur_kernel", "shift_chunk32_kernel"} <= set(KERNELS)


@pytest.mark.parametrize("kernel", KERNELS)
def test_no_read_only_loads_of_what_the_kernel_before_wrote(kernel):
    params, body = _function(TXT, kernel)
    assert "step_begin()" in body
    for p in params.split(","):
        if "const" in p and "__restrict__" in p:
            assert p.split()[-1] in CONSTANT, p.strip()
    for arg in re.findall(r"__ldg\(([^;]*)", body):
        assert arg.startswith("u +") or arg.startswith("u+"), arg      # u: the link pointer


@pytest.mark.parametrize("helper", ["fx_hop", "fx_hops", "ufx_stage", "reduce_partials"])
def test_nor_in_what_they_call(helper):
    params, body = _function(TXT, helper)
    assert "__ldg" not in body
    for p in params.split(","):
        assert not ("const" in p and "__restrict__" in p), p.strip()


@pytest.mark.parametrize("storage", ["P32", "H2"])
def test_nor_in_the_spinor_loads(storage):
    """SpinorIO<P32>::load and Spinor16::load, the loads of dslash_cta_kernel."""
    head = "struct SpinorIO<P32> {" if storage == "P32" else "struct Spinor16 {"
    at = TXT.index(head)
    body = TXT[at:_close(TXT, at + len(head) - 1, "{", "}")]
    assert "__ldg" not in body


def test_the_recurrences_acquire_the_qr_before_they_read_it():
    """small_recur_kernel runs beside V = W S: it may start before its wait only
    once it has acquired the word that the QR released for this step."""
    _, recur = _function(TXT, "small_recur_kernel")
    _, qr = _function(TXT, "small_qr_kernel")
    first = recur.index("shift_recurrence")
    assert "ld_acquire(" in recur[:first] and "step_begin()" in recur[:first]
    assert "cget(" not in recur[:recur.index("ld_acquire(")]
    assert "st_release(" in qr

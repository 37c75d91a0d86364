"""Kernels that are launched before the kernel ahead of them has finished: every one of them waits, in every thread and
unconditionally, before anything that touches global memory, and none reads through the read-only path, whose loads need
not stay behind the wait (the rule stated at pdl_wait in csrc/pvt_internal.h).  Read from the sources, since a violation
is a race that no run has to show."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_14852_b200", "csrc")

# what reads or writes global memory without naming an array element
CALLS = r"\b(__ld\w+|__st\w+|load8|store8|bulk_g2s|fetch_image|form_target(16)?|load_codeword|load_cb|rank_pair|codeword)\s*[(<]"


def sources():
    return sorted(os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*.cu")))


def code_of(name):
    text = open(os.path.join(CSRC, name)).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def kernels(text):
    """name -> (parameters, body) of every kernel of the file"""
    out = {}
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^()]*\)\s*)?(\w+)\s*\(([^{}]*?)\)\s*\{", text):
        depth, at = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[at], 0)
            at += 1
        out[m.group(1)] = (m.group(2), text[m.end():at - 1])
    return out


def dependent_kernels(text):
    """those that are not launched the plain way"""
    plain = set(re.findall(r"(\w+_kernel)\s*(?:<[^;{}()]*>)?\s*<<<", text))
    return {n: k for n, k in kernels(text).items() if n not in plain}


def test_the_kernels_are_found():
    found = {n for f in sources() for n in kernels(code_of(f))}
    assert {"select_keys_kernel", "encode_m1_tc_kernel", "dequant_kernel", "rescore_m1_kernel", "cut_kernel",
            "pstep_grad_small_kernel"} <= found
    assert "pstep_grad_small_kernel" not in dependent_kernels(code_of("pvt_pstep.cu"))
    assert "dequant_kernel" in dependent_kernels(code_of("pvt_dequant.cu"))


@pytest.mark.parametrize("name", sources())
def test_dependent_kernels_wait_before_they_touch_memory(name):
    for kernel, (params, body) in dependent_kernels(code_of(name)).items():
        at = body.find("pdl_wait()")
        assert at >= 0, f"{kernel} never waits"
        ahead = body[:at]
        assert ahead.count("{") == ahead.count("}"), f"{kernel} waits in some of its threads or paths only"
        pointers = re.findall(r"\*\s*(?:__restrict__\s+)?(\w+)\s*(?:,|$)", params)
        unary = r"(?:[=(,;{}+\-!&|?:<>]|\breturn)\s*\*\s*"  # what a dereferencing star can follow
        touch = [CALLS, r"\bp\.\w+\s*(\[|->)", unary + r"p\.\w+", r"\batomic\w+\(\s*&?\s*p\."]
        touch += [rf"\b{q}\s*(\[|->)|{unary}{q}\b" for q in pointers]
        for pattern in touch:
            hit = re.search(pattern, ahead)
            assert not hit, f"{kernel} touches memory ahead of its wait: {hit.group(0)!r}"


@pytest.mark.parametrize("name", sources() + ["pvt_encode_m1.cuh"])
def test_dependent_kernels_do_not_read_through_the_read_only_path(name):
    text = code_of(name)
    for kernel, (params, _) in dependent_kernels(text).items():
        hit = re.search(r"const\s+[\w<>, ]+\*\s*__restrict__\s+\w+", params)
        assert not hit, f"{kernel}: {hit.group(0)}"
    # what is left of the file without the kernels that are launched the plain way and what only they call
    late = dependent_kernels(text)
    for kernel, (params, body) in kernels(text).items():
        if kernel not in late:
            text = text.replace(body, "")
    if name == "pvt_pstep.cu":
        text = re.sub(r"void group_codes\(.*?\n}\n", "", text, flags=re.S)
    assert "__ldg" not in text


def test_grids_follow_the_device():
    """The multiprocessor count that stands in when the device cannot be asked sizes no grid by itself."""
    assert [f for f in sources() if "kSmCountFallback" in code_of(f)] == ["pvt_api.cu"]

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
CALLS = r"\b(__ld\w+|__st\w+)\s*[(<]"
# device functions of the library that touch no global memory (prefetch_l2 brings a line to the L2 and reads nothing)
HARMLESS = {"pdl_trigger", "smem_u32", "mbar_init", "tmem_alloc", "tmem_relinquish", "tc_fence_after", "tc_fence_before",
            "prefetch_l2", "staged_bytes", "small_blocks"}


def sources():
    return sorted(os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*.cu")))


def headers():
    return sorted(os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def code_of(name):
    text = open(os.path.join(CSRC, name)).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def kernels(text):
    """name -> (parameters, body) of every kernel of the file"""
    out = {}
    bounds = r"(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?"
    for m in re.finditer(r"__global__\s+void\s+" + bounds + r"(\w+)\s*\(([^{}]*?)\)\s*\{", text):
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
    assert {"select_keys_kernel", "encode_m1_tc_kernel", "encode_beam_kernel", "refine_group_kernel", "dequant_kernel",
            "rescore_m1_kernel", "cut_kernel", "pstep_grad_small_kernel"} <= found
    assert "pstep_grad_small_kernel" not in dependent_kernels(code_of("pvt_pstep.cu"))
    assert "dequant_kernel" in dependent_kernels(code_of("pvt_dequant.cu"))


def device_functions():
    text = "".join(code_of(f) for f in sources() + headers())
    return set(re.findall(r"__device__[^;{}()]*?\b(\w+)\s*\(", text)) - {"__align__"}


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
        called = set(re.findall(r"\b(\w+)\s*(?:<[^;{}()]*>)?\s*\(", ahead)) & device_functions()
        assert called <= HARMLESS, f"{kernel} calls {sorted(called - HARMLESS)} ahead of its wait"


def read_only_loads(text):
    """what of a file that dependent kernels reach could be read through the read-only path"""
    late = dependent_kernels(text)
    found = []
    for kernel, (params, _) in late.items():
        found += re.findall(r"const\s+[\w<>, ]+\*\s*__restrict__\s+\w+", params)
    # any function may be called by a dependent kernel: only the bodies of kernels that are launched the plain way are left out
    for kernel, (params, body) in kernels(text).items():
        if kernel not in late:
            text = text.replace(body, "")
    return found + re.findall(r"__ldg\w*|\bld\.global\.nc\b", text)


@pytest.mark.parametrize("name", sources() + headers())
def test_dependent_kernels_do_not_read_through_the_read_only_path(name):
    assert read_only_loads(code_of(name)) == []


@pytest.mark.parametrize("name,at", [
    ("pvt_encode_m1.cuh", "load_codeword("),  # device code in a header
    ("pvt_pstep.cu", "group_codes("),         # called by a kernel that is launched the plain way and by one that is not
    ("pvt_refine.cu", "target_of("),
])
def test_a_read_only_load_in_a_function_is_found(name, at):
    text = code_of(name)
    body = text.index("{", text.index(at)) + 1
    assert read_only_loads(text[:body] + " __ldg(p); " + text[body:]) == ["__ldg"]


def test_grids_follow_the_device():
    """The multiprocessor count that stands in when the device cannot be asked sizes no grid by itself."""
    assert [f for f in sources() if "kSmCountFallback" in code_of(f)] == ["pvt_api.cu"]

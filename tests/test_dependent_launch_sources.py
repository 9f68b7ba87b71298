"""Kernels launched behind the one before start while that one still runs, so what it writes is not
read-only for their whole duration: a load that the compiler may take for one (`const T* __restrict__`,
`__ldg`) may go through the non-coherent path or move ahead of the wait.  Checked in the sources: only
the caller's inputs, which are complete before a call's first kernel starts, are declared so."""
import re

from paper_1806_02637_gb300 import build as ecc_build

INPUTS = {"images", "pairs"}


def _functions(text, marker):
    """(signature, body) of the functions whose definitions start with marker."""
    for m in re.finditer(marker, text):
        i = text.index("{", m.end())
        if ";" in text[m.end():i]:   # a declaration
            continue
        depth, j = 0, i
        while True:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
            if depth == 0:
                break
        yield text[m.start():i], text[i:j]


def test_what_earlier_kernels_write_is_not_declared_read_only():
    found = set()
    for src in ecc_build.sources():
        text = re.sub(r"//[^\n]*", "", open(src).read())
        for signature, body in _functions(text, r"__global__"):
            if "wait_for_previous()" not in body:
                continue
            name = re.search(r"(\w+)\s*\((?!.*__launch_bounds__)[^()]*\)\s*$", signature, re.S).group(1)
            found.add(name)
            declared = set(re.findall(r"\bconst\s+[\w:]+\s*\*\s*__restrict__\s+(\w+)", signature))
            assert declared <= INPUTS, (name, declared)
            assert "__ldg" not in body, name
        for signature, body in _functions(text, r"__device__"):
            assert "__ldg" not in body or "joseph" not in signature, signature
    assert {"joseph_kernel", "radon_views_kernel", "weight_kernel", "weight_views_kernel", "absmax_kernel",
            "quantize_f16_kernel", "reduce_kernel", "pair_grad_q_kernel", "view_grad_theta_kernel",
            "view_grad_P_kernel"} <= found

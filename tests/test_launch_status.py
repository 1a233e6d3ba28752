"""Every product reports a launch that failed: no caller drops the status of a launch function.  (A product that is
not launched leaves its output as it was, and CUDA's own last error does not tell: the launch functions return errors
of their own, and clear it.)"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1601_07384_gb300", "csrc")


def declared():
    src = open(os.path.join(CSRC, "dev.cuh")).read()
    return re.findall(r"(\[\[nodiscard\]\] )?cudaError_t (launch_\w+|fx_scales)\(", src)


def test_launch_functions_are_declared_nodiscard():
    names = declared()
    assert len(names) >= 12
    assert [n for attr, n in names if not attr] == []


def test_no_caller_drops_a_status():
    names = "|".join(n for _, n in declared())
    for fn in sorted(os.listdir(CSRC)):
        if not fn.endswith((".cu", ".cuh", ".cpp", ".h")):
            continue
        code = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, fn)).read())
        # a call that is a statement of its own: after ; { } or ) of an if, and not part of an expression
        dropped = re.findall(r"[;{}]\s*((?:%s)\s*\([^;]*\);)" % names, code)
        dropped += re.findall(r"\)\s+((?:%s)\s*\([^;]*\);)" % names, code)
        assert dropped == [], (fn, dropped)


def test_the_first_launch_of_a_product_is_checked_before_the_second():
    code = open(os.path.join(CSRC, "fxops.cu")).read()
    body = code[code.index("cudaError_t fx_launch_t"):code.index("cudaError_t fx_launch_n")]
    first = re.search(r"(\w+) = cudaLaunchKernelEx\(&cfg, k_fx_vec<N, NG>", body)
    assert first and re.match(r"[^;]*;\s*if \(%s != cudaSuccess\) return %s;" % (first[1], first[1]), body[first.start():])
    assert "return cudaLaunchKernelEx(&cfg, k_fx<P, N, NG>" in body

"""The FP32 collision and injection that the march forms, one node per thread, the
on-chip form and the batch share have their rounding in the source: in
march_dev.cuh no product meets a sum but through mul_ / fma_ / add_ (products by
1/2, exact, aside), so that no compiler chooses which is rounded."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1812_05711_gb300", "csrc")


def _functions():
    text = open(os.path.join(SRC, "march_dev.cuh")).read()
    start = text.index("__device__ __forceinline__ void trt_f2(")
    return text[start:text.index("// Charge density of one node from its new populations")]


def test_no_plain_product_in_a_sum():
    body = re.sub(r"//[^\n]*", "", _functions())
    for stmt in re.split(r"[;{}]", body):
        s = stmt.strip()
        if "=" not in s or "(" not in s and "*" not in s:
            continue
        rhs = s.split("=", 1)[1].replace("R(0.5) *", "half ")
        # arguments of the named operations may hold products (they are rounded there)
        prev = None
        while prev != rhs:
            prev = rhs
            rhs = re.sub(r"\b(?:mul_|fma_|add_|one)\([^()]*\)", "T", rhs)
            rhs = re.sub(r"\bR\([^()]*\)", "c", rhs)
        flat = re.sub(r"\(R\)", "", rhs)
        plus = re.search(r"(?<![eE(,*])\s[+-]\s", flat)
        assert not ("*" in flat and plus), s

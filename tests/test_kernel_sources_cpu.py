"""Rules of CUDA C++ that hold by the text of the kernels and that a GPU need not
break visibly."""
import os

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2412_10084_gb300", "csrc")


def block(text, start):
    """The text from `start` on to the brace that closes its first one."""
    i = text.index(start)
    depth, j = 0, text.index("{", i)
    while True:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
        if depth == 0:
            return text[i:j]


def test_regulariser_step_has_no_barrier_of_its_own():
    """Warps of one CTA choose different instances of the regulariser's step, so
    its barrier has to come before that choice."""
    with open(os.path.join(CSRC, "regularize.cu")) as f:
        kernel = block(f.read(), "sdf_reg_kernel(SdfReg P)")
    step = block(kernel, "auto step = [&](auto inner")
    assert "__syncthreads" not in step
    loop = block(kernel, "for (int zs = zb;")
    assert loop.count("__syncthreads") == 1
    assert loop.index("__syncthreads") < loop.index("if (full")

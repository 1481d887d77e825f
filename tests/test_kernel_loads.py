"""Non-coherent loads (ld.global.nc: __ldg, ld_stream, ld_keep) in the kernel
sources.  PTX defines them only for memory that nothing writes while the
kernel runs, and lets the compiler move them ahead of any wait.  Such a fault
depends on timing, so it is looked for in the source and not on a GPU."""
import os
import re

from paper_2110_04175_gb300 import build as rs_build

NON_COHERENT = ("__ldg", "ld_stream", "ld_keep")


def _source(name: str) -> str:
    with open(os.path.join(rs_build.CSRC, name)) as f:
        text = f.read()
    return re.sub(r"//[^\n]*", "", text)


def _argument(text: str, open_paren: int) -> str:
    """The text between the parenthesis at `open_paren` and its partner."""
    depth = 0
    for k in range(open_paren, len(text)):
        depth += {"(": 1, ")": -1}.get(text[k], 0)
        if depth == 0:
            return text[open_paren + 1:k]
    raise AssertionError("unbalanced parentheses")


def _non_coherent_arguments(text: str) -> list:
    return [_argument(text, m.end() - 1) for m in re.finditer(r"\b(?:%s)\(" % "|".join(NON_COHERENT), text)
            if not text[m.end():].lstrip().startswith("const float* p)")]  # the helpers' definitions


def test_the_scan_sees_the_loads():
    found = _non_coherent_arguments(_source("step_kernels.cu"))
    assert any("a.msg_in" in arg for arg in found) and any("a.mu" in arg for arg in found)


def test_counters_are_not_read_through_the_non_coherent_path():
    """relay_step launches the step kernel as a programmatic dependent of the
    counter kernel, which writes the counters while the step kernel may run."""
    for name in ("device.cuh", "step_kernels.cu", "relaysum.cu"):
        for arg in _non_coherent_arguments(_source(name)):
            assert "counts" not in arg, (name, arg)


def _body(text: str, name: str) -> str:
    """The body of the function `name`."""
    at = re.search(r"\b%s\([^;{]*\)\s*\{" % name, text).end()
    depth = 1
    for k in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[at:k]
    raise AssertionError("unbalanced braces")


def test_multi_step_kernel_reads_what_it_writes_with_ordinary_loads():
    """relay_steps leaves the messages of its last two steps in both message
    buffers, the one it starts from included, and updates the models and the
    optimiser state in place: only the centres stay as they are."""
    text = _source("step_kernels.cu")
    args = []
    for name in ("fused_steps", "fused_steps_wide", "relay_fused_steps_kernel"):
        args += _non_coherent_arguments(_body(text, name))
    assert args and all(arg.startswith("a.mu ") for arg in args), args

"""Rules of the CUDA sources that no single run shows."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_20012_gb300", "csrc")


def functions_calling(name):
    """(file, function) of every call of `name`: the function is the last one that
    opens at the start of a line."""
    out = []
    for f in sorted(os.listdir(CSRC)):
        fn = None
        for line in open(os.path.join(CSRC, f)):
            m = re.match(r"(?!//|#|template|using|namespace|struct|\s)[\w:<>,&*\s]*?(\w+)\(", line)
            if m:
                fn = m.group(1)
            if name in line.split("//")[0]:
                out.append((f, fn))
    return out


def test_function_attributes_are_set_at_initialisation_only():
    """A kernel's shared-memory limit is one value per device for the whole process:
    set to a plan's own size before a launch, it can fall below what another
    thread's launch, set just before, asks for.  Handles may live on different
    threads, so it is set once, to the device's limit."""
    calls = functions_calling("cudaFuncSetAttribute")
    assert len(calls) >= 3
    assert [c for c in calls if not c[1].startswith(("init_", "set_smem"))] == []


def test_checked_build_covers_the_streaming_kernels():
    """Every kernel that gathers by an index, or streams a range, that it reads from
    memory checks both in FO_CHECKED builds."""
    text = "".join(open(os.path.join(CSRC, f)).read() for f in ("fredopt_kernels.cu", "fredopt_sweep.cu"))
    body = {}
    for m in re.finditer(r"__global__ [^{;]*?(k_\w+)\([^{;]*\{", text):
        body[m.group(1)] = text[m.end():text.index("\n}\n", m.end())]
    for kernel in ("k_forward", "k_backward", "k_sweep_rows", "k_sweep_cols", "k_sweep_con"):
        assert "checked_index(" in body[kernel], kernel
    for kernel in ("k_sweep_rows", "k_sweep_cols"):
        assert "checked_end(" in body[kernel], kernel

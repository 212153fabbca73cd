"""What holds for one device must not be remembered for the whole process: the
leave for more than 48 KB of dynamic shared memory is given per kernel and
device, so a second device (or two threads with a context each) must not find it
ticked off. Read from the sources: one place asks for it, and it keeps its record
in the context."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1802_05421_gb300", "csrc")


def _sources():
    return {f: open(os.path.join(CSRC, f)).read() for f in os.listdir(CSRC) if f.endswith((".cu", ".h", ".cuh"))}


def test_shared_memory_leave_is_kept_per_context():
    calls = {f: s.count("cudaFuncSetAttribute(") for f, s in _sources().items()}
    assert {f: c for f, c in calls.items() if c} == {"api.cu": 1}
    body = re.search(r"int allow_smem_of\(.*?\n}\n", _sources()["api.cu"], re.S).group(0)
    assert "static" not in body and "ctx->smem_kernels" in body


def test_no_process_wide_answers_of_one_device():
    for f, s in _sources().items():
        found = re.findall(r"static\s+(?:bool|int)\s+\w+\s*=\s*[^;]*;", s)
        # whether the driver has the tensor-map encoder does not depend on the device
        assert all("tried" in x for x in found), (f, found)

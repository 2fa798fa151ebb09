"""Launch attributes are per device: every kernel of a variant that is launched with
dynamic shared memory gets its allowance in set_smem, which runs for each context
(and for cr_step_noalloc per device), and occupancies are kept per device in atomics
(threads may set up contexts at the same time).  Read from the source, since one
device cannot show a second one's launch failing.
"""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_02125_gb300", "csrc",
                   "cr_variant.cuh")


def test_every_kernel_gets_its_allowance_per_device():
    with open(SRC) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    launched = {m[0] for m in re.findall(r"\b(k_\w+)<[^;]*?<<<([^;]*?)>>>", code) if "bytes()" in m[1]}
    launched |= set(re.findall(r"cudaLaunchKernelEx\([^,]*,\s*(k_\w+)", code))
    assert len(launched) >= 8, launched
    body = re.search(r"static cudaError_t set_smem\(\) \{(.*?)\n  \}", code, re.S).group(1)
    assert launched <= set(re.findall(r"allow\((k_\w+)", body)), launched - set(re.findall(r"allow\((k_\w+)", body))


def test_no_process_wide_occupancy():
    with open(SRC) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    assert not re.findall(r"static int \w+ = ", code)
    assert "std::atomic<int>[" in code

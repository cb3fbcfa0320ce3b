"""Kernels that start before their predecessor has ended (programmatic dependent launch) load what that predecessor
writes with ordinary loads: the read-only path (__ldg, ld.global.nc) is defined only for data that nothing writes
while the kernel lives.  A stale value would show on the GPU at best now and then, so the rule is checked in the
source: the read-only path serves the slot map alone, which no kernel of a time step writes."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_12955_gb300", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_step_kernels_use_the_read_only_path_for_the_slot_map_only():
    for name in ("kernels.cuh", "launch.cuh", "runtime.cu"):
        text = _code(name)
        for m in re.finditer(r"__ldg\s*\(|ld\.global\.nc|__ldcg\s*\(", text):
            assert text[m.end():].lstrip().startswith("a.slot "), (name, text[m.start():m.start() + 60])


def test_no_step_kernel_takes_mutable_state_through_a_restrict_pointer():
    # const __restrict__ parameters are loaded through the read-only path too: the ensemble kernels' arguments,
    # constants and work lists, which the host writes and synchronises before the launch
    allowed = {"args", "coefs", "tiles", "list", "heads", "partials", "out", "flags", "v"}
    for name in ("kernels.cuh", "runtime.cu"):
        found = set(re.findall(r"__restrict__\s+(\w+)", _code(name)))
        assert found <= allowed, (name, found - allowed)

"""Kernels launched with programmatic stream serialisation begin while the one
before still writes, so what they read from it is not read-only for their
lifetime: no const __restrict__ parameters, and __ldg only on beta, an argument
of the call.  By reading the sources: a load that the compiler moves above the
wait is a race that no run shows reliably."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2609_36835_gb300" / "csrc"
SOURCES = {p.name: re.sub(r"//.*", "", p.read_text()) for p in sorted(CSRC.glob("*.cu*"))}


def test_no_chained_kernel_declares_its_inputs_read_only():
    for name, text in SOURCES.items():
        for m in re.finditer(r"__global__[^{;]*\{", text):
            found = re.findall(r"const [\w:]+\* ?__restrict__ ?\w+", m.group(0))
            assert not found, (name, found)


def test_non_coherent_loads_are_of_arguments():
    loads = {(name, arg.strip()) for name, text in SOURCES.items() for arg in re.findall(r"__ldg\(([^)+]*)", text)}
    assert loads <= {("joint_attend.cu", "a.beta"), ("attend.cu", "s.be")}, loads

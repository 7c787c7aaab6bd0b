"""What the sources of the kernels have to keep to and no run can show (CPU)."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2607_08786_b200" / "csrc"


def test_tensor_memory_waits_name_the_registers():
    """A tcgen05.wait::ld that does not have the loaded registers as operands leaves the compiler free to
    read them in front of it."""
    waits = []
    for f in sorted(CSRC.glob("*.cu*")):
        for m in re.finditer(r'asm volatile\("tcgen05\.wait::ld[^;]*;"(.*?)\);', f.read_text(), re.S):
            waits.append((f.name, m[1]))
    assert waits
    for name, operands in waits:
        assert operands.count('"+r"') in (16, 32), (name, operands)

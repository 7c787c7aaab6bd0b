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


def test_the_hand_over_outlasts_the_waits_it_depends_on():
    """The decode warps of the wide kernel wait for the epilogue, whose own waits (2 s each) have to be the
    ones that give up: a missing contributor is status 11.  And no lane leaves on its own reading of the
    abort flag, in front of votes of the whole warp."""
    device, wide = (CSRC / "tl3_device.cuh").read_text(), (CSRC / "tl3_spmm_wide.cu").read_text()
    assert int(re.search(r"kHandOverLimitNs = (\d+) \* kWaitLimitNs", device)[1]) >= 4
    waits = re.findall(r"mbar_wait\(bar\(kBarReduce, 0\)[^;]*?\)\)", wide)
    assert len(waits) == 1 and "kHandOverLimitNs" in waits[0]
    decode = wide[wide.index("decode (Algorithm 1)"):wide.index("} else if (warp >= kEpilogueWarp0)")]
    assert "abort_flag" not in decode

"""Every bounded wait of the CUDA sources reports when it runs out.  A wait's
result may go unused only where the failure has just been recorded in the error
word, as the second wait that lets copies land before a block leaves; a result
dropped anywhere else would let a kernel go on with whatever its shared memory
held."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2312_14789_gb300", "csrc")


def _bare_waits(code):
    """Positions of waits that are statements of their own, in code without comments."""
    return [m.end(1) for m in re.finditer(r"((?:[;{}]|\bif \([^;{}]*\)|\belse)\s*)(?:dev::)?mbar_wait\(", code)]


def test_no_bounded_wait_is_dropped():
    waits = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        code = re.sub(r"//[^\n]*|/\*.*?\*/", " ", open(path).read(), flags=re.S)
        waits += len(re.findall(r"mbar_wait\(", code))
        for at in _bare_waits(code):
            recorded = code.rfind("atomicExch(err", 0, at)
            assert recorded >= 0 and "}" not in code[recorded:at], (os.path.basename(path), code[at:at + 60])
    assert waits >= 15

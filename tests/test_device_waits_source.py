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


def test_lattice_is_handed_out_with_its_buffers_set():
    code = re.sub(r"//[^\n]*|/\*.*?\*/", " ", open(os.path.join(CSRC, "lattice.cu")).read(), flags=re.S)
    init = code[code.index("mlbm_lattice_init("):code.index("void mlbm_lattice_destroy(")]
    assert "cudaStreamNonBlocking" in init
    last = max(m.end() for m in re.finditer(r"cudaMem(?:set|cpy)\(", init))
    assert "cudaStreamSynchronize(nullptr)" in init[last:init.index("*out = L")]

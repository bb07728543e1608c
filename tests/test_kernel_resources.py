"""What the compiler reports about kernels whose speed hangs on it.  Compiles, runs nothing."""
import re
import subprocess

from paper_2507_11959_b200 import build


def test_two_bit_uniform_twin_does_not_spill(tmp_path):
    """The GEMV of the uniform twin at 2 bits with two CTAs per SM (64 registers per thread): with spills 4096 x 4096 took 5.7
    instead of 4.2 us."""
    src = tmp_path / "twin.cu"
    src.write_text('#include "common.cuh"\n#include "layout.cuh"\n#include "stream.cuh"\n'
                   "template pot_status_t pot::launch_stream<2, pot::SK_UINT, 1, 16, 2, 0>(const void*, const void*, const void*, int64_t, int64_t, int, "
                   "const void*, int, void*, void*, int*, cudaStream_t);\n")
    flags = [f for f in build.NVCC_FLAGS if f != "--use_fast_math=false"]
    r = subprocess.run([build._nvcc(), *flags, "-I", str(build.CSRC), "-Xptxas", "-v", "-c", str(src), "-o", str(tmp_path / "twin.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    spills = re.findall(r"(\d+) bytes spill stores, (\d+) bytes spill loads", r.stderr)
    assert spills and all(s == ("0", "0") for s in spills), spills

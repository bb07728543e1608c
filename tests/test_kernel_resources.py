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


def test_sums_of_a_cluster_that_may_be_incomplete_are_not_stored():
    """A tile that may hold the sums of a CTA whose bounded wait gave up is not stored.  The CTAs of a cluster add up each other's sums, and
    one may give up after a peer has looked at the error word: it leaves a mark in the place of its sums, which every CTA looks for
    in what it adds up.  By reading, because no wait gives up unless something is broken."""
    text = re.sub(r"//[^\n]*", "", (build.CSRC / "gemm_prefill.cu").read_text())
    kernel = text[text.index("pot_gemm_prefill_kernel(const"):]
    barrier = kernel.index("pf_cluster_sync();")
    look = kernel.index("const bool gave_up = err != nullptr && *reinterpret_cast<volatile int*>(err) != 0;")
    mark = kernel.index("if (gave_up) {", look)
    leave = kernel.index("dst[i * PF_BN] = __uint_as_float(v[i]);", mark)
    assert kernel.index("mbar_wait(accum, 0)") < look < mark < leave < barrier and "v[i] = PF_NO_SUM;" in kernel[mark:leave]
    add_up = text[text.index("pf_add_up_of(const"):text.index("pf_add_up(const")]
    assert add_up.index("p[u][z].x != PF_NO_SUM") < add_up.index("if (!complete) continue;") < add_up.index("uint16_t* dst = a.Y")
    pattern = int(re.search(r"PF_NO_SUM = (0x[0-9A-F]+)u", text).group(1), 16)
    assert 0x7F800000 < pattern < 0x7FC00000   # a signaling NaN: sums of products, and NaN that additions pass on, are none
    mark = int(re.search(r"SK_SUM_MARK = (0x[0-9A-F]+)u", (build.CSRC / "stream_even.cuh").read_text()).group(1), 16)
    assert 0x7F800000 < mark < 0x7FC00000 and mark != pattern   # (looked for where such sums may lie)


def test_the_scale_search_does_not_spill(tmp_path):
    """At 2 bits under 64 registers it did: 2048 x 2048, groups of 64, 36.7 -> 39.0 us."""
    flags = [f for f in build.NVCC_FLAGS if f != "--use_fast_math=false"]
    r = subprocess.run([build._nvcc(), *flags, "-Xptxas", "-v", "-c", str(build.CSRC / "quantize.cu"), "-o", str(tmp_path / "q.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    found = re.findall(r"Compiling entry function '\S*pot_search_kernel.*?(\d+) bytes spill stores, (\d+) bytes spill loads", r.stderr, re.S)
    assert len(found) == 6 and all(s == ("0", "0") for s in found), found

"""The C-ABI library: builds, loads, exports what include/pot.h declares, validates arguments on
the host before touching the GPU, and its layout map is a bijection.  No kernel is launched."""
import ctypes
import re
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent


@pytest.fixture(scope="module")
def L():
    from paper_2507_11959_b200 import build
    build.build()
    from paper_2507_11959_b200 import binding
    return binding.lib()


def declared_functions():
    text = (ROOT / "include" / "pot.h").read_text()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b((?:pot|uint)_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(L):
    names = declared_functions()
    assert {"pot_quantize_ref", "pot_dequant", "pot_gemv", "pot_gemm", "uint_dequant", "uint_gemv"} <= set(names)
    for name in names:
        assert hasattr(L, name), name
    from paper_2507_11959_b200 import binding
    assert set(binding.EXPORTS) == set(names)


def test_size_helpers(L):
    assert L.pot_packed_bytes(4096, 4096, 3) == 4096 * 1536
    assert L.pot_packed_bytes(4096, 4096, 2) == 4096 * 1024
    assert L.pot_packed_bytes(4096, 4100, 3) == 0       # K % 128
    assert L.pot_packed_bytes(4096, 4096, 5) == 0
    assert L.pot_scales_bytes(4096, 4096, 128) == 4096 * 32 * 2
    assert L.pot_scales_bytes(4096, 4096, 64) == 4096 * 64 * 2
    assert L.pot_scales_bytes(4096, 4096, 32) == 0
    # one unit (128 columns) per row block: every warp writes whole row blocks, nothing to combine; longer rows
    # need an arrival counter per row block and FP32 partial slots
    assert L.pot_gemv_workspace_bytes(12288, 128, 3, 128) == 0
    ws = L.pot_gemv_workspace_bytes(4096, 11008, 3, 128)
    assert ws >= 1024 + 256 * 2 * 16 * 4 and ws % 16 == 0
    wg = L.pot_gemm_workspace_bytes(4, 4096, 11008, 3, 128)   # small batch: eight token columns per slot
    assert wg >= 1024 + 256 * 2 * 16 * 8 * 4 and wg % 16 == 0
    # 2 to 8 tokens run the streaming kernel (one workspace size for all of them) while their activations fit in
    # shared memory; 5 to 8 tokens of a longer K run the tcgen05 kernel; one token runs the GEMV kernel
    assert L.pot_gemm_workspace_bytes(8, 12288, 4096, 3, 128) == L.pot_gemm_workspace_bytes(2, 12288, 4096, 3, 128)
    assert L.pot_gemm_workspace_bytes(2, 4096, 11008, 3, 128) == wg
    assert L.pot_gemm_workspace_bytes(8, 4096, 11008, 3, 128) == 256 + 32 * 4 * 8 * 128 * 4   # (see the tcgen05 sizes below)
    assert L.pot_gemm_workspace_bytes(1, 4096, 11008, 3, 128) >= ws
    # Larger M runs the tcgen05 kernel.  It needs scratch only for the tiles it splits along K: all of them when they
    # cover at most half of the SMs (32 tiles -> 4 splits of 32 token rows x 128 features), or those of a last
    # wave that fills at most half of the 148 CTA slots (640 tiles -> 48 tail tiles x 3 splits x 256 rows).
    assert L.pot_gemm_workspace_bytes(32, 4096, 11008, 3, 128) == 256 + 32 * 4 * 32 * 128 * 4
    assert L.pot_gemm_workspace_bytes(2048, 10240, 8192, 3, 128) == 256 + 48 * 3 * 256 * 128 * 4
    assert L.pot_gemm_workspace_bytes(2048, 8192, 28672, 3, 128) == 512 + 68 * 2 * 256 * 128 * 4  # 512 tiles: 68 in the last wave
    assert L.pot_gemm_workspace_bytes(2048, 3584, 8192, 3, 128) == 0     # 224 tiles: the last wave is 51 % full


def test_status_strings(L):
    seen = set()
    for code in range(8):
        s = L.pot_status_string(code).decode()
        assert s and s != "unknown status"
        seen.add(s)
    assert len(seen) == 8
    assert L.pot_status_string(99).decode() == "unknown status"


def test_argument_errors_are_reported_before_any_launch(L):
    before = L.pot_launch_count()
    a = ctypes.c_void_p(0x1000)      # never dereferenced: all of these fail validation on the host
    odd = ctypes.c_void_p(0x1008)
    null = ctypes.c_void_p(0)
    assert L.pot_dequant(null, a, 16, 128, 3, 128, 0, a, null) == 1
    assert L.pot_dequant(a, a, 16, 128, 5, 128, 0, a, null) == 2
    assert L.pot_dequant(a, a, 16, 128, 3, 32, 0, a, null) == 2
    assert L.pot_dequant(a, a, 16, 128, 3, 128, 7, a, null) == 2
    assert L.pot_dequant(a, a, 16, 100, 3, 128, 0, a, null) == 3
    assert L.pot_dequant(a, a, 0, 128, 3, 128, 0, a, null) == 3
    assert L.pot_dequant(a, a, 16, 128, 3, 128, 0, odd, null) == 4
    assert L.pot_gemv(a, a, 24, 128, 3, 128, 1, a, a, null, 0, null) == 3     # tiled needs N % 16 == 0
    assert L.pot_gemv(a, a, 4096, 11008, 3, 128, 1, a, a, null, 0, null) == 5  # split-K without workspace
    assert L.pot_gemv(a, a, 4096, 11008, 3, 128, 1, a, a, a, 64, null) == 5    # workspace too small
    assert L.pot_gemv(a, a, 16, 128, 3, 128, 9, a, a, null, 0, null) == 2
    assert L.pot_gemm(a, a, 16, 128, 3, 128, 0, a, 0, a, null, 0, null) == 3
    assert L.pot_gemm(a, null, 16, 128, 3, 128, 0, a, 4, a, null, 0, null) == 1
    assert L.pot_quantize_ref(a, 16, 128, 3, 128, 9, a, a, null) == 2
    assert L.pot_repack(a, a, 24, 128, 3, 0, null) == 3
    assert L.uint_dequant(a, a, null, 16, 128, 3, 128, 0, a, null) == 1
    assert L.uint_dequant(a, a, a, 16, 128, 3, 128, 5, a, null) == 2
    assert L.pot_validate_scales(a, 0, 3, a, null) == 3
    assert L.pot_launch_count() == before


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("kind", [0, 1])
def test_tiled_layout_map_is_a_bijection_with_pairs_16_apart(L, bits, kind):
    from paper_2507_11959_b200 import binding
    seen = {}
    for q in range(128):
        for b in range(bits):
            w, bit = binding.pot_layout_bit(bits, kind, q, b)
            assert 0 <= w < 4 * bits and 0 <= bit < 32
            assert (w, bit) not in seen
            seen[(w, bit)] = (q, b)
    assert len(seen) == 128 * bits == 4 * bits * 32        # exactly n bits per weight, nothing unused
    for q in range(0, 128, 2):                             # the two codes of a pair: same word, 16 bits apart
        for b in range(bits):
            w0, b0 = binding.pot_layout_bit(bits, kind, q, b)
            w1, b1 = binding.pot_layout_bit(bits, kind, q + 1, b)
            assert w0 == w1 and (b1 - b0) % 32 == 16
    with pytest.raises(binding.PotError):
        binding.pot_layout_bit(bits, kind, 128, 0)


def test_units_of_one_group_reserve_nothing_beside_the_activations(L):
    """K at the edge of what fits beside the rings: with G = 128 the GEMV keeps no zeros behind x, which would cost the longer
    slots at one K, the second CTA per SM at another and x its place in shared memory at a third."""
    from paper_2507_11959_b200 import binding
    assert binding.pot_debug_gemv_plan(1024, 4736, 3, 128)["units_per_slot"] == 4
    assert binding.pot_debug_gemv_plan(1024, 30336, 3, 128)["ctas_per_sm"] == 2
    assert binding.pot_debug_gemv_plan(1024, 95360, 2, 128)["x_in_smem"] == 1


def test_canonical_tiles_are_cut_into_clusters_that_are_resident_at_once(L):
    """How many clusters fit depends on the chip's GPCs: a tile more than that takes the next smaller cluster."""
    from paper_2507_11959_b200 import binding
    usual, fewer = [15, 22, 26, 33, 45, 74], [12, 18, 24, 32, 44, 72]
    splits = lambda tiles, K, r: binding.pot_debug_canonical_splits(tiles, K, r)
    assert [splits(t, 11008, usual) for t in (1, 15, 16, 22, 23, 26, 27, 33, 34, 45, 46, 74, 75, 5000)] == [8, 8, 6, 6, 5, 5, 4, 4, 3, 3, 2, 2, 1, 1]
    assert [splits(t, 11008, fewer) for t in (12, 13, 32, 33, 73)] == [8, 6, 4, 3, 1]
    assert [splits(1, K, usual) for K in (128, 896, 1024, 1536, 2048, 2560, 3072, 4096)] == [1, 1, 2, 3, 4, 5, 6, 8]  # four column blocks per CTA


def test_calls_through_the_extension_module_are_those_through_ctypes(L):
    """The binding's per-token calls: the same argument errors, in the same order, for pointers that are null, misaligned or plain
    addresses, for lengths, widths and layouts that are refused; a wrong number or type of arguments raises."""
    from paper_2507_11959_b200 import binding
    f = binding._load_fast()
    ok = dict(packed=4096, scales=4096, N=64, K=256, bits=3, group=128, layout=1, x=4096, y=4096, ws=None, ws_bytes=0, stream=0)
    bad = [dict(packed=None), dict(x=None), dict(y=0), dict(bits=5), dict(group=32), dict(K=100), dict(N=0), dict(N=-1), dict(layout=7), dict(N=63),
           dict(packed=4097), dict(x=4098), dict(N=2 ** 40)]  # (nothing that would be launched)
    for change in bad:
        a = dict(ok, **change)
        gemv = (a["packed"], a["scales"], a["N"], a["K"], a["bits"], a["group"], a["layout"], a["x"], a["y"], a["ws"], a["ws_bytes"], a["stream"])
        gemm = gemv[:8] + (40,) + gemv[8:]
        for name, args, call in (("pot_gemv", gemv, f.gemv), ("pot_gemv_bf16", gemv, f.gemv), ("pot_gemm", gemm, f.gemm), ("pot_gemm_bf16", gemm, f.gemm)):
            status = getattr(L, name)(*args)
            assert status != 0 and call(getattr(f, name), *args) == status, (name, change)
        if set(change) & {"packed", "y", "bits", "group", "K", "N"} and a["N"] != 63:
            args = gemv[:6] + (0, a["y"], 0)
            status = L.pot_dequant(*args)
            assert status != 0 and f.dequant(f.pot_dequant, *args) == status, change
    with pytest.raises(TypeError):
        f.gemv(f.pot_gemv, 1, 2, 3)
    with pytest.raises(TypeError):
        f.dequant(f.pot_dequant, 4096, 4096, 1.5, 256, 3, 128, 0, 4096, 0)


def test_arguments_that_the_extension_module_does_not_take_are_refused_or_taken_as_ctypes_does(L):
    """None is a null pointer, never a number (as a layout or a type it would be 0, a value that exists); what only ctypes takes (its own
    objects) still gets there."""
    import types
    import torch
    from paper_2507_11959_b200 import binding as B
    f = B._load_fast()
    gemv = [4096, 4096, 64, 256, 3, 128, 0, 4096, 4098, None, 0, None]
    for name, args, call, numbers in (("pot_gemv", gemv, f.gemv, (2, 3, 4, 5, 6, 10)), ("pot_gemm", gemv[:8] + [40] + gemv[8:], f.gemm, (2, 3, 4, 5, 6, 8, 11)),
                                      ("pot_dequant", gemv[:6] + [0, 4098, None], f.dequant, (2, 3, 4, 5, 6))):
        assert call(getattr(f, name), *args) == getattr(L, name)(*args) == 4   # (misaligned: nothing is launched)
        for i, value in [(i, None) for i in numbers] + [(i, 2.0) for i in range(len(args))] + [(0, "4096"), (7, b"4096")]:
            with pytest.raises(TypeError):
                call(getattr(f, name), *args[:i], value, *args[i + 1:])
    packed, scales = torch.zeros(64, 96, dtype=torch.uint8), torch.zeros(64, 2, dtype=torch.float16)
    x, here = torch.zeros(256, dtype=torch.float16), types.SimpleNamespace(cuda_stream=0)
    out = torch.zeros(64 * 256 + 8, dtype=torch.float16)[1:]   # misaligned
    for call in (lambda **k: B.pot_dequant(packed, scales, k.get("K", 256), 3, 128, k.get("form", 0), out=out, stream=k.get("stream", here)),
                 lambda **k: B.pot_gemv(packed, scales, k.get("K", 256), 3, 128, x, k.get("form", B.CANONICAL), y=out, stream=k.get("stream", here)),
                 lambda **k: B.pot_gemm(packed, scales, k.get("K", 256), 3, 128, x.view(1, 256), k.get("form", B.CANONICAL), Y=out, stream=k.get("stream", here))):
        for bad in (dict(form=None), dict(K=None), dict(K=256.0), dict(stream=types.SimpleNamespace(cuda_stream=1.5))):
            with pytest.raises(ctypes.ArgumentError):
                call(**bad)
        for good in (dict(), dict(K=ctypes.c_int64(256)), dict(stream=types.SimpleNamespace(cuda_stream=ctypes.c_void_p(0)))):
            with pytest.raises(B.PotError, match="aligned"):
                call(**good)


def test_the_library_needs_no_extension_module(L, tmp_path, monkeypatch):
    """The extension module belongs to one kind of interpreter and its name says so.  Without a compiler or the Python headers the
    library is built all the same, no module of older sources is left behind, and the binding calls by ctypes."""
    import sys
    import sysconfig
    from paper_2507_11959_b200 import binding as B
    from paper_2507_11959_b200 import build
    tag = sysconfig.get_config_var("EXT_SUFFIX")
    assert build.FASTCALL == B._FASTCALL_PATH and build.FASTCALL.name == "_fastcall" + tag and tag != ".so"
    with monkeypatch.context() as m:
        m.setattr(build, "FASTCALL", tmp_path / build.FASTCALL.name)
        for compiler in ("false", str(tmp_path / "there-is-none")):
            m.setenv("CC", compiler)
            build.FASTCALL.write_bytes(b"of older sources")
            assert build.build_fastcall(force=True) is None and not list(tmp_path.iterdir())
            assert build.build() == build.LIB   # (is up to date)
    with monkeypatch.context() as m:
        m.setattr(B, "_FASTCALL_PATH", tmp_path / "none.so")
        m.setattr(B, "_fast", None)
        f = B._load_fast()
        args = (4096, 4096, 64, 256, 3, 128, 0, 4096, 4098, None, 0, None)
        assert f.gemv(f.pot_gemv, *args) == f.gemv(f.pot_gemv_bf16, *args) == 4 and f.gemm(f.pot_gemm, *args[:8], 40, *args[8:]) == 4
        assert f.dequant(f.pot_dequant, *args[:6], 0, 4098, None) == 4
        with pytest.raises(ctypes.ArgumentError):
            f.gemv(f.pot_gemv, *args[:6], None, *args[7:])


def test_the_clusters_of_tiled_codes_do_not_depend_on_the_chip(L):
    """Host arithmetic, which asks no GPU: the splits decide in which order a tile's sums are added, and GPUs that hold different numbers
    of clusters must agree on them.  The cluster never has more CTAs than the workspace holds splits; 0: the last CTA adds up."""
    from paper_2507_11959_b200 import binding as B
    expected = {(256, 4096, 4096): 4, (16, 4096, 4096): 4, (32, 2048, 8192): 6, (32, 1024, 4096): 8, (300, 144, 4096): 8, (260, 6400, 8192): 2, (260, 9472, 8192): 2,
                (32, 5120, 13824): 3, (32, 1024, 28672): 0, (400, 2048, 8192): 0, (301, 11024, 4096): 0, (2048, 28672, 8192): 0, (4, 4096, 4096): 0, (40, 144, 384): 0}
    for (M, N, K), cluster in expected.items():
        plans = [B.pot_debug_gemm_plan(M, N, K, 3, 128, bf16) for bf16 in (False, True)]
        assert [p["cluster"] for p in plans] == [cluster, cluster], (M, N, K, plans)
        assert all(p["cluster"] <= p["splits"] and (p["cluster"] == 0 or p["split_tiles"] == p["tiles"]) for p in plans)
    assert [B.pot_debug_gemm_plan(48, 1024, 28672, 4, 64, bf16)["cluster"] for bf16 in (False, True)] == [8, 0]   # (a BF16 stage takes longer)
    source = (ROOT / "paper_2507_11959_b200" / "csrc" / "gemm_prefill.cu").read_text()
    launch = source[source.index("pot_status_t gemm_prefill_launch("):source.index("pot_status_t gemm_canonical_launch(")]
    assert "tiled_cluster(" in launch and "cluster_splits(" not in launch   # (what the runtime says only rules clusters out)


def test_one_bf16_token_takes_the_decode_without_the_scale_where_that_is_faster(L):
    """What decides is how many units a warp has to get the making of FP16 numbers of x back on: shapes at which either decode was measured
    to be the faster one, at 2, 3 and 4 bits."""
    from paper_2507_11959_b200 import binding as B
    expected = {(4096, 4096): "000", (7104, 4096): "000", (7120, 4096): "000", (8192, 4096): "011", (9472, 4096): "111", (10656, 4096): "001", (11008, 4096): "001",
                (12288, 4096): "111", (18944, 2048): "111", (16576, 2048): "000", (20000, 2048): "001", (28672, 1152): "001", (15360, 5120): "111", (5120, 13824): "111",
                (2816, 13824): "000", (1024, 28672): "000", (2032, 28672): "000", (2400, 28672): "001", (2368, 28672): "111", (8192, 28672): "111", (28672, 8192): "111", (9472, 16384): "111"}
    for (N, K), want in expected.items():
        for G in (64, 128):
            got = "".join(str(B.pot_debug_gemv_decode(N, K, bits, G, True)["unscaled"]) for bits in (2, 3, 4))
            assert got == ("011" if G == 64 and (N, K) in ((10656, 4096), (11008, 4096)) else want), (N, K, G, got)   # (two scales per unit)
        assert all(B.pot_debug_gemv_decode(N, K, bits, 128, False)["unscaled"] == 1 for bits in (2, 3, 4))   # (FP16 numbers to begin with)


def test_four_warp_ctas_of_the_canonical_gemv_where_they_deal_the_row_blocks_out_better(L):
    """Shapes at which CTAs of four or of eight warps were measured to be the faster ones, at 2, 3 and 4 bits; the other ways to share a row
    block have eight."""
    from paper_2507_11959_b200 import binding as B
    expected = {(2363, 2944): "444", (2379, 2944): "888", (4099, 2048): "888", (4099, 2944): "888", (6000, 2944): "844", (9472, 2944): "844", (9472, 8192): "888",
                (9473, 8192): "444", (10007, 4096): "444", (11840, 8192): "444", (11841, 8192): "888", (12000, 4096): "844", (12000, 16384): "888", (10500, 16384): "844",
                (16000, 8192): "444", (18900, 8192): "888", (10500, 24576): "844", (10500, 28672): "888"}
    for (N, K), want in expected.items():
        plans = [B.pot_debug_canonical_gemv_plan(N, K, bits) for bits in (2, 3, 4)]
        assert "".join(str(p[1]) for p in plans) == want and all(p[0] == 4 and p[2] == 1 for p in plans), (N, K, plans)
    assert [B.pot_debug_canonical_gemv_plan(N, K, 3) for N, K in ((38001, 512), (18993, 1152), (1001, 4096), (555, 11008), (96, 28672), (9, 65536), (5, 65664))] == [
        (1, 8, 1), (2, 8, 1), (8, 8, 1), (8, 8, 2), (8, 8, 4), (8, 8, 4), (0, 8, 0)]


def test_the_units_are_dealt_out_evenly_where_that_is_faster(L):
    """Shapes at which whole row blocks per CTA (0), or the even split (2), were measured to be the faster ones; the even split wherever whole row blocks do not
    divide."""
    from paper_2507_11959_b200 import binding as B
    split = lambda M, N, K, bits, G, bf16: B.pot_debug_gemv_split(M, N, K, bits, G, bf16)
    one = {(28672, 8192, 3, 128, False): 2, (15360, 8192, 3, 128, False): 2, (18944, 8192, 3, 128, False): 2, (28672, 8192, 2, 128, True): 0, (7104, 21760, 3, 64, False): 0,
           (4352, 28672, 3, 64, False): 0, (9200, 20352, 2, 128, False): 0, (8192, 28672, 3, 128, False): 2, (12288, 4096, 3, 128, False): 0, (5120, 13824, 3, 128, False): 2}
    assert {k: split(1, *k) for k in one} == one
    several = {(2, 15360, 5120, 3, 128, False): 2, (2, 4096, 11008, 3, 128, False): 0, (4, 15360, 5120, 3, 128, False): 2, (4, 15360, 5120, 4, 128, False): 0, (4, 6240, 6528, 2, 128, False): 0,
               (4, 13200, 9088, 3, 128, False): 0, (4, 13200, 9088, 3, 128, True): 2, (3, 8288, 6016, 2, 128, False): 0, (4, 8784, 9472, 3, 128, False): 0, (4, 9200, 22656, 3, 64, False): 2,
               (4, 10288, 4096, 3, 64, False): 0, (3, 8096, 9088, 3, 128, False): 0, (3, 14336, 3456, 2, 128, False): 0, (4, 15440, 4352, 4, 128, False): 0, (5, 15360, 5120, 3, 128, False): 0, (8, 3552, 5888, 3, 64, False): 2}
    assert {k: split(*k) for k in several} == several

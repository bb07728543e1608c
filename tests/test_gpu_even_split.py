"""The streaming kernel with the units dealt out evenly to the CTAs: row blocks that two CTAs share, whose sums go from one to the other."""
import numpy as np
import pytest

from tests.gpu_util import GuardedBinding, PotCase, bf16_dev, bits_of, f16_bits_to_bf16_bits, f16_dev, gate, to_dev

pytestmark = pytest.mark.gpu

# (N, K): row blocks per CTA from just above one to many; K of few and odd numbers of column blocks; shared row blocks of which the second CTA
# has a single unit or all but one; x that does not fit into shared memory (4 tokens x 14336
# at 4 bits); a last CTA whose units all lie in a row block that the one before it began (2528 x 2432: 18 units of 19, 2480 x 4992: 37 of 39)
SHAPES = [(2480, 2048), (2992, 1792), (3088, 4224), (2720, 4224), (13024, 384), (7136, 1152), (5200, 2048), (2400, 8192), (2528, 14336), (2528, 2432), (2480, 4992)]


@pytest.fixture(scope="module")
def B():
    return GuardedBinding()


def _acts(M, K, seed):
    from paper_2507_11959_b200 import synth
    return synth.activations(synth.rng_for(4, seed), M, K)


@pytest.mark.parametrize("N,K", SHAPES)
@pytest.mark.parametrize("bits,G", [(2, 64), (3, 128), (4, 64)])
def test_even_split_matches_oracle(B, oracle, N, K, bits, G):
    from paper_2507_11959_b200 import binding
    c = PotCase(N, K, bits, G, dist="t5", seed=(4, 900 + bits))
    tiled, scales = c.tiled(), c.tiled_S()
    for M in (1, 2, 4, 8):
        X = _acts(M, K, 900 + M)
        for bf16 in (False, True):
            Xb = f16_bits_to_bf16_bits(X) if bf16 else X
            if binding.pot_debug_gemm_plan(M, N, K, bits, G, bf16)["streaming"] == 0:
                continue
            assert binding.pot_debug_gemv_split(M, N, K, bits, G, bf16) == 2
            Y, A = oracle.matmul(c.packed, c.S, K, bits, G, Xb, dtype=oracle.BF16 if bf16 else oracle.F16)
            ws = B.new_workspace(binding.pot_gemm_workspace_bytes(M, N, K, bits, G))
            Xd = bf16_dev(Xb) if bf16 else f16_dev(Xb)
            first = None
            for _ in range(3):  # the marks have to be gone after every call; sums in a fixed order
                y = bits_of(B.pot_gemm(tiled, scales, K, bits, G, Xd, binding.TILED, workspace=ws))
                first = y if first is None else first
                assert np.array_equal(y, first), (M, bf16)
            ok, worst, tight = gate(first, Y, A, bf16)
            assert ok and tight < 4.0, (M, bf16, worst, tight)
            assert not ws[:148 * 16 * (1 if M == 1 else 8) * 8].any(), (M, bf16)


# One CTA per SM, whose ring is filled behind the activations: slots of 8 units (2 and 3 bits) and of 4; row blocks shared by two CTAs and not;
# BF16 with and without the scale (2 bits keep whole row blocks)
@pytest.mark.parametrize("N,K", [(28672, 8192), (18944, 8192), (15376, 9088)])
@pytest.mark.parametrize("bits,G", [(2, 64), (2, 128), (3, 64), (3, 128), (4, 64), (4, 128)])
def test_one_token_with_one_cta_per_sm_matches_oracle(B, oracle, N, K, bits, G):
    from paper_2507_11959_b200 import binding
    small = PotCase(1009, K, bits, G, dist="t5", seed=(4, 1200 + bits))
    row = np.arange(N) % small.N     # the matrix repeats the rows of a small one
    tiled, scales = binding.pot_repack(to_dev(small.packed[row]), K, bits, 0), binding.pot_repack_scales(f16_dev(small.S[row]), K, G, 0)
    X = _acts(1, K, 1210)
    for bf16 in (False, True):
        plan = binding.pot_debug_gemv_decode(N, K, bits, G, bf16)
        if plan["ctas_per_sm"] != 1:
            assert N * K < 28672 * 8192
            continue
        assert binding.pot_debug_gemv_split(1, N, K, bits, G, bf16) == (0 if bf16 and bits == 2 else 2)
        Xb = f16_bits_to_bf16_bits(X) if bf16 else X
        Y, A = oracle.matmul(small.packed, small.S, K, bits, G, Xb, dtype=oracle.BF16 if bf16 else oracle.F16)
        ws = B.new_workspace(binding.pot_gemv_workspace_bytes(N, K, bits, G))
        y = [bits_of(B.pot_gemv(tiled, scales, K, bits, G, bf16_dev(Xb[0]) if bf16 else f16_dev(Xb[0]), binding.TILED, workspace=ws)) for _ in range(3)]
        assert np.array_equal(y[0], y[1]) and np.array_equal(y[0], y[2]) and not ws[:148 * 16 * 8].any()
        ok, worst, tight = gate(y[0], Y[0][row], A[0][row], bf16)
        assert ok and tight < 4.0, (bf16, worst, tight)


def test_even_split_repeats_itself_in_a_chain(B):
    """Forty launches behind one another that share a workspace, every one with other numbers: no sum of one call reaches the next."""
    import torch
    from paper_2507_11959_b200 import binding
    N, K, bits, G = 2992, 1792, 3, 128
    c = PotCase(N, K, bits, G, dist="t5", seed=(4, 950))
    tiled, scales = c.tiled(), c.tiled_S()
    assert binding.pot_debug_gemv_split(1, N, K, bits, G) == 2
    ws = binding.new_workspace(binding.pot_gemv_workspace_bytes(N, K, bits, G))
    xs = [f16_dev(_acts(1, K, 960 + i)[0]) for i in range(8)]
    alone = []
    for x in xs:
        alone.append(binding.pot_gemv(tiled, scales, K, bits, G, x, binding.TILED, workspace=ws).clone())
        torch.cuda.synchronize()
    ys = [torch.empty_like(alone[0]) for _ in range(40)]
    for i, y in enumerate(ys):
        binding.pot_gemv(tiled, scales, K, bits, G, xs[i % 8], binding.TILED, y=y, workspace=ws)
    torch.cuda.synchronize()
    assert all(torch.equal(y, alone[i % 8]) for i, y in enumerate(ys))
    # the fixed scratch of pot_gemv_noalloc, after a call that leaves partial sums in it
    small = PotCase(1024, 4096, bits, G, dist="t5", seed=(4, 951))
    binding.pot_gemv_noalloc(small.tiled(), small.tiled_S(), 4096, bits, G, f16_dev(_acts(1, 4096, 970)[0]), torch.empty(1024, dtype=torch.float16, device="cuda"))
    y = binding.pot_gemv_noalloc(tiled, scales, K, bits, G, xs[0], torch.empty_like(alone[0]))
    assert torch.equal(y, alone[0])
    assert binding.pot_debug_errors() == (0, 0, 0)


@pytest.mark.parametrize("M", [1, 4])
def test_even_split_among_streams(B, M):
    """Launches of four streams at once, with a product of 2048 tokens beside them: CTAs of a launch start at very different times, and whichever of
    two that share a row block comes second adds the sums.  The same bits as alone, and nothing left in the workspaces."""
    import torch
    from paper_2507_11959_b200 import binding
    N, K, bits, G = (2400, 8192, 3, 128) if M == 1 else (15360, 5120, 3, 128)
    c = PotCase(N, K, bits, G, dist="t5", seed=(4, 980 + M))
    tiled, scales, x = c.tiled(), c.tiled_S(), f16_dev(_acts(M, K, 981))
    assert binding.pot_debug_gemv_split(M, N, K, bits, G) == 2
    need = binding.pot_gemm_workspace_bytes(M, N, K, bits, G)
    alone = binding.pot_gemm(tiled, scales, K, bits, G, x, binding.TILED, workspace=binding.new_workspace(need)).clone()
    big, wide = f16_dev(_acts(2048, K, 982)), binding.new_workspace(binding.pot_gemm_workspace_bytes(2048, N, K, bits, G))
    streams = [torch.cuda.Stream() for _ in range(4)]
    spaces = [binding.new_workspace(need) for _ in streams]
    ys = [[torch.empty_like(alone) for _ in range(12)] for _ in streams]
    torch.cuda.synchronize()
    for i in range(12):
        for s, ws, y in zip(streams, spaces, ys):
            with torch.cuda.stream(s):
                binding.pot_gemm(tiled, scales, K, bits, G, x, binding.TILED, Y=y[i], workspace=ws)
        if i % 4 == 0:
            binding.pot_gemm(tiled, scales, K, bits, G, big, binding.TILED, workspace=wide)
    torch.cuda.synchronize()
    assert all(torch.equal(v, alone) for y in ys for v in y)
    assert not any(ws[:148 * 16 * (1 if M == 1 else 8) * 8].any() for ws in spaces)
    assert binding.pot_debug_errors() == (0, 0, 0)


@pytest.mark.parametrize("M", [5, 6, 7, 8])
@pytest.mark.parametrize("bits,G", [(2, 128), (3, 64), (4, 128)])
def test_even_split_of_five_to_eight_tokens(B, oracle, M, bits, G):
    """Three or four sums per lane, the last of them with half of its lanes: the same bits from three calls on one workspace, no marks left in it."""
    from paper_2507_11959_b200 import binding
    for i, (N, K) in enumerate([(2480, 2048), (3552, 5888)]):
        c = PotCase(N, K, bits, G, dist="t5", seed=(4, 1100 + 10 * bits + i))
        X = _acts(M, K, 1110 + M)
        for bf16 in (False, True):
            assert binding.pot_debug_gemm_plan(M, N, K, bits, G, bf16)["streaming"] == 1 and binding.pot_debug_gemv_split(M, N, K, bits, G, bf16) == 2
            Xb = f16_bits_to_bf16_bits(X) if bf16 else X
            Y, A = oracle.matmul(c.packed, c.S, K, bits, G, Xb, dtype=oracle.BF16 if bf16 else oracle.F16)
            ws = B.new_workspace(binding.pot_gemm_workspace_bytes(M, N, K, bits, G))
            y = [bits_of(B.pot_gemm(c.tiled(), c.tiled_S(), K, bits, G, bf16_dev(Xb) if bf16 else f16_dev(Xb), binding.TILED, workspace=ws)) for _ in range(3)]
            assert np.array_equal(y[0], y[1]) and np.array_equal(y[0], y[2]) and not ws[:148 * 16 * 8 * 8].any()
            ok, worst, tight = gate(y[0], Y, A, bf16)
            assert ok and tight < 4.0, (N, bf16, worst, tight)

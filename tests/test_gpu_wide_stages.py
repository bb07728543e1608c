"""The tcgen05 kernel with stages of 128 columns for 65 to 256 tokens: three or four of them, filled by three producer groups in turn."""
import pytest

from tests.gpu_util import GuardedBinding, PotCase, bf16_dev, bits_of, f16_bits_to_bf16_bits, f16_dev, gate

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    return GuardedBinding()


# one X tile that both issuers share (K >= 512) and not; h at the edges of four stages; fewer stages than the ring has, one more, many
@pytest.mark.parametrize("M,stages", [(65, 4), (112, 4), (128, 4), (129, 4), (224, 4), (225, 3), (256, 3)])
@pytest.mark.parametrize("K", [384, 512, 640, 1664, 4096])
def test_wide_stages_match_oracle(B, oracle, M, K, stages):
    from paper_2507_11959_b200 import synth
    for bits, G, bf16, N in ((3, 128, False, 400), (4, 64, True, 144), (2, 64, False, 2320)):
        c = PotCase(N, K, bits, G, dist="t5", seed=(4, 990 + bits))
        X = synth.activations(synth.rng_for(4, 991 + M), M, K)
        X = f16_bits_to_bf16_bits(X) if bf16 else X
        plan = B.pot_debug_gemm_plan(M, N, K, bits, G, bf16)
        assert plan["stage_columns"] == 128 and plan["ring_stages"] == (3 if M <= 128 and K < 512 else stages), plan
        Y, A = oracle.matmul(c.packed, c.S, K, bits, G, X, dtype=oracle.BF16 if bf16 else oracle.F16)
        Xd = bf16_dev(X) if bf16 else f16_dev(X)
        for layout, P, S in ((B.TILED, c.tiled(), c.tiled_S()), (B.CANONICAL, c.d_packed, c.d_S)):
            ok, worst, tight = gate(bits_of(B.pot_gemm(P, S, K, bits, G, Xd, layout)), Y, A, bf16)
            assert ok and tight < 4.0, (layout, bits, bf16, worst, tight)

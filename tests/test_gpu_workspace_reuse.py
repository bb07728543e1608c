"""One workspace per matrix, zeroed once, for calls with any number of tokens: what one call leaves in it is not taken for anything by the next."""
import pytest
import torch

from paper_2507_11959_b200 import binding as B

pytestmark = pytest.mark.gpu


def run_sequence(N, K, bits, G, tokens):
    """FP16 and BF16 products in turn on one workspace, each compared bit for bit with the same product on a workspace of its own."""
    gen = torch.Generator(device="cuda").manual_seed(N + K + bits)
    packed, scales = B.pot_quantize_ref((torch.randn(N, K, generator=gen, device="cuda", dtype=torch.float16) * 0.02), bits, G, B.SCALE_TOP)
    packed, scales = B.pot_repack(packed, K, bits, 0), B.pot_repack_scales(scales, K, G, 0)
    X = torch.randn(max(tokens), K, generator=gen, device="cuda", dtype=torch.float16)
    Xs = (X, X.to(torch.bfloat16))
    need = {M: B.pot_gemm_workspace_bytes(M, N, K, bits, G) for M in tokens}
    shared = B.new_workspace(max(need.values()))
    alone = {}
    for i, M in enumerate(tokens):
        for x in Xs[::1 - 2 * (i & 1)]:
            def product(workspace):
                Y = torch.full((M, N), 0x7E5A, dtype=torch.int16, device="cuda")  # (a NaN: an element that is not written shows)
                B.pot_gemm(packed, scales, K, bits, G, x[:M], B.TILED, Y=Y.view(x.dtype), workspace=workspace)
                return Y
            if (M, x.dtype) not in alone:
                alone[M, x.dtype] = product(B.new_workspace(need[M]))
            assert torch.equal(product(shared), alone[M, x.dtype]), (i, M, x.dtype)
    torch.cuda.synchronize()
    assert B.pot_debug_errors() == (0, 0, 0)


@pytest.mark.parametrize("N,K,bits,G,tokens", [
    (28672, 8192, 3, 128, (2048, 4, 1, 16, 2, 300, 8, 512, 1, 4)), (8192, 28672, 2, 128, (64, 4, 1, 16, 2, 300, 8, 1, 4)),
    (22016, 4096, 4, 64, (512, 4, 1, 16, 2, 300, 8, 1, 4)), (5120, 13824, 3, 64, (32, 4, 1, 16, 2, 300, 8, 1, 4)), (6400, 8192, 3, 128, (32, 4, 1, 4, 64, 2))])
def test_even_split_after_partial_sums_of_more_tokens(N, K, bits, G, tokens):
    """The sums that go from CTA to CTA lie where products of more tokens leave partial sums: those are no marks."""
    plans = [(M, B.pot_debug_gemm_plan(M, N, K, bits, G)) for M in tokens]
    assert any(p["split_tiles"] for _, p in plans) and any(p["streaming"] and B.pot_debug_gemv_split(M, N, K, bits, G) == 2 for M, p in plans)
    run_sequence(N, K, bits, G, tokens)


@pytest.mark.parametrize("N,K,bits,G,tokens", [
    (2048, 8192, 3, 128, (32, 4, 1, 300, 2, 512, 8, 1)), (2400, 1152, 2, 64, (64, 4, 1, 16, 8, 2, 1)), (1536, 4608, 4, 128, (16, 4, 1, 300, 2, 1))])
def test_unit_split_after_partial_sums_of_more_tokens(N, K, bits, G, tokens):
    """Arrival counters of the row blocks, of which there may be more than 64: partial sums of more tokens lie behind them."""
    plans = [(M, B.pot_debug_gemm_plan(M, N, K, bits, G)) for M in tokens]
    assert any(p["split_tiles"] for _, p in plans) and all(B.pot_debug_gemv_split(M, N, K, bits, G) == 1 for M, p in plans if p["streaming"])
    run_sequence(N, K, bits, G, tokens)


@pytest.mark.parametrize("N,K,bits,G,tokens", [(8192, 28672, 2, 128, (16, 2048, 16)), (1024, 28672, 3, 64, (32, 7680, 32, 7680))])
def test_more_than_64_split_tiles_after_partial_sums_of_fewer(N, K, bits, G, tokens):
    """The arrival counters of up to 74 split tiles, the last ten of which lie where products of other token counts leave partial sums."""
    plans = {M: B.pot_debug_gemm_plan(M, N, K, bits, G) for M in tokens}
    assert any(p["split_tiles"] > 64 and p["cluster"] == 0 for p in plans.values()) and any(0 < p["split_tiles"] <= 64 for p in plans.values())
    run_sequence(N, K, bits, G, tokens)

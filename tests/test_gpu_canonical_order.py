"""The canonical GEMV asks for codes and scales before it waits for its predecessor in the stream."""
import pytest
import torch

from paper_2507_11959_b200 import binding as B
from paper_2507_11959_b200 import synth
from tests.gpu_util import f16_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,N,K", [(2, 1000, 4096), (3, 4099, 1152), (4, 37, 28672)])
def test_canonical_gemv_behind_the_quantizer_and_behind_itself(bits, N, K):
    """Weights quantized just before the product, then a chain in which every product reads what the one before it wrote: new weights and inputs
    every time, nothing synchronised, eagerly and from a graph, against the same steps one by one."""
    G, R = 128, 5
    Ws = [f16_dev(synth.weights(synth.rng_for(8, 700 + r), N, K, "t5")) for r in range(R)]
    xs = [f16_dev(synth.activations(synth.rng_for(8, 720 + r), 1, K)[0]) for r in range(R)]
    W, x = torch.empty_like(Ws[0]), torch.empty_like(xs[0])
    S = torch.empty(N, K // G, dtype=torch.float16, device="cuda")
    packed = torch.empty(N, K * bits // 8, dtype=torch.uint8, device="cuda")
    ys, mid = [torch.empty(N, dtype=torch.float16, device="cuda") for _ in range(3)], torch.zeros(K, dtype=torch.float16, device="cuda")

    def chain(sync):
        p, s = B.pot_quantize_ref(W, bits, G, B.SCALE_TOP)
        B.pot_gemv(p, s, K, bits, G, x, B.CANONICAL, y=ys[0])
        for a, b in ((0, 1), (1, 2)):
            if sync:
                torch.cuda.synchronize()
            mid[:min(N, K)].copy_(ys[a][:min(N, K)].clamp(-8, 8))
            B.pot_gemv(p, s, K, bits, G, mid, B.CANONICAL, y=ys[b])
        return p, s

    ref = []
    for r in range(R):
        W.copy_(Ws[r])
        x.copy_(xs[r])
        p, s = B.pot_quantize_ref(W, bits, G, B.SCALE_TOP)
        torch.cuda.synchronize()
        packed.copy_(p.view(packed.shape))
        S.copy_(s)
        torch.cuda.synchronize()
        first = B.pot_gemv(packed, S, K, bits, G, x, B.CANONICAL).clone()
        torch.cuda.synchronize()
        chain(True)
        torch.cuda.synchronize()
        assert torch.equal(ys[0], first)
        ref.append([y.clone() for y in ys])
    assert not torch.equal(ref[0][2], ref[1][2])
    for it in range(6 * R):
        r = (3 * it + 1) % R
        W.copy_(Ws[r])
        x.copy_(xs[r])
        chain(False)
        assert all(torch.equal(a, b) for a, b in zip(ys, ref[r])), (it, r)
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            chain(False)
        for it in range(3 * R):
            r = (2 * it + 1) % R
            W.copy_(Ws[r])
            x.copy_(xs[r])
            graph.replay()
            st.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(ys, ref[r])), ("graph", it, r)
    assert B.pot_debug_errors() == (0, 0, 0)

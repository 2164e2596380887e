"""Small batches, which the FFN and the combine group by themselves: mask-word
and chunk edges (32, 64 and 96 tokens), pools that are not whole chunks of 32
experts, the largest pool and selection, the shared expert."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_34117_gb300 as sw
from paper_2609_34117_gb300 import synth

pytestmark = pytest.mark.gpu

DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sw.build.build()
    oracle.build()


@pytest.mark.parametrize("B,E,k,shared", [(31, 33, 3, 0), (32, 16, 2, 128), (33, 100, 8, 0),
                                          (64, 1024, 32, 0), (65, 40, 4, 128), (96, 1024, 8, 0),
                                          (95, 16, 16, 0), (97, 40, 4, 128)])
def test_layer_small_batches(B, E, k, shared):
    H, I = 256, 128
    shape = synth.LayerShape(hidden=H, num_experts=E, inter=I, top_k=k)
    w_gu, w_d = synth.expert_weights(shape, 1)
    wr = synth.router_weight(shape, 1)
    x = synth.hidden_states(B, shape, 2)
    args = [t.to(DEV) for t in (x, wr)] + [None] + [t.to(DEV) for t in (w_gu, w_d)] + [k]
    host = [synth.bf16_bits(x), wr.numpy(), None, synth.bf16_bits(w_gu), synth.bf16_bits(w_d), k]
    if shared:
        w_sg, gu, dn = synth.shared_expert(H, shared, 3)
        out = sw.slimwise_moe_decode_shared(*args, w_sg.to(DEV), gu.to(DEV), dn.to(DEV))
        ref = oracle.moe_decode_shared(*host, w_sg.numpy(), synth.bf16_bits(gu), synth.bf16_bits(dn))
    else:
        out = sw.slimwise_moe_decode_full(args[0], args[1], *args[3:])
        ref = oracle.moe_decode(*host)
    got = out.float().cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref["out"]) <= 1e-2 * np.linalg.norm(ref["out"])
    assert np.abs(got - ref["out"]).max() <= 3e-2
    # in place: the output may be the hidden rows' own buffer
    if not shared:
        y = sw.slimwise_moe_decode_full(args[0], args[1], *args[3:], out=args[0])
        assert torch.equal(y, out)


# hidden rows that leave a routing CTA no room for its static shared memory at
# the usual tokens per cluster: fewer tokens, not a refused launch
@pytest.mark.parametrize("B", [40, 70])
def test_routing_of_rows_that_fill_shared_memory(B):
    H, E, k = 28928, 128, 2
    shape = synth.LayerShape(hidden=H, num_experts=E, inter=64, top_k=k)
    x, wr = synth.hidden_states(B, shape, 1), synth.router_weight(shape, 2)
    r = sw.slimwise_moe_route(x.to(DEV), wr.to(DEV), None, k, E)
    idx, gates = oracle.route(oracle.router_logits(synth.bf16_bits(x), wr.numpy()),
                              np.arange(E, dtype=np.int32), k)
    assert np.array_equal(r["topk_idx"].cpu().numpy(), idx)
    np.testing.assert_allclose(r["topk_gate"].cpu().numpy(), gates, rtol=4e-6, atol=1e-7)


# 65 tokens of the largest pool: the combine's CTAs find no room beside the
# FFN's.  The chained launches must not take longer than plain stream ordering:
# 0.92 of its time, and 1.19 when the combine was signalled early all the same
def test_chained_launches_of_a_large_pool_overlap():
    E, H, I, k, B = 1024, 512, 64, 8, 65
    shape = synth.LayerShape(hidden=H, num_experts=E, inter=I, top_k=k)
    w_gu, w_d = synth.expert_weights(shape, 1, device=DEV)
    wr, x = synth.router_weight(shape, 2, device=DEV), synth.hidden_states(B, shape, 3, device=DEV)
    ret = torch.arange(256, dtype=torch.int32, device=DEV)
    ws, out = sw.alloc_workspace(B, H, E, I, k, DEV), torch.empty_like(x)

    def best_of_9(**opts):  # replayed from a graph: no host time
        def call():
            sw.slimwise_moe_decode_ex(x, wr, ret, w_gu, w_d, k, out=out, workspace=ws, **opts)
        call()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for _ in range(50):
                call()
        times = []
        for _ in range(9):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            graph.replay()
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    assert best_of_9() <= 1.05 * best_of_9(disable_pdl=True)

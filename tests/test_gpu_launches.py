"""The kernels per call that bench.py reports are those that the library
launches, on both sides of each rule that changes their number."""
import pytest
import torch
from torch.profiler import ProfilerActivity, profile

import bench
import paper_2609_34117_gb300 as sw
from paper_2609_34117_gb300 import synth

pytestmark = pytest.mark.gpu

DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sw.build.build()
    # a process's first profile can come back empty
    for _ in range(5):
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            torch.ones(8, device=DEV).add_(1)
            torch.cuda.synchronize()
        if any("kernel" in e.name for e in p.events()):
            return
    pytest.skip("the profiler records no kernels")


@pytest.mark.parametrize("H,E,k,B,m_prime,ffn_items", [
    (256, 16, 2, 4, 8, 0), (256, 16, 2, 96, 8, 0), (256, 16, 2, 97, 8, 0), (256, 16, 2, 96, 8, 1),
    (384, 16, 2, 96, 8, 1), (256, 16, 2, 256, 8, 0), (256, 16, 2, 257, 8, 0),
    (256, 16, 2, 767, 8, 0), (256, 16, 2, 768, 8, 0), (256, 128, 2, 191, 128, 0),
    (256, 128, 2, 192, 128, 0), (256, 256, 2, 63, 256, 0), (256, 256, 2, 64, 256, 0),
    (256, 512, 2, 1, 257, 0), (128, 1024, 1, 800, 1024, 0), (2048, 128, 8, 2048, 128, 0)])
def test_reported_launches_are_the_library_s(H, E, k, B, m_prime, ffn_items):
    shape = synth.LayerShape(hidden=H, num_experts=E, inter=128, top_k=k)
    w_gu, w_d = synth.expert_weights(shape, 1, device=DEV)
    wr, x = synth.router_weight(shape, 2, device=DEV), synth.hidden_states(B, shape, 3, device=DEV)
    ret = torch.arange(m_prime, dtype=torch.int32, device=DEV)
    ws, out = sw.alloc_workspace(B, H, E, 128, k, DEV), torch.empty_like(x)

    def call():
        sw.slimwise_moe_decode_ex(x, wr, ret, w_gu, w_d, k, out=out, workspace=ws, ffn_items=ffn_items)
    call()
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        call()
        torch.cuda.synchronize()
    kernels = [e for e in p.events() if "slimwise::" in e.name]
    assert len(kernels) == bench.layer_launches(shape, B, m_prime, 0, ffn_items), \
        [e.name for e in kernels]

"""Two host threads that call layers of different sizes at the same time, each
with its own workspace: what one thread sets up for its launches must not
refuse the other's.  The kernels themselves are ordered on one stream."""
import threading

import pytest
import torch

import paper_2609_34117_gb300 as sw
from paper_2609_34117_gb300 import synth

pytestmark = pytest.mark.gpu

DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sw.build.build()


# (H, E, B, k): the same kernels with different shared memory -- cluster routing
# of narrow and wide rows; the FFN and tiled grouping of large and small pools
@pytest.mark.parametrize("a,b", [((256, 16, 8, 2), (4096, 16, 8, 2)),
                                 ((128, 1024, 800, 1), (128, 16, 800, 1))])
def test_threads_with_different_shapes(a, b):
    stream = torch.cuda.Stream()
    errors, n = [], 6000

    def work(H, E, B, k, out):
        try:
            shape = synth.LayerShape(hidden=H, num_experts=E, inter=64, top_k=k)
            w_gu, w_d = synth.expert_weights(shape, 1, device=DEV)
            wr = synth.router_weight(shape, 2, device=DEV)
            x = synth.hidden_states(B, shape, 3, device=DEV)
            ws = sw.alloc_workspace(B, H, E, 64, k, DEV)
            y = torch.empty_like(x)
            torch.cuda.synchronize()
            start.wait()
            for _ in range(n):
                sw.slimwise_moe_decode_full(x, wr, w_gu, w_d, k, out=y, workspace=ws, stream=stream)
            stream.synchronize()
            assert sw.slimwise_moe_device_status(ws, stream) == 0
            out.append((y, sw.slimwise_moe_decode_full(x, wr, w_gu, w_d, k, stream=stream)))
            stream.synchronize()
        except Exception as e:  # reported by the test's own thread
            errors.append(e)
            start.abort()

    start = threading.Barrier(2)
    outs = [[], []]
    threads = [threading.Thread(target=work, args=(*s, o)) for s, o in zip((a, b), outs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for o in outs:
        assert torch.equal(*o[0])

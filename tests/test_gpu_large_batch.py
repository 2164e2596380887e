"""Large batches (prompt chunks, calibration batches) against the oracle: the
tiled grouping kernels at the edges of their range and of their tiles, and
whole layers whose experts take several work entries."""
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


# 768 tokens is where the tiled kernels start; tiles are 128 tokens up to
# 8192 of them, then 256 (8193: one token in the last tile's first block)
@pytest.mark.parametrize("B,E,k", [(767, 16, 2), (768, 16, 2), (769, 128, 8), (1025, 1024, 32),
                                   (4097, 256, 8), (8192, 128, 8), (8193, 16, 1),
                                   (20000, 100, 4)])
def test_group_large_batches(B, E, k):
    rng = np.random.default_rng(B)
    sel = np.argsort(rng.random((B, E)) * np.linspace(0.2, 1.0, E), axis=1)[:, :k].astype(np.int32)
    g = sw.slimwise_moe_group(torch.from_numpy(sel).to(DEV), E)
    ref = oracle.group_by_expert(sel, E)
    U = ref["union_size"]
    assert int(g["union_size"].item()) == U
    for name in ("counts", "offsets", "perm", "pos"):
        assert np.array_equal(g[name].cpu().numpy(), ref[name]), name
    ids = g["union_ids"].cpu().numpy()
    assert np.array_equal(ids[:U], ref["union_ids"]) and np.all(ids[U:] == -1)


def _check(got, ref):
    got = got.float().cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) <= 1e-2 * np.linalg.norm(ref)
    assert np.abs(got - ref).max() <= 3e-2


# grouped rows of a ragged hidden width; experts of several entries with an
# odd remainder, one of them selected by every token; the shared expert
@pytest.mark.parametrize("H,E,I,k,B,shared", [(640, 24, 192, 3, 777, 0), (256, 16, 128, 2, 1031, 0),
                                              (256, 16, 128, 2, 1500, 128), (512, 8, 128, 4, 2051, 0)])
def test_layer_large_batches(H, E, I, k, B, shared):
    shape = synth.LayerShape(hidden=H, num_experts=E, inter=I, top_k=k)
    w_gu, w_d = synth.expert_weights(shape, 1)
    wr = synth.router_weight(shape, 1)
    bias = torch.zeros(E)
    bias[E // 2] = 20.0
    x, wr = synth.apply_popularity_bias(synth.hidden_states(B, shape, 2), wr, bias)
    args = [t.to(DEV) for t in (x, wr)] + [None] + [t.to(DEV) for t in (w_gu, w_d)] + [k]
    host = [synth.bf16_bits(x), wr.numpy(), None, synth.bf16_bits(w_gu), synth.bf16_bits(w_d), k]
    toks = np.sort(np.random.default_rng(B).choice(B, size=200, replace=False)).astype(np.int32)
    if shared:
        w_sg, gu, dn = synth.shared_expert(H, shared, 3)
        out = sw.slimwise_moe_decode_shared(*args, w_sg.to(DEV), gu.to(DEV), dn.to(DEV))
        ref = oracle.moe_decode_shared(*host, w_sg.numpy(), synth.bf16_bits(gu), synth.bf16_bits(dn), toks)
    else:
        out = sw.slimwise_moe_decode_full(args[0], args[1], *args[3:])
        ref = oracle.moe_decode_sampled(*host, toks)
    _check(out[toks], ref["out"])
    r = sw.slimwise_moe_route(args[0], args[1], None, k, E)
    assert np.array_equal(r["topk_idx"].cpu().numpy(), ref["idx"])


# Tiled routing in tiles of 32, 16 and 8 tokens x 16 experts with ragged edges, the three top-k forms, a pool whose logits do not
# fit the scratch rows (the cluster kernel keeps it), any order of the ids
@pytest.mark.parametrize("H,E,k,B,m_prime", [(256, 16, 2, 609, 8), (2048, 512, 8, 33, 511),
                                             (2048, 1024, 8, 1, 1024), (2048, 128, 8, 257, 121),
                                             (256, 16, 2, 5000, 8), (640, 40, 3, 769, 33),
                                             (2048, 128, 8, 800, 128), (384, 256, 8, 1055, 201),
                                             (256, 512, 32, 777, 300), (128, 1024, 1, 800, 1024)])
def test_tiled_routing_equals_oracle_and_small_batches(H, E, k, B, m_prime):
    shape = synth.LayerShape(hidden=H, num_experts=E, inter=64, top_k=k)
    x, wr = synth.hidden_states(B, shape, 3), synth.router_weight(shape, 4)
    wr[E // 2] = wr[E // 3]  # equal logits: ties to the lowest id
    ret = synth.retained_set(E, m_prime, 5, shuffle=True)
    xd, wd, rd = x.to(DEV), wr.to(DEV), ret.to(DEV)
    r = sw.slimwise_moe_route(xd, wd, rd, k, E)
    idx, gates = oracle.route(oracle.router_logits(synth.bf16_bits(x), wr.numpy()), ret.numpy(), k)
    assert np.array_equal(r["topk_idx"].cpu().numpy(), idx)
    np.testing.assert_allclose(r["topk_gate"].cpu().numpy(), gates, rtol=4e-6, atol=1e-7)
    # bit for bit what the cluster kernel gives (small batches), special values
    # among them
    xd[5 % B], xd[B - 1, 7], xd[30 % B, 9] = 0.0, float("inf"), float("nan")
    r = sw.slimwise_moe_route(xd, wd, rd, k, E)
    step = 28
    for t0 in range(0, B, step):
        s = sw.slimwise_moe_route(xd[t0:t0 + step].contiguous(), wd, rd, k, E)
        assert torch.equal(s["topk_idx"], r["topk_idx"][t0:t0 + step])
        assert torch.equal(s["topk_gate"].view(torch.int32),
                           r["topk_gate"][t0:t0 + step].view(torch.int32))


# Routing that bounds the logits on the tensor cores and evaluates those that
# can be selected: at the smallest sizes of its range, with ragged tiles of
# tokens and experts, an odd pool (unpaired stores), K in 4 parts and in one,
# ids in any order, and where no bound holds (values that are not finite, norms
# that leave the range, tied and repeated experts)
@pytest.mark.parametrize("H,E,k,B,m_prime", [(2048, 128, 8, 2048, 128), (2048, 256, 8, 1025, 256),
                                             (640, 200, 8, 5001, 177), (256, 256, 16, 8193, 256),
                                             (2048, 160, 1, 2050, 129)])
def test_filtered_routing_equals_oracle_and_small_batches(H, E, k, B, m_prime):
    shape = synth.LayerShape(hidden=H, num_experts=E, inter=64, top_k=k)
    x, wr = synth.hidden_states(B, shape, 3), synth.router_weight(shape, 4)
    wr[E // 2] = wr[E // 3]  # equal logits: ties to the lowest id
    wr[E // 4] = wr[E // 5] * (1 + 1e-6)  # closer than any bound of the filter
    ret = synth.retained_set(E, m_prime, 5, shuffle=True)
    xd, wd, rd = x.to(DEV), wr.to(DEV), ret.to(DEV)
    r = sw.slimwise_moe_route(xd, wd, rd, k, E)
    idx, gates = oracle.route(oracle.router_logits(synth.bf16_bits(x), wr.numpy()), ret.numpy(), k)
    assert np.array_equal(r["topk_idx"].cpu().numpy(), idx)
    np.testing.assert_allclose(r["topk_gate"].cpu().numpy(), gates, rtol=4e-6, atol=1e-7)
    # bit for bit what the cluster kernel gives (small batches)
    xd[5], xd[B - 1, 7], xd[30, 9] = 0.0, float("inf"), float("nan")
    xd[31], xd[32] = xd[31] * 1e36, xd[32] * 1e-30
    rep = rd.clone()
    rep[1::2] = rep[0::2][:len(rep[1::2])]  # every id twice
    big = wd.clone()
    big[E // 6, 3] = float("inf")
    rows = np.r_[0:64, B // 2:B // 2 + 64, B - 65:B]
    for w, ids in [(wd, rd), (wd, rep), (big, rd), (torch.zeros_like(wd), rd), (wd * 1e-30, rd),
                   (wd[:1] + 1e-5 * wd, rd)]:
        r = sw.slimwise_moe_route(xd, w, ids, k, E)
        s = [sw.slimwise_moe_route(xd[rows[i:i + 28]].contiguous(), w, ids, k, E)
             for i in range(0, len(rows), 28)]
        assert torch.equal(torch.cat([v["topk_idx"] for v in s]), r["topk_idx"][rows])
        assert torch.equal(torch.cat([v["topk_gate"] for v in s]).view(torch.int32),
                           r["topk_gate"][rows].view(torch.int32))


def _rows(kind, shape, g):
    """normal, of one sign (sums without cancellation), elements over e^+-6"""
    r = torch.randn(shape, generator=g, device=DEV)
    if kind == "sign":
        r = r.abs()
    elif kind == "wide":
        r = r.sign() * torch.exp(12 * torch.rand(shape, generator=g, device=DEV) - 6)
    return r


def _filter_bound(H):
    return 2.0**-17 + H / 8 * 2.0**-21 + (H / 32 + 6) * 2.0**-23


# The filter's bound allows the tensor core's sum a rounding that its
# documentation does not give; what it really has is seen here: the approximate
# logits (left in the workspace's last region by a routing-only call) against
# 64 bits, K in one part.  At most a quarter of the bound.
@pytest.mark.parametrize("kind", ["normal", "sign", "wide"])
@pytest.mark.parametrize("H,k", [(2048, 8), (8192, 8), (32768, 2)])
def test_tensor_core_logits_stay_well_inside_their_bound(H, k, kind):
    B, E = 5120, 256
    assert torch.cuda.get_device_properties(0).multi_processor_count < 2 * 2 * B // 128
    g = torch.Generator(device=DEV).manual_seed(H)
    x = _rows(kind, (B, H), g).to(torch.bfloat16)
    wr = 0.02 * _rows(kind, (E, H), g)
    ws = sw.alloc_workspace(B, H, E, 64, k, DEV)
    sw.slimwise_moe_route(x, wr, None, k, E, 64, workspace=ws)
    y0 = ws.numel() - (B * k * H * 2 + 1023) // 1024 * 1024
    z = ws[y0:y0 + B * E * 4].view(torch.float32).view(B, E)[64:].double()  # grouping wrote the first
    x, wr = x[64:].double(), wr.double()
    norms = x.norm(dim=1)[:, None] * wr.norm(dim=1)[None, :]
    ratio = ((z - x @ wr.T).abs() / (norms * _filter_bound(H))).max().item()
    assert 0 < ratio <= 0.25, ratio


# every token's selections are those of small batches bit for bit, for rows of
# each kind and long sums: the bound is then up to several gaps between the
# logits wide.  Half of the experts are one row spread over three bounds.
@pytest.mark.parametrize("copies", [False, True])
@pytest.mark.parametrize("kind", ["normal", "sign", "wide"])
@pytest.mark.parametrize("H,B,E", [(4096, 1030, 256), (8192, 2050, 128), (8192, 5120, 256)])
def test_filtered_routing_of_long_rows(H, B, E, kind, copies):
    k = 8
    g = torch.Generator(device=DEV).manual_seed(B)
    x = _rows(kind, (B, H), g).to(torch.bfloat16)
    wr = 0.02 * _rows(kind, (E, H), g)
    if copies:
        spread = 3 * _filter_bound(H) * torch.rand((E // 2, 1), generator=g, device=DEV)
        noise = 1e-5 * torch.randn((E // 2, H), generator=g, device=DEV)
        wr[::2] = wr[:1] * (1 + spread) * (1 + noise)
    r = sw.slimwise_moe_route(x, wr, None, k, E)
    for t0 in range(0, B, 28):
        s = sw.slimwise_moe_route(x[t0:t0 + 28].contiguous(), wr, None, k, E)
        assert torch.equal(s["topk_idx"], r["topk_idx"][t0:t0 + 28])
        assert torch.equal(s["topk_gate"].view(torch.int32),
                           r["topk_gate"][t0:t0 + 28].view(torch.int32))


@pytest.mark.parametrize("B,E,k", [(1, 16, 1), (5, 1024, 32), (300, 96, 8)])
def test_routing_outputs_may_be_left_out(B, E, k):
    # any output may be NULL; one written alone equals the same one among all
    from paper_2609_34117_gb300 import binding
    import ctypes
    shape = synth.LayerShape(hidden=256, num_experts=E, inter=64, top_k=k)
    x = synth.hidden_states(B, shape, 3).to(DEV)
    wr = synth.router_weight(shape, 4).to(DEV)
    r = sw.slimwise_moe_route(x, wr, None, k, E)
    names = ("topk_idx", "topk_gate", "counts", "offsets", "union_ids", "union_size", "perm", "pos")
    ws = sw.alloc_workspace(B, 256, E, 64, k)
    s = binding.Shape(B, 256, E, 64)
    for i, n in enumerate(names):
        alone = torch.full_like(r[n], -7)
        ptrs = [alone.data_ptr() if j == i else None for j in range(8)]
        rc = binding.load().slimwise_moe_route(
            x.data_ptr(), wr.data_ptr(), None, 0, k, torch.cuda.current_stream().cuda_stream,
            ctypes.byref(s), ws.data_ptr(), ws.numel(), *ptrs)
        assert rc == 0
        assert torch.equal(alone, r[n]), n

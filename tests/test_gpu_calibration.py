"""Importance statistics where the summing kernels can go wrong: experts with
no row, with fewer rows than a summing CTA has threads and with several per
thread, and row widths that are not a whole batch of loads."""
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


@pytest.mark.parametrize("H,E,I,k,B,hot", [(256, 16, 128, 2, 1, False), (256, 16, 128, 2, 300, True),
                                           (640, 24, 64, 3, 129, False), (4224, 8, 64, 2, 70, False)])
def test_statistics_of_ragged_rows_and_popular_experts(H, E, I, k, B, hot):
    shape = synth.LayerShape(hidden=H, num_experts=E, inter=I, top_k=k)
    w_gu, w_d = synth.expert_weights(shape, 1)
    wr = synth.router_weight(shape, 1)
    x = synth.hidden_states(B, shape, 2)
    if hot:  # one expert takes every token, one none
        bias = torch.zeros(E)
        bias[3], bias[5] = 30.0, -30.0
        x, wr = synth.apply_popularity_bias(x, wr, bias)
    stats, _ = sw.slimwise_moe_expert_stats(x.to(DEV), wr.to(DEV), w_gu.to(DEV), w_d.to(DEV), k)
    got = stats.cpu().numpy()
    ref = oracle.expert_stats(synth.bf16_bits(x), wr.numpy(), synth.bf16_bits(w_gu),
                              synth.bf16_bits(w_d), k)
    assert np.array_equal(got[:, 0], ref[:, 0])
    # gates are fp32 (a few ulp); a norm carries the bf16 roundings of the
    # activations and of its own row, 2^-9 each at most
    np.testing.assert_allclose(got[:, 1], ref[:, 1], rtol=1e-6, atol=1e-12)
    np.testing.assert_allclose(got[:, 2:], ref[:, 2:], rtol=4e-3, atol=1e-12)


@pytest.mark.parametrize("m", [1, 7, 32])
def test_selection_of_special_scores(m):
    # infinities rank as numbers, -0 ties with 0, negative scores below
    st = np.zeros((32, 4))
    st[:, 0] = 1.0
    st[:, 1] = np.where(np.arange(32) % 5 == 0, -0.0, np.arange(32) % 7 - 3.0)
    st[4, 1], st[9, 1] = np.inf, -np.inf
    ids = sw.slimwise_moe_select_retained(torch.from_numpy(st).to(DEV), m, "mass").cpu().numpy()
    assert np.array_equal(ids, oracle.select_retained(st, m, "mass"))


@pytest.mark.parametrize("m", [1, 7, 32])
def test_selection_with_nan_scores(m):
    # a NaN score is neither above nor below another: its expert is kept beside
    # the m highest of the others, and the lowest m ids of those are written
    st = np.zeros((32, 4))
    st[:, 0], st[:, 1] = 1.0, (np.arange(32) * 7) % 32
    nan = np.array([2, 19, 31])
    st[nan, 1] = np.nan
    ids = sw.slimwise_moe_select_retained(torch.from_numpy(st).to(DEV), m, "mass").cpu().numpy()
    rest = np.setdiff1d(np.arange(32), nan)
    best = rest[np.argsort(-st[rest, 1], kind="stable")[:m]]
    assert np.array_equal(ids, np.sort(np.concatenate([best, nan]))[:m])

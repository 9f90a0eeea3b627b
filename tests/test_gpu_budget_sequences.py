"""Counts, their sum and the error word for several sequences, into words that
hold something else before the call: alone, with and without a malformed
sequence, and inside a step (the words cleared by the forward's first
kernel)."""
import numpy as np
import pytest
import torch

import gpu_cases as G
from paper_2608_01784_gb300 import _binding as B
from paper_2608_01784_gb300 import api
from paper_2608_01784_gb300 import workloads as W


def _state(n_seq, seed):
    cfg = W.CONFIGS["llada_moe_b32"].with_(n_seq=n_seq, prompt_len=5, gen_len=64)
    return cfg, W.make_state(cfg, seed)


@pytest.mark.gpu
@pytest.mark.parametrize("n_seq", [2, 33])
@pytest.mark.parametrize("bad", [False, True])
def test_sum_and_error_word(n_seq, bad):
    cfg, state = _state(n_seq, 11 + n_seq)
    p = G.params_of(cfg)
    ref = G.oracle_allocate(state, p)
    if bad:
        state["active_block"][n_seq - 1] = 0  # flagged; the counts are K of far blocks
    ds = api.state_to_device(state)
    k_sum = torch.full((1,), 12345, dtype=torch.int64, device="cuda")
    status = torch.full((1,), 7, dtype=torch.int32, device="cuda")
    k, k_sum, status = api.allocate(ds, p, k_sum=k_sum, status=status)
    torch.cuda.synchronize()
    got = k.cpu().numpy()
    good = slice(0, got.size if not bad else got.size - cfg.seq_len)
    assert np.array_equal(got[good], ref[good])
    assert int(k_sum.item()) == int(got.sum())
    assert (B.reflex_read_status(status) == B.REFLEX_OK) == (not bad)


@pytest.mark.gpu
@pytest.mark.parametrize("n_seq", [2, 33])
def test_step_clears_the_words(n_seq):
    cfg, state = _state(n_seq, 3)
    cfg = cfg.with_(d=256, E=8, inter=128, k_max=8, weight_std=0.05)
    layer = W.make_layer(cfg, 5)
    dl = api.layer_to_device(layer, cfg.dtype)
    moe = api.MoELayer(dl, dtype="bf16", d=256, E=8, inter=128, shared_inter=0, k_max=8,
                       max_tokens=cfg.T)
    p = G.params_of(cfg)
    k_sum = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    status = torch.full((1,), 3, dtype=torch.int32, device="cuda")
    for _ in range(2):
        moe.step(api.state_to_device(state), p, dl["hidden"], k_sum=k_sum, status=status)
        torch.cuda.synchronize()
        assert int(k_sum.item()) == int(G.oracle_allocate(state, p).sum())
        assert B.reflex_read_status(status) == B.REFLEX_OK

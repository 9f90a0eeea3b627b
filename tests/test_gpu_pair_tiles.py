"""The CTA-pair expert GEMMs at the edges of their token tiles: row counts
either side of 32, 64, 96, 128 and 256 (the MMA's N, the row boxes, a second
tile of one row), whole and partial 32-row output chunks, both GEMM modes and
the dense shared expert, copied and gathered rows, against the oracle."""
import numpy as np
import pytest

import gpu_cases as G
from paper_2608_01784_gb300 import _binding as B
from paper_2608_01784_gb300 import workloads as W


@pytest.mark.gpu
@pytest.mark.parametrize("rows", [1, 16, 31, 32, 33, 63, 64, 65, 96, 97, 128, 129, 255, 256,
                                  257, 288, 511, 513])
def test_rows_of_an_expert(rows):
    # expert 0 of two gets `rows` tokens, expert 1 the others: the router
    # weights follow one hidden column, whose sign picks the expert
    T, d, inter = 2 * 513 + 10, 256, 128
    cfg = W.LayerConfig(name="pair", dtype="bf16", d=d, E=2, inter=inter, shared_inter=128,
                        k_min=1, k_base=1, k_max=1, delta_role=0, delta_cur=0, w_cf=0.3,
                        n_seq=1, prompt_len=T, gen_len=0, block=32, weight_std=0.05,
                        conf="uniform", mask_rule="half")
    layer = W.make_layer(cfg, rows, T=T)
    h = W.bf16_bits_to_f32(layer["hidden"]).reshape(T, d)
    w = np.zeros((2, d), np.float32)
    w[0, 0], w[1, 0] = 1.0, -1.0
    h[:, 0] = -1.0
    h[np.random.default_rng(rows).permutation(T)[:rows], 0] = 1.0
    layer["hidden"], layer["w_router"] = W.to_bf16_bits(h), W.to_bf16_bits(w)
    k = np.ones(T, np.int32)
    ref = G.oracle_layer(cfg, layer, k)
    assert int(ref["offsets"][1]) == rows
    outs = []
    for flags in (0, B.REFLEX_FLAG_GATHER_IN_GEMM):
        out, rec, status = G.GpuLayer(cfg, layer).forward(
            k, flags=B.REFLEX_FLAG_RENORM_TOPK | flags)
        assert status == B.REFLEX_OK
        G.check_routing(rec, ref, k, cfg.E)
        rel, mx = G.out_errors(out, ref["out"])
        assert rel <= G.BF16_REL_L2 and mx <= G.BF16_MAX_ABS, (rel, mx)
        outs.append(out)
    assert np.array_equal(outs[0], outs[1])

"""Router scores of short batches, bit for bit against the oracle's chain:
the resident-rows tiles at the edges of their bands (the last CTA count that
fits, one token more), partial token and expert tiles, long rows that leave
one CTA per SM, and the ring tiles behind them."""
import numpy as np
import pytest

import gpu_cases as G
import oracle
from paper_2608_01784_gb300 import _binding as B
from paper_2608_01784_gb300 import workloads as W


@pytest.mark.gpu
@pytest.mark.parametrize("T,E,d", [
    (1, 1, 256), (1, 17, 512), (3, 64, 2048),
    (304, 64, 256), (305, 64, 256),      # 4 x 16 tiles: 304 CTAs, one more row of them
    (608, 64, 512), (609, 64, 512),      # 8 x 16 tiles
    (528, 64, 2048), (529, 64, 2048),    # 97 KB per CTA: 7 CTAs on four SMs, then the ring
    (152, 64, 4096), (153, 64, 4096),    # 164 KB per CTA: one per SM
    (608, 64, 2048), (609, 64, 2048),    # the ring's one CTA per SM, then 16 x 32 tiles
    (470, 160, 1024),                    # 16 x 32 tiles, five expert tiles
    (1216, 64, 256), (1217, 64, 256),    # 16 x 32 tiles, then the ring
    (70, 250, 768), (1300, 8, 256), (4000, 8, 64),
    (300, 64, 192), (380, 64, 192),      # rows of no whole chunks: 1 x 1, 1 x 2 ring tiles
    (3100, 64, 256), (1100, 180, 128),   # 2 x 2 ring tiles
    (4096, 64, 256), (1400, 250, 256), (1700, 250, 256),  # 4 x 4, 2 x 2, 2 x 4 ring tiles
    (6475, 96, 128), (2060, 250, 128),   # 2 x 2 with eight CTAs per SM, 4 x 4
    (30000, 10, 128),
])
def test_scores_bit_exact(T, E, d):
    cfg = W.LayerConfig(name="scores", dtype="bf16", d=d, E=E, inter=128, shared_inter=0,
                        k_min=1, k_base=1, k_max=1, delta_role=0, delta_cur=0, w_cf=0.3,
                        n_seq=1, prompt_len=T, gen_len=0, block=32, weight_std=0.05,
                        conf="uniform", mask_rule="half")
    layer = W.make_layer(cfg, T + E + d, T=T)
    gl = G.GpuLayer(cfg, layer)
    _, rec, status = gl.forward(np.ones(T, np.int32),
                                flags=B.REFLEX_STAGE_ROUTE | B.REFLEX_FLAG_SIMT_EXPERTS |
                                B.REFLEX_FLAG_EXACT_SCORES)
    assert status == B.REFLEX_OK
    z = oracle.router_logits(layer["hidden"], layer["w_router"])
    assert np.array_equal(rec["scores"].view(np.uint32), z.view(np.uint32))

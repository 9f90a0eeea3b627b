"""The shared expert's tiles carried by the routed 1-SM GEMM launches, against
the oracle: row counts at the edges of a 128-row tile, a shared width unlike
the routed one (another reduction length in the same down launch), both tile
widths, and a shared width that the wide tiles do not divide (its own
launches)."""
import numpy as np
import pytest

import gpu_cases as G
from paper_2608_01784_gb300 import _binding as B
from paper_2608_01784_gb300 import workloads as W


@pytest.mark.gpu
@pytest.mark.parametrize("T,E,inter,shared", [
    (1, 8, 128, 128),
    (127, 8, 256, 128),
    (129, 64, 128, 384),
    (300, 512, 512, 128),   # 256-wide tiles
    (300, 512, 512, 64),    # 256-wide tiles, 64 shared columns: own launches
    (2100, 128, 128, 256),  # 2048 tokens and more: pair tiles before
])
def test_shared_expert_in_the_routed_launch(T, E, inter, shared):
    cfg = W.LayerConfig(name="shared", dtype="bf16", d=256, E=E, inter=inter,
                        shared_inter=shared, k_min=1, k_base=2, k_max=4, delta_role=1,
                        delta_cur=1, w_cf=0.3, n_seq=1, prompt_len=T, gen_len=0, block=32,
                        weight_std=0.05, conf="uniform", mask_rule="half")
    layer = W.make_layer(cfg, 7 + T, T=T)
    k = np.random.default_rng(T).integers(1, 5, T).astype(np.int32)
    out, rec, status = G.GpuLayer(cfg, layer).forward(k)
    assert status == B.REFLEX_OK
    ref = G.oracle_layer(cfg, layer, k)
    G.check_routing(rec, ref, k, cfg.E)
    rel, mx = G.out_errors(out, ref["out"])
    assert rel <= G.BF16_REL_L2 and mx <= G.BF16_MAX_ABS, (rel, mx)

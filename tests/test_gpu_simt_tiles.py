"""The SIMT expert GEMMs at the edges of their tiles (16 x 64 and 64 x 128
outputs, k blocks of 64 and 16, 128-row group tiles), against the oracle:
one row, one row either side of a tile, column counts that leave a partial
last tile, and both tile sizes of the dispatch.  The tolerances are the fp32
and bf16 layer tolerances (a dot product of K terms errs by at most
K 2^-24 sum |x w|; 32-term chunks keep it far below)."""
import numpy as np
import pytest

import gpu_cases as G
from paper_2608_01784_gb300 import _binding as B
from paper_2608_01784_gb300 import workloads as W


def _case(dtype, T, E, kmax, d, inter, shared, seed):
    cfg = W.LayerConfig(name="simt", dtype=dtype, d=d, E=E, inter=inter, shared_inter=shared,
                        k_min=1, k_base=1, k_max=kmax, delta_role=0, delta_cur=0, w_cf=0.3,
                        n_seq=1, prompt_len=T, gen_len=0, block=32,
                        weight_std=None if dtype == "f32" else 0.02, conf="uniform",
                        mask_rule="half")
    return cfg, W.make_layer(cfg, seed, T=T)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("T,E,kmax,d,inter,shared", [
    (1, 1, 1, 64, 64, 0),
    (15, 1, 1, 64, 64, 64),       # one row short of a small tile
    (17, 2, 2, 128, 192, 0),
    (65, 1, 1, 320, 64, 0),
    (129, 3, 2, 192, 64, 64),     # a second 128-row group tile of one row
    (128, 1, 1, 64, 128, 0),
    (20, 40, 2, 256, 320, 0),     # about one row per expert: warp-per-dot kernels
    (700, 20, 2, 128, 256, 0),    # small tiles, two CTAs per SM
    (2500, 1, 1, 64, 512, 0),     # large tiles: 64 x 128
    (1999, 5, 4, 192, 320, 0),    # ragged groups, partial column tiles
    (2048, 1, 1, 1024, 640, 64),  # 32 chunks of 32 products
])
def test_tile_edges(dtype, T, E, kmax, d, inter, shared):
    cfg, layer = _case(dtype, T, E, kmax, d, inter, shared, seed=T + d)
    k = np.random.default_rng(T).integers(1, kmax + 1, T).astype(np.int32)
    gl = G.GpuLayer(cfg, layer)
    out, rec, status = gl.forward(k, flags=B.REFLEX_FLAG_RENORM_TOPK |
                                  B.REFLEX_FLAG_SIMT_EXPERTS)
    assert status == B.REFLEX_OK
    ref = G.oracle_layer(cfg, layer, k)
    G.check_routing(rec, ref, k, cfg.E)
    rel, mx = G.out_errors(out, ref["out"])
    if dtype == "f32":
        assert rel <= G.F32_REL_L2 and mx <= G.F32_MAX_ABS, (rel, mx)
    else:
        assert rel <= G.BF16_REL_L2 and mx <= G.BF16_MAX_ABS, (rel, mx)


@pytest.mark.gpu
@pytest.mark.parametrize("T,inter", [(40, 64), (2500, 512)])
def test_an_overflowing_sum_stays_infinite(T, inter):
    # up weights of 1e38: every up sum of 64 ones is +inf, the gate sums are
    # 64, so act = 64 * inf and y, with positive down weights, is +inf
    d = 64
    cfg, layer = _case("f32", T, 1, 1, d, inter, 0, seed=T)
    layer["hidden"][:] = 1.0
    layer["w_gate_up"][:, :inter] = 1.0
    layer["w_gate_up"][:, inter:] = 1e38
    layer["w_down"][:] = 1.0
    gl = G.GpuLayer(cfg, layer)
    out, _, status = gl.forward(np.ones(T, np.int32))
    assert status == B.REFLEX_OK
    assert np.all(np.isposinf(out))

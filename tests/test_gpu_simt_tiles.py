"""The SIMT expert GEMMs at the edges of their tiles (16 x 64 and 64 x 128
outputs, k blocks of 64 and 32, 128-row group tiles), against the oracle:
one row, one row either side of a tile, column counts that leave a partial
last tile (64 of the 128 columns of a large down tile: every other tile width
divides the widths that the layer takes), both tile sizes of the dispatch and
the dot kernels.  The tolerances are the fp32 and bf16 layer tolerances (a dot
product of K terms errs by at most K 2^-24 sum |x w|; running sums of 8 or 16
products and their carried rounding keep it far below)."""
import numpy as np
import pytest
import torch

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
    (96, 32, 4, 128, 256, 0),     # six expected rows: the last for bf16's dot kernels
    (97, 32, 4, 128, 256, 0),
    (31, 32, 4, 256, 512, 0),     # below two expected rows: the last for fp32's
    (32, 32, 4, 256, 512, 0),
    (700, 20, 2, 128, 256, 0),    # small tiles, two CTAs per SM
    (2500, 1, 1, 64, 512, 0),     # large tiles: 64 x 128
    (1999, 5, 4, 192, 320, 0),    # ragged groups, small tiles
    (4000, 5, 4, 192, 64, 0),     # large down tiles, the last of 64 columns
    (5200, 4, 1, 320, 64, 64),    # the same in the dense shared expert
    (2048, 1, 1, 1024, 640, 64),  # 32 k blocks
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


@pytest.mark.gpu
@pytest.mark.parametrize("T,inter", [(40, 64), (2500, 512)])
def test_rows_without_finite_sums_leave_the_others_alone(T, inter):
    # up weights of 1e38: rows of ones overflow to +inf (as above), rows of
    # 1e-3 do not; a NaN in a row makes its outputs NaN
    d = 64
    cfg, layer = _case("f32", T, 1, 1, d, inter, 0, seed=T)
    h = layer["hidden"].reshape(T, d)
    h[:] = np.float32(1e-3) * (1 + np.arange(T, dtype=np.float32)[:, None] / T)
    layer["w_gate_up"][:, :inter] = 1.0
    layer["w_gate_up"][:, inter:] = 1e38
    layer["w_down"][:] = 1e-3
    clean, _, status = G.GpuLayer(cfg, layer).forward(np.ones(T, np.int32))
    assert status == B.REFLEX_OK and np.all(np.isfinite(clean))
    big, nan = np.arange(0, T, 9), np.arange(4, T, 9)
    h[big] = 1.0
    h[nan, 7] = np.nan
    out, _, status = G.GpuLayer(cfg, layer).forward(np.ones(T, np.int32))
    assert status == B.REFLEX_OK
    assert np.all(np.isposinf(out[big])) and np.all(np.isnan(out[nan]))
    rest = np.setdiff1d(np.arange(T), np.concatenate([big, nan]))
    assert np.array_equal(out[rest].view(np.uint32), clean[rest].view(np.uint32))


@pytest.mark.gpu
@pytest.mark.parametrize("where", ["rows", "weights"])
def test_values_without_finite_sums_cost_little(where):
    # 14 times the layer's time for a NaN in every row and 6.5 times for an
    # infinity in a gate row of every expert (all outputs NaN or infinite)
    # where single threads summed the outputs again; 1.1 and 3.8 with warps
    T, E, d, inter = 1024, 16, 1024, 512
    cfg, layer = _case("f32", T, E, 2, d, inter, 0, seed=3)
    gl = G.GpuLayer(cfg, layer)
    k = torch.full((T,), 2, dtype=torch.int32, device="cuda")
    out = torch.empty_like(gl.dev["hidden"])

    def us():
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        best = 1e9
        for _ in range(4):
            a.record()
            for _ in range(10):
                gl.moe.forward(gl.dev["hidden"], k, out)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 100)
        return best

    clean = us()
    if where == "rows":
        gl.dev["hidden"][:, 3] = float("nan")
    else:
        gl.moe.w["w_gate_up"][:, 7, 5] = float("inf")
    bad = us()
    assert gl.moe.status() == B.REFLEX_OK and not bool(torch.isfinite(out).any())
    assert bad <= (2.0 if where == "rows" else 5.0) * clean, (clean, bad)

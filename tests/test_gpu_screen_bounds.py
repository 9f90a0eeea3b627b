"""Screened routing where the score intervals say nothing: rows with an
infinity or a NaN, rows whose sum of squares leaves the fp32 range at either
end, router rows of the same kinds.  Ids, weights and the selected scores are
those of REFLEX_FLAG_EXACT_SCORES bit for bit, in the batched recheck (either
side of its two instantiations) and in the per-token recheck (above 256
experts)."""
import numpy as np
import pytest

import gpu_cases as G
from paper_2608_01784_gb300 import _binding as B
from paper_2608_01784_gb300 import api
from paper_2608_01784_gb300 import workloads as W


def _layer(T, E, d, kmax, seed):
    cfg = W.LayerConfig(name="screen", dtype="bf16", d=d, E=E, inter=128, shared_inter=0,
                        k_min=1, k_base=1, k_max=kmax, delta_role=0, delta_cur=0, w_cf=0.3,
                        n_seq=1, prompt_len=T, gen_len=0, block=32, weight_std=0.05,
                        conf="uniform", mask_rule="half")
    return cfg, W.make_layer(cfg, seed, T=T)


def _same_as_exact(cfg, layer, k):
    assert cfg.E > 256 or api.screens_in_batches(k.size, cfg.E, cfg.d, cfg.k_max)
    gl = G.GpuLayer(cfg, layer)
    flags = B.REFLEX_FLAG_RENORM_TOPK | B.REFLEX_STAGE_ROUTE
    _, s, st_s = gl.forward(k, flags=flags)
    _, e, st_e = gl.forward(k, flags=flags | B.REFLEX_FLAG_EXACT_SCORES)
    assert st_s == st_e == B.REFLEX_OK
    used = np.arange(cfg.k_max)[None, :] < k[:, None]
    assert np.all((e["ids"] >= 0) == used)
    assert np.array_equal(s["ids"], e["ids"])
    np.testing.assert_array_equal(s["alpha"], e["alpha"])  # NaN where the exact path has NaN
    rows, cols = np.nonzero(used)
    ids = e["ids"][rows, cols]
    np.testing.assert_array_equal(s["scores"][rows, ids], e["scores"][rows, ids])


# a token's row: what its first values, or all of them, are
TOKENS = {"overflow": lambda h: h * np.float32(1e19), "largest": lambda h: h * np.float32(1e38),
          "inf": lambda h: np.where(np.arange(h.size) == 5, np.float32(np.inf), h),
          "-inf": lambda h: np.where(np.arange(h.size) == h.size - 1, np.float32(-np.inf), h),
          "both": lambda h: np.where(np.arange(h.size) < 2, np.float32([np.inf, -np.inf] * (h.size // 2)), h),
          "nan": lambda h: np.where(np.arange(h.size) == 9, np.float32(np.nan), h),
          "zero": lambda h: h * 0, "tiny": lambda h: h * np.float32(2.0 ** -80)}


@pytest.mark.gpu
@pytest.mark.parametrize("T,E,d", [(1025, 256, 2048), (5000, 64, 1024), (2500, 65, 2048),
                                   (1800, 300, 256)])
@pytest.mark.parametrize("router", ["finite", "overflow", "largest", "inf", "nan"])
def test_rows_without_a_bound(T, E, d, router):
    kmax = 12
    cfg, layer = _layer(T, E, d, kmax, seed=T + E)
    h = W.bf16_bits_to_f32(layer["hidden"]).reshape(T, d)
    w = W.bf16_bits_to_f32(layer["w_router"]).reshape(E, d)
    with np.errstate(over="ignore", invalid="ignore"):
        for i, t in enumerate([0, 3, 7, 8, 31, 40, 100, T - 1]):
            h[t] = list(TOKENS.values())[i](h[t])
        if router != "finite":
            for e in (0, E // 2, E - 1):
                w[e] = TOKENS[router](w[e])
        layer["hidden"], layer["w_router"] = W.to_bf16_bits(h), W.to_bf16_bits(w)
    k = np.random.default_rng(T).integers(1, kmax + 1, T).astype(np.int32)
    k[:8] = kmax
    _same_as_exact(cfg, layer, k)


@pytest.mark.gpu
@pytest.mark.parametrize("T,E,d", [(1025, 256, 2048), (5000, 64, 1024), (1800, 300, 256)])
@pytest.mark.parametrize("eh,ew", [(-80, 0), (0, -80), (-70, -60), (-100, -22)])
def test_rows_whose_squares_underflow(T, E, d, eh, ew):
    # scores far below the products they are summed from, of rows scaled by
    # powers of two until their squares (and, last, the products) are subnormal
    rng = np.random.default_rng(T + E)
    kmax = 8
    cfg, layer = _layer(T, E, d, kmax, seed=T)
    x = W.bf16_bits_to_f32(W.to_bf16_bits(rng.standard_normal((T, d // 2))))
    y = W.bf16_bits_to_f32(W.to_bf16_bits(rng.standard_normal((E, d // 2))))
    eps = (1e-3 * rng.standard_normal((E, d // 2))).astype(np.float32)
    h, w = np.concatenate([x, x], 1), np.concatenate([y, eps - y], 1)
    layer["hidden"] = W.to_bf16_bits(h * np.float32(2.0 ** eh))
    layer["w_router"] = W.to_bf16_bits(w * np.float32(2.0 ** ew))
    _same_as_exact(cfg, layer, rng.integers(1, kmax + 1, T).astype(np.int32))

"""The batched router screen at the edges of its token blocks, against the
oracle's scores and selection (bit for bit): a block of one token, the last
token count of a single wave of CTAs and the first of the next, expert counts
either side of the two instantiations, and odd counts of candidates per token
(a duo without a second chain)."""
import numpy as np
import pytest

import gpu_cases as G
import oracle
from paper_2608_01784_gb300 import _binding as B
from paper_2608_01784_gb300 import api
from paper_2608_01784_gb300 import workloads as W


@pytest.mark.gpu
@pytest.mark.parametrize("T,E,d,kmax", [
    (2049, 256, 256, 12),
    (8100, 65, 128, 7),     # 65 experts, blocks of 56 tokens
    (2049, 256, 128, 12),   # blocks of 16 tokens
    (1217, 256, 1024, 12),  # blocks of 8 tokens: the first that are screened, d = 1024
    (9728, 128, 128, 4),    # one wave of 152 blocks of 64
    (9729, 200, 128, 12),   # two waves
    (9729, 64, 256, 12),    # 32-token blocks, the last of one token
    (9760, 33, 128, 1),
    (38552, 17, 128, 4),    # up to 32 experts: the first that are screened below d = 1024
])
def test_block_edges(T, E, d, kmax):
    assert api.screens_in_batches(T, E, d, kmax)
    cfg = W.LayerConfig(name="screen", dtype="bf16", d=d, E=E, inter=128, shared_inter=0,
                        k_min=1, k_base=1, k_max=kmax, delta_role=0, delta_cur=0, w_cf=0.3,
                        n_seq=1, prompt_len=T, gen_len=0, block=32, weight_std=0.05,
                        conf="uniform", mask_rule="half")
    layer = W.make_layer(cfg, T + E, T=T)
    k = np.random.default_rng(T).integers(1, kmax + 1, T).astype(np.int32)
    gl = G.GpuLayer(cfg, layer)
    _, rec, status = gl.forward(k, flags=B.REFLEX_FLAG_RENORM_TOPK | B.REFLEX_STAGE_ROUTE)
    assert status == B.REFLEX_OK
    z = oracle.router_logits(layer["hidden"], layer["w_router"])
    ids, alpha = oracle.select(z, k, kmax)
    assert np.array_equal(rec["ids"], ids)
    valid = ids >= 0
    np.testing.assert_allclose(rec["alpha"][valid], alpha[valid], rtol=G.ALPHA_RTOL, atol=1e-7)
    rows = np.nonzero(valid)[0]
    assert np.array_equal(rec["scores"][rows, ids[valid]].view(np.uint32),
                          z[rows, ids[valid]].view(np.uint32))

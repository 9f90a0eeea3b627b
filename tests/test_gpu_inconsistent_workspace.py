"""Expert stages on a workspace whose row offsets and tile prefixes hold
anything: the values are unspecified, but no access leaves the buffers.  The
workspace, the output and the token rows lie in one buffer with guard zones
between them, which the stages must leave as they are."""
import numpy as np
import pytest
import torch

import gpu_cases as G
from paper_2608_01784_gb300 import _binding as B
from paper_2608_01784_gb300 import workloads as W

GUARD = 1 << 20
EXTREMES = np.array([-2**31, -2**31 + 1, -2**24, -129, -1, 0, 1, 127, 128, 2**24, 2**30,
                     2**31 - 128, 2**31 - 1], np.int64)
RENORM = B.REFLEX_FLAG_RENORM_TOPK
SIMT = RENORM | B.REFLEX_FLAG_SIMT_EXPERTS


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,T,E,inter,flags", [
    ("f32", 40, 4, 128, RENORM),     # 16-row tiles
    ("f32", 2500, 2, 512, RENORM),   # 64-row tiles
    ("f32", 20, 40, 320, RENORM),    # warp-per-dot kernels
    ("bf16", 300, 4, 128, SIMT),
    ("bf16", 300, 4, 128, RENORM),   # 1-SM tiles
    ("bf16", 1100, 4, 128, RENORM),  # CTA-pair tiles
    ("bf16", 1100, 4, 128, RENORM | B.REFLEX_FLAG_GATHER_IN_GEMM),
    ("bf16", 600, 40, 128, RENORM),
])
def test_expert_stages_stay_in_their_buffers(dtype, T, E, inter, flags):
    d, kmax = 256, 2
    cfg = W.LayerConfig(name="ws", dtype=dtype, d=d, E=E, inter=inter, shared_inter=0,
                        k_min=1, k_base=1, k_max=kmax, delta_role=0, delta_cur=0, w_cf=0.3,
                        n_seq=1, prompt_len=T, gen_len=0, block=32, weight_std=0.05,
                        conf="uniform", mask_rule="half")
    gl = G.GpuLayer(cfg, W.make_layer(cfg, T, T=T))
    moe = gl.moe
    es = 4 if dtype == "f32" else 2
    sizes = [moe.ws_bytes, T * d * es]
    buf = torch.full((sum(sizes) + 3 * GUARD + 1024,), 0x5a, dtype=torch.uint8, device="cuda")
    at, views, guards = 0, [], []
    for n in sizes:
        guards.append(buf[at:at + GUARD])
        start = (at + GUARD + 255) // 256 * 256
        views.append(buf[start:start + n])
        at = start + n
    guards.append(buf[at:at + GUARD])
    moe.ws = views[0]
    out = views[1].view(moe.tdtype).view(T, d)
    k = torch.full((T,), kmax, dtype=torch.int32, device="cuda")
    moe.forward(gl.dev["hidden"], k, out, flags=flags)
    torch.cuda.synchronize()
    assert moe.status() == B.REFLEX_OK
    # offsets, then the two tile prefixes, up to the pair permutation
    words = moe._view(moe.rec.offsets, (moe.rec.perm - moe.rec.offsets) // 4)
    good = words.clone()
    rng = np.random.default_rng(T + E)
    for trial in range(40):
        bad = good.cpu().numpy().astype(np.int64)
        hit = rng.random(bad.size) < (1.0 if trial % 4 == 0 else rng.uniform(0.01, 0.5))
        bad[hit] = rng.choice(EXTREMES, int(hit.sum()))
        words.copy_(torch.from_numpy(bad.astype(np.int32)))
        moe.forward(gl.dev["hidden"], k, out, flags=flags | B.REFLEX_STAGE_EXPERT_UP |
                    B.REFLEX_STAGE_EXPERT_DOWN)
        torch.cuda.synchronize()
    for g in guards:
        assert bool((g == 0x5a).all())
    # and a consistent workspace again
    moe.forward(gl.dev["hidden"], k, out, flags=flags)
    torch.cuda.synchronize()
    assert moe.status() == B.REFLEX_OK

"""The network kernel where its three warpgroups per CTA have uneven numbers of 128-row tiles
(none, one, several), against the BF16 restatement and its 2e-3 bar (only the FP32 sums and rare
rounding flips differ)."""
import numpy as np
import pytest

from gpu_common import need_gpu
from test_gpu_learned import bf16_net, bf16_round

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 129, 385, 60001, 120000])
def test_mlp_tiles(rows):
    torch, cb = need_gpu()
    rng = np.random.default_rng(rows)
    p = (rng.standard_normal(5127) * 0.25).astype(np.float32)
    feat = rng.standard_normal((rows, 7)).astype(np.float32)
    gout = rng.standard_normal((rows, 7)).astype(np.float32)
    emu, gemu = bf16_net(feat.astype(np.float64), bf16_round(p), gout.astype(np.float64))
    out = cb.mlp_forward(torch.from_numpy(feat).cuda(), p).cpu().numpy()
    grad = cb.mlp_backward(torch.from_numpy(feat).cuda(), p, torch.from_numpy(gout).cuda())
    assert np.linalg.norm(out - emu) <= 2e-3 * np.linalg.norm(emu)
    assert np.linalg.norm(grad - gemu) <= 2e-3 * np.linalg.norm(gemu)
    # every parameter block, so that a small one cannot hide behind a large one
    for a, b in ((0, 448), (448, 512), (512, 4608), (4608, 4672), (4672, 5120), (5120, 5127)):
        assert np.linalg.norm(grad[a:b] - gemu[a:b]) <= 1e-2 * np.linalg.norm(gemu[a:b]), (a, b)

"""The multi-vector product on a basis, and in a workspace, between 16-byte boundaries: the same
bits as from one (the same products in the same order; the bulk copies give way to loads of
single codes)."""
import numpy as np
import pytest

from gpu_common import FORMATS, need_gpu

pytestmark = pytest.mark.gpu

BYTES = {"f64": 8, "f32": 4, "i32": 4, "f16": 2, "bf16": 2, "i16": 2, "e4m3": 1}


@pytest.mark.parametrize("fmt", FORMATS)
@pytest.mark.parametrize("n,ncols,k", [(4096, 1, 1), (5000, 17, 3), (70001, 33, 8), (300001, 130, 5)])
def test_any_code_alignment(fmt, n, ncols, k):
    torch, cb = need_gpu()
    ld = (n + 4095) // 4096 * 4096
    g = torch.Generator(device="cuda")
    g.manual_seed(n + k)
    v = torch.rand(ncols, ld, dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    v[:, n:] = 0.0
    V = torch.stack([cb.encode(fmt, c, 1.0)[0] for c in v]).contiguous()
    flat = V.view(torch.uint8).reshape(-1)
    W = torch.randn(k, n, dtype=torch.float64, device="cuda", generator=g)
    scales = torch.rand(ncols, dtype=torch.float64, device="cuda", generator=g)
    need = cb.lib().cbg_basis_dot_multi_workspace(ld, ncols, k)
    want = cb.basis_dot_multi(fmt, n, V, ld, scales, W, path="cuda")
    room = torch.empty(flat.numel() + 16, dtype=torch.uint8, device="cuda")
    work = torch.empty(need + 16, dtype=torch.uint8, device="cuda")
    assert room.data_ptr() % 16 == 0 and work.data_ptr() % 16 == 0
    bs = BYTES[fmt]
    for off in sorted({bs % 16, 8, 16 - bs}):
        U = room[off: off + flat.numel()]
        U.copy_(flat)
        got = cb.basis_dot_multi(fmt, n, U.reshape(ncols, -1), ld, scales, W, path="cuda", workspace=work[off: off + need])
        assert torch.equal(got, want), (fmt, off)
    if fmt == "f16" and ncols <= 128:                  # the tensor path needs the boundary: auto does without it
        assert torch.equal(cb.basis_dot_multi(fmt, n, U.reshape(ncols, -1), ld, scales, W), want)
        with pytest.raises(cb.CbgError) as e:
            cb.basis_dot_multi(fmt, n, U.reshape(ncols, -1), ld, scales, W, path="tensor")
        assert e.value.status == -6

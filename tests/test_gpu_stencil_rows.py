"""fsl_mlp_stencils writes its BF16 rows to any address of a BF16 value: rows at
byte offsets 2, 4 and 6 of an 8-byte boundary equal the aligned ones, and nothing
before or after them is touched; an odd address is refused."""
import ctypes

import numpy as np
import pytest


def _call(F, t, n, x, target, sub=4):
    p = lambda a: ctypes.c_void_p(a)
    return F.lib().fsl_mlp_stencils(n, *[p(t[k].data_ptr()) for k in ("axes", "quat", "dir", "delta", "invert")], sub, 1e-3, 9,
                                    p(x), p(target), None)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 5, 33, 20000])
@pytest.mark.parametrize("off", [1, 2, 3, 4, 5])
def test_rows_at_every_bf16_address(n, off):
    import torch
    from paper_1509_07691_gb300 import fsl as F
    from paper_1509_07691_gb300 import synthetic as S
    q = S.mlp_sample_params(17, n)
    t = {k: torch.from_numpy(np.ascontiguousarray(q[k], np.int32 if k == "invert" else np.float32)).cuda()
         for k in ("axes", "quat", "dir", "delta", "invert")}
    want, target = F.mlp_stencils(q, sub=4, noise=1e-3, noise_seed=9)
    buf = torch.full((off + 128 * n + 64,), 7.0, dtype=torch.bfloat16, device="cuda")
    tgt = torch.empty(n, dtype=torch.float32, device="cuda")
    assert _call(F, t, n, buf.data_ptr() + 2 * off, tgt.data_ptr()) == F.OK
    torch.cuda.synchronize()
    assert torch.equal(buf[off: off + 128 * n].view(n, 128), want)
    assert torch.all(buf[:off] == 7) and torch.all(buf[off + 128 * n:] == 7)
    assert torch.equal(tgt, target)


def test_odd_address_is_refused():
    from paper_1509_07691_gb300 import build
    build.build()
    from paper_1509_07691_gb300 import fsl as F
    fake = ctypes.c_void_p(1 << 20)  # never dereferenced
    args = (1, fake, fake, fake, fake, fake, 4, 0.0, 0)
    assert F.lib().fsl_mlp_stencils(*args, ctypes.c_void_p((1 << 20) + 1), fake, None) == F.EINVAL
    assert F.lib().fsl_mlp_stencils(0, *args[1:], ctypes.c_void_p((1 << 20) + 2), fake, None) == F.OK

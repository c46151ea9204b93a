"""Fill levels by sub-sampling at the edges of the kernel's decisions: every
shape, inside and outside, sample counts per axis around the 4^3 blocks, odd
grids; the counts equal the oracle's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = {
    "sphere": dict(c=(11.3, 9.8, 10.1), R=6.4),
    "small": dict(kind="sphere", c=(11.3, 9.8, 10.1), R=0.4),
    "mode2": dict(c=(11.0, 9.5, 10.25), R=5.5, eps2=0.3),
    "mode2_core": dict(kind="mode2", c=(11.0, 9.5, 10.0), R=1.6, eps2=-0.4),
    "cap": dict(c=(11.3, 9.8, 0.5), R=7.2, zw=0.5),
    "cap_fine": dict(kind="cap", c=(11.3, 9.8, 3.0), R=7.2, zw=3.03125),
    "two_spheres": dict(c=(7.2, 9.8, 10.1), R=4.4, c2=(14.9, 9.1, 10.3), R2=3.7),
    "pool": dict(h0=9.6, amp=2.0, wavelength=9.0),
    "plane": dict(n=(0.3, -0.5, 0.7), d=4.2),
}


@pytest.mark.parametrize("sub", [1, 3, 4, 5, 16, 17])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_fill_levels_of_every_shape(orc, name, sub):
    import torch
    from paper_1509_07691_gb300 import fsl as F
    kw = dict(SHAPES[name])
    kind = kw.pop("kind", name)
    for shape, invert in (((21, 20, 23), 0), ((19, 18, 131), 1)):
        ref = orc.fill(orc.geom(kind, sub=sub, invert=invert, **kw), shape)
        phi = torch.full(shape, -1.0, device="cuda")
        F.fill_geometry(F.make_params(shape), F.make_geometry(kind, sub=sub, invert=invert, **kw), phi)
        assert np.array_equal(phi.cpu().numpy(), ref.astype(np.float32))

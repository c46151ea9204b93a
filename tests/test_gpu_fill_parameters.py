"""Fill levels at parameters off the ordinary range: negative radii (whole cells are
decided by the radius as it is, the samples of the others by its square), mode-2
amplitudes of either sign (every cell as the sampling has it), half-spaces whose
normal is far from unit length.  Counts equal the oracle's sampling."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPE = (27, 26, 29)
C, C2 = (13.3, 12.8, 14.1), (16.2, 13.1, 12.9)


def _fill(kind, sub, invert, **kw):
    import torch
    from paper_1509_07691_gb300 import fsl as F
    phi = torch.full(SHAPE, -1.0, device="cuda")
    F.fill_geometry(F.make_params(SHAPE), F.make_geometry(kind, sub=sub, invert=invert, **kw), phi)
    return phi.cpu().numpy()


def _sampled(orc, kind, sub, invert, **kw):
    return np.asarray(orc.fill(orc.geom(kind, sub=sub, invert=invert, **kw), SHAPE)).astype(np.float32)


def _whole(kind, invert, c=C, R=0.0, eps2=0.0, c2=(0, 0, 0), R2=0.0, zw=0.0):
    """1 inside, -1 outside, 0 sampled, by the distance of a cell's centre."""
    z, y, x = np.meshgrid(*[np.arange(n, dtype=np.float64) for n in SHAPE], indexing="ij")
    d = lambda p: np.sqrt((x - p[0]) ** 2 + (y - p[1]) ** 2 + (z - p[2]) ** 2)
    r, q, e = d(c), d(c2), abs(eps2)
    lo, hi = (R * (1 - 0.5 * e), R * (1 + e)) if kind == "mode2" else (R, R)
    into, out = r + 1 < lo, r - 1 > hi
    if kind == "cap":
        into, out = into & (z - 1 > zw), out | (z + 1 < zw)
    if kind == "two_spheres":
        into, out = into | (q + 1 < R2), out & (q - 1 > R2)
    w = np.where(into, 1, np.where(out, -1, 0))
    return -w if invert else w


NEGATIVE = {
    "sphere_below_one": ("sphere", dict(c=C, R=-0.4)), "sphere_near_one": ("sphere", dict(c=C, R=-0.95)),
    "sphere": ("sphere", dict(c=C, R=-5.0)), "mode2": ("mode2", dict(c=C, R=-2.3, eps2=0.4)),
    "mode2_wide": ("mode2", dict(c=C, R=-1.2, eps2=-3.0)), "cap": ("cap", dict(c=C, R=-0.7, zw=14.0)),
    "two_first": ("two_spheres", dict(c=C, R=-6.0, c2=C2, R2=5.0)),
    "two_second": ("two_spheres", dict(c=C, R=6.0, c2=C2, R2=-4.5)),
    "two_both": ("two_spheres", dict(c=C, R=-0.6, c2=C2, R2=-0.8)),
}


@pytest.mark.parametrize("sub", [1, 4, 9])
@pytest.mark.parametrize("invert", [0, 1])
@pytest.mark.parametrize("name", sorted(NEGATIVE))
def test_negative_radii(orc, name, invert, sub):
    kind, kw = NEGATIVE[name]
    w = _whole(kind, invert, **kw)
    want = np.where(w > 0, np.float32(1), np.where(w < 0, np.float32(0), _sampled(orc, kind, sub, invert, **kw)))
    assert np.array_equal(_fill(kind, sub, invert, **kw), want)


@pytest.mark.parametrize("sub", [1, 5, 16])
@pytest.mark.parametrize("invert", [0, 1])
@pytest.mark.parametrize("scale", [1e-320, 1e-300, 1e-160, 7e-44, 3e-42, 1e-39, 1e-30, 1.0, 1e30, 1e160, 1e300, 0.0])
def test_half_space_normals_of_any_length(orc, scale, invert, sub):
    n = tuple(scale * v for v in (0.31, -0.52, 0.73))
    kw = dict(n=n, d=scale * 7.4)
    assert np.array_equal(_fill("plane", sub, invert, **kw), _sampled(orc, "plane", sub, invert, **kw))


SHAPES = {
    "sphere": dict(c=C, R=7.3), "mode2": dict(c=C, R=5.5, eps2=0.3), "cap": dict(c=C, R=8.1, zw=14.0),
    "two_spheres": dict(c=C, R=4.4, c2=C2, R2=5.2), "pool": dict(h0=13.6, amp=3.0, wavelength=1.7),
    "plane": dict(n=(0.31, -0.52, 0.73), d=7.4),
}


@pytest.mark.parametrize("invert", [0, 1])
@pytest.mark.parametrize("sub", [1, 2, 3])
@pytest.mark.parametrize("kind", sorted(SHAPES))
def test_few_samples(orc, kind, sub, invert):
    """A thread per cell up to 2^3 samples, a warp per open cell from 3^3 on."""
    assert np.array_equal(_fill(kind, sub, invert, **SHAPES[kind]), _sampled(orc, kind, sub, invert, **SHAPES[kind]))


@pytest.mark.parametrize("sub", [1, 4])
def test_pool_without_a_wavelength(sub):
    """No sample is inside (the phase is no number), whole cells below the crests are."""
    z = np.broadcast_to(np.arange(SHAPE[0], dtype=np.float64)[:, None, None], SHAPE)
    want = (z + 1 < 13.6 - 2.0).astype(np.float32)
    assert np.array_equal(_fill("pool", sub, 0, h0=13.6, amp=2.0, wavelength=0.0), want)


def test_one_sample_costs_less_than_many():
    """Cells of one sample are not taken by a warp each: 0.03 of the time of 6^3 samples
    on a pool of short waves, with a warp per cell 0.7 (256 x 256 x 24)."""
    import torch
    from paper_1509_07691_gb300 import fsl as F
    shape = (24, 256, 256)
    phi = torch.empty(shape, device="cuda")

    def ms(sub):
        g, P = F.make_geometry("pool", h0=12.3, amp=6.0, wavelength=1.7, sub=sub), F.make_params(shape)
        v = []
        for _ in range(6):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            for _ in range(5):
                F.fill_geometry(P, g, phi)
            e[1].record()
            torch.cuda.synchronize()
            v.append(e[0].elapsed_time(e[1]))
        return min(v)

    a, b = ms(1), ms(6)
    assert a < 0.6 * b, (a, b)

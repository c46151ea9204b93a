"""Training stencils whose quaternions are not of unit length (the matrix of the
formula is taken as it is) and whose semi-axes are negative (only their squares
enter): the rows hold the fill levels of the oracle's sampling of every point.
The values of a row are compared in ascending order: which of two axes comes first
is open where the normal's components tie, and at 6^3 samples several do.

Tolerance of a value: one sub-sample (the FP32 sample test against FP64) plus one
BF16 step."""
import numpy as np
import pytest

from paper_1509_07691_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [0.3, 0.9, 1.15, 1.3, 2.0, 4.0])
def test_quaternions_of_any_length(scale):
    _check(dict(S.mlp_sample_params(41, 200)), quat=scale)


@pytest.mark.parametrize("signs", [(1, -1, 1), (-1, -1, -1)])
def test_negative_semi_axes(signs):
    _check(dict(S.mlp_sample_params(42, 200)), axes=np.array(signs, np.float32))


@pytest.mark.parametrize("sub", [7, 8, 13, 32])
@pytest.mark.parametrize("n", [1, 3, 760, 761])
def test_small_sets_equal_the_same_rows_of_a_large_one(n, sub):
    """A block per stencil and a warp per stencil give the same rows and targets."""
    import torch
    from paper_1509_07691_gb300 import fsl as F
    p = S.mlp_sample_params(43, 1200)
    X, t = F.mlp_stencils(p, sub=sub, noise=1e-3, noise_seed=4)
    Xs, ts = F.mlp_stencils({k: v[:n] for k, v in p.items()}, sub=sub, noise=1e-3, noise_seed=4)
    assert torch.equal(X[:n], Xs) and torch.equal(t[:n], ts)


def test_a_few_fine_stencils_are_not_left_to_single_warps():
    """100 stencils at 32^3 samples against 1520, which fill the GPU a warp each: 0.26 of
    their time with a block per stencil, 0.7 with a warp per stencil."""
    import torch
    from paper_1509_07691_gb300 import fsl as F

    def us(n):
        p = S.mlp_sample_params(44, n)
        F.mlp_stencils(p, sub=32)
        v = []
        for _ in range(5):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            F.mlp_stencils(p, sub=32)
            e[1].record()
            torch.cuda.synchronize()
            v.append(e[0].elapsed_time(e[1]))
        return min(v)

    assert us(100) < 0.5 * us(1520)


def _check(p, quat=1.0, axes=1.0):
    import oracle.mlp as M
    from paper_1509_07691_gb300 import fsl as F
    p["quat"] = np.asarray(p["quat"], np.float32) * np.float32(quat)
    p["axes"] = np.asarray(p["axes"], np.float32) * axes
    n, sub = p["quat"].shape[0], 6
    X, _ = F.mlp_stencils(p, sub=sub, noise=0.0)
    X = X.float().cpu().numpy().astype(np.float64)
    bad = 0
    for k in range(n):
        C = M.shape_centre(p["axes"][k], p["quat"][k].astype(np.float64), p["dir"][k], p["delta"][k])
        s = M.stencil_fill(p["axes"][k], p["quat"][k].astype(np.float64), C, int(p["invert"][k]), sub)
        bad += np.max(np.abs(np.sort(X[k, :125]) - np.sort(M.bf16(2.0 * s.reshape(-1) - 1.0)))) > 2.0 / sub ** 3 + 2 ** -7
    assert bad == 0

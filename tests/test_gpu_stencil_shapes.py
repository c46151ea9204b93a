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

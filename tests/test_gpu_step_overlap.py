"""Kernels of a step that are dispatched before their predecessor has drained: the
interface list's blocks spread over the GPU behind the learned curvature's network."""
import time

import pytest

pytestmark = pytest.mark.gpu


def test_interface_pass_spreads_behind_the_network():
    """Ten steps with the learned curvature against ten without curvature, a bubble in
    48^3: 1.5 times; 1.77 with the interface pass's blocks on the first SMs to drain."""
    import numpy as np
    import torch
    from paper_1509_07691_gb300 import fsl as F
    from paper_1509_07691_gb300 import synthetic as S
    net = F.Mlp({k: np.asarray(v, np.float64) for k, v in S.mlp_init_weights(3).items()})
    n = 48
    ms = {}
    for model in (F.CURV_NONE, F.CURV_MLP):
        P = F.make_params((n, n, n), tau=0.7, sigma=5e-4, curv_model=model)
        phi = torch.empty((n, n, n), device="cuda")
        F.fill_geometry(P, F.make_geometry("sphere", c=(n / 2 + .3, n / 2 - .2, n / 2 + .1), R=n * 0.2, invert=1, sub=8), phi)
        sim = F.Sim(P, phi0=phi)
        if model == F.CURV_MLP:
            sim.attach_mlp(net)
        sim.prescribe_flow(1.0, (0.03, 0.015, -0.02))
        sim.step(60)
        v = []
        for _ in range(15):
            torch.cuda.synchronize()
            t = time.perf_counter()
            sim.step(10)
            torch.cuda.synchronize()
            v.append(time.perf_counter() - t)
        ms[model] = sorted(v)[len(v) // 2]
        assert sim.status() == 0
        sim.close()
    assert ms[F.CURV_MLP] < 1.68 * ms[F.CURV_NONE], ms

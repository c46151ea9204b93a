"""Initial PDFs of both buffers on grids whose directions start at every 16-byte
phase, and steps in pairs against single steps."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("shape", [(3, 3, 3), (5, 7, 9), (6, 8, 11), (16, 16, 16)])
def test_initial_pdfs_fill_both_buffers(shape, storage):
    import torch
    from paper_1509_07691_gb300 import fsl as F
    phi = torch.zeros(shape, device="cuda")
    phi[1, 1, 1] = 0.5
    sim = F.Sim(F.make_params(shape, storage=storage), phi0=phi)
    w = torch.tensor([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, dtype=torch.float32, device="cuda").view(19, 1, 1, 1)
    for f in sim.f:
        want = w.expand_as(f) if storage == F.F32 else torch.zeros_like(f)
        assert torch.equal(f, want.to(f.dtype))
    assert sim.stats()[1] == 1
    sim.close()


@pytest.mark.parametrize("calls", [(1, 1, 1, 1, 1), (5,), (2, 3), (1, 4), (3, 2)])
def test_steps_in_pairs_equal_single_steps(calls):
    import torch
    from paper_1509_07691_gb300 import fsl as F
    shape, out = (24, 22, 26), []
    phi = torch.zeros(shape, device="cuda")
    P = F.make_params(shape, sigma=1e-3, tau=0.7)
    F.fill_geometry(P, F.make_geometry("sphere", c=(12.3, 11.1, 12.4), R=6.5, sub=8), phi)
    for seq in ((1,) * 5, calls):
        sim = F.Sim(P, phi0=phi)
        sim.prescribe_flow(1.0, (0.05, 0.02, -0.03))
        for n in seq:
            sim.step(n)
        out.append((sim.parity, sim.f_current().clone(), sim.flags_current().clone(), sim.mass.clone(), sim.phi.clone()))
        assert sim.status() == 0
        sim.close()
    assert out[0][0] == out[1][0] == 1
    for a, b in zip(out[0][1:], out[1][1:]):
        assert torch.equal(a, b)

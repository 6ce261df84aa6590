"""Fused against separate PM passes at the meshes whose fused deposit or line
passes have compile-time forms of their own, with ragged particle counts per tile."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1509_04685_gb300 as C  # noqa: E402


def _force(nq, ng, path=0, tile=0):
    L = 100.0
    sim = C.Simulation(C.make_config(nq, ng, L, 0.05, 1.0, 40))
    sim.init_tables()
    g = torch.Generator(device="cuda").manual_seed(ng + nq)
    sim.d.copy_(torch.randn(sim.d.shape, generator=g, device="cuda") * 4.0)
    assert C.LIB.cola_pm_set_path(path) == 0
    C.cola_fft_set_tile(ng, tile)
    try:
        f = sim.force(1.0).double()
    finally:
        C.LIB.cola_pm_set_path(0)
        C.cola_fft_set_tile(ng, 0)
    assert sim.status() == 0
    return f


@pytest.mark.parametrize("nq,ng", [(64, 64), (40, 96), (128, 128), (108, 160), (64, 192), (160, 256), (128, 384)])
def test_fused_force_equals_separate(nq, ng):
    a, b = _force(nq, ng, path=1), _force(nq, ng, path=2)
    # each path is within 1e-5 of the oracle in the parity tests
    assert float((a - b).norm() / b.norm()) < 2e-5


@pytest.mark.parametrize("nq,ng", [(64, 512), (128, 1024)])
def test_force_at_the_estimator_meshes(nq, ng):
    # the same transforms by the runtime line passes (four columns per tile)
    a, b = _force(nq, ng), _force(nq, ng, tile=4)
    assert float((a - b).norm() / b.norm()) < 2e-5

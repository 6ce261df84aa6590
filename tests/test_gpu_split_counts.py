"""The fused deposit's split 32-bit counters around their limit of 4095 particles
per tile: a crowd on one point just below, at and above it, the other particles
spread out.  An overflowing counter would change the crowd's mass grossly, which
the force on the others shows; both PM paths (the separate one adds 64-bit
counts in global memory) must give it alike."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1509_04685_gb300 as C  # noqa: E402


@pytest.mark.parametrize("crowd", [2000, 4090, 4095, 4096, 12000])
def test_force_of_a_crowded_cell(crowd):
    nq, ng, L = 32, 768, 64.0
    sim = C.Simulation(C.make_config(nq, ng, L, 0.05, 1.0, 40))
    sim.init_tables()
    i = torch.arange(nq, device="cuda", dtype=torch.float32) * (L / nq)
    q = torch.stack(torch.meshgrid(i, i, i, indexing="ij")).reshape(3, -1)
    g = torch.Generator(device="cuda").manual_seed(crowd)
    sim.d.copy_(torch.randn(q.shape, generator=g, device="cuda"))
    sim.d[:, :crowd] = 20.3 - q[:, :crowd]
    force = []
    for path in (1, 2):
        assert C.LIB.cola_pm_set_path(path) == 0
        try:
            force.append(sim.force(1.0)[:, crowd:].double())
        finally:
            C.LIB.cola_pm_set_path(0)
        assert sim.status() == 0
    # each path is within 1e-5 of the oracle in the parity tests
    assert float((force[0] - force[1]).norm() / force[1].norm()) < 2e-5

"""The fused deposit's split 32-bit counters with a crowd exactly on a cell corner,
where every particle's whole weight 2^40 falls on one cell: the upper counter,
2^20 per particle, wraps to zero at 4096 particles, so a limit on the split form
above 4095 would lose the crowd's mass.  Crowds at, just above and up to three
times the limit, in the warp-row pass (768) and the block-tile passes (64, 1152);
the separate path, which adds 64-bit counts in global memory, is the reference."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1509_04685_gb300 as C  # noqa: E402

# corner coordinate x with x ng / L + 1/2 a whole number (nq = 32, L = 64)
CORNER = {64: 20.5, 768: 20.375, 1152: 20.25}


@pytest.mark.parametrize("ng", sorted(CORNER))
@pytest.mark.parametrize("crowd", [4095, 4096, 5000, 8191, 8192, 12288])
def test_force_of_a_crowd_on_a_cell_corner(ng, crowd):
    nq, L = 32, 64.0
    sim = C.Simulation(C.make_config(nq, ng, L, 0.05, 1.0, 40))
    sim.init_tables()
    i = torch.arange(nq, device="cuda", dtype=torch.float32) * (L / nq)
    q = torch.stack(torch.meshgrid(i, i, i, indexing="ij")).reshape(3, -1)
    g = torch.Generator(device="cuda").manual_seed(crowd)
    sim.d.copy_(torch.randn(q.shape, generator=g, device="cuda"))
    sim.d[:, :crowd] = CORNER[ng] - q[:, :crowd]  # exact in FP32
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

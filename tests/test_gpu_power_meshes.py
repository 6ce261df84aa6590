"""Transforms and shell sums at the estimator meshes with passes of their own
(512, 1024) and at meshes smaller than one block's share of modes, against
64-bit torch on the GPU."""
import math

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1509_04685_gb300 as C  # noqa: E402


@pytest.mark.parametrize("n", [512, 1024])
def test_fft3d_of_the_estimator_meshes(n):
    P = C.cola_fft_pitch(n)
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn((n, n, n), generator=g, device="cuda")
    buf = torch.zeros((n, n, 2 * P), device="cuda")
    buf[:, :, :n] = x
    ws = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
    C.cola_fft3d_r2c(n, buf, ws)
    ref = torch.view_as_real(torch.fft.rfftn(x.double()))
    got = buf.view(n, n, P, 2)[:, :, : n // 2 + 1]
    num = sum(float((got[i].double() - ref[i]).square().sum()) for i in range(n))
    assert math.sqrt(num / float(ref.square().sum())) < 1e-6  # the FFT parity tolerance
    del ref
    C.cola_fft3d_c2r(n, buf, ws)
    back = buf[:, :, :n] / n**3
    assert float((back - x).double().norm() / x.double().norm()) < 1e-6


@pytest.mark.parametrize("nq,ng", [(8, 4), (16, 6), (16, 30), (64, 512), (64, 1024)])
def test_shell_sums_of_the_density(nq, ng):
    L = 100.0
    sim = C.Simulation(C.make_config(nq, ng, L, 0.05, 1.0, 40))
    sim.init_tables()
    g = torch.Generator(device="cuda").manual_seed(3)
    sim.d.copy_(torch.randn(sim.d.shape, generator=g, device="cuda") * 3.0)
    k, p0, p2, p4, n = sim.multipoles(ng, a_out=0.05, node=0)  # v = psi = 0: real space
    k1, p, n1 = sim.power(ng, a_out=0.05, node=0)
    assert sim.status() == 0
    dk = torch.fft.rfftn(sim.density().double())
    i = torch.fft.fftfreq(ng, 1.0 / ng, device="cuda", dtype=torch.float64)
    kz = torch.arange(ng // 2 + 1, device="cuda", dtype=torch.float64)
    w = torch.where((kz == 0) | (kz == ng // 2), 1.0, 2.0)
    s = torch.zeros(4, ng, dtype=torch.float64, device="cuda")
    for x in range(ng):
        n2 = i[x] ** 2 + i[:, None] ** 2 + kz[None, :] ** 2
        b = torch.floor(n2.sqrt() + 0.5).long()
        pw = dk[x].abs() ** 2 * (L**3 / float(ng) ** 6)
        mu2 = kz**2 / n2.clamp(min=1.0)
        for q, v in enumerate((torch.ones_like(n2), n2.sqrt(), pw, pw * (1.5 * mu2 - 0.5))):
            s[q].scatter_add_(0, b.reshape(-1), (v * w).reshape(-1))
    s = s[:, 1: ng // 2 + 1]
    assert torch.equal(n, s[0]) and torch.equal(n1, s[0])
    for kk, pp in ((k, p0), (k1, p)):
        torch.testing.assert_close(kk, s[1] / s[0] * (2 * math.pi / L), rtol=2e-6, atol=0.0)
        torch.testing.assert_close(pp, s[2] / s[0], rtol=2e-5, atol=0.0)  # the P(k) parity tolerance
    torch.testing.assert_close(p2, 5 * s[3] / s[0], rtol=0.0, atol=1e-4 * float((s[2] / s[0]).max()))


@pytest.mark.parametrize("ng", [768, 1024, 1152, 1536])
def test_power_of_blocked_rows(ng):
    # the blocked estimator mesh and its x pass against the plain mesh (four columns per tile)
    nq, L = 64, 100.0
    sim = C.Simulation(C.make_config(nq, ng, L, 0.05, 1.0, 40))
    sim.init_tables()
    g = torch.Generator(device="cuda").manual_seed(ng)
    sim.d.copy_(torch.randn(sim.d.shape, generator=g, device="cuda") * 3.0)
    k, p, n = sim.power(ng, a_out=0.05, node=0)
    C.cola_fft_set_tile(ng, 4)
    try:
        k4, p4, n4 = sim.power(ng, a_out=0.05, node=0)
    finally:
        C.cola_fft_set_tile(ng, 0)
    assert sim.status() == 0
    assert torch.equal(n, n4)
    torch.testing.assert_close(k, k4, rtol=2e-6, atol=0.0)
    torch.testing.assert_close(p, p4, rtol=2e-5, atol=0.0)  # the P(k) parity tolerance

"""P(k) while another thread changes the column width of the same mesh: the width
is a matter of speed, so a call that has laid its mesh out for one width is
neither refused nor wrong when it changes in between."""
import threading

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1509_04685_gb300 as C  # noqa: E402


def test_power_while_the_column_width_changes():
    nq, ng, L = 32, 768, 100.0
    sim = C.Simulation(C.make_config(nq, ng, L, 0.05, 1.0, 40))
    sim.init_tables()
    g = torch.Generator(device="cuda").manual_seed(5)
    sim.d.copy_(torch.randn(sim.d.shape, generator=g, device="cuda") * 3.0)
    want = [t.clone() for t in sim.power(ng, a_out=0.05, node=0)]
    stop = threading.Event()

    def toggle():
        while not stop.is_set():
            for width in (4, 0):
                C.cola_fft_set_tile(ng, width)

    t = threading.Thread(target=toggle)
    t.start()
    try:
        got = [[t.clone() for t in sim.power(ng, a_out=0.05, node=0)] for _ in range(200)]
    finally:
        stop.set()
        t.join()
        C.cola_fft_set_tile(ng, 0)
    assert sim.status() == 0
    for k, p, n in got:
        assert torch.equal(n, want[2])
        torch.testing.assert_close(k, want[0], rtol=2e-6, atol=0.0)
        torch.testing.assert_close(p, want[1], rtol=2e-5, atol=0.0)  # the P(k) parity tolerance

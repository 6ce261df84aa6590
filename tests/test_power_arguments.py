"""P(k) and multipoles refuse an output time that is not finite: the number of
integration steps to it has no value (no GPU needed: nothing is launched)."""
import ctypes

import pytest


@pytest.mark.parametrize("a_out", [float("inf"), -float("inf"), 0.0, -0.5])
def test_output_time_has_to_be_positive_and_finite(a_out):
    import paper_1509_04685_gb300 as C
    L = C.LIB
    cfg = C.make_config(8, 24, 32.0, 0.05)
    size = C.cola_workspace_size(cfg)
    fake = 1 << 40  # never dereferenced
    st = C.cola_state(fake, fake, fake, fake)
    n = C.cola_launch_count()
    assert L.cola_power_spectrum(ctypes.byref(cfg), ctypes.byref(st), 0, a_out, 24, 0, fake, fake, fake, 12, fake,
                                 size, None) == -1
    assert L.cola_power_multipoles(ctypes.byref(cfg), ctypes.byref(st), 0, a_out, 24, 0, fake, fake, fake, fake, fake,
                                   12, fake, size, None) == -1
    assert C.cola_launch_count() == n

"""Power-law time sampling whose first node underflows to a = 0 is refused: ln a, and
with it the number of integration steps, is infinite there (no GPU needed)."""
import pytest


@pytest.mark.parametrize("a_init,p,ok", [(0.05, 0.5, True), (0.05, 4.0, True), (0.05, 200.0, True),
                                         (0.05, 246.0, True), (0.05, 250.0, False), (0.05, 400.0, False), (1e-300, 1.0, True),
                                         (1e-300, 2.0, False), (0.05, 1e-300, True)])
def test_first_node_has_to_be_a_number_above_zero(a_init, p, ok):
    import paper_1509_04685_gb300 as C
    cfg = C.make_config(8, 24, 32.0, a_init, sampling=C.SAMPLING_POW, sampling_p=p)
    if ok:
        assert C.cola_workspace_size(cfg) > 0
    else:
        with pytest.raises(C.ColaError) as e:
            C.cola_workspace_size(cfg)
        assert e.value.code == -1

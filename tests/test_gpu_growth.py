"""The FP64 time tables against the oracle where their maps are cut: node counts
around the tiles of the row kernel (64 maps, 256 rows), a run that ends before
a = 1 (a last span to the normalisation) and a start close to the ODEs' own."""
import numpy as np
import pytest

from oracle import cosmology as cm
from gpu_util import host

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1509_04685_gb300 as C  # noqa: E402
COSMO = cm.Cosmology()


@pytest.mark.parametrize("n,a_init,a_final,flags", [
    (2, 0.05, 1.0, 0), (64, 0.05, 1.0, 0), (65, 0.02, 1.0, C.FLAG_MODIFIED_KDK), (256, 0.05, 1.0, 0),
    (257, 0.05, 1.0, C.FLAG_MODIFIED_KDK), (20, 0.05, 0.4, 0), (40, 0.01, 1.0, 0)])
def test_step_table_at_the_edges_of_its_tiles(n, a_init, a_final, flags):
    cfg = C.make_config(8, 16, 64.0, a_init, a_final, n, flags=flags)
    sim = C.Simulation(cfg)
    sim.init_tables()
    got = host(sim.table())
    t = cm.step_table(COSMO, cm.time_nodes(a_init, a_final, n), cm.Growth(COSMO),
                      modified=bool(flags & C.FLAG_MODIFIED_KDK))
    for col, name in enumerate(C.TABLE_COLUMNS):
        ref = getattr(t, name)
        # the tolerance of the step-table parity test
        np.testing.assert_allclose(got[:, col], ref, rtol=1e-9, atol=1e-12 * np.abs(ref).max(), err_msg=name)

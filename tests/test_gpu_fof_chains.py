"""Friends-of-friends on long chains of first friends (filaments around the whole
box along each axis and along the diagonal, closed and cut) and at the smallest
lattices with linking lengths near one half, where the neighbour cells of a
particle wrap on both sides; labels equal to the oracle's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fof

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1509_04685_gb300 as C  # noqa: E402

from gpu_util import dev  # noqa: E402


def _labels(nq, L, x, b):
    """GPU and oracle labels of particles at positions x (3, nq^3), in mean spacings"""
    d = ((x - fof.lattice_sites(nq)) * (L / nq)).astype(np.float32)
    s = C.Simulation(C.make_config(nq, 3 * nq, L, 0.05))
    s.d.copy_(dev(d))
    g, _, _ = s.fof(b, 2)
    return g.cpu().numpy(), fof.fof_groups(d, nq, L, b)


@pytest.mark.parametrize("order", ["along", "against", "shuffled"])
@pytest.mark.parametrize("cut", [False, True])
@pytest.mark.parametrize("step", [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 1)])
def test_filaments_around_the_box(step, cut, order):
    # one filament of nq^3 / 16 particles on each of 16 lines, four cells apart
    nq, L = 16, 64.0
    n, per = nq**3, nq**3 // 16
    m = np.arange(n)
    if order == "against":
        m = m[::-1]
    elif order == "shuffled":
        m = np.random.default_rng(3).permutation(m)
    line, t = m // per, (m % per + 0.5) * (nq / per)
    across = [a for a in range(3) if not step[a]] or [0, 1]  # the axes the lines are spread over
    x = np.zeros((3, n))
    x[across[0]] = 4 * (line // 4) + 1.3
    x[across[1]] = 4 * (line % 4) + 2.6
    for a in range(3):
        x[a] = (x[a] + step[a] * t) % nq
    if cut:  # the links at t = 5 and at t = 11 are missing
        gap = (np.abs(t - 5.0) < 1.0) | (np.abs(t - 11.0) < 1.0)
        x[:, gap] = np.array([[3.3], [0.6], [0.4]])
    dist = nq / per * np.linalg.norm(step)
    got, want = _labels(nq, L, x, 1.4 * dist)
    assert len(np.unique(want)) == (33 if cut else 16)
    np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("nq", [4, 6, 8, 10])
@pytest.mark.parametrize("b", [0.05, 0.3, 0.49])
def test_smallest_lattices(nq, b):
    for seed in range(8):
        rng = np.random.default_rng(100 * nq + seed)
        x = rng.uniform(0, nq, (3, nq**3))
        if seed % 2:  # most of them near the faces and corners
            x = np.where(rng.uniform(size=x.shape) < 0.7, rng.normal(0, 0.3, x.shape) % nq, x)
        got, want = _labels(nq, 2.0 * nq, x, b)
        np.testing.assert_array_equal(got, want)

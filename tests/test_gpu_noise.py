"""The normal draw of the white noise (csrc/noise.cuh) against extended precision:
random words, the tails (u1 near 0 and 1), the quadrant edges of the cosine, and
powers of two and square roots of two, where a logarithm is split.

Bound: CUDA documents log within 1 ulp, sqrt rounded correctly and cospi within
2 ulp, an ulp being at most 2 units of 2^-53 of the value; the root halves the
logarithm's error.  1 + 1 + 4, and 1 for the product: 7 units, 8 with room for
the second order."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1509_04685_gb300 import build as B  # noqa: E402

SRC = r"""
#include "noise.cuh"
__global__ void k_draw(const uint4* w, double* out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (double)cola::box_muller(w[i]);
}
extern "C" int draw(const void* w, void* out, int n) {
    k_draw<<<(n + 255) / 256, 256>>>((const uint4*)w, (double*)out, n);
    return (int)cudaDeviceSynchronize();
}
"""
LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


def _reference(m1, m2):
    """sqrt(-2 ln(m1 2^-53)) cos(2 pi m2 2^-53) in extended precision."""
    top = m1 > 1 << 52
    near = np.log1p(-((1 << 53) - m1).astype(LD) / LD(1 << 53))
    far = np.log(m1.astype(LD) / LD(1 << 53))
    k = (m2 + (1 << 50)) >> 51  # quarter turns, and the rest of the angle
    r = (m2 - (k << 51)).astype(LD) * PI / LD(1 << 52)
    c = np.where(k % 2 == 1, np.sin(r), np.cos(r))
    c = np.where((k == 1) | (k == 2), -c, c)
    return np.sqrt(-2 * np.where(top, near, far)) * c


@pytest.fixture(scope="module")
def draw(tmp_path_factory):
    d = tmp_path_factory.mktemp("noise")
    src, lib = d / "draw.cu", d / "libdraw.so"
    src.write_text(SRC)
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-I", B.CSRC, "-shared", "-o", str(lib), str(src)], check=True)
    lib = ctypes.CDLL(str(lib))

    def run(m1, m2):
        a, b = m1 - 1, m2 - 1
        w = np.stack([a >> 26 << 5, (a & 0x3ffffff) << 6, b >> 26 << 5, (b & 0x3ffffff) << 6], 1).astype(np.uint32)
        w = torch.from_numpy(w.view(np.int32)).cuda()
        out = torch.empty(len(m1), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert lib.draw(ctypes.c_void_p(w.data_ptr()), ctypes.c_void_p(out.data_ptr()), len(m1)) == 0
        return out.cpu().numpy()

    return run


def _random(rng, n):
    return rng.integers(1, (1 << 53) + 1, n, dtype=np.int64)


def _near(rng, centres, n):
    """integers around each centre, at distances spread over the powers of two up to 2^40"""
    off = rng.integers(-(1 << 40), 1 << 40, n, dtype=np.int64) >> rng.integers(0, 41, n)
    return np.clip(rng.choice(np.asarray(centres, dtype=np.int64), n) + off, 1, 1 << 53)


CASES = {
    "random": lambda g, n: (_random(g, n), _random(g, n)),
    "u1 near 0": lambda g, n: (_random(g, n) >> g.integers(1, 53, n) | 1, _random(g, n)),
    "u1 near 1": lambda g, n: (_near(g, [1 << 53], n), _random(g, n)),
    "u1 at split points": lambda g, n: (
        _near(g, [int(2.0 ** (52.0 - e / 2.0)) for e in range(20)], n), _random(g, n)),
    "quadrant edges": lambda g, n: (_random(g, n), _near(g, [k << 50 for k in range(9)], n)),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_draw_is_full_fp64(draw, case):
    n = 1 << 18
    m1, m2 = CASES[case](np.random.default_rng(11), n)
    want = _reference(m1, m2)
    got = draw(m1, m2).astype(LD)
    assert np.all(np.abs(got - want) <= 8 * LD(2.0) ** -53 * np.abs(want))


def test_draw_at_the_ends(draw):
    m1 = np.array([1, 1, 1 << 53, 1 << 53, (1 << 53) - 1], dtype=np.int64)
    m2 = np.array([1 << 53, 1 << 51, 1 << 53, 1, 1 << 52], dtype=np.int64)  # 2 pi, pi / 2, 2 pi, ~0, pi
    got = draw(m1, m2)
    assert np.isfinite(got).all()
    assert got[0] == pytest.approx(float(np.sqrt(2 * 53 * np.log(2.0))), rel=1e-15)
    assert got[1] == 0.0 and got[2] == 0.0 and got[3] == 0.0
    assert got[4] == pytest.approx(-(2.0 ** -26), rel=1e-15)  # sqrt(2 2^-53)

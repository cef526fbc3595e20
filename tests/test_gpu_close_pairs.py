"""FP64 pair forces keep their precision however close two atoms are.

The reciprocal of r^2 starts from the top 32 bits of the separation, of which a
pair closer than some 1e-3 leaves few.  Separations from 1 to 4e-8 of random
direction in a box of side 16 (exact in the fixed-point positions), against exact
integers: within 1e-13 (a dozen roundings of 1e-16, s^7 of one of them)."""
from fractions import Fraction

import numpy as np
import pytest

import oracle as O
from paper_0812_1633_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def re():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0812_1633_gb300 import build
    build.build()
    import paper_0812_1633_gb300 as m
    m.lib()
    return m


def exact(d):
    """Force on the first of two atoms from the separation d (to the second), and the energy."""
    d = [Fraction(float(c)) for c in d]
    s = 1 / sum(c * c for c in d)
    fs = s ** 4 * (24 - 48 * s ** 3)
    rc6 = Fraction(5, 2) ** 6
    return [float(fs * c) for c in d], float(4 * (s ** 6 - s ** 3) - 4 * (1 / rc6 ** 2 - 1 / rc6))


@pytest.mark.parametrize("alloc", [True, False])
def test_two_atoms(re, alloc):
    import torch
    rng = np.random.default_rng(4)
    for k in range(25):
        for _ in range(4):
            a = 5.0 + rng.integers(0, 2 ** 46, 3) * 2.0 ** -47
            u = rng.normal(size=3)
            step = np.rint(u / np.linalg.norm(u) * 2.0 ** (48 - k)) * 2.0 ** -48
            x = np.stack([a, a + step])
            d = x[1] - x[0]  # exact: multiples of 2^-48 below 8
            want, uw = exact(d)
            f, U = (re.lj_forces_device if alloc else re.lj_forces_device_noalloc)(torch.tensor(x, device="cuda"), 16.0)
            f = f.cpu().numpy()
            scale = np.abs(want).max()
            assert np.abs(f[0] - want).max() < 1e-13 * scale, k
            assert np.abs(f[1] + want).max() < 1e-13 * scale, k
            assert abs(U.item() - uw) < 1e-13 * abs(uw), k


@pytest.mark.parametrize("P", [1, 2, 4, 8])
def test_close_pair_in_a_replica(re, P):
    N = 256
    L = inputs.box_length(N)
    ctx = re.Context(N, L, 2.5, [1.0], 3, precision="fp64", atom_threads=P, cluster=4)
    x, _ = ctx.get_state()
    x[7] = x[40] + np.array([3.1e-6, -1.7e-6, 2.2e-6])
    ctx.set_state(x)
    f = ctx.forces()
    xg, _ = ctx.get_state()
    fo, uo = O.forces_brute(xg, L)[:2]
    # the positions read back are rounded to 1e-15, 1e-9 of the separation: s^7 1e-8
    assert np.abs(f - fo).max() < 1e-7 * np.abs(fo).max()
    assert ctx.energies()[0][0] == pytest.approx(uo, rel=1e-7)
    ctx.close()

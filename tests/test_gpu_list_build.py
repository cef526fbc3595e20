"""The batched kernel's list builds and pair loops at the edges of their ranges.

The list of an atom comes from testing every atom (up to 256 atoms per thread
of an atom) or from the screened build (above); both must give every pair
inside the cutoff whatever the atom count (rows of 32 atoms, the last one
partly filled), the threads per atom and the room for noted candidates.  After
a few steps (lists rebuilt every step at skin 0.05) forces and energies at the
reached positions are compared with a brute-force FP64 sum: FP64 within 1e-12
of the rms force, mixed within 1e-5 (the parity tests' tolerances).

Pairs within 1e-8 of the cutoff, where the force jumps, must fall on the side
of the FP64 distance."""
import numpy as np
import pytest

import oracle as O
from paper_0812_1633_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "mixed": 1e-5}


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


def check_forces(ctx, N, L, R, prec):
    x, _ = ctx.get_state()
    f = ctx.forces()
    U = ctx.energies()[0]
    for r in range(R):
        fo, uo = O.forces_brute(x[r * N:(r + 1) * N], L)[:2]
        rms = np.sqrt((fo ** 2).sum(1).mean())
        err = np.sqrt(((f[r * N:(r + 1) * N] - fo) ** 2).sum(1)).max() / rms
        assert err < TOL[prec], (r, err)
        assert U[r] == pytest.approx(uo, rel=1e-10 if prec == "fp64" else 1e-6)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("N,P,cluster,skin,cap", [
    (256, 1, 8, 0.05, 0), (256, 8, 8, 0.5, 0),      # one row past nothing; 32 and 4 atoms a warp
    (500, 1, 1, 0.5, 0), (500, 2, 2, 0.05, 0),      # screened and direct; last row of 20 atoms
    (1372, 1, 2, 0.05, 0), (1372, 2, 4, 0.5, 0), (1372, 4, 8, 0.05, 0),  # last row of 28 atoms
    (2048, 1, 2, 0.3, 104), (2048, 2, 4, 0.5, 0),   # room for 26 notes: tested in parts
    (2048, 4, 8, 0.6, 0),                           # full rows, four lanes an atom
])
def test_forces_after_rebuilds(re, N, P, cluster, skin, cap, prec):
    if prec == "fp64" and N == 1372 and cluster == 2:
        pytest.skip("one of the sizes is enough for the slow path")
    L, R = inputs.box_length(N), 2
    ctx = re.Context(N, L, 2.5, [1.0, 2.0], 17, precision=prec, skin=skin, cluster=cluster,
                     atom_threads=P, nbr_capacity=cap)
    for n in (1, 40):
        ctx.advance(n)
        check_forces(ctx, N, L, R, prec)
    ctx.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("P", [1, 2, 4])
def test_pairs_at_the_cutoff(re, P, prec):
    """A liquid with, every 50 atoms, one moved radially to r = 2.5 (1 -+ 1e-8)
    of an atom far away from its own neighbours' cores."""
    N = 864
    L = inputs.box_length(N)
    ctx = re.Context(N, L, 2.5, [1.2], 3, precision=prec, cluster=4, atom_threads=P)
    ctx.advance(60)
    x, _ = ctx.get_state()
    moved = 0
    for i in range(0, N, 50):
        d = x - x[i]
        d -= L * np.rint(d / L)
        r = np.sqrt((d ** 2).sum(1))
        j = int(np.argmin(np.abs(r - 2.5)))
        if abs(r[j] - 2.5) < 0.02:
            want = 2.5 * (1 + (1e-8 if moved % 2 else -1e-8))
            x[j] = (x[i] + d[j] * (want / r[j])) % L
            moved += 1
    assert moved >= 6
    ctx.set_state(x)
    check_forces(ctx, N, L, 1, prec)
    ctx.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("P,cluster", [(4, 4), (2, 2)])
def test_result_does_not_depend_on_the_register_build(re, P, cluster, prec):
    """More clusters than fit at once take the build with fewer registers; the
    same replicas in a smaller context take the other one: equal bit for bit,
    also with uneven budgets (which keep the larger build)."""
    N = 500
    L = inputs.box_length(N)
    temps = [1.0 + 0.01 * k for k in range(160)]
    state = []
    for R in (160, 12):
        ctx = re.Context(N, L, 2.5, temps[:R], 23, precision=prec, cluster=cluster, atom_threads=P)
        ctx.advance(12)
        ctx.advance(np.arange(R) % 5 + 1)
        x, v = ctx.get_state()
        state.append((x[:12 * N], v[:12 * N], ctx.energies()[0][:12]))
        ctx.close()
    for a, b in zip(*state):
        np.testing.assert_array_equal(a, b)

"""Sub-lists must not depend on how the caller numbers its atoms.

The builds give an atom's lanes their entries by the atoms' numbers.  An order
that takes the atoms of b spatial domains in turn puts most neighbours of an
atom into one residue class, far beyond one sub-list's room (six standard
deviations above an even share); a capacity given by the caller may hold an
atom's whole list and still not an uneven share.  Both must be accepted, with
forces and energies at the brute-force FP64 sum's (FP64 within 1e-12 of the rms
force, mixed within 1e-5, the parity tests' tolerances), and with results that
do not depend on the cluster size; a list that is too long as a whole is
reported as before.  sort_interval=-1: the lists follow the caller's numbering
(by default such an order is replaced by one in space before the lists are built)."""
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


def liquid(N, seed):
    """A jittered FCC lattice."""
    L = inputs.box_length(N)
    k = round((N / 4) ** (1 / 3))
    basis = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]])
    cells = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 1, 3)
    x = (cells + basis).reshape(-1, 3) * (L / k)
    return (x + np.random.default_rng(seed).uniform(-0.07, 0.07, x.shape)) % L, L


def reorder(x, L, order, seed):
    N = len(x)
    if order == "random":
        return x[np.random.default_rng(seed).permutation(N)]
    if order == "octants":
        o = (x > L / 2) @ np.array([4, 2, 1])
        y = x[np.argsort(o, kind="stable")]
        b = 8
    else:  # so many slabs
        y = x[np.argsort(x[:, 0], kind="stable")]
        b = int(order)
    assert N % b == 0
    return y.reshape(b, N // b, 3).swapaxes(0, 1).reshape(N, 3)


def check(ctx, N, L, R, prec):
    x, _ = ctx.get_state()
    f = ctx.forces()
    U = ctx.energies()[0]
    for r in range(R):
        fo, uo = O.forces_brute(x[r * N:(r + 1) * N], L)[:2]
        rms = np.sqrt((fo ** 2).sum(1).mean())
        err = np.sqrt(((f[r * N:(r + 1) * N] - fo) ** 2).sum(1)).max() / rms
        assert err < TOL[prec], (r, err)
        assert U[r] == pytest.approx(uo, rel=1e-10 if prec == "fp64" else 1e-6)


@pytest.mark.parametrize("smem", [-1, 1])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("N,P,cluster,order", [
    (256, 8, 2, "4"), (500, 4, 4, "4"), (864, 8, 8, "octants"),   # every atom tested
    (864, 4, 4, "octants"), (864, 2, 2, "octants"),               # the same, and screened
    (1372, 4, 8, "4"), (1372, 2, 4, "2"),                         # last row partly filled
    (2048, 4, 8, "4"), (2048, 4, 8, "16"), (2048, 4, 8, "random"), (2048, 2, 4, "32"),
])
def test_any_numbering(re, N, P, cluster, order, prec, smem):
    x, L = liquid(N, N)
    R = 2
    xs = np.concatenate([reorder(x, L, order, 1), reorder(x, L, order, 2)])
    ctx = re.Context(N, L, 2.5, [1.0, 1.3], 5, precision=prec, cluster=cluster, atom_threads=P,
                     sort_interval=-1, lists_smem=smem)
    ctx.set_state(xs)
    check(ctx, N, L, R, prec)
    ctx.advance(30)
    assert (ctx.counters()[1] >= 1).all()
    check(ctx, N, L, R, prec)
    ctx.close()


def test_cluster_size_changes_nothing(re):
    """Dealt and undealt sub-lists in one warp: bit-equal for every cluster size."""
    N = 864
    x, L = liquid(N, 3)
    y = reorder(x, L, "octants", 0)
    y[N // 2:] = y[N // 2:][np.argsort(y[N // 2:, 1], kind="stable")]
    out = []
    for cluster in (4, 8):
        ctx = re.Context(N, L, 2.5, [1.1], 5, precision="mixed", cluster=cluster, atom_threads=4,
                         sort_interval=-1)
        ctx.set_state(y)
        ctx.advance(25)
        out.append(ctx.get_state())
        ctx.close()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])


def test_tight_capacity_at_the_default_shape(re):
    """120 neighbours per atom hold every list (about 95 entries); an eighth of
    them does not hold every eighth of a list by number."""
    N, R = 256, 4
    L = inputs.box_length(N)
    ctx = re.Context(N, L, 2.5, [0.9, 1.1, 1.3, 1.6], 7, precision="fp64", nbr_capacity=120)
    ctx.advance(300)
    check(ctx, N, L, R, "fp64")
    ctx.close()


@pytest.mark.parametrize("P", [2, 4, 8])
def test_too_long_as_a_whole_is_reported(re, P):
    N = 500
    x, L = liquid(N, 2)
    with pytest.raises(re.REError) as e:
        ctx = re.Context(N, L, 2.5, [1.0], 5, precision="mixed", cluster=4, atom_threads=P, nbr_capacity=64)
        ctx.set_state(x)
        ctx.forces()
    assert e.value.code == re.RE_EOVERFLOW


@pytest.mark.parametrize("order", ["random", "slabs", "lattice"])
def test_default_renumbering_keeps_the_callers_order(re, order):
    """Default options: the state reads back in the caller's order, and its
    forces are the brute-force ones, whether the atoms were renumbered or not."""
    N = 1372
    x, L = liquid(N, 4)
    y = x if order == "lattice" else reorder(x, L, order if order == "random" else "4", 5)
    v = np.random.default_rng(6).normal(0.0, 1.0, (N, 3))
    ctx = re.Context(N, L, 2.5, [1.0], 5, precision="mixed")
    ctx.set_state(y, v)
    xg, vg = ctx.get_state()
    d = xg - y
    assert np.abs(d - L * np.rint(d / L)).max() < 1e-12
    assert np.abs(vg - v).max() < 1e-12
    check(ctx, N, L, 1, "mixed")
    ctx.close()

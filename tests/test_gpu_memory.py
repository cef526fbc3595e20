"""Device memory of a batched context: the state, one set of neighbour lists and
the fixed words, at the default capacity and at one that leaves no room in the
lists' array (where the build's notes get an array of their own, and the lists
are the same), also after the autotuner has gone through shapes that need one."""
import numpy as np
import pytest

from paper_0812_1633_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,skin", [(864, 0.3), (2048, 0.5), (4000, 0.5)])
def test_one_set_of_lists(N, skin):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0812_1633_gb300 as re
    R, L = 500000 // N, inputs.box_length(N)
    temps = [0.8 + 0.001 * k for k in range(R)]
    re.Context(256, inputs.box_length(256), 2.5, [1.0], 1).close()  # modules loaded
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx = re.Context(N, L, 2.5, temps, 3, skin=skin)
    ctx.advance(12)
    ctx.energies()
    used = before - torch.cuda.mem_get_info()[0]
    ctx.close()
    m = N / L ** 3 * 4 / 3 * np.pi * (2.5 + skin) ** 3  # neighbours of an atom
    lists = 2 * 8 * (int(np.ceil(m / 8 + 6 * np.sqrt(m / 8) + 4)) + 3) // 4 * 4
    # 260 bytes of state an atom, 9 KB a replica, allocation granularity
    assert used < N * R * (lists + 260) + R * 9216 + (48 << 20)


@pytest.mark.parametrize("cap", [128, 160])
def test_capacity_without_room_for_notes(cap):
    """128: every layout of the lists fills the array; the trajectories are those
    of a capacity with room."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0812_1633_gb300 as re
    for N, P, cluster in ((864, 2, 2), (2048, 4, 8), (1372, 1, 2)):
        L = inputs.box_length(N)
        out = []
        for c in (cap, 0):
            ctx = re.Context(N, L, 2.5, [0.9, 1.2], 3, precision="mixed", atom_threads=P,
                             cluster=cluster, nbr_capacity=c)
            ctx.advance(40)
            out.append(ctx.get_state()[0])
            ctx.close()
        if P == 1:  # several lanes: a dealt sub-list has another order
            np.testing.assert_array_equal(out[0], out[1])
        else:
            d = out[0] - out[1]
            assert np.abs(d - L * np.rint(d / L)).max() < 1e-3


def test_shapes_with_and_without_the_array():
    """The tuner goes through shapes with and without room for notes, and a
    free-running launch may take another one between replays of a cached graph."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0812_1633_gb300 as re
    N, R = 1372, 12
    L, temps = inputs.box_length(N), [0.9 + 0.1 * k for k in range(R)]
    a = re.Context(N, L, 2.5, temps, 5, skin=0.3)
    cfg = a.autotune(steps=5)
    b = re.Context(N, L, 2.5, temps, 5, skin=0.3, cluster=cfg["cluster"], atom_threads=cfg["atom_threads"])
    assert np.array_equal(a.get_state()[0], b.get_state()[0])
    for ctx in (a, b):
        ctx.run(4, graph=True)
        ctx.run_free(2, 5)
        ctx.run(4, graph=True)
        assert np.isfinite(ctx.energies()[0]).all()
    a.close()
    b.close()

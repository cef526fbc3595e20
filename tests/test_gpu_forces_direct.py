"""re_lj_forces_device and re_lj_forces_device_noalloc at the edges of their
ranges (odd atom counts, fewer atoms than a warp, one more or less than a row of
32, the largest), against the oracle's brute-force sum: FP64 within 1e-12 of the
rms force, mixed within 1e-5 (the parity tests' tolerances); coincident and
crowded atoms refused; calls from several threads and streams independent."""
import threading

import numpy as np
import pytest

import oracle as O

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


def configuration(N, seed, spacing=1.08):
    """N atoms on a jittered cubic grid of this spacing, some of its sites empty."""
    rng = np.random.default_rng(seed)
    k = max(int(np.ceil(N ** (1 / 3))), 6)
    sites = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.5
    x = sites[rng.permutation(k ** 3)[:N]] * spacing
    L = k * spacing
    return (x + rng.uniform(-0.06, 0.06, x.shape)) % L, L


def check(f, U, x, L, prec):
    fo, uo = O.forces_brute(x, L)[:2]
    rms = np.sqrt((fo ** 2).sum(1).mean())
    assert np.sqrt(((f - fo) ** 2).sum(1)).max() <= TOL[prec] * rms
    assert abs(U - uo) <= (1e-12 if prec == "fp64" else 1e-6) * max(abs(uo), 1.0)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("N", [2, 31, 33, 217, 987, 1217, 2433, 4001])
def test_edges(re, N, prec):
    import torch
    x, L = configuration(N, N)
    xt = torch.tensor(x, device="cuda")
    f, U = re.lj_forces_device(xt, L, precision=prec)
    check(f.cpu().numpy(), U.item(), x, L, prec)
    if prec == "fp64":
        f, U = re.lj_forces_device_noalloc(xt, L)
        check(f.cpu().numpy(), U.item(), x, L, prec)


def test_refusals(re):
    import torch
    x, L = configuration(300, 1)
    y = x.copy()
    y[7] = y[200]
    for call in (lambda a: re.lj_forces_device(a, L), lambda a: re.lj_forces_device_noalloc(a, L)):
        with pytest.raises(re.REError) as e:
            call(torch.tensor(y, device="cuda"))
        assert e.value.code == re.RE_ENUMERIC
    crowded = (x * 0.45) % (2 * L)  # eleven times the density its box has on average
    for call in (lambda a: re.lj_forces_device(a, 2 * L), lambda a: re.lj_forces_device_noalloc(a, 2 * L)):
        with pytest.raises(re.REError) as e:
            call(torch.tensor(crowded, device="cuda"))
        assert e.value.code == re.RE_EOVERFLOW
    with pytest.raises(re.REError) as e:  # more than a replica of the batched path holds
        re.lj_forces_device(torch.zeros((9000, 3), device="cuda", dtype=torch.float64), 40.0)
    assert e.value.code == re.RE_EINVAL


def test_threads_and_streams(re):
    import torch
    cases = [configuration(n, n) for n in (500, 1100, 700, 987)]
    xs = [torch.tensor(x, device="cuda") for x, _ in cases]
    want = [re.lj_forces_device(a, L)[0].cpu().numpy() for a, (_, L) in zip(xs, cases)]
    torch.cuda.synchronize()
    bad = []

    def work(k):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            for _ in range(20):
                f, _ = re.lj_forces_device(xs[k], cases[k][1])
                if not np.array_equal(f.cpu().numpy(), want[k]):
                    bad.append(k)

    ts = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not bad

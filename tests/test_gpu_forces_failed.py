"""A force call that fails (coincident atoms, more neighbours than the limit)
leaves the caller's f and U as they were; f over x, which such a call then leaves
too, gives the forces of a call with an array of its own."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def call(re, alloc, x, f, U, L, prec):
    import torch
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    n = x.shape[0]
    if alloc:
        return re.lib().re_lj_forces_device(n, L, 2.5, 1, re.PREC[prec], x.data_ptr(), f.data_ptr(), U.data_ptr(), st)
    return re.lib().re_lj_forces_device_noalloc(n, L, 2.5, 1, x.data_ptr(), f.data_ptr(), U.data_ptr(), st)


@pytest.mark.parametrize("alloc,prec", [(True, "fp64"), (True, "mixed"), (False, "fp64")])
@pytest.mark.parametrize("N", [64, 987, 3001])
def test_failed_call_and_in_place(alloc, prec, N):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0812_1633_gb300 as re
    rng = np.random.default_rng(N)
    k = max(int(np.ceil(N ** (1 / 3))), 7)
    grid = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)
    x = (grid[rng.permutation(k ** 3)[:N]] + 0.5) * 1.1 + rng.uniform(-0.06, 0.06, (N, 3))
    L = 1.1 * k
    same = x.copy()
    same[3] = same[40]
    crowded = x * 0.3 if N > 500 else None
    for y, box, code in ((same, L, re.RE_ENUMERIC), (crowded, L, re.RE_EOVERFLOW)):
        if y is None:
            continue
        xt = torch.tensor(y, device="cuda")
        f = torch.full_like(xt, 7.0)
        U = torch.full((1,), 9.0, dtype=torch.float64, device="cuda")
        assert call(re, alloc, xt, f, U, box, prec) == code
        assert (f == 7.0).all() and U.item() == 9.0
        before = xt.clone()
        assert call(re, alloc, xt, xt, U, box, prec) == code
        assert torch.equal(xt, before)
    xt = torch.tensor(x, device="cuda")
    f = torch.empty_like(xt)
    U = torch.zeros(1, dtype=torch.float64, device="cuda")
    V = torch.zeros(1, dtype=torch.float64, device="cuda")
    assert call(re, alloc, xt, f, U, L, prec) == re.RE_OK
    assert call(re, alloc, xt, xt, V, L, prec) == re.RE_OK
    assert torch.equal(xt, f) and torch.equal(U, V)

"""The stateless exchange with its outputs over its inputs (T_out = T, lam_out =
lam): the same partners, decisions and values as with arrays of its own, which
equal the oracle's.  Ladders of one CTA, of a cluster with one pair across two
CTAs' slices, and of the largest size; equal energies, so that every pair is
accepted and every T moves, and energies that differ."""
import ctypes as C

import numpy as np
import pytest

import oracle as O
from paper_0812_1633_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [2, 128, 129, 1000, 4096])
@pytest.mark.parametrize("use_lam", [False, True])
@pytest.mark.parametrize("equal_u", [True, False])
def test_in_place(R, use_lam, equal_u):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0812_1633_gb300 as re
    rng = np.random.default_rng(R)
    T = rng.permutation(inputs.geometric_ladder(0.7, 3.0, R))
    lam = rng.uniform(0.9, 1.0, R) if use_lam else np.ones(R)
    U = lam * 7.0 if equal_u else -6.0 * R + rng.normal(0.0, 2.0, R)
    for attempt in range(6):
        Tn, ln, po, ao, vo, uo = O.exchange_h(T, lam, U, 11, attempt, 0, 1)[:6]
        t = torch.tensor(T, device="cuda")
        lt = torch.tensor(lam, device="cuda")
        u = torch.tensor(U, device="cuda")
        partner = torch.empty(R, dtype=torch.int32, device="cuda")
        acc = torch.empty(R, dtype=torch.uint8, device="cuda")
        vs = torch.empty(R, dtype=torch.float64, device="cuda")
        st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
        if use_lam:  # uscale over U as well
            rc = re.lib().re_exchange_device_h(R, t.data_ptr(), lt.data_ptr(), u.data_ptr(), 11, attempt, 0, 1,
                                               t.data_ptr(), lt.data_ptr(), partner.data_ptr(), acc.data_ptr(),
                                               vs.data_ptr(), u.data_ptr(), st)
        else:
            rc = re.lib().re_exchange_device(R, t.data_ptr(), u.data_ptr(), 11, attempt, 0, t.data_ptr(),
                                             partner.data_ptr(), acc.data_ptr(), vs.data_ptr(), st)
        assert rc == re.RE_OK
        assert np.array_equal(partner.cpu().numpy(), po)
        assert np.array_equal(acc.cpu().numpy(), ao)
        assert np.array_equal(t.cpu().numpy(), Tn)
        if equal_u:
            assert np.array_equal(ao == 1, po >= 0)
        if use_lam:
            assert np.array_equal(lt.cpu().numpy(), ln)
            assert np.allclose(u.cpu().numpy(), uo, rtol=1e-15)
        assert np.allclose(vs.cpu().numpy(), vo, rtol=1e-15)

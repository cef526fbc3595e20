"""No common relative error in the mixed energies.

A pair's FP32 roundings are its own and average out over many pairs; a rounded
constant of the box does not.  Hot dense liquids, where the r^-12 part weighs most:
the mean relative error over 32 configurations stays below 2e-8 (the roundings of
an atom's energy, some 5e-7, make 6e-9 over 32 x 256 atoms)."""
import numpy as np
import pytest

from paper_0812_1633_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [256, 864, 2048])
def test_mean_energy_error(N):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0812_1633_gb300 as re
    L, R = inputs.box_length(N), 32
    ctx = re.Context(N, L, 2.5, inputs.geometric_ladder(2.0, 3.0, R), 21, precision="mixed")
    ctx.advance(200)
    x, _ = ctx.get_state()
    ctx.close()
    err = []
    for r in range(R):
        xt = torch.tensor(x[r * N:(r + 1) * N], device="cuda")
        u, w = (re.lj_forces_device(xt, L, precision=p)[1].item() for p in ("mixed", "fp64"))
        err.append(u / w - 1.0)
    assert abs(np.mean(err)) < 2e-8

"""The memory that the force call's pool keeps: at most 64 MB after calls from
several threads, and none of it once a context's allocation fails for lack of
memory (a context far larger than the device, which is refused as before)."""
import threading

import numpy as np
import pytest

from paper_0812_1633_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_pool_is_bounded_and_given_back():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0812_1633_gb300 as re
    N = 4000
    L = inputs.box_length(N)
    re.Context(256, inputs.box_length(256), 2.5, [1.0], 1).close()  # modules loaded
    rng = np.random.default_rng(1)
    x = torch.tensor((np.stack(np.meshgrid(*[np.arange(16)] * 3, indexing="ij"), -1).reshape(-1, 3)[:N] + 0.5) * (L / 16)
                     + rng.uniform(-0.05, 0.05, (N, 3)), device="cuda")

    def work():
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(5):
                re.lj_forces_device(x, L)

    work()
    ts = [threading.Thread(target=work) for _ in range(6)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    kept = torch.cuda.mem_get_info()[0]
    with pytest.raises(re.REError) as e:  # lists of 4096 x 6912 x 6912 entries: 391 GB in one piece
        re.Context(6912, inputs.box_length(6912), 2.5, list(1.0 + 0.001 * np.arange(4096)), 1, path="plain",
                   nbr_capacity=6912)
    assert e.value.code == re.RE_ENOMEM
    given = torch.cuda.mem_get_info()[0] - kept
    assert 0 < given <= 64 << 20
    re.lj_forces_device(x, L)  # and it starts anew

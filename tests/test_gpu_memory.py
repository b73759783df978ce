"""Device memory that a grid keeps for speed gives way to memory that a call needs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def msh():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1210_5246_gb300 import msh as m
    m.load()
    return m


def _grid(msh, steps):
    n = (64, 48, 40)
    rng = np.random.default_rng(4)
    W = np.zeros((10,) + n[::-1])
    W[0] = rng.uniform(0.8, 1.2, n[::-1])
    W[1:4] = rng.uniform(-0.2, 0.2, (3,) + n[::-1])
    W[4] = W[7] = W[9] = 1.0
    g = msh.Grid(n, (0.0,) * 3, (1.0,) * 3, ((0, 0),) * 3, 0.4, msh.FP64)
    g.set_state(W, msh.PRIMITIVE)
    g.run(max_steps=steps)
    return g


@pytest.mark.parametrize("call", ["tape", "adjoint"])
def test_staging_buffers_are_given_back_to_a_call_out_of_memory(msh, call):
    """A call that needs more device memory than there is fails; the buffers of the staged step (8
    states and 6 sides of ghosts here) were freed before the second attempt.  The next steps allocate
    them again and go on to the same bits."""
    import torch
    ref = _grid(msh, 3)
    ref.run(max_steps=3)
    want, t = ref.get_state(), ref.time()
    ref.close()
    g = _grid(msh, 3)
    staging = 8 * 10 * 8 * int(np.prod(g.n))
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    with pytest.raises(msh.MshError) as ei:
        if call == "tape":
            g.set_tape(1, 10 ** 7)  # 10^7 states: 98 TB
        else:
            U = g.get_state()
            g.adjoint_run(U, np.full(10 ** 6, 1e-4), U, K=1)  # 10^6 checkpoints: 9.8 TB
    assert ei.value.status == msh.MSH_E_NOMEM
    assert torch.cuda.mem_get_info()[0] - free0 >= 0.9 * staging
    g.run(max_steps=3)
    np.testing.assert_array_equal(g.get_state(), want)
    assert g.time() == t
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info()[0] <= 0.1 * staging
    g.close()

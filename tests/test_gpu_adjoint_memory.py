"""Memory that adjoint runs at the default checkpoint interval hold: contexts that keep every
state take at most 1/16 of the device's memory together, later ones go back to checkpoints, and
destroying contexts gives the share back."""

import numpy as np
import pytest

from paper_1712_08288_gb300 import binding as B
from paper_1712_08288_gb300 import workloads as W
from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def test_kept_states_of_many_contexts_are_bounded():
    torch = require_gpu()
    n, T = 64, 200
    N = n ** 3
    state = 19 * N * 4
    mask, ut = np.ones(N, bool), np.full((N, 3), 0.01)
    free, total = torch.cuda.mem_get_info()
    every = T * state                                       # 3.98e9 bytes, under 4 GiB
    share = total // 16
    count = share // every + 3                              # three more than the share holds
    small = (2 * int(np.ceil(np.sqrt(T))) + 12) * state     # checkpoints, a segment, working arrays
    if free < 16 * every + count * every:
        pytest.skip("needs free device memory")

    def adjoint():
        sim = B.Lbm("D3Q19", (n, n, n), W.relaxation_rates("D3Q19", 1.0), "f32", 1.0)
        sim.set_force((1e-6, 0.0, 0.0))
        sim.init_equilibrium()
        before = torch.cuda.mem_get_info()[0]
        grad = sim.adjoint(T, mask, ut)[1]
        return sim, grad, before - torch.cuda.mem_get_info()[0]

    sims, grads, used = zip(*(adjoint() for _ in range(count)))
    assert used[0] >= every and used[-1] <= small
    assert sum(used) <= share + count * small
    for g in grads:
        assert np.abs(g - grads[0]).max() <= 1e-4 * np.abs(grads[0]).max()
    # the same call again takes nothing more
    before = torch.cuda.mem_get_info()[0]
    sims[0].adjoint(T, mask, ut)
    sims[-1].adjoint(T, mask, ut)
    assert before - torch.cuda.mem_get_info()[0] <= small
    for sim in sims:
        sim.close()
    sim, _, again = adjoint()
    assert again >= every
    sim.close()

"""A batch of more problems than the y and z axes of a launch grid can count
(65 535): every per-problem kernel has to take its problems along x."""
import numpy as np
import pytest

from paper_1402_5618_gb300 import workloads as W

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("checked", [False, True])
def test_more_problems_than_65535(checked):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_5618_gb300 import binding as B
    B.lib()
    nprob = 65600
    kinds = [W.random_smooth_1d(8 + k, stream=700 + k) for k in range(3)]
    cfgs = [B.config_from_problem(p, cfl_positivity_cap=checked) for p in kinds]
    one = []
    for c, p in zip(cfgs, kinds):
        s = B.Solver(None, batch=[c])
        s.set_state(p.U0.ravel().copy())
        s.step()
        one.append(s.get_state()[0].copy())
        s.close()
    s = B.Solver(None, batch=[cfgs[k % 3] for k in range(nprob)])
    s.set_state(np.concatenate([kinds[k % 3].U0.ravel() for k in range(nprob)]))
    s.step()
    out = s.get_state()[0]
    s.close()
    period = sum(u.size for u in one)
    full = np.concatenate(one)
    whole = out[:out.size // period * period].reshape(-1, period)
    assert np.array_equal(whole, np.broadcast_to(full, whole.shape))
    assert np.array_equal(out[whole.size:], full[:out.size - whole.size])

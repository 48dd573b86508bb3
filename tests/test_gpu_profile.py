"""hrm_set_profiling brackets every kernel of a step: with the list kernels, the unchanged cells' kernel and the deferred
midpoints' ones counted, the brackets hold as many kernels as the step launches."""
from collections import Counter

import pytest

from paper_2208_04488_gb300 import problems as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hrm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2208_04488_gb300 import build, hrm as H
    build.build()
    return H


@pytest.mark.parametrize("pr,lists", [(P.shock_tube_1d_baseline(400), False), (P.shock_bubble_2d(64, 32), False),
                                      (P.shock_bubble_2d(400, 200), True), (P.interface_3d(41), True)],
                         ids=["400", "64x32", "400x200", "41^3"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("gate", [False, True], ids=["plain", "gate"])
def test_brackets_cover_every_kernel(hrm, pr, lists, precision, gate):
    fp32 = precision == "fp32"
    prm = dict(cfl=0.4, check=0, precision=hrm.FP32 if fp32 else hrm.FP64)
    s = hrm.Solver.from_problem(pr, params=hrm.params_default(**prm))
    if gate:
        s.set_detector(hrm.Detector(capacity=1 << 14, seed=1))
        s.set_params(hrm.params_default(learned=hrm.LEARNED_GATE, **prm))
    s.set_profiling(True)
    s.step(0.0, 2)
    prof = s.profile_read()
    n = Counter(k for k, _ in prof)
    assert n[hrm.KERNEL_SWEEPS] == n[hrm.KERNEL_UPDATE] == 3 and n[hrm.KERNEL_FINALIZE] == 1
    assert n[hrm.KERNEL_LISTS] == (3 if lists else 0)
    assert n[hrm.KERNEL_KEEP] == (3 if fp32 and lists else 0)
    assert n[hrm.KERNEL_FIX] == (3 * pr.D if fp32 else 0)
    assert n[hrm.KERNEL_GATE] == (3 * pr.D if gate and not fp32 else 0)
    kernels = sum(n.values()) - n[hrm.KERNEL_SWEEPS] + n[hrm.KERNEL_LISTS]  # two kernels in each list bracket
    assert kernels == s.step_launches()
    assert all(ms >= 0.0 for _, ms in prof)
    s.close()


def test_a_call_beside_the_step_takes_no_bracket(hrm):
    """hrm_rhs and stages one at a time use the same kernels outside the traced step."""
    import torch
    pr = P.shock_bubble_2d(400, 200)
    s = hrm.Solver.from_problem(pr, params=hrm.params_default(cfl=0.4, check=0))
    s.set_profiling(True)
    s.step(0.0, 1)
    n = len(s.profile_read())
    s.rhs([1e-8, 1e-8], torch.empty((pr.M, pr.ncells), dtype=torch.float64, device="cuda"))
    s.begin_step(s.step_tau())
    for k in range(s.stages()):
        s.stage(k)
    s.step(0.0, 1)
    assert len(s.profile_read()) == n
    s.close()

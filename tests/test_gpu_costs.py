"""What a call may cost beside another one on the same state, by medians of device times: guards against work that a
call's result does not need."""
import numpy as np
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


def median_ms(f, n=9):
    import torch
    f()
    t = []
    for _ in range(n):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        t.append(a.elapsed_time(b))
    return float(np.median(t))


def test_first_order_step_forms_no_primitives_that_nothing_uses(hrm):
    """Precision form, 1024x512 water column after 20 steps: the first-order flux reads two nodes' planes and solves one
    Riemann problem. With the nodes' FP64 primitives formed and not used a step took 1.54 times one of the whole scheme."""
    import torch
    torch.cuda.current_stream().synchronize()
    pr = P.shock_water_column_2d(1024, 512)
    s = hrm.Solver.from_problem(pr, params=hrm.params_default(cfl=0.4, check=0, precision=hrm.FP32))
    s.step(0.0, 20)
    W = torch.from_numpy(s.get(hrm.FIELD_W)).cuda()

    def steps():
        s.set(W)
        s.step(0.0, 4)

    high = median_ms(steps)
    s.set_params(hrm.params_default(cfl=0.4, check=0, precision=hrm.FP32, scheme=1))
    assert median_ms(steps) < 1.25 * high
    s.close()

"""States that a step cannot digest -- vacuum, NaN, infinities, fluxes beyond the
number range, a time step that is not a number -- must come out of the list-driven
kernels as out of the arithmetic written out: a cell between two uniform faces takes
its own flux twice, and the difference of two infinite or undefined fluxes is NaN,
not zero."""
import numpy as np
import pytest

from paper_2208_04488_gb300 import problems as P

pytestmark = pytest.mark.gpu

GRIDS = [[40], [45, 33], [22, 20, 21]]
N = 3


@pytest.fixture(scope="module")
def hrm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2208_04488_gb300 import build, hrm as H
    build.build()
    return H


def uniform(n, bc=0):
    D, cells = len(n), int(np.prod(n))
    gamma, pinf, cv, q = P._species([P.BENCH_WATER, P.BENCH_AIR, P.BENCH_HELIUM])
    one = np.ones(cells)
    prim = P._assemble(N, D, [0.3 * one, 0.5 * one], [(20.0 - 15.0 * d) * one for d in range(D)], 1.2e5 * one, 310.0 * one)
    return P.Problem("uniform", gamma, pinf, cv, q, list(n), [0.0] * D, [1.0 + 0.3 * d for d in range(D)], [bc] * (2 * D), prim,
                     cfl=0.4)


def spoilt(W, n, what):
    """W with one value per plane written into a block of cells that holds whole stencils."""
    D = len(n)
    block = np.ones(n[::-1], bool)
    for x, m in zip(np.meshgrid(*[np.arange(v) for v in n[::-1]], indexing="ij"), n[::-1]):
        block &= (x >= m // 4) & (x < m // 4 + max(9, m // 2))
    mom, en, al = N, N + D, N + D + 1
    planes = {"vacuum": {0: 0.0, 1: 0.0, 2: 0.0}, "nan": {mom: np.nan}, "nan_alpha": {al: np.nan}, "inf_energy": {en: np.inf},
              "inf_density": {0: np.inf}, "overflow": {en: 1e302, mom: -1e10}, "overflow32": {en: 1e36, mom: 1e7},
              "negative": {0: -1.0}}[what]
    X = W.copy()
    for m, v in planes.items():
        X[m, block.reshape(-1)] = v
    return X


@pytest.mark.parametrize("n", GRIDS, ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("bc", [0, 1], ids=["transmissive", "periodic"])
@pytest.mark.parametrize("what", ["vacuum", "nan", "nan_alpha", "inf_energy", "inf_density", "overflow"])
def test_fp64_step_and_rhs_equal_the_oracle(hrm, orc, n, bc, what):
    import torch
    pr = uniform(n, bc)
    f, g, W0 = orc.setup(pr)
    dt, _ = orc.dt(f, g, W0, 0.4)
    lam = orc.lambdas(f, g, W0, dt)
    W = spoilt(W0, n, what)
    s = hrm.Solver.from_problem(pr, params=hrm.params_default(cfl=0.4, check=0))
    s.set(W)
    rhs = s.rhs(lam, torch.empty((pr.M, pr.ncells), dtype=torch.float64, device="cuda")).cpu().numpy()
    with np.errstate(all="ignore"):
        np.testing.assert_array_equal(rhs, orc.rhs(f, orc.make_params(), g, W, lam))
        for relax in (hrm.RELAX_STAGE, hrm.RELAX_OFF):
            s.set_params(hrm.params_default(cfl=0.4, check=0, relax_mode=relax))
            for steps in (1, 2):
                s.set(W)
                s.step(dt, steps)
                np.testing.assert_array_equal(s.get(hrm.FIELD_W), orc.step(f, orc.make_params(relax_mode=relax), g, W, dt, steps))
    s.close()


@pytest.mark.parametrize("n", GRIDS, ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("what", ["vacuum", "nan", "inf_energy", "overflow", "overflow32"])
@pytest.mark.parametrize("relax", [0, 1])
def test_precision_form_step_equals_its_stages(hrm, n, what, relax):
    pr = uniform(n)
    prm = hrm.params_default(cfl=0.4, check=0, precision=hrm.FP32, relax_mode=relax)
    a, b = hrm.Solver.from_problem(pr, params=prm), hrm.Solver.from_problem(pr, params=prm)
    dt, tau = a.dt(0.4)
    W = spoilt(a.get(hrm.FIELD_W), n, what)
    a.set(W)
    b.set(W)
    a.step(dt, 1)
    b.begin_step(tau, dt)
    for k in range(b.stages()):
        b.stage(k)
    Wa = a.get(hrm.FIELD_W)
    np.testing.assert_array_equal(Wa, b.get(hrm.FIELD_W))
    assert np.isnan(Wa).any()
    a.close()
    b.close()


@pytest.mark.parametrize("n", GRIDS, ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("scheme", ["wcns", "hllc1"])
def test_undefined_time_step_reaches_every_cell(hrm, n, precision, scheme):
    """Cells of negative density have no sound speed: the CFL step of the first step
    after the state was written is not a number, and so are all cells after it."""
    pr = uniform(n)
    s = hrm.Solver.from_problem(pr, params=hrm.params_default(cfl=0.4, check=0, scheme=1 if scheme == "hllc1" else 0,
                                                              precision=hrm.FP64 if precision == "fp64" else hrm.FP32))
    s.set(spoilt(s.get(hrm.FIELD_W), n, "negative"))
    s.step(0.0, 1)
    assert np.isnan(s.get(hrm.FIELD_W)).all()
    s.close()

"""List-driven sweeps: uniform faces are found by comparing neighbouring cells and
only the other midpoints run the midpoint body. On grids around the sizes of the
blocks and warps that build the lists, in every dimension and with every kind of
side, a uniform state with a few disturbed cells -- the corners, the middle, or
none -- must step exactly as the oracle, which tests every midpoint's six nodes."""
import numpy as np
import pytest

from paper_2208_04488_gb300 import problems as P

pytestmark = pytest.mark.gpu

GRIDS = [[3], [7], [255], [256], [257], [33, 3], [5, 64], [257, 4], [3, 4, 5], [9, 3, 8]]


@pytest.fixture(scope="module")
def hrm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2208_04488_gb300 import build, hrm as H
    build.build()
    return H


def disturbed(n, bc, where, N=3):
    """A uniform moving state with disturbed cells (and a boundary state of its own on Dirichlet sides)."""
    D, cells = len(n), int(np.prod(n))
    fl = [P.BENCH_WATER, P.BENCH_AIR, P.BENCH_HELIUM][:N]
    gamma, pinf, cv, q = P._species(fl)
    one = np.ones(cells)
    prim = P._assemble(N, D, [0.3 * one, 0.5 * one][:N - 1], [(20.0 - 15.0 * d) * one for d in range(D)], 1.2e5 * one, 310.0 * one)
    at = {"none": [], "first": [0], "last": [cells - 1], "middle": [cells // 2], "ends": [0, cells // 3, cells - 1]}[where]
    for i, c in enumerate(at):
        prim[0, c] += 0.05 * (i + 1)
        prim[N - 1 + (i % D), c] += 3.0
        prim[N + D - 1, c] *= 1.01
    pr = P.Problem("disturbed", gamma, pinf, cv, q, list(n), [0.0] * D, [1.0 + 0.3 * d for d in range(D)], [bc] * (2 * D), prim,
                   cfl=0.4)
    if bc == 2:  # half of the sides continue the interior state, the others differ
        for b in range(2 * D):
            ns = cells // n[b // 2]
            s = P._assemble(N, D, [np.full(ns, 0.3), np.full(ns, 0.5)][:N - 1],
                            [np.full(ns, 20.0 - 15.0 * d) for d in range(D)], np.full(ns, 1.2e5), np.full(ns, 310.0))
            if b % 2:
                s[N + D, : (ns + 1) // 2] += 5.0
            pr.boundary[b] = s
    return pr


@pytest.mark.parametrize("n", GRIDS, ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("bc", [0, 1, 2], ids=["transmissive", "periodic", "dirichlet"])
@pytest.mark.parametrize("where", ["none", "first", "last", "middle", "ends"])
def test_step_and_rhs_equal_the_oracle(hrm, orc, n, bc, where):
    import torch
    pr = disturbed(n, bc, where)
    f, g, W = orc.setup(pr)
    s = hrm.Solver.from_problem(pr, params=hrm.params_default(cfl=0.4, check=0))
    dt, _ = orc.dt(f, g, W, 0.4)
    lam = orc.lambdas(f, g, W, dt)
    rhs = s.rhs(lam, torch.empty((pr.M, pr.ncells), dtype=torch.float64, device="cuda")).cpu().numpy()
    np.testing.assert_array_equal(rhs, orc.rhs(f, orc.make_params(), g, W, lam))
    s.step(dt, 3)
    np.testing.assert_array_equal(s.get(hrm.FIELD_W), orc.step(f, orc.make_params(), g, W, dt, 3))
    s.close()


@pytest.mark.parametrize("n", GRIDS, ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("bc", [0, 1, 2], ids=["transmissive", "periodic", "dirichlet"])
@pytest.mark.parametrize("where", ["none", "ends"])
def test_precision_form_step_equals_its_stages(hrm, n, bc, where):
    """The step's updates form uniform faces' fluxes from the cell's own planes; the
    stages taken one at a time write and read every midpoint's flux."""
    pr = disturbed(n, bc, where)
    prm = hrm.params_default(cfl=0.4, check=0, precision=hrm.FP32)
    a, b = hrm.Solver.from_problem(pr, params=prm), hrm.Solver.from_problem(pr, params=prm)
    for _ in range(3):
        a.step(0.0, 1)
        b.begin_step(b.step_tau())
        for k in range(b.stages()):
            b.stage(k)
    np.testing.assert_array_equal(a.get(hrm.FIELD_W), b.get(hrm.FIELD_W))
    a.close()
    b.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("where", ["none", "ends"])
def test_batch_of_small_instances_equals_single_contexts(hrm, precision, where):
    """The stage kernel's lists over instances smaller than a warp's, a tile's or a
    work item's share, of both species counts."""
    ps = [disturbed(n, bc, where, N) for n in ([3, 3], [33, 3], [5, 64], [257, 4]) for bc in (0, 1) for N in (2, 3)]
    prm = hrm.params_default(cfl=0.4, check=0, precision=hrm.FP64 if precision == "fp64" else hrm.FP32)
    b = hrm.BatchSolver(ps, params=prm)
    b.step(3)
    for i, pr in enumerate(ps):
        s = hrm.Solver.from_problem(pr, params=prm)
        s.step(0.0, 3)
        np.testing.assert_array_equal(b.get(i), s.get(hrm.FIELD_W))
        s.close()


@pytest.mark.parametrize("n", [[70], [40, 24], [130, 80], [12, 10, 9]], ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("low", [-140, -330], ids=["2^-465", "subnormal"])
def test_decaying_velocities_equal_the_oracle(hrm, orc, n, low):
    """Velocities of every exponent down to zero beside ordinary ones, alone and within one stencil."""
    pr = disturbed(n, 0, "ends")
    rng = np.random.default_rng(20)
    D, cells = len(n), int(np.prod(n))
    for d in range(D):
        exponent = rng.uniform(low, 1.0, cells) if d else np.linspace(1.0, low, cells) + rng.uniform(-9.0, 0.0, cells)
        u = rng.choice([-1.0, 1.0], cells) * 10.0 ** exponent
        pr.prim[pr.N - 1 + d] = np.where(rng.random(cells) < 0.1, 0.0, u)
    f, g, W = orc.setup(pr)
    s = hrm.Solver.from_problem(pr, params=hrm.params_default(cfl=0.4, check=0))
    dt, _ = orc.dt(f, g, W, 0.4)
    W1 = orc.step(f, orc.make_params(), g, W, dt, 2)
    s.step(dt, 2)
    np.testing.assert_array_equal(s.get(hrm.FIELD_W), W1)
    s.close()


@pytest.mark.parametrize("cells", [4607, 4608, 13311, 13312, 20479, 20480])
def test_shared_midpoints_equal_the_oracle(hrm, orc, cells):
    """Lists around the lengths at which 8, 4, 2 and 1 lanes take a midpoint (no stencil is uniform)."""
    pr = disturbed([cells], 0, "none")
    rng = np.random.default_rng(cells)
    pr.prim[0] += 0.01 * rng.random(cells)
    pr.prim[pr.N - 1] += rng.random(cells)
    f, g, W = orc.setup(pr)
    s = hrm.Solver.from_problem(pr, params=hrm.params_default(cfl=0.4, check=0))
    dt, _ = orc.dt(f, g, W, 0.4)
    s.step(dt, 2)
    np.testing.assert_array_equal(s.get(hrm.FIELD_W), orc.step(f, orc.make_params(), g, W, dt, 2))
    s.close()

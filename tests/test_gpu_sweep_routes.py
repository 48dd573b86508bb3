"""Which sweep a grid takes -- lists of the non-uniform midpoints or, on small grids and with the first-order scheme, all
midpoints with their own test -- and how many lanes share an FP64 midpoint must not show in the results: FP64 against the
oracle on grids around the sizes where the rules switch, with every option of the midpoint body and states that set its
limiters off; the precision form against the batched form, which finds its uniform midpoints by tiles, and against its
own stages one at a time, which read every flux."""
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


def blocks(n, bc, N=3, rough=0.0, seed=3):
    """A uniform moving state with blocks of other states; `rough`: the share of cells with a random state of their own,
    volume fractions at both ends included."""
    rng = np.random.default_rng(seed)
    D, cells = len(n), int(np.prod(n))
    gamma, pinf, cv, q = P._species([P.BENCH_WATER, P.BENCH_AIR, P.BENCH_HELIUM][:N])
    one = np.ones(cells)
    prim = P._assemble(N, D, [0.3 * one, 0.5 * one][:N - 1], [(20.0 - 15.0 * d) * one for d in range(D)], 1.2e5 * one, 310.0 * one)
    x = np.meshgrid(*[np.arange(v) / v for v in n[::-1]], indexing="ij")[::-1]
    inside = np.ones_like(x[0], bool)
    for v in x:
        inside &= (v > 0.3) & (v < 0.55)
    inside = inside.reshape(-1)
    prim[0, inside] = 0.45
    prim[N + D - 1, inside] *= 1.3
    pick = rng.random(cells) < rough
    k = int(pick.sum())
    a = rng.choice([1e-8, 0.2, 0.6, 1.0 - 3e-8], k)
    prim[0, pick] = a
    if N == 3:
        prim[1, pick] = (1.0 - a) * rng.choice([1e-8, 0.5, 1.0 - 1e-8], k)
    for d in range(D):
        prim[N - 1 + d, pick] = rng.normal(0.0, 60.0, k)
    prim[N + D - 1, pick] = 10.0 ** rng.uniform(4.8, 5.6, k)
    pr = P.Problem("blocks", gamma, pinf, cv, q, list(n), [0.0] * D, [1.0 + 0.3 * d for d in range(D)], [bc] * (2 * D), prim,
                   cfl=0.4)
    if bc == 2:
        for b in range(2 * D):
            m = cells // n[b // 2]
            pr.boundary[b] = P._assemble(N, D, [np.full(m, 0.3), np.full(m, 0.5)][:N - 1],
                                         [np.full(m, 20.0 - 15.0 * d) for d in range(D)], np.full(m, 1.2e5), np.full(m, 310.0))
            pr.boundary[b][N + D, : (m + 1) // 2] += 5.0 * (b % 2)
    return pr


def ids(n):
    return "x".join(map(str, n))


OPTIONS = {"default": {}, "no_blend": {"blend": 0}, "no_limiters": {"limiters": 0}, "first_order": {"scheme": 1}, "gate": {}}


# no lists with 8, 4 and 2 lanes a midpoint; lists, all midpoints in them: 2 lanes and 1
@pytest.mark.parametrize("n", [[3000], [66, 60], [17, 15, 14], [9000], [100, 90], [21, 20, 22], [16384], [128, 128], [16, 32, 30],
                               [18001], [140, 129], [24, 25, 31], [22001], [150, 151], [31, 30, 29]], ids=ids)
@pytest.mark.parametrize("option", list(OPTIONS))
@pytest.mark.parametrize("N", [2, 3])
def test_fp64_bodies_equal_the_oracle(hrm, orc, n, option, N):
    import torch
    pr = blocks(n, 0, N, rough=1.0)
    f, g, W = orc.setup(pr)
    dt, _ = orc.dt(f, g, W, 0.4)
    kw = OPTIONS[option]
    s = hrm.Solver.from_problem(pr, params=hrm.params_default(cfl=0.4, check=0, **kw))
    gates = None
    if option == "gate":
        gates = [(np.random.default_rng(d).random(s.face_count(d)) < 0.5).astype(np.uint8) for d in range(pr.D)]
        for d in range(pr.D):
            s.set_gate(d, gates[d])
        s.set_params(hrm.params_default(cfl=0.4, check=0, learned=hrm.LEARNED_FIXED))
    s.step(dt, 2)
    with np.errstate(all="ignore"):
        ref = orc.step(f, orc.make_params(**kw), g, W, dt, 2, gates=gates, omp=gates is None)
    np.testing.assert_array_equal(s.get(hrm.FIELD_W), ref)
    s.close()


@pytest.mark.parametrize("n", [[16384], [16385], [128, 128], [257, 65], [25, 26, 25], [26, 26, 25]], ids=ids)
@pytest.mark.parametrize("bc", [0, 1, 2], ids=["transmissive", "periodic", "dirichlet"])
@pytest.mark.parametrize("rough", [0.0, 0.02])
def test_fp64_routes_equal_the_oracle(hrm, orc, n, bc, rough):
    import torch
    pr = blocks(n, bc, rough=rough)
    f, g, W = orc.setup(pr)
    dt, _ = orc.dt(f, g, W, 0.4)
    lam = orc.lambdas(f, g, W, dt)
    s = hrm.Solver.from_problem(pr, params=hrm.params_default(cfl=0.4, check=0))
    rhs = s.rhs(lam, torch.empty((pr.M, pr.ncells), dtype=torch.float64, device="cuda")).cpu().numpy()
    np.testing.assert_array_equal(rhs, orc.rhs(f, orc.make_params(), g, W, lam))
    s.step(dt, 3)
    np.testing.assert_array_equal(s.get(hrm.FIELD_W), orc.step(f, orc.make_params(), g, W, dt, 3, omp=True))
    s.close()


@pytest.mark.parametrize("n", [[256, 256], [257, 256], [513, 129]], ids=ids)
@pytest.mark.parametrize("bc", [0, 1], ids=["transmissive", "periodic"])
@pytest.mark.parametrize("rough", [0.0, 0.02, 1.0])
@pytest.mark.parametrize("N", [2, 3])
def test_precision_form_equals_the_batched_form(hrm, n, bc, rough, N):
    pr = blocks(n, bc, N, rough=rough)
    prm = hrm.params_default(cfl=0.4, check=0, precision=hrm.FP32)
    b = hrm.BatchSolver([pr], params=prm)
    b.step(3)
    s = hrm.Solver.from_problem(pr, params=prm)
    s.step(0.0, 3)
    np.testing.assert_array_equal(s.get(hrm.FIELD_W), b.get(0))
    s.close()


@pytest.mark.parametrize("n", [[3000], [100, 90], [20, 21, 22], [65536], [65537], [511, 129], [41, 40, 41]], ids=ids)
@pytest.mark.parametrize("bc", [0, 1, 2], ids=["transmissive", "periodic", "dirichlet"])
@pytest.mark.parametrize("option", ["default", "no_screen", "first_order", "gate", "euler"])
def test_precision_form_step_equals_its_stages(hrm, n, bc, option):
    pr = blocks(n, bc, rough=0.02)
    kw = {"no_screen": {"screen": 0}, "first_order": {"scheme": 1}, "euler": {"integrator": hrm.EULER}}.get(option, {})
    prm = hrm.params_default(cfl=0.4, check=0, precision=hrm.FP32, **kw)
    a, b = hrm.Solver.from_problem(pr, params=prm), hrm.Solver.from_problem(pr, params=prm)
    if option == "gate":
        for s in (a, b):
            for d in range(pr.D):
                s.set_gate(d, (np.random.default_rng(d).random(s.face_count(d)) < 0.5).astype(np.uint8))
            s.set_params(hrm.params_default(cfl=0.4, check=0, precision=hrm.FP32, learned=hrm.LEARNED_FIXED))
    for _ in range(3):
        a.step(0.0, 1)
        b.begin_step(b.step_tau())
        for k in range(b.stages()):
            b.stage(k)
    np.testing.assert_array_equal(a.get(hrm.FIELD_W), b.get(hrm.FIELD_W))
    a.close()
    b.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_route_follows_the_options_of_a_context(hrm, precision):
    """One context stepped with and without lists in turn (the first-order scheme has none) equals contexts that were
    given the same states."""
    pr = blocks([300, 231], 0, rough=0.02)
    prec = hrm.FP64 if precision == "fp64" else hrm.FP32
    s = hrm.Solver.from_problem(pr, params=hrm.params_default(cfl=0.4, check=0, precision=prec))
    for k in range(4):
        W = s.get(hrm.FIELD_W)
        prm = hrm.params_default(cfl=0.4, check=0, precision=prec, scheme=k % 2)
        s.set_params(prm)
        s.set(W)
        s.step(0.0, 2)
        o = hrm.Solver.from_problem(pr, params=prm)
        o.set(W)
        o.step(0.0, 2)
        np.testing.assert_array_equal(s.get(hrm.FIELD_W), o.get(hrm.FIELD_W))
        o.close()
    s.close()

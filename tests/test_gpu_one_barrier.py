"""The one-barrier solver's share shapes against the two-barrier schedule.

Both solve the same convex problem to the same residual, so their steps
agree within the tolerances of the oracle parity tests (centres 1e-6 D in
float64 at tol 1e-10, 2e-5 D mixed at tol 1e-6).  The sizes sit at the edges of the
kernel's layout: one block and its neighbours (32 rods a block until every SM has
one), the last share whose rods get eight lanes (96 rods a block at 768
workers) and the first that get two, a rod count just past a warp, shapes
with and without a warp for the block sums (768 and 256; 1024; two and four
blocks an SM), walls (the zero velocity row) and springs (bilateral slots), and a
solve_lcp in the caller's order (a halo of nearly every slot's other end).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2109_08206_gb300 as A  # noqa: E402
from paper_2109_08206_gb300 import workloads as W  # noqa: E402

from test_gpu_parity import dev, host, periodic_diff  # noqa: E402

pytestmark = pytest.mark.gpu

BAR = {A.FP64: (1e-10, 1e-6), A.MIXED: (1e-6, 2e-5)}
SOLVER_ONE, SOLVERS_TWO = 1, (2, 3)


@pytest.fixture(scope="module", autouse=True)
def _built():
    A.build()
    assert torch.cuda.is_available()


def system(n, seed=5, phi=0.06):
    box = max(W.box_for_fraction(n, 1.0, 10.0, phi), 12.5)
    return W.random_system(seed, n, box, forces="thermal", tol=1e-6)


def steps(s, precision, threads, bps, walls=None, springs=None):
    tol, bar = BAR[precision]
    out = []
    for barriers in (1, 2):
        nb = 0 if springs is None else len(springs["kappa"])
        with A.Context(A.params_of(s, precision=precision, tol=tol), s.n, max(64, 16 * s.n + nb)) as ctx:
            ctx.set_launch(threads, bps)
            ctx.set_solver_schedule(barriers)
            if walls is not None:
                ctx.set_walls(*walls)
            if springs is not None:
                ctx.set_springs(dev(springs["ends"], torch.int32), dev(springs["arms"]), dev(springs["kappa"]),
                                dev(springs["rest"]))
            x, q = dev(s.x), dev(s.quat)
            info = ctx.step(x, q, dev(s.f_nc))
            if info.n_pairs + nb > 0:
                assert info.solver == SOLVER_ONE if barriers == 1 else info.solver in SOLVERS_TWO
            out.append((host(x), host(q)))
    (x1, q1), (x2, q2) = out
    assert np.abs(periodic_diff(x1, x2, s.box)).max() <= bar
    assert np.abs(q1 - q2).max() <= bar


@pytest.mark.parametrize("precision", [A.FP64, A.MIXED])
@pytest.mark.parametrize("n", [2, 32, 33, 65, 96 * 152, 97 * 152])
def test_sizes(n, precision):
    steps(system(n), precision, 768, 0)


@pytest.mark.parametrize("precision", [A.FP64, A.MIXED])
@pytest.mark.parametrize("threads,bps", [(256, 1), (992, 1), (1024, 1), (512, 2), (256, 4)])
def test_launch_shapes(threads, bps, precision):
    steps(system({1: 3000, 2: 10000, 4: 20000}[bps]), precision, threads, bps)   # (every SM full of blocks)


@pytest.mark.parametrize("precision", [A.FP64, A.MIXED])
def test_walls_and_springs(precision):
    s = system(700)
    steps(s, precision, 768, 0, springs=W.spring_set(s, 300, seed=3, kappa=30.0))
    lo, hi = 2.0, s.box[2] - 14.0
    s.x[:, 2] = lo + 6.0 + s.x[:, 2] / s.box[2] * (hi - lo - 12.0)
    s.f_nc[:, 2] -= 3000.0
    steps(s, precision, 768, 0, walls=(2, lo, hi))


@pytest.mark.parametrize("n", [500, 30000])
def test_solve_lcp_in_caller_order(n):
    s = system(n)
    gam = []
    tol, _ = BAR[A.MIXED]
    for barriers in (1, 2):
        with A.Context(A.params_of(s, precision=A.MIXED, tol=tol), n, 12 * n) as ctx:
            ctx.set_solver_schedule(barriers)
            x, q, f = dev(s.x), dev(s.quat), dev(s.f_nc)
            pairs = ctx.build_neighbors(x, q)
            _, dgeom, lq = ctx.assemble_constraints(x, q, f, pairs)
            g, info = ctx.solve_lcp(q, pairs, dgeom, lq)
            assert info.solver == SOLVER_ONE if barriers == 1 else info.solver in SOLVERS_TWO
            # velocity D gamma, which is unique where gamma is not
            i, j = pairs[:, 0].long(), pairs[:, 1].long()
            F = torch.zeros((n, 6), dtype=torch.float64, device="cuda")
            F.index_add_(0, i, torch.cat([dgeom[:, 0:3], dgeom[:, 3:6]], 1) * g[:, None])
            F.index_add_(0, j, torch.cat([-dgeom[:, 0:3], -dgeom[:, 6:9]], 1) * g[:, None])
            gam.append(host(F))
    assert np.linalg.norm(gam[0] - gam[1]) <= 1e-3 * np.linalg.norm(gam[1])


def test_shapes_in_turn_on_one_context():
    s = system(20000)   # shares past the 48 KB a kernel may use without asking
    tol, _ = BAR[A.MIXED]
    shapes = [(768, 0), (1024, 0), (256, 1), (768, 0)]

    def one(ctx, threads, bps):
        ctx.set_launch(threads, bps)
        x, q = dev(s.x), dev(s.quat)
        assert ctx.step(x, q, dev(s.f_nc)).solver == SOLVER_ONE
        return host(x)

    params = A.params_of(s, precision=A.MIXED, tol=tol)
    with A.Context(params, s.n, 12 * s.n) as ctx:
        got = [one(ctx, *shape) for shape in shapes]
    for shape, x in zip(shapes, got):
        with A.Context(params, s.n, 12 * s.n) as ctx:
            assert np.array_equal(one(ctx, *shape), x)


@pytest.mark.parametrize("shape", [(768, 0), (1024, 0)])
def test_recorded_step_repeats_the_eager_one(shape):
    s = system(20000)   # past the line between the kernels with and without the barrier
    with A.Context(A.params_of(s, precision=A.MIXED, tol=1e-6), s.n, 12 * s.n) as ctx:
        ctx.set_launch(*shape)
        ctx.set_step_graph(True)
        x, q, f = dev(s.x), dev(s.quat), dev(s.f_nc)
        got = []
        for _ in range(4):   # eager, recorded, replayed twice
            x.copy_(dev(s.x))
            q.copy_(dev(s.quat))
            assert ctx.step(x, q, f).solver == SOLVER_ONE
            got.append(host(x).copy())
    assert all(np.array_equal(got[0], g) for g in got[1:])

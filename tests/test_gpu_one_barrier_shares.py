"""The one-barrier solver's launches: kernel, shared memory and what they cost."""
import pytest

torch = pytest.importorskip("torch")

import paper_2109_08206_gb300 as A  # noqa: E402

from test_gpu_one_barrier import SOLVER_ONE, SOLVERS_TWO, system  # noqa: E402
from test_gpu_parity import dev  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = {A.FP64: 1e-6, A.MIXED: 1e-5}


@pytest.fixture(scope="module", autouse=True)
def _built():
    A.build()
    assert torch.cuda.is_available()


def us_per_iteration(call, repeats=7):
    """Least solve time per iteration over the repeats, and the last call's info."""
    infos = [call() for _ in range(repeats)]
    return min(i.ms_solve for i in infos) * 1e3 / infos[-1].iters, infos[-1]


def timed_step(s, precision, threads, bps, barriers=1, graph=False):
    with A.Context(A.params_of(s, precision=precision, tol=TOL[precision]), s.n, 12 * s.n) as ctx:
        ctx.set_launch(threads, bps)
        ctx.set_solver_schedule(barriers)
        ctx.set_step_graph(graph)
        x, q, f = dev(s.x), dev(s.quat), dev(s.f_nc)
        x0, q0 = x.clone(), q.clone()

        def call():
            x.copy_(x0)
            q.copy_(q0)
            return ctx.step(x, q, f)

        if graph:
            call(), call()   # eager, recorded
        return us_per_iteration(call)


def timed_lcp(s, precision, barriers=1):
    with A.Context(A.params_of(s, precision=precision, tol=TOL[precision]), s.n, 12 * s.n) as ctx:
        ctx.set_solver_schedule(barriers)
        x, q, f = dev(s.x), dev(s.quat), dev(s.f_nc)
        pairs = ctx.build_neighbors(x, q)
        _, dgeom, lq = ctx.assemble_constraints(x, q, f, pairs)
        return us_per_iteration(lambda: ctx.solve_lcp(q, pairs, dgeom, lq)[1])


def test_float64_shares_leave_l1_for_the_spills():
    """An iteration of the one-barrier solver is no longer than one of the
    two-barrier schedule it stands in for (a tenth for the clock): where the
    launch took all the shared memory, the registers that the kernel spills
    went to L2 and this one was half as long again."""
    s = system(16000, phi=0.10)
    one, info = timed_lcp(s, A.FP64)
    two, info2 = timed_lcp(s, A.FP64, barriers=2)
    assert info.solver == SOLVER_ONE and info2.solver in SOLVERS_TWO
    assert one <= 1.1 * two, (one, two)


def test_shares_that_fill_an_sm_of_several_blocks_meet_at_a_barrier():
    """The same bound: here the share itself leaves no L1, and the kernel without
    spills is the faster one."""
    s = system(50000, phi=0.10)
    one, info = timed_step(s, A.MIXED, 256, 4)
    two, info2 = timed_step(s, A.MIXED, 256, 4, barriers=2)
    assert info.solver == SOLVER_ONE and info2.solver in SOLVERS_TWO
    assert one <= 1.1 * two, (one, two)


def test_recorded_step_asks_for_the_eager_steps_shared_memory():
    """The recorded solve is the eager one (a quarter for the clock and for what
    runs beside it)."""
    s = system(10000, phi=0.10)
    eager, info = timed_step(s, A.MIXED, 256, 4)
    recorded, info2 = timed_step(s, A.MIXED, 256, 4, graph=True)
    assert info.solver == info2.solver == SOLVER_ONE and info.iters == info2.iters
    assert recorded <= 1.25 * eager, (recorded, eager)


@pytest.mark.parametrize("precision", [A.FP64, A.MIXED])
def test_recorded_step_outgrown_by_its_shares(precision):
    """Rods that close in until their shares no longer fit what the recorded
    step asked for: that step runs eagerly, the next is recorded anew, and all of
    them give what eager steps give, on the way back as well."""
    s = system(3000)
    scales = [1.0, 1.0, 1.0, 0.6, 0.6, 0.6, 0.6, 1.0]
    got = []
    for graph in (False, True):
        with A.Context(A.params_of(s, precision=precision, tol=TOL[precision], max_iter=1_000_000), s.n, 64 * s.n) as ctx:
            ctx.set_step_graph(graph)
            x, q, f = dev(s.x), dev(s.quat), dev(s.f_nc)
            x0, q0 = x.clone(), q.clone()
            out = []
            for scale in scales:
                x.copy_(x0 * scale)
                q.copy_(q0)
                info = ctx.step(x, q, f)
                assert info.solver == SOLVER_ONE
                out.append((info, x.clone(), q.clone()))
            got.append(out)
    eager, recorded = got
    assert eager[3][0].n_pairs > 3 * eager[0][0].n_pairs
    for (a, xa, qa), (b, xb, qb) in zip(eager, recorded):
        assert (a.n_pairs, a.iters, a.residual) == (b.n_pairs, b.iters, b.residual)
        assert torch.equal(xa, xb) and torch.equal(qa, qb)
    launches = [info.launches for info, _, _ in recorded]
    replay, plain = launches[2], eager[2][0].launches
    assert replay != plain
    assert launches == [plain, replay, replay, plain, replay, replay, replay, replay]


@pytest.mark.parametrize("precision", [A.FP64, A.MIXED])
@pytest.mark.parametrize("threads", [768, 1024])   # with and without a warp of the sums' own
def test_waits_for_words_that_never_come_run_out(threads, precision):
    """A block that leaves after the first grid barrier: the others' waits for its
    velocities and sums run out, nothing moves, and the context goes on."""
    s = system(3000)
    with A.Context(A.params_of(s, precision=precision, tol=TOL[precision]), s.n, 12 * s.n) as ctx:
        ctx.set_launch(threads)
        x, q, f = dev(s.x), dev(s.quat), dev(s.f_nc)
        x0, q0 = x.clone(), q.clone()
        want = ctx.step(x, q, f)
        moved = x.clone(), q.clone()
        x.copy_(x0)
        q.copy_(q0)
        ctx.set_wait_limit(0.2)
        ctx.inject_fault(4)
        assert ctx.step(x, q, f, check=False).status == 4
        assert torch.equal(x, x0) and torch.equal(q, q0)
        ctx.set_wait_limit(5.0)
        info = ctx.step(x, q, f)
        assert info.solver == SOLVER_ONE and info.iters == want.iters
        assert torch.equal(x, moved[0]) and torch.equal(q, moved[1])

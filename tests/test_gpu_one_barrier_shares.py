"""The one-barrier solver's launches: kernel, shared memory and what they cost.

Its two kernels (tagged words, and the barrier form that large systems in the
caller's order take) and every layout of a block's share (velocities of other
blocks' rods in rows or polled slot by slot, the step's delta and g in shared or
global memory) sum in one order, so their solutions agree bit for bit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2109_08206_gb300 as A  # noqa: E402

from test_gpu_one_barrier import BAR, SOLVER_ONE, SOLVERS_TWO, steps, system  # noqa: E402
from test_gpu_parity import dev, host  # noqa: E402

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


# ------------------------------------------------------------ same bits
def cell_order(s):
    """The rods in the step's order: Morton order of their cells, then by id."""
    box = np.asarray(s.box)
    nc = np.maximum(1, np.floor(box / ((s.length + s.diameter + s.delta_c) * (1.0 + 1e-9)))).astype(int)
    cell = np.minimum(((s.x - box * np.floor(s.x / box)) / (box / nc)).astype(int), nc - 1)
    key = np.zeros(s.n, dtype=np.int64)
    for bit in range(10):
        for k in range(3):
            key |= ((cell[:, k] >> bit) & 1) << (3 * bit + k)
    return np.argsort(key, kind="stable")


def layouts(pairs, n, esize, blocks):
    """Of a launch of one block an SM (152 of them): the largest share's bytes, and for how many
    blocks the velocities of other blocks' rods, and delta and g, find room."""
    def up(b):
        return (b + 15) // 16 * 16

    P, Q = pairs[:, 0].astype(np.int64), pairs[:, 1].astype(np.int64)
    row_p = np.concatenate([[0], np.cumsum(np.bincount(P, minlength=n))])
    row_q = np.concatenate([[0], np.cumsum(np.bincount(Q, minlength=n))])
    work = row_p + 2 * row_q + 2 * np.arange(n + 1)
    start = [int(np.searchsorted(work, work[n] * b // blocks)) for b in range(blocks)] + [n]
    by_q = np.argsort(Q, kind="stable")
    need, shares = 0, []
    for r0, r1 in zip(start, start[1:]):
        c0, c1 = row_p[r0], row_p[r1]
        other = by_q[row_q[r0]:row_q[r1]]
        ghosts = other[(other < c0) | (other >= c1)]
        far = Q[c0:c1]
        halo = len(np.unique(np.concatenate([far[(far < r0) | (far >= r1)], P[ghosts]])))
        nc, nr, nq, ng = c1 - c0, r1 - r0, len(other), len(ghosts)
        nt = nc + ng
        per_rod = np.diff(row_p[r0:r1 + 1]) + np.diff(row_q[r0:r1 + 1])
        entries = int((4 * ((per_rod + 3) // 4)).sum())
        need = max(need, up(4 * ((blocks + 3) // 4 * 4) * esize) + up((13 * nt + 9 * nr) * esize) +
                   up((nt + ng + 2 * nr + 2) * 4) + up((nt + nq + nr) * 2))
        used = up((12 * (nt + 1) + 3 * nr) * esize + 4 * nt + 2 * entries + 4 * nr + 24) + 6 * (nr + 1) * esize
        shares.append((used, 6 * halo * esize, 2 * nc * esize))
    room = need + need * 8 // 13
    for kb in (164, 196):
        most = kb * 1024 - 2048 - 1200
        if need <= most:
            room = min(room, most)
            break
    room = min(room, 230000)
    rows = [used + h <= room for used, h, _ in shares]
    spare = [used + (h if fits else 0) + d <= room for (used, h, d), fits in zip(shares, rows)]
    return int(need), sum(rows), sum(spare)


@pytest.mark.parametrize("n,precision,spills", [(17000, A.FP64, False), (17000, A.MIXED, False),
                                                (35500, A.FP64, True), (72000, A.MIXED, True)])
def test_barrier_form_repeats_the_tagged_form(n, precision, spills):
    """Rods numbered in the step's order make solve_lcp (the barrier form above
    16,000 rods) the solve of step (tagged words), with shares that hold all of
    their data in shared memory and shares that leave delta and g to global memory
    or poll the other blocks' velocities."""
    s = system(n, phi=0.10)
    order = cell_order(s)
    tol = TOL[precision]
    x, q, f = dev(s.x[order]), dev(s.quat[order]), dev(s.f_nc[order])
    rows = 12 * n
    with A.Context(A.params_of(s, precision=precision, tol=tol), n, rows) as ctx:
        pairs = ctx.build_neighbors(x, q)
        _, dgeom, lq = ctx.assemble_constraints(x, q, f, pairs)
        got, lcp = ctx.solve_lcp(q, pairs, dgeom, lq)
        _, halos, spares = layouts(host(pairs), n, 8 if precision == A.FP64 else 4, 152)
        assert (spares < 152) == spills   # (of the float64 ones a block polls as well: halos is 151)
        listed = torch.zeros((rows, 3), dtype=torch.int32, device="cuda")
        want = torch.zeros(rows, dtype=torch.float64, device="cuda")
        step = ctx.step(x, q, f, pairs_out=listed, gamma_out=want)
    assert step.solver == lcp.solver == SOLVER_ONE
    assert torch.equal(listed[:step.n_pairs], pairs)
    assert (step.iters, step.residual) == (lcp.iters, lcp.residual) and lcp.residual <= tol
    assert torch.equal(want[:step.n_pairs], got)


# ------------------------------------------- against the two-barrier schedule
def displacement(s, q, pairs, dgeom, g):
    """h M D gamma of the centres, unique where gamma is not."""
    i, j = pairs[:, 0].long(), pairs[:, 1].long()
    F = torch.zeros((s.n, 3), dtype=torch.float64, device="cuda")
    F.index_add_(0, i, dgeom[:, 0:3] * g[:, None])
    F.index_add_(0, j, -dgeom[:, 0:3] * g[:, None])
    qs = q / q.norm(dim=1, keepdim=True)
    w, a, b, c = qs.unbind(1)
    p = torch.stack([2 * (a * c + w * b), 2 * (b * c - w * a), w * w - a * a - b * b + c * c], 1)
    perp = 4 * np.pi * s.viscosity * s.length / np.log(2 * s.length / s.diameter)
    return host(s.dt / perp * (F + p * (p * F).sum(1, keepdim=True)))


@pytest.mark.parametrize("n,precision,phi", [(16001, A.FP64, 0.06), (16001, A.MIXED, 0.06), (30000, A.FP64, 0.06),
                                             (16000, A.FP64, 0.10), (16000, A.MIXED, 0.20)])
def test_solve_lcp_in_caller_order(n, precision, phi):
    """The barrier form (above 16,000 rods), and the tagged one where some blocks
    poll the other blocks' velocities for want of room."""
    s = system(n, phi=phi)
    tol, bar = BAR[precision]
    got = []
    for barriers in (1, 2):
        with A.Context(A.params_of(s, precision=precision, tol=tol), n, 12 * n) as ctx:
            ctx.set_solver_schedule(barriers)
            x, q, f = dev(s.x), dev(s.quat), dev(s.f_nc)
            pairs = ctx.build_neighbors(x, q)
            _, dgeom, lq = ctx.assemble_constraints(x, q, f, pairs)
            if n <= 16000:
                _, halos, _ = layouts(host(pairs), n, 8 if precision == A.FP64 else 4, 152)
                assert halos < 152
            g, info = ctx.solve_lcp(q, pairs, dgeom, lq)
            assert info.solver == SOLVER_ONE if barriers == 1 else info.solver in SOLVERS_TWO
            assert info.residual <= tol
            got.append(displacement(s, q, pairs, dgeom, g))
    if phi < 0.2:
        assert np.abs(got[0] - got[1]).max() <= bar
    else:   # a dense pack: forces far from unique, motion in the mean
        assert np.linalg.norm(got[0] - got[1]) <= 1e-3 * np.linalg.norm(got[1])


@pytest.mark.parametrize("precision", [A.FP64, A.MIXED])
def test_two_rods_in_contact(precision):
    """One block, one slot."""
    s = system(2, seed=2)
    with A.Context(A.params_of(s, precision=precision), 2, 64) as ctx:
        assert len(ctx.build_neighbors(dev(s.x), dev(s.quat))) == 1
    steps(s, precision, 768, 0)

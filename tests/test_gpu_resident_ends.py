"""Where the resident PCG ends or has to give way: whatever it cannot do, the phase kernels do,
with the results that they had, and what one call does leaves others as they were."""
import threading

import numpy as np
import pytest

import oracle
from paper_2511_06824_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PHYS = inputs.phys_vector()


@pytest.fixture(scope="module")
def g():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_06824_gb300 import build, gmaf
    build.build()
    gmaf.load()
    return gmaf


def resident(info):
    """Whether the solve took the resident kernel (ids 50000000 + 1000 VEC + 10 RR)."""
    return info["kernel_variant"] // 10000000 == 5


def system(nth, nz, K, seed):
    rng = np.random.default_rng(seed)
    tex = inputs.dimple_texture(rng)
    st, *arrs = oracle.assemble_joint(nth, nz, PHYS, tex, [inputs.random_state(rng) for _ in range(K)])
    assert st == 0
    return [torch.from_numpy(np.ascontiguousarray(a).ravel()).cuda() for a in arrs]


def solve(g, nth, nz, K, arrs, budget=0, start=None, allow=None, **opts):
    """Status, iterations, true residual, details and solution, in a context of its own."""
    p = torch.full((K * nth * nz,), 5.0, dtype=torch.float64, device="cuda")
    if start is not None:
        p.copy_(start)
        opts["zero_init"] = 0
    with g.Context(hbm_budget_bytes=budget) as c:
        st, it, rel = g.gmaf_solve_joint(c.handle, nth, nz, K, *arrs, p, g.solver_opts(**{"eps": 1e-10, **opts}),
                                         allow=allow or (g.GMAF_OK,))
        info = g.gmaf_last_solve_info(c.handle)
    return st, it, rel, info, p


def rel_l2(a, b):
    return float(torch.linalg.norm(a - b) / torch.linalg.norm(b))


def test_threads_with_contexts_of_their_own(g):
    """Threads, each with a context and a stream, solve grids that take the same kernel with
    different amounts of shared memory, over and over: no launch fails, and every result is bit for
    bit that of the solve alone."""
    shapes = [(60, 40, 9), (128, 64, 4), (512, 304, 1), (60, 40, 2)]
    kw = dict(eps=1e-6, max_iter=2)
    arrs = [system(*s, 3) for s in shapes]
    refs = [solve(g, *s, a, allow=(g.GMAF_NOT_CONVERGED,), **kw)[4] for s, a in zip(shapes, arrs)]
    failed = []

    def work(q):
        try:
            stream = torch.cuda.Stream()
            p = torch.zeros_like(refs[q])
            torch.cuda.synchronize()
            with g.Context(stream=stream.cuda_stream) as c:
                for _ in range(4000):
                    st, _, _ = g.gmaf_solve_joint(c.handle, *shapes[q], *arrs[q], p, g.solver_opts(**kw),
                                                  allow=tuple(range(-8, 1)))
                    if st != g.GMAF_NOT_CONVERGED:
                        failed.append((q, g.status_string(st)))
                        break
                if not resident(g.gmaf_last_solve_info(c.handle)) or not torch.equal(p, refs[q]):
                    failed.append((q, "result"))
        except Exception as e:                      # noqa: BLE001
            failed.append((q, repr(e)))

    ts = [threading.Thread(target=work, args=(q,)) for q in range(len(shapes))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not failed, failed


# norms whose squares are subnormal, just above that, where only the residual's are, and next to
# the largest double
@pytest.mark.parametrize("power", [-520, -485, -440, 505])
@pytest.mark.parametrize("precision,criterion", [(0, 0), (0, 1), (1, 0)])
def test_sources_at_the_ends_of_the_range(g, monkeypatch, power, precision, criterion):
    """The sums over blocks are fixed-point numbers whose scale is a normal exponent some way from
    either end: beyond, the phase kernels solve the system, from the same start."""
    nth, nz, K = 64, 20, 3
    D, aE, aN, S = system(nth, nz, K, 9)
    unit = 2.0 ** -np.floor(np.log2(float(D.max())))            # a diagonal of order one
    S = S * 2.0 ** (power - np.floor(np.log2(float(torch.linalg.norm(S)))))
    arrs = [D * unit, aE * unit, aN * unit, S]
    start = 0.5 * S
    kw = dict(precision=precision, criterion=criterion, start=start, max_iter=20000,
              allow=(g.GMAF_OK, g.GMAF_NOT_CONVERGED, g.GMAF_NONFINITE))
    monkeypatch.setenv("GMAF_NO_TUNE", "1")
    a = solve(g, nth, nz, K, arrs, **kw)
    monkeypatch.setenv("GMAF_VARIANT", "604322" if precision else "2322")
    b = solve(g, nth, nz, K, arrs, **kw)
    assert not resident(b[3])
    assert a[0] == b[0] and bool(a[4].any())
    if resident(a[3]):
        assert rel_l2(a[4], b[4]) <= 1e-8
    else:
        assert a[1] == b[1] and torch.equal(a[4], b[4])
    if power == -440:
        assert a[0] == g.GMAF_OK


@pytest.mark.parametrize("fill", [0.95, 0.5, 0.999])
def test_sums_with_the_largest_low_limbs(g, monkeypatch, fill):
    """152 full blocks whose warps all have the same sum of squares, its bits below the 22 leading
    ones `fill` of the most they can be: the low halves of the blocks' fixed-point sums are then as
    large as they get.  ||r|| / ||b|| of a start, without an iteration, to rounding."""
    nth, nz, K = 512, 304, 1
    D, aE, aN, _ = system(nth, nz, K, 4)
    # 64 cells a warp: a sum of 1 + fill / 2^22
    S = torch.full((K * nth * nz,), float(np.sqrt((1.0 + fill * 2.0 ** -22) / 64.0)), dtype=torch.float64, device="cuda")
    start = torch.linspace(0.0, 1.0, K * nth * nz, dtype=torch.float64, device="cuda") / float(D.max())
    kw = dict(start=start, max_iter=0, allow=(g.GMAF_NOT_CONVERGED,))
    a = solve(g, nth, nz, K, [D, aE, aN, S], **kw)[3]
    monkeypatch.setenv("GMAF_VARIANT", "1001003")
    b = solve(g, nth, nz, K, [D, aE, aN, S], **kw)[3]
    assert resident(a) and not resident(b)
    assert abs(a["rel_residual"] / b["rel_residual"] - 1.0) <= 1e-13


@pytest.mark.parametrize("nth,nz,K,precision,criterion,forced", [
    (64, 32, 1, 0, 0, 2322), (132, 45, 9, 1, 0, 604322), (130, 45, 9, 0, 1, 2322),
    (512, 250, 9, 0, 0, 2322), (640, 200, 9, 1, 0, 604322), (700, 300, 9, 1, 0, 604322),
])
def test_a_wait_that_runs_out_gives_way_to_the_phase_kernels(g, monkeypatch, nth, nz, K, precision,
                                                             criterion, forced):
    """A block that waits longer than the limit (here one poll) ends the resident run, as it would
    when other work kept some of the blocks off the GPU: the phase kernels then solve the system,
    from the start that was given, and the context goes on."""
    arrs = system(nth, nz, K, 8)
    kw = dict(precision=precision, criterion=criterion, eps=1e-8)
    monkeypatch.setenv("GMAF_NO_TUNE", "1")
    monkeypatch.setenv("GMAF_RESIDENT_POLLS", "1")
    p = torch.full((K * nth * nz,), 5.0, dtype=torch.float64, device="cuda")
    with g.Context() as c:
        for _ in range(2):
            st, it, _ = g.gmaf_solve_joint(c.handle, nth, nz, K, *arrs, p, g.solver_opts(**kw))
            assert st == 0 and g.gmaf_last_solve_info(c.handle)["kernel_variant"] == forced
    monkeypatch.delenv("GMAF_RESIDENT_POLLS")
    monkeypatch.setenv("GMAF_VARIANT", str(forced))
    ref = solve(g, nth, nz, K, arrs, **kw)
    assert it == ref[1] and torch.equal(p, ref[4])
    monkeypatch.delenv("GMAF_VARIANT")
    assert resident(solve(g, nth, nz, K, arrs, **kw)[3])


# a small system that takes the resident run, and a large one with the budget that the phase kernels
# need for it; the first one's scaled matrix, with ASSOR-I's diagonal, takes more than that
@pytest.mark.parametrize("small,large,forced,opts", [
    ((256, 128, 4), (1000, 250, 4), 2322, dict(precond=2)),
    ((512, 250, 9), (640, 300, 9), 2322, {}),
    ((256, 128, 9), (640, 300, 9), 2322, dict(criterion=1)),
    ((512, 250, 9), (1028, 290, 9), 604322, dict(precision=1)),
    ((640, 200, 9), (700, 300, 9), 604322, dict(precision=1)),
])
def test_budgets_that_were_enough_still_are(g, monkeypatch, small, large, forced, opts):
    """A budget of what the phase kernels hold, to the byte: the solve succeeds, also after a smaller
    one in the same context, and stays within it."""
    sizes = (small, large)
    arrs = [system(*s, 2) for s in sizes]
    ps = [torch.zeros_like(a[3]) for a in arrs]
    o = g.solver_opts(eps=1e-6, **opts)
    monkeypatch.setenv("GMAF_NO_TUNE", "1")
    monkeypatch.setenv("GMAF_VARIANT", str(forced))
    with g.Context() as c:
        for k in (0, 1):
            g.gmaf_solve_joint(c.handle, *sizes[k], *arrs[k], ps[k], o)
            if opts.get("criterion", 0) == 0:
                assert g.gmaf_last_solve_info(c.handle)["kernel_variant"] == forced
        held = g.gmaf_workspace_bytes(c.handle)
    refs = [p.clone() for p in ps]
    monkeypatch.delenv("GMAF_VARIANT")
    with g.Context() as c:
        g.gmaf_solve_joint(c.handle, *sizes[0], *arrs[0], ps[0], o)
        assert resident(g.gmaf_last_solve_info(c.handle))
    for order in ((1,), (0, 1, 0, 1)):
        with g.Context(hbm_budget_bytes=held) as c:
            for k in order:
                ps[k].fill_(7.0)
                st, _, _ = g.gmaf_solve_joint(c.handle, *sizes[k], *arrs[k], ps[k], o, allow=tuple(range(-8, 1)))
                assert st == 0, (order, k, g.status_string(st))
                assert g.gmaf_workspace_bytes(c.handle) <= held
                assert rel_l2(ps[k], refs[k]) <= 1e-3


# grids and tolerances at which a scaled run ends between 1.25 and 10 times its tolerance
@pytest.mark.parametrize("nth,nz,K,eps,criterion", [
    (512, 250, 9, 3e-14, 0), (1000, 250, 4, 1e-13, 0), (1000, 250, 4, 4e-14, 0), (1024, 250, 9, 5e-14, 0),
    (1000, 250, 4, 1e-13, 1), (1000, 250, 4, 5e-14, 1),
])
def test_a_restart_that_is_cut_off_takes_nothing_back(g, nth, nz, K, eps, criterion):
    """A first run that ends within ten times the tolerance is the solution, whether or not there
    are iterations left for the restart that would bring it closer."""
    arrs = system(nth, nz, K, nth)
    kw = dict(eps=eps, criterion=criterion, allow=(g.GMAF_OK, g.GMAF_NOT_CONVERGED))
    end = solve(g, nth, nz, K, arrs, **kw)
    assert end[0] == 0 and end[3]["restarts"] >= 1
    # the first run's count: the smallest budget that is enough
    lo, hi = 1, end[1]
    while lo < hi:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if solve(g, nth, nz, K, arrs, max_iter=mid, **kw)[0] == 0 else (mid + 1, hi)
    first = solve(g, nth, nz, K, arrs, max_iter=lo, **kw)
    assert first[0] == 0 and first[2] <= 10.0 * eps
    for more in (1, 2, 5, 20):
        st, it, rel, info, p = solve(g, nth, nz, K, arrs, max_iter=lo + more, **kw)
        assert st == 0 and rel <= first[2], (more, info)
        assert criterion == 1 or rel < first[2] or torch.equal(p, first[4])
    for more in range(1, min(40, lo)):
        assert solve(g, nth, nz, K, arrs, max_iter=lo - more, **kw)[0] == g.GMAF_NOT_CONVERGED


# (n_theta, n_z, resident for a diagonal that is the couplings' sum)
@pytest.mark.parametrize("nth,nz,fits", [(700, 300, True), (1028, 290, False)])
@pytest.mark.parametrize("where", ["everywhere", "one cell"])
def test_a_diagonal_with_a_term_of_its_own(g, monkeypatch, nth, nz, fits, where):
    """Forms that rebuild the diagonal from the couplings are for systems whose diagonal is their
    sum: with anything added to it (here 2 %) the diagonal is read, and the solve converges to what
    FP64 gives."""
    K = 9
    D, aE, aN, S = system(nth, nz, K, nth)
    monkeypatch.setenv("GMAF_VARIANT", "10604322")
    plain = solve(g, nth, nz, K, [D, aE, aN, S], precision=1)[3]
    assert plain["kernel_variant"] == 10604322
    monkeypatch.delenv("GMAF_VARIANT")
    assert resident(solve(g, nth, nz, K, [D, aE, aN, S], precision=1)[3]) == fits
    more = D.clone()
    if where == "everywhere":
        more *= 1.02
    else:
        more[(K - 1) * nth * nz + (nz // 2) * nth + 7] *= 1.02
    arrs = [more, aE, aN, S]
    kw = dict(max_iter=20000, allow=(g.GMAF_OK, g.GMAF_NOT_CONVERGED, g.GMAF_NONFINITE))
    ref = solve(g, nth, nz, K, arrs, **kw)
    for variant in (None, "10604322"):
        if variant:
            monkeypatch.setenv("GMAF_VARIANT", variant)
        st, it, rel, info, p = solve(g, nth, nz, K, arrs, precision=1, **kw)
        assert st == 0 and info["kernel_variant"] not in (10604322, 50004160)
        assert rel_l2(p, ref[4]) <= 1e-6


@pytest.mark.parametrize("nth,nz,K", [(64, 32, 1), (96, 48, 9), (132, 45, 9), (256, 128, 9), (512, 256, 9), (640, 200, 9)])
@pytest.mark.parametrize("iters", [1, 3, 30, 100000])
def test_mixed_runs_are_those_of_the_phase_kernels(g, monkeypatch, nth, nz, K, iters):
    """Resident runs of up to 8 rows and the phase kernels of four columns a lane take the same
    FP32 operations in the same order, and the norm of the FP64 residual is added up in that
    kernel's order.  The grid's other sums are added in another order, but agree once they are
    rounded to FP32: the same solution, to the last bit."""
    arrs = system(nth, nz, K, nth)
    kw = dict(precision=1, eps=1e-13, max_iter=iters, allow=(g.GMAF_OK, g.GMAF_NOT_CONVERGED))
    a = solve(g, nth, nz, K, arrs, **kw)
    monkeypatch.setenv("GMAF_VARIANT", "604322")
    b = solve(g, nth, nz, K, arrs, **kw)
    assert resident(a[3]) and b[3]["kernel_variant"] == 604322
    assert a[0] == b[0] and a[1] == b[1] and torch.equal(a[4], b[4])

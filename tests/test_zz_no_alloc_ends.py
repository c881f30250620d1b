"""Where the resident run of the allocation-free solve ends or gives way, as gmaf_solve_joint's does.

The file name puts it after the test that first loads the scratch array."""
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


def system(nth, nz, K, seed):
    rng = np.random.default_rng(seed)
    tex = inputs.dimple_texture(rng)
    st, *arrs = oracle.assemble_joint(nth, nz, PHYS, tex, [inputs.random_state(rng) for _ in range(K)])
    assert st == 0
    return [torch.from_numpy(np.ascontiguousarray(a).ravel()).cuda() for a in arrs]


@pytest.mark.parametrize("power", [-520, -485, -440, 505])
def test_sources_at_the_ends_of_the_range(g, monkeypatch, power):
    """Where sums of squares leave the range of the resident run's sums, the phase kernels solve the
    system from the same start, as in gmaf_solve_joint."""
    nth, nz, K = 64, 20, 3
    D, aE, aN, S = system(nth, nz, K, 9)
    unit = 2.0 ** -np.floor(np.log2(float(D.max())))            # a diagonal of order one
    S = S * 2.0 ** (power - np.floor(np.log2(float(torch.linalg.norm(S)))))
    arrs = [D * unit, aE * unit, aN * unit, S]
    opts = g.solver_opts(eps=1e-10, zero_init=0, max_iter=20000)
    allow = (g.GMAF_OK, g.GMAF_NOT_CONVERGED, g.GMAF_NONFINITE)
    monkeypatch.setenv("GMAF_VARIANT", "2322")
    p, q = 0.5 * S, 0.5 * S
    with g.Context() as c:
        st, it, rel = g.gmaf_solve_joint(c.handle, nth, nz, K, *arrs, p, opts, allow=allow)
    stq, itq, relq = g.gmaf_solve_joint_noalloc(nth, nz, K, *arrs, q, opts, allow=allow)
    assert stq == st and itq == it and bool(q.any())
    if st == g.GMAF_OK and power > -500:
        assert float(torch.linalg.norm(p - q) / torch.linalg.norm(p)) <= 1e-8


@pytest.mark.parametrize("nth,nz,K", [(64, 32, 1), (512, 250, 9)])
def test_a_wait_that_runs_out_gives_way_to_the_phase_kernels(g, monkeypatch, nth, nz, K):
    """A resident run whose blocks wait longer than the limit (here one poll) ends, and the phase
    kernels solve the system; the next call takes the resident run again."""
    arrs = system(nth, nz, K, 8)
    opts = g.solver_opts(eps=1e-8)
    p, q, r = (torch.full((K * nth * nz,), 3.0, dtype=torch.float64, device="cuda") for _ in range(3))
    monkeypatch.setenv("GMAF_VARIANT", "2322")
    with g.Context() as c:
        st, it, rel = g.gmaf_solve_joint(c.handle, nth, nz, K, *arrs, p, opts)
    monkeypatch.setenv("GMAF_RESIDENT_POLLS", "1")
    stq, itq, relq = g.gmaf_solve_joint_noalloc(nth, nz, K, *arrs, q, opts)
    monkeypatch.delenv("GMAF_RESIDENT_POLLS")
    str_, itr, relr = g.gmaf_solve_joint_noalloc(nth, nz, K, *arrs, r, opts)
    assert st == stq == str_ == 0 and itq == it and abs(itr - it) <= 2 and relq <= 1e-7
    assert float(torch.linalg.norm(p - q) / torch.linalg.norm(p)) <= 1e-10
    assert not torch.equal(q, r) and float(torch.linalg.norm(p - r) / torch.linalg.norm(p)) <= 1e-6


@pytest.mark.parametrize("eps", [1e-13, 4e-14])
def test_a_restart_that_is_cut_off_takes_nothing_back(g, eps):
    """A first run that ends within ten times the tolerance is the solution, whether or not there
    are iterations left for the restart that would bring it closer."""
    nth, nz, K = 1000, 250, 4
    arrs = system(nth, nz, K, nth)
    p = torch.zeros(K * nth * nz, dtype=torch.float64, device="cuda")

    def run(max_iter):
        return g.gmaf_solve_joint_noalloc(nth, nz, K, *arrs, p, g.solver_opts(eps=eps, max_iter=max_iter),
                                          allow=(g.GMAF_OK, g.GMAF_NOT_CONVERGED))

    st, hi, _ = run(100000)
    assert st == 0
    lo, most = 1, hi
    while lo < hi:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if run(mid)[0] == 0 else (mid + 1, hi)
    st, it, first = run(lo)
    assert st == 0 and it == lo < most and first <= 10.0 * eps
    q = p.clone()
    for more in (1, 2, 5, 20):
        st, it, rel = run(lo + more)
        assert st == 0 and (rel < first or torch.equal(p, q))
    for more in range(1, 40):
        assert run(lo - more)[0] == g.GMAF_NOT_CONVERGED

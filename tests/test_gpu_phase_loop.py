"""The phase kernels' own loops on systems that fit on the SMs, where a solve takes the resident run
unless a variant is asked for: graph against host loop, event timing, the loop guard of finish_b, and
the refinement driven from the host.  Every arm asserts the variant that it ran."""
import numpy as np
import pytest

import oracle
from paper_2511_06824_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PHYS = inputs.phys_vector()
FORMS = [(0, 2322), (0, 202322), (0, 1001003), (1, 604322), (1, 4322), (1, 10604322)]


@pytest.fixture(scope="module")
def g():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_06824_gb300 import build, gmaf
    build.build()
    gmaf.load()
    return gmaf


@pytest.fixture(scope="module")
def problem():
    nth, nz, K = 132, 45, 9
    rng = np.random.default_rng(31)
    tex = inputs.dimple_texture(rng)
    st, *host = oracle.assemble_joint(nth, nz, PHYS, tex, [inputs.random_state(rng) for _ in range(K)])
    assert st == 0
    return (nth, nz, K), host, [torch.from_numpy(np.ascontiguousarray(a).ravel()).cuda() for a in host]


def run(g, c, problem, variant, allow=(), **opts):
    (nth, nz, K), _, arrs = problem
    p = torch.zeros(K * nth * nz, dtype=torch.float64, device="cuda")
    st, it, rel = g.gmaf_solve_joint(c.handle, nth, nz, K, *arrs, p, g.solver_opts(**opts), allow=allow)
    info = g.gmaf_last_solve_info(c.handle)
    assert info["kernel_variant"] == variant and info["status"] == st
    return p, st, it, rel, info


@pytest.mark.parametrize("precision,variant", FORMS)
def test_graph_host_loop_and_event_timing_agree_bitwise(g, monkeypatch, problem, precision, variant):
    monkeypatch.setenv("GMAF_VARIANT", str(variant))
    outs = []
    with g.Context() as c:
        outs += [run(g, c, problem, variant, precision=precision)[0] for _ in range(2)]
        g.gmaf_set_phase_timing(c.handle, True)
        p, _, it, _, _ = run(g, c, problem, variant, precision=precision)
        t = g.gmaf_phase_timing(c.handle)
        outs.append(p)
        g.gmaf_set_phase_timing(c.handle, False)
        outs.append(run(g, c, problem, variant, precision=precision)[0])
    monkeypatch.setenv("GMAF_NO_GRAPH", "1")
    with g.Context() as c:
        outs.append(run(g, c, problem, variant, precision=precision)[0])
    assert all(torch.equal(p, outs[0]) for p in outs)
    # one launch of either phase an iteration, as the events counted them
    assert t["phase_a"][1] >= it and t["phase_b"][1] >= it and t["phase_a"][0] > 0
    assert t["resid64"][1] >= 1


@pytest.mark.parametrize("no_graph", ["0", "1"])
@pytest.mark.parametrize("precision,variant", FORMS)
def test_loop_guard_expires_in_the_phase_kernels(g, monkeypatch, problem, precision, variant, no_graph):
    monkeypatch.setenv("GMAF_VARIANT", str(variant))
    monkeypatch.setenv("GMAF_NO_GRAPH", no_graph)
    monkeypatch.setenv("GMAF_LOOP_GUARD", "5")
    with g.Context() as c:
        _, st, _, _, info = run(g, c, problem, variant, allow=(g.GMAF_TIMEOUT,), precision=precision, eps=1e-12)
    assert st == g.GMAF_TIMEOUT and info["iterations"] <= 8
    monkeypatch.delenv("GMAF_LOOP_GUARD")
    with g.Context() as c:
        _, st, it, rel, _ = run(g, c, problem, variant, precision=precision, eps=1e-12)
    assert st == g.GMAF_OK and it > 8 and rel <= 1e-11


@pytest.mark.parametrize("restart,delta", [("1", "0.1"), ("0", "0.1"), ("0", "0.3"), ("0", "0.001")])
@pytest.mark.parametrize("variant", [604322, 4322])
def test_refinement_from_the_host_matches_the_oracle(g, monkeypatch, problem, restart, delta, variant):
    monkeypatch.setenv("GMAF_VARIANT", str(variant))
    monkeypatch.setenv("GMAF_MIXED_RESTART", restart)
    monkeypatch.setenv("GMAF_RELIABLE_DELTA", delta)
    (nth, nz, K), host, _ = problem
    st, po, ito, _, _ = oracle.solve_joint(nth, nz, *host, precond=1, omega=1.2, eps=1e-10)
    assert st == 0
    with g.Context() as c:
        p, _, it, rel, info = run(g, c, problem, variant, precision=1, eps=1e-10)
    assert rel <= 1e-10 and info["outer_iterations"] >= 2
    assert np.linalg.norm(p.cpu().numpy() - po.ravel()) <= 1e-6 * np.linalg.norm(po)
    if restart == "0" and delta != "0.001":
        assert it <= 1.1 * ito + 10

"""The allocation-free solve on systems that fit on the SMs: the same resident runs as
gmaf_solve_joint's, in every form of the kernel (registers, tensor memory, couplings streamed),
just beyond its fit (the host-driven loop), from a start, through a restart, and without a byte of
device memory taken after the first call.

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


def _problem(nth, nz, K, seed):
    rng = np.random.default_rng(seed)
    tex = inputs.dimple_texture(rng)
    st, *a = oracle.assemble_joint(nth, nz, PHYS, tex, [inputs.random_state(rng) for _ in range(K)])
    assert st == 0
    return [torch.from_numpy(np.ascontiguousarray(x).ravel()).cuda() for x in a]


def test_forms_match_solve_joint_and_allocate_nothing(g):
    small = _problem(64, 32, 1, 0)
    p = torch.empty(64 * 32, dtype=torch.float64, device="cuda")
    g.gmaf_solve_joint_noalloc(64, 32, 1, *small, p, g.solver_opts(eps=1e-10))
    for nth, nz, K, precond in [(64, 32, 1, 1), (131, 45, 9, 0), (256, 128, 9, 1), (512, 200, 9, 1),
                                (700, 200, 4, 2), (700, 384, 5, 1), (640, 300, 9, 1)]:
        arrs = _problem(nth, nz, K, nth + nz)
        n = K * nth * nz
        ref = torch.zeros(n, dtype=torch.float64, device="cuda")
        p = torch.full((n,), 7.0, dtype=torch.float64, device="cuda")
        with g.Context() as c:
            opts = g.solver_opts(eps=1e-10, precond=precond)
            st, it, _ = g.gmaf_solve_joint(c.handle, nth, nz, K, *arrs, ref, opts)
            # a recurrence that ends far below what the true residual can reach: a restart, then an end
            deep = g.solver_opts(eps=1e-17, precond=precond, max_iter=3 * it)
            std, itd, reld = g.gmaf_solve_joint(c.handle, nth, nz, K, *arrs, ref.clone(), deep,
                                                allow_not_converged=True)
        q = torch.empty_like(p)
        warm = g.solver_opts(eps=1e-9, precond=precond, zero_init=0)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        st2, it2, rel2 = g.gmaf_solve_joint_noalloc(nth, nz, K, *arrs, p, opts)
        q.copy_(p)
        st3, it3, _ = g.gmaf_solve_joint_noalloc(nth, nz, K, *arrs, q, warm)
        same = torch.equal(p, q)
        st4, it4, rel4 = g.gmaf_solve_joint_noalloc(nth, nz, K, *arrs, q, deep,
                                                    allow=(g.GMAF_OK, g.GMAF_NOT_CONVERGED))
        torch.cuda.synchronize()
        left = torch.cuda.mem_get_info()[0]
        assert st == st2 == 0 and abs(it2 - it) <= 1 + it // 100 and rel2 <= 1e-9
        assert float((p - ref).norm() / ref.norm()) <= 1e-9
        assert st3 == 0 and it3 == 0 and same
        assert st4 == std and rel4 <= 10.0 * max(reld, 1e-15)
        assert left >= free - (2 << 20)         # (torch.equal's own temporary)

"""Assembly and loads against the oracle where the column-marching kernels can go wrong:
fewer columns than a warp's 31, exactly 31, 32 and 124, segments of rows that are not full,
batches of conditions of the same eccentricities (more than one batch holds, and in any
order), and dimples so dense that two lattice rows reach a level.

The tolerances are those of the kernels' other tests: coefficients to rounding (1e-11), the
source to 1e-9 of its interior size (it is a difference of film thicknesses), loads to 1e-11
of the largest part."""
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


def conditions(K, shared, seed):
    """K states; the conditions listed in `shared` have the eccentricities of the first of them."""
    rng = np.random.default_rng(seed)
    c = [inputs.random_state(rng) for _ in range(K)]
    for k in shared[1:]:
        c[k][:4] = c[shared[0]][:4]
    return c


@pytest.mark.parametrize("nth,nz,K,shared,density", [
    (3, 2, 1, (), 0.2), (30, 3, 2, (), 0.85), (31, 33, 3, (1, 2), 0.2), (32, 40, 2, (0, 1), 0.85),
    (124, 65, 5, (), 0.2), (125, 2, 9, (0, 5, 6, 7, 8), 0.2), (257, 70, 4, (3, 0, 1), 0.85),
    (64, 31, 14, (12, 2, 3, 5, 7, 11, 13), 0.2), (40, 129, 64, tuple(range(0, 64, 2)), 0.5),
])
def test_assembly_and_loads_match_the_oracle(g, nth, nz, K, shared, density):
    rng = np.random.default_rng(nth + nz)
    tex = inputs.dimple_texture(rng, density=density)
    conds = conditions(K, shared, nth)
    so, *want = oracle.assemble_joint(nth, nz, PHYS, tex, conds)
    n = K * nth * nz
    out = [torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(4)]
    p = 2e7 * (1.0 - np.linspace(0.0, 0.99, nz)[:, None]) + 1e6 * rng.random((K, nz, nth))
    loads = torch.zeros(12 * K, dtype=torch.float64, device="cuda")
    with g.Context() as c:
        assert g.gmaf_assemble(c.handle, nth, nz, PHYS, tex, conds, *out) == so == 0
        for _ in range(2):            # the second call finds the first one's tickets at zero
            loads.fill_(7.0)
            g.gmaf_integrate_loads(c.handle, nth, nz, PHYS, tex, conds,
                                   torch.from_numpy(p.ravel().copy()).cuda(), loads)
        torch.cuda.synchronize()
    D, aE, aN, S = (x.cpu().numpy().reshape(K, nz, nth) for x in out)
    for a, b in zip((D, aE, aN), want[:3]):
        np.testing.assert_allclose(a, b, rtol=1e-11)
    scale = np.abs(want[3][:, 1:-1]).max() if nz > 2 else np.abs(want[3]).max()
    np.testing.assert_allclose(S, want[3], rtol=1e-9, atol=1e-9 * scale)
    got = loads.cpu().numpy().reshape(K, 12)
    ref = np.stack([oracle.loads(nth, nz, PHYS, tex, cond, p[k])[1] for k, cond in enumerate(conds)])
    for part in (slice(0, 6), slice(6, 12)):
        x, y = got[:, part], ref[:, part]
        big = np.maximum(np.abs(y), 1e-3 * np.linalg.norm(y, axis=1, keepdims=True))
        assert np.max(np.abs(x - y) / big) <= 1e-11

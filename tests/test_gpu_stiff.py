"""Stiff pairs (eps / sigma far above 1) in the fixed-point kernel (needs a GPU):
contributions of far pairs, whose force is many powers of ten below the
coefficients' scale.  Isolated pairs of atoms, so that each force is one
contribution: within a count (2^-44) and 2^-46 of the exact force per component.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2508_13523_gb300 as md  # noqa: E402
from paper_2508_13523_gb300 import synth as S  # noqa: E402


@pytest.mark.parametrize("kind", [md.MD_LIST_HALF, md.MD_LIST_FULL])
@pytest.mark.parametrize("nt", [1, 2])
@pytest.mark.parametrize("eps, rc", [(30.0, 6.5), (100.0, 8.0), (1e4, 8.0), (1e6, 10.0)])
def test_far_contributions_of_stiff_pairs(eps, rc, nt, kind):
    # 6^3 pairs 24 apart, separations 1.5 .. rc in random directions
    g = np.stack(np.meshgrid(*[np.arange(6)] * 3, indexing="ij"), -1).reshape(-1, 3) * 24.0 + 6.0
    m = len(g)
    u = S.normal(41, 3 * m).reshape(m, 3)
    u /= np.linalg.norm(u, axis=1)[:, None]
    x = np.concatenate([g, g + u * (1.5 + (rc - 1.5) * S.uniform(42, m))[:, None]])
    box = np.full(3, 144.0)
    t = np.arange(2 * m, dtype=np.int32) // m % nt
    with md.LJMD(x, np.zeros_like(x), t, box, np.full((nt, nt), eps), np.ones((nt, nt)),
                 np.full((nt, nt), rc), np.ones(nt), list_kind=kind, threads_per_atom=1) as ctx:
        ctx.set_kernel(1, -1, 2, 0)
        ctx.compute_forces(0)
        xw, _, f = ctx.get_state(host=True)
    d = xw[m:].astype(np.longdouble) - xw[:m]
    d -= box * np.round(d / box)
    r2 = (d * d).sum(1)
    s6 = 1 / r2 ** 3
    fj = (24 * np.longdouble(eps) * s6 * (2 * s6 - 1) / r2)[:, None] * d
    mag = np.abs(24 * eps * s6 * (2 * s6 + 1) / r2)[:, None] * np.abs(d)
    tol = 2.0 ** -44 + 2.0 ** -46 * mag
    assert (np.abs(f[m:] - fj) <= tol).all(), np.max(np.abs(f[m:] - fj) / tol)
    assert (np.abs(f[:m] + fj) <= tol).all()

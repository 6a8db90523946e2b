"""Fixed-point positions in boxes with one long edge (needs a GPU): grids on
either side of the rule that picks their step, atoms at the faces and the corner,
drifts out of the box.

Bound per component as in the tests of the kernel's other ranges: one count (2^-44)
per contribution plus 2^-46 of the sum of the contributions' magnitudes.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle as O  # noqa: E402
import paper_2508_13523_gb300 as md  # noqa: E402
from paper_2508_13523_gb300 import synth as S  # noqa: E402


@pytest.mark.parametrize("kind", [md.MD_LIST_FULL, md.MD_LIST_HALF])
@pytest.mark.parametrize("axis", [0, 2])
@pytest.mark.parametrize("edge", [10.4, 290.0, 296.0, 584.0, 590.0, 1170.0, 1176.0, 2100.0])
def test_forces_in_a_long_box(edge, axis, kind):
    x, b, _ = S.fcc(6, 0.8442)
    x = x + 0.2 * (S.uniform(61, x.size).reshape(x.shape) - 0.5)
    x[:, axis] -= 0.5 * b[0]  # across the long axis' boundary, periodic along the others
    box = b.copy()
    box[axis] = edge
    with md.LJMD(x, np.zeros_like(x), None, box, 1.0, 1.0, 2.5, 1.0, list_kind=kind,
                 threads_per_atom=1) as ctx:
        ctx.set_kernel(1, -1, 2, 0)
        for drift in (0.0, 0.09, -0.12):  # wrapped, and with the kept list out of the box
            x0, v0, _ = ctx.get_state()
            if drift:
                x0[:, axis] += drift
                ctx.set_state(x0, v0, keep_list=True)
            ctx.compute_forces(0)
            xw, _, f = ctx.get_state(host=True)
            lj = O.LJ()
            fref, _, _ = O.forces(xw, box, lj, skin=0.3)
            i, j = O.pairs_brute(xw % box, box, 2.5)
            d = xw[j] - xw[i]
            d -= box * np.round(d / box)
            s6 = (1.0 / (d * d).sum(1)) ** 3
            g = 24 * s6 * np.abs(2 * s6 - 1) / np.sqrt((d * d).sum(1))
            n = len(xw)
            cnt = np.bincount(i, minlength=n) + np.bincount(j, minlength=n)
            mag = np.bincount(i, g, n) + np.bincount(j, g, n)
            bound = (cnt * 2.0 ** -44 + mag * 2.0 ** -46)[:, None]
            assert np.all(np.abs(f - fref) <= bound), np.max(np.abs(f - fref) / bound)

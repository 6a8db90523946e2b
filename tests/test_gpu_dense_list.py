"""Lists so dense that the fixed-point sums take smaller contributions (needs a
GPU): the coefficients follow the list, back and forth, through the captured
segments.
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


@pytest.mark.parametrize("nt", [1, 2])
@pytest.mark.parametrize("kind", [md.MD_LIST_HALF, md.MD_LIST_FULL])
def test_context_between_thin_and_dense_lists(kind, nt):
    """6,912 small atoms with a long cutoff: spread over the box (about 360 stencil
    candidates) or in one corner of it (about 2,700, above 2^11).  Each state
    run three times in turn in one context gives, bit for bit, the run of a context
    of its own; forces against the oracle."""
    x, box, _ = S.fcc(12, 0.42)
    x = x + 0.05 * (S.uniform(5, x.size).reshape(x.shape) - 0.5)
    v = S.maxwell_boltzmann(np.ones(len(x)), 0.3, 6)
    t = np.arange(len(x), dtype=np.int32) % nt
    tab = lambda a: np.full((nt, nt), a)
    states = (x, 0.5 * x)

    def context(x):
        ctx = md.LJMD(x, v, t, box, tab(1.0), tab(0.5), tab(2.8), np.ones(nt), list_kind=kind,
                      dt=0.001, rebuild_every=5, threads_per_atom=1)
        ctx.set_kernel(1, -1, 2, 0)
        return ctx

    def run(ctx, x):
        ctx.set_state(torch.as_tensor(x, device="cuda"), torch.as_tensor(v, device="cuda"))
        ctx.step(12)
        return ctx.get_state(host=True)

    alone = []
    for s in states:
        with context(s) as ctx:
            alone.append(run(ctx, s))
    with context(x) as ctx:
        for _ in range(3):
            for s, want in zip(states, alone):
                for a, b in zip(run(ctx, s), want):
                    np.testing.assert_array_equal(a, b)
        xw, _, f = ctx.get_state(host=True)
    fref, _, _ = O.forces(xw, box, O.LJ(tab(1.0), tab(0.5), tab(2.8), ntypes=nt), type_=t, skin=0.3)
    assert np.abs(f - fref).max() <= 1e-11 * np.abs(fref).max()

"""Reverse mode through steps whose list is rebuilt between its checkpoints
(check_disp, needs a GPU): a rebuild sorts the atoms anew in the middle of a
segment.  Against the oracle's reverse mode with a list of every step; bounds as
for the runs without such rebuilds (1e-10 on the final forces, 1e-9 of the rms on
the derivatives, mixed precision 1e-2).
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


def rel(a, b):
    return float(np.abs(a - b).max() / np.sqrt(np.mean(np.sum(b * b, axis=-1))))


@pytest.mark.parametrize("prec", [md.MD_PREC_FP64, md.MD_PREC_MIXED])
@pytest.mark.parametrize("kind", [md.MD_LIST_FULL, md.MD_LIST_HALF])
@pytest.mark.parametrize("nsteps", [19, 33])
def test_traj_vjp_with_rebuilds_inside_a_segment(nsteps, kind, prec):
    p = S.binary_mixture_params(rebuild_every=20)
    x, box, _ = S.fcc(6, 1.2)
    x = x + 0.05 * (S.uniform(81, x.size).reshape(x.shape) - 0.5)
    t = (S.uniform(82, len(x)) >= 0.8).astype(np.int32)
    v = S.maxwell_boltzmann(np.ones(len(x)), 8.0, 83)  # half the skin in some 8 steps
    lj = O.LJ(p.eps, p.sigma, p.rc, ntypes=2)
    cot = S.normal(93, x.size).reshape(x.shape)
    with md.LJMD(x, v, t, box, p.eps, p.sigma, p.rc, p.mass, dt=p.dt, list_kind=kind,
                 precision=prec, rebuild_every=20, check_disp=True, threads_per_atom=2) as ctx:
        x0, v0, _ = ctx.get_state(host=True)
        ckx, ckv, fK = ctx.traj_forward(x0, v0, nsteps, 20)
        x0b, v0b, g = ctx.traj_vjp(nsteps, 20, ckx, ckv, cot)
        ctx.set_state(torch.as_tensor(x0, device="cuda"), torch.as_tensor(v0, device="cuda"))
        ctx.step(19)
        assert ctx.stats()["builds"] > 1  # the displacement does ask for rebuilds
    _, _, fo, _ = O.run(x0, v0, box, lj, p.mass, type_=t, nsteps=nsteps, rebuild_every=1)
    xr, vr, gr = O.traj_vjp(x0, v0, box, lj, p.mass, cot, type_=t, nsteps=nsteps, rebuild_every=1)
    tol = 1e-9 if prec == md.MD_PREC_FP64 else 1e-2
    if prec == md.MD_PREC_FP64:
        assert rel(fK.cpu().numpy(), fo) <= 1e-10
    assert rel(x0b.cpu().numpy(), xr) <= tol
    assert rel(v0b.cpu().numpy(), vr) <= tol
    assert np.abs(g - gr).max() <= tol * np.abs(gr).max()

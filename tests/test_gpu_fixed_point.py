"""The FP64 contexts' fixed-point pair kernel at the edges of its ranges
(needs a GPU).

Forces, energy and virial against the oracle for: every number of lanes per
atom that the dispatch picks by the box's size, boxes barely larger than two
cutoffs (every pair may cross the boundary), one type in the general form
(a long cutoff in units of sigma), several types with different ratios, forces
far above and far below the counts' unit, overlapping atoms (the FP64 path),
atoms without a fixed-point position (a box of more than 409 length units),
atoms with more than 2^11 stencil candidates, and rows whose skin part comes
into range as a whole (several rounds of the lanes' slots).

Bound per component: one count (2^-44) per contribution for its rounding,
plus 2^-46 of the sum of the contributions' magnitudes (128 ulps: r^2 within
3 ulps on either side enters the force with a power of at most 7, and FP64
separations across the boundary carry the rounding of coordinates that are up
to 8 times as large).
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


def lattice(n, density, amp, seed):
    x, box, _ = S.fcc(n, density)
    return x + amp * (S.uniform(seed, x.size).reshape(x.shape) - 0.5), box


def pair_sums(x, box, eps, sigma, rc, t):
    """Contributions per atom and the sum of their magnitudes."""
    i, j = O.pairs_cells(x, box, float(np.max(rc))) if len(x) > 3000 else \
        O.pairs_brute(x, box, float(np.max(rc)))
    d = x[j] - x[i]
    d -= box * np.round(d / box)
    r2 = (d * d).sum(1)
    e, s, c = (np.broadcast_to(w, (2, 2))[t[i], t[j]] for w in (eps, sigma, rc))
    keep = r2 < c * c
    i, j, r2, e, s = i[keep], j[keep], r2[keep], e[keep], s[keep]
    s6 = (s * s / r2) ** 3
    f = 24 * e * s6 * np.abs(2 * s6 - 1) / np.sqrt(r2)
    cnt = np.bincount(i, minlength=len(x)) + np.bincount(j, minlength=len(x))
    mag = np.bincount(i, f, len(x)) + np.bincount(j, f, len(x))
    return cnt, mag


def check(ctx, x, box, eps, sigma, rc, t, skin):
    nt = 1 if np.ndim(eps) == 0 else 2
    f = ctx.get_state()[2].cpu().numpy()
    th = ctx.energy()
    lj = O.LJ(eps, sigma, rc, ntypes=nt)
    fref, E, W = O.forces(x, box, lj, type_=t if nt > 1 else None, skin=skin)
    cnt, mag = pair_sums(x, box, eps, sigma, rc, t)
    bound = (cnt * 2.0 ** -44 + mag * 2.0 ** -46)[:, None]
    assert np.all(np.abs(f - fref) <= bound), np.max(np.abs(f - fref) / np.maximum(bound, 1e-300))
    # the virial is summed over atoms from the rounded forces, and one type's
    # energy over its trace: 1e-12 plus 6 sigma of the contributions' roundings
    # (each below 2^-45, independent) at positions within half the box
    noise = 6 * np.sqrt(cnt.sum()) * 2.0 ** -45 * 0.5 * float(np.max(box))
    assert abs(th.pe - E) <= 1e-12 * max(abs(E), np.abs(W).max()) + noise
    assert np.abs(th.virial - W).max() <= 1e-12 * np.abs(W).max() + noise


MIX = dict(eps=np.array([[1.0, 1.5], [1.5, 0.5]]), sigma=np.array([[1.0, 0.8], [0.8, 0.88]]),
           rc=np.array([[2.5, 2.0], [2.0, 2.2]]))
WIDE = dict(eps=np.array([[1.0, 0.3], [0.3, 2.0]]), sigma=np.array([[0.25, 0.6], [0.6, 1.0]]),
            rc=np.array([[2.5, 1.5], [1.5, 1.2]]))

CASES = {
    # name: (cells, density, jitter, eps, sigma, rc)
    "8 lanes, box of two cutoffs": (3, 0.8442, 0.15, 1.0, 1.0, 2.5),
    "8 lanes, ragged warp": (5, 0.8442, 0.2, 1.0, 1.0, 2.5),
    "4 lanes": (16, 0.8442, 0.2, 1.0, 1.0, 2.5),
    "2 lanes": (35, 0.8442, 0.2, 1.0, 1.0, 2.5),
    "general form, one type": (9, 0.8442, 0.2, 1.0, 0.3, 2.5),
    "long cutoff": (8, 0.8442, 0.2, 1.0, 1.0, 5.5),
    "large forces": (8, 0.8442, 0.3, 100.0, 1.0, 2.5),
    "small forces": (8, 0.8442, 0.2, 1e-4, 1.0, 2.5),
    "overlaps": (8, 0.8442, 1.2, 1.0, 1.0, 2.5),
    "mixture": (8, 1.2, 0.3, MIX["eps"], MIX["sigma"], MIX["rc"]),
    "mixture of very different sizes": (8, 0.9, 0.3, WIDE["eps"], WIDE["sigma"], WIDE["rc"]),
    "dense": (9, 40.0, 0.03, 1.0, 0.3, 1.2),
}


@pytest.mark.parametrize("kind", [md.MD_LIST_FULL, md.MD_LIST_HALF])
@pytest.mark.parametrize("case", CASES)
def test_forces_energy_virial(case, kind):
    cells, density, amp, eps, sigma, rc = CASES[case]
    x, box = lattice(cells, density, amp, 50 + cells)
    t = (S.uniform(7, len(x)) < 0.3).astype(np.int32) if np.ndim(eps) else \
        np.zeros(len(x), np.int32)
    nt = 2 if np.ndim(eps) else 1
    with md.LJMD(x, np.zeros_like(x), t, box, eps, sigma, rc, np.ones(nt), list_kind=kind,
                 threads_per_atom=1) as ctx:
        ctx.set_kernel(1, -1, 2, 0)
        ctx.compute_forces(0)
        xw = ctx.get_state()[0].cpu().numpy()
        check(ctx, xw, box, eps, sigma, rc, t, 0.3)


@pytest.mark.parametrize("kind", [md.MD_LIST_FULL, md.MD_LIST_HALF])
def test_atoms_without_fixed_point_position(kind):
    """A 1,500-wide box holding a lattice block around the origin corner: the
    grid of its positions is too coarse for coordinates below 2, which take
    the FP64 path (and so do their partners)."""
    x, b = lattice(6, 0.8442, 0.2, 61)
    x -= 0.5 * b[0]
    box = np.full(3, 1500.0)
    t = np.zeros(len(x), np.int32)
    with md.LJMD(x, np.zeros_like(x), t, box, 1.0, 1.0, 2.5, 1.0, list_kind=kind,
                 threads_per_atom=1) as ctx:
        ctx.set_kernel(1, -1, 2, 0)
        ctx.compute_forces(0)
        xw = ctx.get_state()[0].cpu().numpy()
        f = ctx.get_state()[2].cpu().numpy()
    fref, _, _ = O.forces(xw, box, O.LJ(), skin=0.3)
    cnt, mag = pair_sums(xw, box, 1.0, 1.0, 2.5, t)
    # across the boundary the FP64 separation is rounded to 2^-43: 2^-44 / 0.8
    # in r enters the force with |dF/dr| <= 14 |F| / r, alike on both sides
    bound = (cnt * 2.0 ** -44 + mag * 2.0 ** -46)[:, None]
    assert np.all(np.abs(f - fref) <= bound)


@pytest.mark.parametrize("kind", [md.MD_LIST_FULL, md.MD_LIST_HALF])
def test_skin_entries_in_range(kind):
    """The kept list of a dense box after a contraction by 0.85: per lane far
    more skin entries in range than it has slots."""
    x, box = lattice(5, 3.0, 0.1, 62)
    t = np.zeros(len(x), np.int32)
    with md.LJMD(x, np.zeros_like(x), t, box, 1.0, 0.5, 2.5, 1.0, skin=1.5, list_kind=kind,
                 threads_per_atom=1) as ctx:
        ctx.set_kernel(1, -1, 2, 0)
        x0, v0, _ = ctx.get_state()
        builds = ctx.stats()["builds"]
        c = torch.as_tensor(0.5 * box, device=x0.device)
        x1 = (c + 0.85 * (x0 - c)).contiguous()
        ctx.set_state(x1, v0, keep_list=True)
        assert ctx.stats()["builds"] == builds
        check(ctx, x1.cpu().numpy(), box, 1.0, 0.5, 2.5, t, 0.0)


COUL = {
    # name: (cells, eps, sigma, rc, q, qqrd2e, rc_coul)
    "weak, one type": (6, 1.0, 1.0, 2.5, [1e-3], 1.0, 2.5),
    "strong": (6, np.ones((2, 2)), np.ones((2, 2)), np.full((2, 2), 2.5), [3.0, -2.0], 10.0, 2.5),
    "one neutral type": (6, np.ones((2, 2)), np.ones((2, 2)), np.full((2, 2), 2.5), [0.5, 0.0],
                         1.0, 1.7),
    "beyond rc of a pair": (6, MIX["eps"], MIX["sigma"], MIX["rc"], [0.5, -0.5], 1.0, 2.45),
    "4 lanes": (17, np.ones((2, 2)), np.ones((2, 2)), np.full((2, 2), 2.5), [0.5, -0.5], 1.0, 2.5),
}


@pytest.mark.parametrize("kind", [md.MD_LIST_FULL, md.MD_LIST_HALF])
@pytest.mark.parametrize("case", COUL)
def test_coulomb(case, kind):
    """lj/cut/coul/cut against the oracle; the bound as above with the
    Coulomb contributions' magnitudes added (two roundings per contribution:
    each term has its own)."""
    cells, eps, sigma, rc, q, qqrd2e, rc_coul = COUL[case]
    x, box = lattice(cells, 0.8442, 0.3, 80 + cells)
    nt = len(q)
    t = (np.arange(len(x)) % 4 >= 2).astype(np.int32) if nt > 1 else np.zeros(len(x), np.int32)
    with md.LJMD(x, np.zeros_like(x), t, box, eps, sigma, rc, np.ones(nt), list_kind=kind,
                 threads_per_atom=1) as ctx:
        ctx.set_coulomb(q, rc_coul, qqrd2e)
        ctx.set_kernel(1, -1, 2, 0)
        ctx.compute_forces(0)
        xw, _, f = (a.cpu().numpy() for a in ctx.get_state())
        th = ctx.energy()
    lj = O.LJ(eps, sigma, rc, ntypes=nt, q=q, rc_coul=rc_coul, qqrd2e=qqrd2e)
    fref, E, W = O.forces(xw, box, lj, type_=t if nt > 1 else None, skin=0.3)
    cnt, mag = pair_sums(xw, box, eps, sigma, rc, t)
    i, j = O.pairs_cells(xw, box, rc_coul) if len(x) > 3000 else O.pairs_brute(xw, box, rc_coul)
    d = xw[j] - xw[i]
    d -= box * np.round(d / box)
    r2 = (d * d).sum(1)
    qt = np.asarray(q)
    fc = qqrd2e * np.abs(qt[t[i]] * qt[t[j]]) / r2
    cnt = cnt + np.bincount(i, minlength=len(x)) + np.bincount(j, minlength=len(x))
    mag = mag + np.bincount(i, fc, len(x)) + np.bincount(j, fc, len(x))
    bound = (2 * cnt * 2.0 ** -44 + mag * 2.0 ** -46)[:, None]
    assert np.all(np.abs(f - fref) <= bound)
    noise = 6 * np.sqrt(2 * cnt.sum()) * 2.0 ** -45 * 0.5 * float(np.max(box))
    ec = (qqrd2e * np.abs(qt[t[i]] * qt[t[j]]) / np.sqrt(r2)).sum()
    assert abs(th.pe - E) <= 1e-12 * max(abs(E), np.abs(W).max(), ec) + noise
    assert np.abs(th.virial - W).max() <= 1e-12 * max(np.abs(W).max(), ec) + noise


@pytest.mark.parametrize("prec", [md.MD_PREC_FP64, md.MD_PREC_MIXED])
@pytest.mark.parametrize("every", [50, 7])
def test_check_disp_segments(prec, every):
    """check_disp runs several steps per launch and stops them on the device
    where a displacement asks for a rebuild: the same builds and, bit for bit,
    the same trajectory as one call per step (order-independent force sums)."""
    x, box = lattice(6, 0.8442, 0.1, 91)
    v = S.maxwell_boltzmann(np.ones(len(x)), 2.0, 92)
    runs = []
    for calls in ([61], [1] * 61, [20, 1, 40]):
        with md.LJMD(x, v, None, box, 1.0, 1.0, 2.5, 1.0, precision=prec, check_disp=True,
                     rebuild_every=every, threads_per_atom=1, list_kind=md.MD_LIST_HALF) as ctx:
            ctx.set_kernel(1, -1, 2 if prec == md.MD_PREC_FP64 else 0, 0)
            ctx.compute_forces(0)  # the initial forces with order-independent sums too
            for k in calls:
                ctx.step(k)
            st = ctx.stats()
            runs.append((st["builds"], st["max_disp"], [a.cpu().numpy() for a in ctx.get_state()]))
    assert runs[0][0] > 61 // every + 2  # builds between the cadence's
    for r in runs[1:]:
        assert r[:2] == runs[0][:2]
        for a, b in zip(r[2], runs[0][2]):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("precision", [md.MD_PREC_FP64, md.MD_PREC_MIXED])
@pytest.mark.parametrize("nt", [3, 8])
def test_tables_of_many_types(nt, precision):
    """The kernels' shared tables hold the types that there are: forces and
    force VJP with an odd number of types and with the most, every pair of
    types with coefficients of its own.  Bounds: 1e-11 (FP64) and 1e-3 (mixed)
    of the largest component, as for two types."""
    x, box = lattice(6, 0.8442, 0.2, 71)
    t = np.arange(len(x), dtype=np.int32) % nt
    u = S.uniform(72, 2 * nt * nt).reshape(2, nt, nt)
    u = 0.5 * (u + u.transpose(0, 2, 1))
    eps, sigma = 0.5 + u[0], 0.8 + 0.2 * u[1]
    rc = 2.5 * sigma
    tol = 1e-11 if precision == md.MD_PREC_FP64 else 1e-3
    cot = S.normal(73, x.size).reshape(x.shape)
    lj = O.LJ(eps, sigma, rc, ntypes=nt)
    with md.LJMD(x, np.zeros_like(x), t, box, eps, sigma, rc, np.ones(nt), precision=precision,
                 list_kind=md.MD_LIST_HALF, threads_per_atom=2) as ctx:
        for compacted in ((0, 2) if precision == md.MD_PREC_FP64 else (0,)):
            ctx.set_kernel(1 if compacted else 2, -1, compacted, 0)
            ctx.compute_forces(0)
            xw, _, f = (w.cpu().numpy() for w in ctx.get_state())
            fref, _, _ = O.forces(xw, box, lj, type_=t, skin=0.3)
            assert np.abs(f - fref).max() <= tol * np.abs(fref).max()
        xbar, g = ctx.force_vjp(cot)
    xref, gref = O.force_vjp(xw, box, lj, cot, type_=t, skin=0.3)
    assert np.abs(xbar.cpu().numpy() - xref).max() <= tol * np.abs(xref).max()
    assert np.abs(g - gref).max() <= tol * np.abs(gref).max()

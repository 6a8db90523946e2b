"""The neighbor list over many rebuilds (needs a GPU): what other calls between
rebuilds may not disturb.  Runs are compared bit for bit: fixed-point force sums
and the stable sort do not depend on the order of additions.
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


def context(n_cells, seed, **kw):
    x, box, _ = S.fcc(n_cells, 0.8442)
    x = x + 0.1 * (S.uniform(seed, x.size).reshape(x.shape) - 0.5)
    v = S.maxwell_boltzmann(np.ones(len(x)), 1.44, seed + 1)
    kw = dict(dict(rebuild_every=10, threads_per_atom=1), **kw)
    ctx = md.LJMD(x, v, None, box, 1.0, 1.0, 2.5, 1.0, **kw)
    if kw.get("precision", md.MD_PREC_FP64) == md.MD_PREC_FP64:
        ctx.set_kernel(1, -1, 2, 0)
    ctx.compute_forces(0)
    return ctx


def final(ctx):
    off, idx = ctx.neighbors()
    return [a.cpu().numpy() for a in (*ctx.get_state(), off, idx)]


@pytest.mark.parametrize("prec", [md.MD_PREC_FP64, md.MD_PREC_MIXED])
@pytest.mark.parametrize("kind", [md.MD_LIST_HALF, md.MD_LIST_FULL])
def test_list_export_between_rebuilds(prec, kind):
    """Exporting the list scans over the atoms, which takes more scratch than the
    scan over the cells (10,976 atoms: 6 tiles against 1); the rebuilds after it
    are one graph by then and keep the address they were captured with.  Other
    contexts take device memory in between."""
    runs = []
    for export in (False, True):
        with context(14, 3, precision=prec, list_kind=kind) as ctx:
            ctx.step(35)  # three rebuilds after the first
            others = []
            if export:
                ctx.neighbors()
                others = [context(4, 7 + k, precision=prec, list_kind=kind) for k in range(4)]
                before = [final(o) for o in others]
            ctx.step(40)
            runs.append(final(ctx))
            for o, b in zip(others, before if export else ()):
                o.compute_forces(0)
                for p, q in zip(final(o), b):
                    np.testing.assert_array_equal(p, q)
                o.close()
    for p, q in zip(*runs):
        np.testing.assert_array_equal(p, q)


@pytest.mark.parametrize("nt", [2, 8])
@pytest.mark.parametrize("kind", [md.MD_LIST_HALF, md.MD_LIST_FULL])
@pytest.mark.parametrize("cells", [3, 5, 8])
def test_partial_chunks_with_several_types(cells, kind, nt):
    """The build tests 32 candidates at a time and looks up a cutoff for the
    types of each; the last chunk of a cell's candidates is seldom full.  The list
    against the oracle's pairs, with types that make every table entry in use."""
    x, box, _ = S.fcc(cells, 0.8442)
    x = (x + 0.2 * (S.uniform(60 + nt, x.size).reshape(x.shape) - 0.5)) % box
    t = np.arange(len(x), dtype=np.int32) % nt
    u = S.uniform(61, nt * nt).reshape(nt, nt)
    rc = 1.5 + 0.25 * (u + u.T)
    with md.LJMD(x, np.zeros_like(x), t, box, np.ones((nt, nt)), np.ones((nt, nt)), rc,
                 np.ones(nt), list_kind=kind, threads_per_atom=1) as ctx:
        off, idx = (a.cpu().numpy() for a in ctx.neighbors())
    rlist = float(rc.max()) + 0.3
    i, j = O.pairs_brute(x, box, rlist)
    want = np.unique(np.minimum(i, j) * len(x) + np.maximum(i, j))
    a = np.repeat(np.arange(len(x)), np.diff(off))
    got = np.sort(np.minimum(a, idx) * len(x) + np.maximum(a, idx))
    np.testing.assert_array_equal(got, want if kind == md.MD_LIST_HALF else np.repeat(want, 2))


@pytest.mark.parametrize("kind", [md.MD_LIST_HALF, md.MD_LIST_FULL])
@pytest.mark.parametrize("cells, density, rc", [
    (24, 0.2, 2.5),    # 12,167 cells of 4.5 atoms: one thread per atom
    (24, 0.3, 2.5),    # 8,000 cells of 6.9: one block per cell
    (9, 0.8442, 4.8),  # one cell of 2,916 atoms: many blocks for it
    (4, 0.8442, 2.2),  # one cell of 256
])
def test_build_routes(cells, density, rc, kind):
    """Both forms of the build on either side of the rule that picks one, and cells
    that take many groups of 32 atoms: the list against the oracle's pairs."""
    x, box, _ = S.fcc(cells, density)
    x = (x + 0.3 * (S.uniform(70, x.size).reshape(x.shape) - 0.5)) % box
    with md.LJMD(x, np.zeros_like(x), None, box, 1.0, 1.0, rc, 1.0, list_kind=kind,
                 threads_per_atom=1) as ctx:
        off, idx = (a.cpu().numpy() for a in ctx.neighbors())
    i, j = O.pairs_cells(x, box, rc + 0.3) if len(x) > 4000 else O.pairs_brute(x, box, rc + 0.3)
    i, j, idx = (q.astype(np.int64) for q in (i, j, idx))  # keys up to n^2
    want = np.sort(np.minimum(i, j) * len(x) + np.maximum(i, j))
    a = np.repeat(np.arange(len(x)), np.diff(off))
    got = np.sort(np.minimum(a, idx) * len(x) + np.maximum(a, idx))
    np.testing.assert_array_equal(got, want if kind == md.MD_LIST_HALF else np.repeat(want, 2))


@pytest.mark.parametrize("prec", [md.MD_PREC_FP64, md.MD_PREC_MIXED])
@pytest.mark.parametrize("kind", [md.MD_LIST_HALF, md.MD_LIST_FULL])
def test_new_coefficients_with_a_captured_rebuild(prec, kind):
    """set_lj and set_kernel keep the captured rebuild (it depends on neither):
    a run with new coefficients is, bit for bit, that of a context created with
    them."""
    with context(10, 21, precision=prec, list_kind=kind) as ctx:
        ctx.step(45)  # four rebuilds: captured by then
        x, v, _ = ctx.get_state()
        ctx.set_lj(1.25, 0.97)
        ctx.set_kernel(2 if prec else 1, -1, 0 if prec else 3, 0)
        ctx.set_state(x, v)
        ctx.step(45)
        got = final(ctx)
    _, box, _ = S.fcc(10, 0.8442)
    with md.LJMD(x, v, None, box, 1.25, 0.97, 2.5, 1.0, precision=prec, list_kind=kind,
                 rebuild_every=10, threads_per_atom=1) as ctx:
        ctx.set_kernel(2 if prec else 1, -1, 0 if prec else 3, 0)
        ctx.set_state(x, v)
        ctx.step(45)
        want = final(ctx)
    for p, q in zip(got, want):
        np.testing.assert_array_equal(p, q)


@pytest.mark.parametrize("kind", [md.MD_LIST_HALF, md.MD_LIST_FULL])
def test_list_without_memory(kind):
    """A list that has to grow and finds no device memory: the call says so, calls
    that would read the list say so until a rebuild succeeds, and the context then
    gives the forces of a new one."""
    with context(20, 9, list_kind=kind) as ctx:
        ctx.step(35)  # with captured segments and rebuild
        x, v, f = ctx.get_state()
        ctx.set_state(x, v)
        want = ctx.get_state()
        dense = 0.25 * x  # rows of thousands of entries: 350 MB and more
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        hold = torch.empty(free - (200 << 20), dtype=torch.uint8, device="cuda")
        try:
            with pytest.raises(md.MDError) as e:
                ctx.set_state(dense, v)
            assert e.value.code == md.MD_ENOMEM
            for call in (lambda: ctx.compute_forces(0), lambda: ctx.step(5), ctx.energy,
                         ctx.neighbor_count, lambda: ctx.force_vjp(v), ctx.build_neighbors,
                         lambda: ctx.set_state(dense, v, keep_list=True)):
                with pytest.raises(md.MDError) as e:
                    call()
                assert e.value.code == md.MD_ENOMEM
            assert ctx.stats()["list_entries"] == 0
        finally:
            del hold
            torch.cuda.empty_cache()
        ctx.set_state(x, v)
        for a, b in zip(ctx.get_state(), want):
            assert torch.equal(a, b)
        ctx.step(25)

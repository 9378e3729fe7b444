"""The device-side setup and its layouts at the edges of their kernels. Galerkin and
interpolation rows that overflow the first column table (more than 512 distinct columns,
plain AMG on P4 matrices), and coarsest inverses whose size is below, at and above a
multiple of the 32-row pivot block, against the oracle; the interleaved slices. Integer
decisions are exact; values are held to the tolerance of the other setup tests (1e-12 of
the largest entry), cycles to 1e-11."""
import numpy as np
import pytest

from paper_1204_2586_gb300.inputs import kappa_lognormal, kuhn_mesh

pytestmark = pytest.mark.gpu


def _close(a, b, tol):
    assert np.abs(a - b).max() <= tol * np.abs(b).max()


def _pair(oracle_mod, k, n, **kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(n, 0.2, 0)
    kap = kappa_lognormal(t.shape[0], 1)
    G, O = Problem(xyz, t, k, kap), oracle_mod.Problem(xyz, t, k, kap)
    G.setup(**kw)
    O.setup(**kw)
    return torch, G, O


@pytest.mark.parametrize("k,n,theta", [(4, 6, 0.004), (3, 7, 0.01)])
def test_rows_with_many_columns(oracle_mod, k, n, theta):
    _, G, O = _pair(oracle_mod, k, n, mode=2, theta=theta, coarse_size=20)
    longest = 0
    assert G.info.levels == O.levels()
    for l in range(O.levels()):
        Lo = O.level(l)
        c, nc = G.colours(l)
        assert np.array_equal(c, Lo["colour"]) and nc == Lo["ncolour"]
        for which, key in ((3 + 2 * l, "A"), (4 + 2 * l, "P")):
            if key not in Lo:
                continue
            ptr, col, val, shape = G.matrix(which)
            assert shape == Lo[key].shape and np.array_equal(ptr, Lo[key].ptr) and np.array_equal(col, Lo[key].col)
            _close(val, Lo[key].val, 1e-12)
        if l > 0:
            longest = max(longest, int(np.diff(Lo["A"].ptr).max()))
    assert longest > 512  # the larger table was needed


@pytest.mark.parametrize("n,coarse_size", [(4, 256), (5, 256), (6, 40), (7, 256), (9, 600)])
def test_coarsest_inverse(oracle_mod, n, coarse_size):
    torch, G, O = _pair(oracle_mod, 2, n, coarse_size=coarse_size, level_smoother=1)
    assert G.info.coarse_rows == O.level(O.levels() - 1)["A"].shape[0]
    b = np.random.default_rng(n).standard_normal(G.nH)
    _close(G.apply_vcycle(torch.tensor(b, device="cuda")).cpu().numpy(), O.vcycle(b), 1e-11)


# one size for each shape of the interleaved slices (lanes, steps, batch), both precisions,
# and the whole-row slices of the multiplicative form's full sweep
@pytest.mark.parametrize("k,n,prec,mode", [(2, 2, 0, 0), (1, 9, 0, 0), (1, 9, 1, 0), (3, 12, 0, 0), (2, 64, 0, 0),
                                           (3, 40, 0, 0), (4, 40, 0, 0), (3, 9, 1, 0), (3, 24, 1, 0), (4, 12, 1, 0),
                                           (4, 40, 1, 0), (2, 5, 0, 1), (3, 12, 0, 1), (4, 10, 1, 1)])
def test_slices_match_rows(k, n, prec, mode):
    """The default sweep over slices against the row layout with 4 lanes (itself held to the
    oracle elsewhere). Both add a row's products in some order: a sum of L terms is off by
    at most L u sum|a y|, and the 2 C phases pass it on."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(n, 0.2, 0)
    P = Problem(xyz, t, k, kappa_lognormal(t.shape[0], 1))
    r = torch.randn(P.nh, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    out = []
    for layout in (4, 0):
        P.setup(smoother_layout=layout, precond_precision=prec, mode=mode, level_smoother=1)
        assert (P.info.smoother_layout > 500) == (layout == 0)
        out.append(P.apply_prec(r) if mode else P.apply_smoother(r))
    longest = 400 if k == 4 else 200
    u = 2.0 ** -24 if prec else 2.0 ** -53
    assert (out[1] - out[0]).norm() <= 2 * P.info.fine_colours * longest * u * out[0].norm()
    P.close()


# cycles whose dense tail starts on the first, the second and a deeper level
@pytest.mark.parametrize("n,level_smoother", [(6, 0), (12, 1), (21, 0), (21, 1), (17, 0)])
def test_cycle_with_dense_tail(oracle_mod, n, level_smoother):
    torch, G, O = _pair(oracle_mod, 1, n, level_smoother=level_smoother)
    assert G.info.levels == O.levels()
    b = np.random.default_rng(n).standard_normal(G.nH)
    ref = O.vcycle(b)
    _close(G.apply_vcycle(torch.tensor(b, device="cuda")).cpu().numpy(), ref, 1e-11)
    # FP32: row sums of up to 5120 terms on the tail, u = 2^-24
    G.setup(level_smoother=level_smoother, precond_precision=1)
    _close(G.apply_vcycle(torch.tensor(b, device="cuda")).cpu().numpy(), ref, 5120 * 2.0 ** -24)


# every block width with rows shared by lane groups and a dense tail, against the
# single-column solve of each column (both to 1e-8: the bound of the other block tests)
@pytest.mark.parametrize("ncols,prec,level_smoother,mode", [(3, 0, 0, 0), (7, 1, 0, 0), (13, 0, 1, 0), (30, 1, 1, 0),
                                                            (41, 0, 0, 1), (60, 1, 0, 0)])
def test_block_widths(ncols, prec, level_smoother, mode):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(6, 0.2, 0)
    P = Problem(xyz, t, 3, kappa_lognormal(t.shape[0], 1))
    P.setup(precond_precision=prec, level_smoother=level_smoother, mode=mode)
    b = torch.randn(P.nh, ncols, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(ncols))
    x, st = P.solve(b)
    assert max(st["true_rel"]) <= 1e-8
    for c in (0, ncols // 2, ncols - 1):
        xc, sc = P.solve(b[:, c].contiguous())
        assert abs(sc["iters"][0] - st["iters"][c]) <= 1
        assert (x[:, c] - xc).norm() <= 1e-8 * xc.norm()
    P.close()


# one size for each shape of the SpMV's slices, and the product between set_kappa and setup
@pytest.mark.parametrize("k,n", [(2, 8), (3, 12), (3, 16), (3, 24), (4, 20)])
def test_spmv_slices(k, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(n, 0.2, 0)
    kap = kappa_lognormal(t.shape[0], 1)
    P = Problem(xyz, t, k, kap)
    x = torch.randn(P.nh, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    y0 = P.spmv(x)  # rows of the CSR form
    P.setup()
    assert P.info.spmv_layout > 500
    # a row sum of L terms is off by at most L u sum |a x|, either way
    bound = 2 * 400 * 2.0 ** -53 * P.spmv(x.abs()).abs().max() * 4
    assert (P.spmv(x) - y0).abs().max() <= bound
    P.set_kappa(kap)
    assert torch.equal(P.spmv(x), y0)
    P.close()


def _sweep_bound(P, prec):
    """Rounding of a symmetric sweep and a dense tail: 2 C phases of sums of up to 400 terms,
    then one of up to 5120, either way."""
    u = 2.0 ** -24 if prec else 2.0 ** -53
    return (2 * 2 * P.info.fine_colours * 400 + 2 * 5120) * u


# the whole preconditioner as one dense product (up to 3400 unknowns; 4913 keep the sweeps)
# against the row layout's sweeps
@pytest.mark.parametrize("k,n,prec,level_smoother", [(2, 8, 0, 0), (2, 8, 1, 1), (4, 4, 0, 1), (3, 5, 1, 0), (2, 9, 0, 0),
                                                     (1, 4, 0, 0)])
def test_dense_preconditioner(k, n, prec, level_smoother):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(n, 0.2, 0)
    P = Problem(xyz, t, k, kappa_lognormal(t.shape[0], 1))
    r = torch.randn(P.nh, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    out = []
    for layout in (4, 0):
        P.setup(smoother_layout=layout, precond_precision=prec, level_smoother=level_smoother)
        out.append(P.apply_prec(r))
    assert (out[1] - out[0]).norm() <= _sweep_bound(P, prec) * out[0].norm()
    P.close()


# the three velocity components in one sweep (above 3400 unknowns) against one at a time
@pytest.mark.parametrize("k,n,prec", [(2, 9, 0), (3, 6, 1)])
def test_stokes_components_share_sweeps(k, n, prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(n, 0.2, 0)
    P = Problem(xyz, t, k)
    out = []
    for layout in (4, 0):
        P.setup(smoother_layout=layout, precond_precision=prec, level_smoother=1)
        P.stokes_setup()
        r = torch.randn(P.stokes_n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
        out.append(P.stokes_prec(r)[: 3 * P.nh])
    assert (out[1] - out[0]).norm() <= _sweep_bound(P, prec) * out[0].norm()
    P.close()


@pytest.mark.parametrize("n", [2, 16, 17, 18])
def test_colouring_in_one_block_and_in_rounds(oracle_mod, n):
    """P1 problems of 1, 3375, 4096 and 4913 rows: up to 4096 the colouring runs in one block."""
    _, G, O = _pair(oracle_mod, 1, n)
    c, nc = G.colours(-1)
    assert np.array_equal(c, O.fine_colour()) and nc == c.max() + 1
    assert np.array_equal(G.colours(0)[0], O.level(0)["colour"])


@pytest.mark.parametrize("k,n,level_smoother", [(2, 8, 0), (1, 16, 1), (2, 5, 0), (1, 9, 0), (3, 5, 1)])
def test_dense_preconditioner_fp32_is_as_exact_as_sweeps(k, n, level_smoother):
    """Each against FP64 on the same vectors: the one product of thousands of terms is no
    further off than the sweeps whose place it takes."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(n, 0.2, 0)
    P = Problem(xyz, t, k, kappa_lognormal(t.shape[0], 1))
    g = torch.Generator("cuda").manual_seed(n)
    rs = [torch.randn(P.nh, dtype=torch.float64, device="cuda", generator=g) for _ in range(4)]
    err = []
    for layout in (4, 0):
        z = []
        for prec in (0, 1):
            P.setup(smoother_layout=layout, precond_precision=prec, level_smoother=level_smoother)
            z.append([P.apply_prec(r) for r in rs])
        err.append(sum(((a - b).norm() / b.norm()).item() for a, b in zip(z[1], z[0])))
    assert err[1] <= err[0]
    P.close()


@pytest.mark.parametrize("n", [7, 9, 12, 16])
def test_dense_tail_fp32_rounds_three_times(n):
    """A cycle that is one dense product (P1 meshes: the tail begins on the finest level) rounds
    its matrix, its input and its result to FP32: each an independent relative error, uniform
    within half a unit of the last place, 2^-24 / sqrt(3) / 1.5 in the mean square over a binade
    (2.3e-8). For entries of random sign the three add up to 4e-8; the bound allows 1.5 times that
    and nothing for the sums."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(n, 0.2, 0)
    P = Problem(xyz, t, 1, kappa_lognormal(t.shape[0], 1))
    g = torch.Generator("cuda").manual_seed(n)
    bs = [torch.randn(P.nH, dtype=torch.float64, device="cuda", generator=g) for _ in range(4)]
    x = []
    for prec in (0, 1):
        P.setup(precond_precision=prec)
        x.append([P.apply_vcycle(b) for b in bs])
    e = max(((a - c).norm() / c.norm()).item() for a, c in zip(x[1], x[0]))
    assert e <= 1.5 * 3 ** 0.5 * 2.3e-8
    P.close()


# blocks on both sides of the line between one dense product and the launches of the levels:
# by width, by rows, by level smoother and precision
@pytest.mark.parametrize("n,ncols,prec,level_smoother,dense", [(17, 3, 0, 0, True), (17, 64, 0, 0, False), (17, 64, 1, 0, True),
                                                               (26, 64, 0, 0, True), (9, 32, 0, 1, False), (11, 3, 0, 1, True),
                                                               (22, 16, 1, 1, True),
                                                               (13, 32, 1, 1, False), (17, 32, 1, 1, False)])
def test_block_cycle_with_and_without_dense_tail(n, ncols, prec, level_smoother, dense):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(n, 0.2, 0)
    P = Problem(xyz, t, 1, kappa_lognormal(t.shape[0], 1))
    P.setup(precond_precision=prec, level_smoother=level_smoother)
    b = torch.randn(P.nh, ncols, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    x, st = P.solve(b)
    i = P.info
    assert i.tail_level < i.levels - 1
    assert i.block_tail_level == (i.tail_level if dense else i.levels - 1)
    assert max(st["true_rel"]) <= 1e-8
    for c in (0, ncols - 1):
        xc, sc = P.solve(b[:, c].contiguous())
        assert abs(sc["iters"][0] - st["iters"][c]) <= 1
        assert (x[:, c] - xc).norm() <= 1e-8 * xc.norm()
    P.close()


# both sides of the line from which a row of the blocked product is a whole warp's, for rows of
# 14 and 27 entries (P3 and P4: test_block_widths and the block tests against the oracle)
@pytest.mark.parametrize("k,n,ncols", [(1, 17, 8), (1, 18, 16), (2, 13, 8), (2, 17, 3)])
def test_block_product_of_short_rows(k, n, ncols):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(n, 0.2, 0)
    P = Problem(xyz, t, k, kappa_lognormal(t.shape[0], 1))
    P.setup(level_smoother=1)
    b = torch.randn(P.nh, ncols, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    x, st = P.solve(b)
    assert max(st["true_rel"]) <= 1e-8
    for c in (0, ncols - 1):
        xc, sc = P.solve(b[:, c].contiguous())
        assert abs(sc["iters"][0] - st["iters"][c]) <= 1
        assert (x[:, c] - xc).norm() <= 1e-8 * xc.norm()
    P.close()


@pytest.mark.parametrize("n,ncols,lanes", [(6, 3, {32}), (6, 8, {32}), (6, 16, {32}), (32, 3, {2, 4}), (32, 8, {4, 8})])
def test_block_lanes_are_those_that_run(n, ncols, lanes):
    """P3: phases of 200 rows take a warp per row, phases of 34,000 the block's own lanes."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(n, 0.2, 0)
    P = Problem(xyz, t, 3)
    P.setup(level_smoother=1, max_iter=2)
    P.solve(torch.ones(P.nh, ncols, dtype=torch.float64, device="cuda"), raise_on_fail=False)
    assert P.info.block_lanes in lanes
    P.close()


def _phase_entries(P):
    i = P.info
    return (i.nnz_h - i.n_h) / 2 / i.fine_colours


# phases that let the next one launch after their own wait (FP64, 80,000 to 750,000 entries a
# phase, both forms of the preconditioner), and FP32 slices of 4 lanes, steps and batches
@pytest.mark.parametrize("k,n,prec,mode,lo,hi,lanes", [(2, 28, 0, 0, 80e3, 750e3, 2), (3, 18, 0, 0, 80e3, 750e3, 2),
                                                       (4, 14, 0, 0, 80e3, 750e3, 2), (2, 26, 0, 1, 80e3, 375e3, 2),
                                                       (3, 17, 0, 1, 80e3, 375e3, 2), (2, 28, 1, 0, 110e3, 2e6, 4),
                                                       (3, 32, 1, 0, 5e5, 2e6, 4)])
def test_late_and_middling_slices_match_rows(k, n, prec, mode, lo, hi, lanes):
    """As test_slices_match_rows, at the sizes of these two forms."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(n, 0.2, 0)
    P = Problem(xyz, t, k, kappa_lognormal(t.shape[0], 1))
    r = torch.randn(P.nh, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    out = []
    for layout in (4, 0):
        P.setup(smoother_layout=layout, precond_precision=prec, mode=mode, level_smoother=1)
        assert P.info.smoother_layout == (500 + lanes if layout == 0 else layout)
        out.append(P.apply_prec(r) if mode else P.apply_smoother(r))
    assert lo <= _phase_entries(P) < hi
    longest = 400 if k == 4 else 200
    u = 2.0 ** -24 if prec else 2.0 ** -53
    assert (out[1] - out[0]).norm() <= 2 * P.info.fine_colours * longest * u * out[0].norm()
    P.close()


def test_stokes_components_share_late_sweeps():
    """As test_stokes_components_share_sweeps, with phases of the late form."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(26, 0.2, 0)
    P = Problem(xyz, t, 2)
    out = []
    for layout in (4, 0):
        P.setup(smoother_layout=layout, level_smoother=1)
        P.stokes_setup()
        r = torch.randn(P.stokes_n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        out.append(P.stokes_prec(r)[: 3 * P.nh])
    assert 80e3 <= _phase_entries(P) < 750e3
    assert (out[1] - out[0]).norm() <= _sweep_bound(P, 0) * out[0].norm()
    P.close()


# problems on both sides of the line from which the whole additive preconditioner is one dense
# product: 3375 unknowns of P2 are, of P4 (too many entries) are not; 2744, 64; 4913, 4096 not
@pytest.mark.parametrize("k,n,prec,kw,dense", [(2, 8, 0, {}, 1), (2, 8, 1, {}, 1), (3, 5, 1, {}, 1), (1, 5, 0, {}, 1),
                                               (4, 3, 0, {}, 1), (4, 4, 0, {}, 0), (2, 9, 0, {}, 0), (1, 17, 1, {}, 0),
                                               (2, 8, 0, dict(smoother_layout=4), 0), (2, 8, 0, dict(spmv_threads=8), 0),
                                               (2, 8, 0, dict(mode=1), 0), (2, 8, 0, dict(smoother=1), 0)])
def test_dense_preconditioner_runs_where_it_should(k, n, prec, kw, dense):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(n, 0.2, 0)
    P = Problem(xyz, t, k)
    P.setup(precond_precision=prec, **kw)
    assert P.info.dense_prec == dense
    P.close()


@pytest.mark.parametrize("n,level_smoother,tail", [(17, 0, 0), (19, 0, 1), (22, 1, 2), (32, 0, 2)])
def test_cycle_with_dense_tail_at_each_level(oracle_mod, n, level_smoother, tail):
    torch, G, O = _pair(oracle_mod, 1, n, level_smoother=level_smoother)
    assert G.info.tail_level == tail < G.info.levels - 1
    b = np.random.default_rng(n).standard_normal(G.nH)
    _close(G.apply_vcycle(torch.tensor(b, device="cuda")).cpu().numpy(), O.vcycle(b), 1e-11)

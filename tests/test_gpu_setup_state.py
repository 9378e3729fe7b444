"""What a problem holds before, between and after its setups: memory that is no longer in use
goes back, and a setup that fails leaves none."""
import pytest

from paper_1204_2586_gb300 import _lib as L
from paper_1204_2586_gb300.inputs import kappa_lognormal, kuhn_mesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _problem(k, n):
    from paper_1204_2586_gb300 import Problem

    xyz, t = kuhn_mesh(n, 0.2, 0)
    return Problem(xyz, t, k, kappa_lognormal(t.shape[0], 1))


def _free(torch):
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


MB = 1 << 20


def test_set_kappa_gives_memory_back(torch_cuda):
    """pkasp_set_kappa discards the setup: of its 36 bytes an entry of A_h (FP32 preconditioner:
    split 16, SpMV slices 12, smoother slices 8) no more than 1 GB stays for the next one."""
    torch = torch_cuda
    P = _problem(4, 32)
    P.setup(precond_precision=1, level_smoother=1)
    held = _free(torch)
    P.set_kappa(kappa_lognormal(P.nt, 2))
    assert _free(torch) - held >= 36 * P.info.nnz_h - 1024 * MB
    P.close()


def test_smaller_setup_gives_memory_back(torch_cuda):
    """A setup with fewer copies of A_h than the one before it holds less: 28 bytes an entry of
    slices are gone (SpMV 12, smoother 8, whole rows 8), 64 MB of it may stay in the pool, as
    much again in the parts of its blocks that the smaller setup uses."""
    torch = torch_cuda
    P = _problem(4, 20)
    P.setup(mode=1, precond_precision=1, level_smoother=1)
    held = _free(torch)
    P.setup(smoother=1, precond_precision=1, spmv_threads=4, level_smoother=1)
    assert _free(torch) - held >= 28 * P.info.nnz_h - 128 * MB
    P.close()


def test_setup_out_of_memory_leaves_no_setup(torch_cuda):
    """A second setup with more and more device memory left to it, from almost none to almost
    enough, so that it fails at every stage, the layouts of the last one included. Every
    failure is reported, and no call that needs a setup runs on what is left of either."""
    torch = torch_cuda
    P = _problem(4, 18)
    b = P.rhs()
    y = P.spmv(b)
    small = dict(smoother=1, spmv_threads=4, level_smoother=1)
    big = dict(mode=1, precond_precision=1, level_smoother=1)
    P.setup(**big)
    x = P.solve(b)[0]
    held = _free(torch)
    P.setup(**small)
    need = _free(torch) - held  # what the larger setup takes on top
    assert need > 100 * MB
    failed = 0
    for part in range(24):
        P.setup(**small)
        ballast = torch.empty(_free(torch) - 16 * MB - part * need // 20, dtype=torch.uint8, device="cuda")
        try:
            P.setup(**big)
        except L.PkaspError as e:
            failed += 1
            assert e.code in (L.PKASP_ENOMEM, L.PKASP_ECUDA)
            for call in (P.solve, P.apply_prec, P.apply_smoother, P.stokes_setup):
                with pytest.raises(L.PkaspError) as e:
                    call() if call == P.stokes_setup else call(b)
                assert e.value.code == L.PKASP_ESTATE
            assert P.info.levels == 0
            assert torch.equal(P.spmv(b), y)  # A_h is the problem's, not the setup's
        del ballast
        torch.cuda.empty_cache()
    assert 8 <= failed < 24
    P.setup(**big)
    assert torch.equal(P.solve(b)[0], x)
    P.close()


@pytest.mark.parametrize("krylov", [0, 1])
def test_history_is_one_block(torch_cuda, krylov):
    """Solves that ask for longer and longer histories: 40 of 0.8 to 32 MB, 656 MB in all, of which
    the longest is held, and what they return does not change."""
    torch = torch_cuda
    P = _problem(2, 6)
    b = P.rhs()
    P.setup(krylov=krylov)
    first = P.solve(b, hist_cap=64)[1]["hist"]
    free = _free(torch)
    for i in range(1, 41):
        assert (P.solve(b, hist_cap=100_000 * i)[1]["hist"] == first).all()
    assert free - _free(torch) <= 64 * MB
    P.close()


def test_failed_block_solve_keeps_the_history(torch_cuda):
    """A blocked solve that ends in an error half-way (here: a capture of its stream, which it
    cannot run under) leaves the single-column solves as they were, also past the blocks' end."""
    import ctypes as C

    torch = torch_cuda
    rt = C.CDLL(next(l.split()[-1] for l in open("/proc/self/maps") if "libcudart" in l))
    P = _problem(2, 6)
    b = P.rhs()
    B = torch.stack([b, 2 * b, 3 * b], dim=1).contiguous()
    P.setup()
    x, st = P.solve(b, hist_cap=64)
    X = P.solve(B)[0]
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    assert rt.cudaStreamBeginCapture(C.c_void_p(s.cuda_stream), 2) == 0  # relaxed: this stream alone
    with pytest.raises(L.PkaspError):
        P.solve(B, torch.zeros_like(B), stream=s)
    g = C.c_void_p()
    rt.cudaStreamEndCapture(C.c_void_p(s.cuda_stream), C.byref(g))
    rt.cudaGetLastError()
    assert torch.equal(P.solve(B)[0], X)
    P.set_kappa(kappa_lognormal(P.nt, 1))  # the blocks' memory goes
    P.setup()
    x2, st2 = P.solve(b, hist_cap=64)
    assert torch.equal(x2, x) and (st2["hist"] == st["hist"]).all()
    P.close()


@pytest.mark.parametrize("k,n,prec,mode", [(2, 8, 0, 0), (2, 8, 1, 0), (2, 4, 0, 0), (2, 9, 0, 0), (2, 8, 0, 1), (2, 6, 0, 2)])
def test_preconditioner_in_place(torch_cuda, k, n, prec, mode):
    """z = B r with z on r, or overlapping it: the result of separate vectors, bit for bit,
    whether B is one dense product, sweeps or a cycle."""
    torch = torch_cuda
    P = _problem(k, n)
    P.setup(precond_precision=prec, mode=mode)
    g = torch.Generator("cuda").manual_seed(n)
    r = torch.randn(P.nh, dtype=torch.float64, device="cuda", generator=g)
    z = P.apply_prec(r)
    s = torch.cuda.current_stream().cuda_stream
    for shift in (0, 1, P.nh // 2, P.nh - 1):
        for first in (0, shift):  # r above z, and z above r
            buf = torch.zeros(P.nh + shift, dtype=torch.float64, device="cuda")
            rv, zv = buf[first:first + P.nh], buf[shift - first:shift - first + P.nh]
            rv.copy_(r)
            L.check(L.load().pkasp_apply_prec(P.h, rv.data_ptr(), zv.data_ptr(), s))
            assert torch.equal(zv, z)
    P.close()

"""GPU: the forms of the matvec and of the QMR update that the size of a request
chooses, and the device loop and stream capture of a request whose kernels start
while the ones before them drain.

Tolerances against the oracle are those of the matvec elsewhere (FP64 1e-12 in the
relative 2-norm)."""
import numpy as np
import pytest

from oracle import green, run
from paper_2208_01348_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dd():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2208_01348_gb300 import eelsdda
    return eelsdda


@pytest.fixture()
def ctx(dd):
    h = dd.eels_create(0)
    yield h
    dd.eels_destroy(h)


# FP64 slabs whose rows a block shares: clusters of two, four and eight blocks,
# lattices shorter than their padding, rows that do not fill the last turn
@pytest.mark.parametrize("dims", [(36, 48, 48), (40, 24, 96), (26, 36, 69), (12, 48, 108), (3, 48, 71), (2, 48, 107),
                                  (1, 80, 125), (1, 125, 40), (1, 120, 119), (2, 128, 100)])
def test_fp64_rows_shared_by_a_block_equal_fft_oracle(dd, ctx, dims):
    eps_h, d_nm, e_eV = 2.1 + 0.1j, 1.5, 2.3
    occ = I.box_occupancy(*dims)
    rng = np.random.default_rng(dims[1] * 1000 + dims[2])
    occ *= (rng.random(occ.shape) < 0.8).astype(np.uint8)
    occ.flat[0] = 1
    dd.eels_set_grid(ctx, occ, d_nm)
    eps_p = [I.drude(e_eV)]
    pt = run.setup(*dims, d_nm, occ, e_eV, eps_p, eps_h, (300.0, 300.0), ekin_keV=100.0)
    op = green.FFTOperator(pt.idx, pt.n_axes, pt.d, pt.k, pt.alpha)
    x = I.random_complex((1, len(pt.r), 3), seed=3)
    y = dd.eels_apply_matrix(ctx, dd.EELS_FP64, e_eV, eps_p, eps_h, x)
    ref = op.matvec(x[0])
    assert np.linalg.norm(y[0] - ref) < 1e-12 * np.linalg.norm(ref)


# 3N entries on both sides of each precision's line between one kernel and three, the
# padded points of an x pass on both sides of its line between three lanes and one
@pytest.mark.parametrize("dims,prec,kernels", [((13, 14, 15), "FP64", 4), ((13, 14, 16), "FP64", 6),
                                               ((2, 3, 3), "FP64", 4), ((16, 16, 16), "FP64", 6),
                                               ((11, 11, 31), "FP64", 6), ((28, 28, 27), "MIXED", 4),
                                               ((28, 28, 28), "MIXED", 6)])
def test_kernels_of_a_qmr2_iteration(dd, ctx, dims, prec, kernels):
    """The three kernels of the matvec, and one or three for the vectors: a solve
    launches what the length of the vectors says, reaches the residual it was asked
    for, and three systems together have the bits of each alone."""
    import torch
    S, eps_h = 3, 1.0 + 0j
    dd.eels_set_grid(ctx, I.box_occupancy(*dims), 1.5)
    n = int(np.prod(dims))
    e = np.array([3.4, 3.7, 4.0])
    eps_p = np.array([[I.drude(v)] for v in e])
    p = getattr(dd, "EELS_" + prec)
    dt, eps = (torch.complex128, 1e-9) if prec == "FP64" else (torch.complex64, 1e-5)
    g = torch.Generator(device="cuda").manual_seed(2)
    b = torch.randn((S, 3, n), generator=g, device="cuda", dtype=dt)
    st = torch.cuda.current_stream().cuda_stream

    def solve(i0, i1, tol, most):
        dd.eels_prepare_operator(ctx, e[i0:i1], eps_p[i0:i1], np.full(i1 - i0, eps_h))
        x = torch.zeros_like(b[i0:i1])
        l0 = dd.eels_kernel_launches()
        status, iters = dd.eels_krylov_solve_dev(ctx, p, dd.EELS_QMR2, b[i0:i1].data_ptr(), x.data_ptr(), i1 - i0, tol,
                                                 most, st)
        torch.cuda.synchronize()
        return x, status, iters, dd.eels_kernel_launches() - l0
    x, status, iters, _ = solve(0, S, eps, 3000)
    assert (status == 1).all()
    r = torch.zeros_like(x)
    dd.eels_matvec_dev(ctx, p, x.data_ptr(), r.data_ptr(), S, st)
    for i in range(S):
        # the quasi-residual underestimates the residual by at most sqrt(iterations + 1) <= 55
        assert float(torch.linalg.vector_norm(r[i] - b[i]) / torch.linalg.vector_norm(b[i])) < 55 * eps
        xi, _, it, n_launch = solve(i, i + 1, eps, 3000)
        assert it[0] == iters[i] and torch.equal(xi[0], x[i])
        # three launches start the solve; a replay is six iterations, and the host looks for the end after 1, 2, 4, 8, 8 ...
        replays, burst = 1, 1
        while 6 * replays < it[0]:
            burst = min(8, 2 * burst)
            replays += burst
        assert n_launch == 3 + replays * 6 * kernels


@pytest.mark.parametrize("solver", ["QMR2", "QMR", "BICGSTAB"])
@pytest.mark.parametrize("dims", [(12, 12, 12), (3, 4, 5), (2, 10, 10)])
def test_device_loop_of_a_request_with_dependent_launches(dd, ctx, dims, solver):
    """One FP64 point on a lattice whose passes have at most one block per SM: its
    kernels start while the ones before them drain, in the body of the device loop's
    WHILE node as in the host's replays, and both loops give the same bits."""
    dd.eels_set_grid(ctx, I.box_occupancy(*dims), 20.0 / 12)
    e = np.array([3.4])
    res = []
    for loop in (0, 1):
        o = dd.eels_default_opts(ekin_keV=100.0, precision=dd.EELS_FP64, eps_it=1e-8,
                                 solver=getattr(dd, "EELS_" + solver), n_dir=162, device_loop=loop)
        r = dd.eels_solve(ctx, o, e, I.drude(e)[:, None], np.full(1, 1.0 + 0j), np.array([[30.0, 0.0]]), want_p=True)
        assert r.converged.all()
        res.append(r)
    for key in ("p_eels", "p_cl", "p_ext", "p_abs", "p", "residual", "iters"):
        assert np.array_equal(getattr(res[0], key), getattr(res[1], key)), key


@pytest.mark.parametrize("dims,prec", [((12, 12, 12), "FP64"), ((12, 12, 12), "MIXED"), ((11, 11, 31), "FP64")])
def test_captured_matvec_gives_the_same_bits(dd, ctx, dims, prec):
    """eels_matvec_dev in a caller's stream capture, after a kernel and after a copy of
    the caller's, with and without dependent launches: replays on other inputs give
    the bits of the direct call."""
    import torch
    dd.eels_set_grid(ctx, I.box_occupancy(*dims), 1.5)
    dd.eels_prepare_operator(ctx, [2.4], [[I.drude(2.4)]], [1.0 + 0j])
    p, dt = getattr(dd, "EELS_" + prec), torch.complex128 if prec == "FP64" else torch.complex64
    g = torch.Generator(device="cuda").manual_seed(8)
    n = int(np.prod(dims))
    src = torch.randn((1, 3, n), generator=g, device="cuda", dtype=dt)
    x, y, z = torch.zeros_like(src), torch.zeros_like(src), torch.zeros_like(src)

    def step():
        st = torch.cuda.current_stream().cuda_stream
        x.copy_(src)
        dd.eels_matvec_dev(ctx, p, x.data_ptr(), y.data_ptr(), 1, st)
        x.mul_(2.0)
        dd.eels_matvec_dev(ctx, p, x.data_ptr(), z.data_ptr(), 1, st)
    step()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    for seed in (1, 2):
        src.copy_(torch.randn((1, 3, n), generator=g, device="cuda", dtype=dt))
        step()
        torch.cuda.synchronize()
        want_y, want_z = y.clone(), z.clone()
        y.zero_()
        z.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, want_y) and torch.equal(z, want_z)

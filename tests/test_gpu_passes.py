"""GPU: the matvec's slab and x passes and the batched D-hat build at the
lattices where their plans change, against the FP64 FFT oracle.

Tolerances are those of the matvec elsewhere: FP64 1e-12, FP32 2e-5 in the
relative 2-norm (the FP32 rounding of the transforms grows like
eps32 * log M; the largest lattices here pad to 256 points per axis)."""
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


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _occ(dims, nmat, contiguous):
    nx, ny, nz = dims
    occ = np.ones((nz, ny, nx), dtype=np.uint8)
    if nmat == 2:
        occ[nz // 2:] = 2
    if not contiguous:
        rng = np.random.default_rng(nx * 10007 + ny * 101 + nz)
        occ *= (rng.random(occ.shape) < 0.7).astype(np.uint8)
        occ.flat[0] = 1
    return occ


def _operator(dims, occ, d_nm, e_eV, eps_p, eps_h):
    pt = run.setup(*dims, d_nm, occ, e_eV, eps_p, eps_h, (300.0, 300.0), ekin_keV=100.0)
    return pt, green.FFTOperator(pt.idx, pt.n_axes, pt.d, pt.k, pt.alpha)


@pytest.mark.parametrize("dims,padded", [
    # slabs of one block, of a few rows and of the longest lines
    ((2, 1, 1), None), ((1, 128, 1), None), ((1, 1, 128), None), ((2, 12, 125), None), ((2, 125, 12), None),
    # slabs split over a cluster: FP64 from 128 x 128 points, FP32 from 180 x 180
    ((2, 64, 65), None), ((2, 90, 90), None), ((1, 128, 128), (2, 256, 256)), ((2, 97, 123), (4, 196, 250)),
    # shared-memory x lines: the longest radices and the ends of the range
    ((16, 3, 5), (32, 6, 10)), ((65, 3, 5), None), ((76, 2, 9), None), ((97, 3, 2), None), ((123, 2, 3), (250, 4, 6)),
    ((128, 2, 3), (256, 4, 6)),
    # register x pass with lone tensor-copied tiles: Mz below, at and above a tile of 16 or 8, last tile partial
    ((32, 3, 7), (64, 6, 14)), ((32, 3, 9), (64, 6, 18)), ((31, 4, 13), (64, 8, 28)), ((20, 5, 24), (64, 10, 48)),
    ((64, 3, 3), (128, 6, 6)), ((64, 2, 5), (128, 4, 10)), ((33, 3, 9), (128, 6, 18)), ((50, 3, 12), (128, 6, 24)),
])
@pytest.mark.parametrize("nmat,contiguous", [(1, True), (2, False)])
def test_matvec_at_plan_edges_equals_fft_oracle(dd, ctx, dims, padded, nmat, contiguous):
    occ, d_nm, e_eV, eps_h = _occ(dims, nmat, contiguous), 1.5, 2.3, 2.0 + 0.1j
    nmat = int(occ.max())
    eps_p = [I.drude(e_eV), 3.0 + 0.4j][:nmat]
    dd.eels_set_grid(ctx, occ, d_nm)
    if padded:
        assert tuple(dd.eels_padded_dims(ctx)) == padded
    pt, op = _operator(dims, occ, d_nm, e_eV, eps_p, eps_h)
    x = I.random_complex((2, len(pt.r), 3), seed=3)
    ref = [op.matvec(v) for v in x]
    y64 = dd.eels_apply_matrix(ctx, dd.EELS_FP64, e_eV, eps_p, eps_h, x)
    y32 = dd.eels_apply_matrix(ctx, dd.EELS_MIXED, e_eV, eps_p, eps_h, x)
    for i in range(2):
        assert rel(y64[i], ref[i]) < 1e-12
        assert rel(y32[i], ref[i]) < 2e-5


@pytest.mark.parametrize("dims", [(3, 4, 5), (9, 14, 11), (32, 5, 12), (64, 3, 9), (20, 33, 7)])
@pytest.mark.parametrize("prec", ["FP64", "MIXED"])
def test_batches_of_energies_and_beams_equal_fft_oracle(dd, ctx, dims, prec):
    """Five energies built together, one to three beams each: every system of the
    batch has its energy's D-hat, whatever shares its block."""
    import torch
    energies, beams = [1.4, 1.9, 2.3, 2.8, 3.4], [2, 1, 3, 1, 2]
    occ, d_nm, eps_h = _occ(dims, 2, False), 1.5, 2.1025 + 0j
    dd.eels_set_grid(ctx, occ, d_nm)
    e = np.repeat(energies, beams)
    eps_p = np.stack([[I.drude(v), 2.25 + 0.1j] for v in e])
    dd.eels_prepare_operator(ctx, e, eps_p, np.full(len(e), eps_h))
    n = int(np.count_nonzero(occ))
    x = I.random_complex((len(e), n, 3), seed=9)
    dt = torch.complex128 if prec == "FP64" else torch.complex64
    idx = _operator(dims, occ, d_nm, e[0], list(eps_p[0]), eps_h)[0].idx
    perm = np.lexsort((idx[:, 2], idx[:, 1], idx[:, 0]))         # the library's order: by ix, then iy, then iz
    xt = torch.from_numpy(np.ascontiguousarray(x[:, perm].transpose(0, 2, 1))).to(dt).cuda()
    yt = torch.full_like(xt, float("nan"))
    dd.eels_matvec_dev(ctx, getattr(dd, "EELS_" + prec), xt.data_ptr(), yt.data_ptr(), len(e),
                       torch.cuda.current_stream().cuda_stream)
    y = yt.cpu().numpy().astype(np.complex128)
    for i, ev in enumerate(e):
        pt, op = _operator(dims, occ, d_nm, ev, list(eps_p[i]), eps_h)
        sa = np.sqrt(pt.alpha / pt.d ** 3)[:, None]
        ref = (sa * op.matvec(sa * x[i]) * pt.d ** 3)[perm].T
        assert rel(y[i], ref) < (1e-12 if prec == "FP64" else 2e-5), ev


@pytest.mark.parametrize("dims", [(5, 4, 6), (2, 64, 65), (2, 90, 90), (32, 5, 12)])
@pytest.mark.parametrize("prec", ["FP64", "MIXED"])
def test_lanczos_sums_of_split_slabs(dd, ctx, dims, prec):
    """The inner solve uses the matvec's own partial sums of p^T A p, one per
    block of a slab: QMR2 reduces the true residual on lattices whose slabs
    are whole and split."""
    import torch
    occ, d_nm, e_eV, eps_h = _occ(dims, 1, True), 1.5, 3.6, 1.0 + 0j
    dd.eels_set_grid(ctx, occ, d_nm)
    eps_p = [I.drude(e_eV)]
    dd.eels_prepare_operator(ctx, [e_eV], [eps_p], [eps_h])
    p = getattr(dd, "EELS_" + prec)
    dt, eps = (torch.complex128, 1e-9) if prec == "FP64" else (torch.complex64, 1e-5)
    g = torch.Generator(device="cuda").manual_seed(4)
    b = torch.randn((1, 3, int(np.count_nonzero(occ))), generator=g, device="cuda", dtype=dt)
    x, r = torch.zeros_like(b), torch.zeros_like(b)
    st = torch.cuda.current_stream().cuda_stream
    status, _ = dd.eels_krylov_solve_dev(ctx, p, dd.EELS_QMR2, b.data_ptr(), x.data_ptr(), 1, eps, 5000, st)
    assert status[0] == 1
    dd.eels_matvec_dev(ctx, p, x.data_ptr(), r.data_ptr(), 1, st)
    # the quasi-residual underestimates the residual by at most sqrt(iterations + 1) <= 71
    assert float(torch.linalg.vector_norm(r - b) / torch.linalg.vector_norm(b)) < 71 * eps


@pytest.mark.parametrize("dims,prec", [((11, 11, 31), "FP64"), ((11, 11, 31), "MIXED"), ((3, 4, 5), "FP64"),
                                       ((24, 20, 30), "FP64"), ((30, 27, 28), "MIXED")])
def test_qmr2_bits_do_not_depend_on_the_batch(dd, ctx, dims, prec):
    """3N entries decide how an iteration's vectors are cut up and whether one kernel
    or three run them: 16 systems together and the first and last of them alone
    give the same bits."""
    import torch
    occ, d_nm, eps_h = _occ(dims, 1, True), 1.5, 1.0 + 0j
    dd.eels_set_grid(ctx, occ, d_nm)
    n, S = int(np.count_nonzero(occ)), 16
    e = np.linspace(3.3, 4.0, S)
    eps_p = np.stack([[I.drude(v)] for v in e])
    p = getattr(dd, "EELS_" + prec)
    dt, eps = (torch.complex128, 1e-9) if prec == "FP64" else (torch.complex64, 1e-5)
    g = torch.Generator(device="cuda").manual_seed(6)
    b = torch.randn((S, 3, n), generator=g, device="cuda", dtype=dt)
    st = torch.cuda.current_stream().cuda_stream

    def solve(i0, i1):
        dd.eels_prepare_operator(ctx, e[i0:i1], eps_p[i0:i1], np.full(i1 - i0, eps_h))
        x = torch.zeros_like(b[i0:i1])
        status, iters = dd.eels_krylov_solve_dev(ctx, p, dd.EELS_QMR2, b[i0:i1].data_ptr(), x.data_ptr(), i1 - i0, eps,
                                                 2000, st)
        torch.cuda.synchronize()
        assert (status == 1).all()
        return x, iters
    x, iters = solve(0, S)
    for i in (0, S - 1):
        xi, it = solve(i, i + 1)
        assert it[0] == iters[i] and torch.equal(xi[0], x[i])

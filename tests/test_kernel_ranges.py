"""Kernels over the rest of their range: matrices beyond the usual survey (rows that no longer fit in
shared memory, columns beyond a warp's registers), the FP32 Gram's skipped padding, and the first and
last levels of a modelling run; against 64-bit references of the same operation."""
import numpy as np
import pytest

import oracle
from test_kernel_edges import _line_ctx
from test_limits import _load_set

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 8, 9, 100, 312, 313, 400, 433, 434, 461])
def test_largest_eigenvalue(n):
    """EGH_MU_REL_MAXEIG against the 64-bit spectrum of the same Hessians: fewer rows than a cluster has
    blocks, rows kept as doubles (to 312), as floats, and read from L2 (from 434).  The transforms have a
    constant part, so that the largest eigenvalue stands well apart and 300 steps reach it; the library's
    sums are FP64 (n 2^-53 each, and the 64-bit reference's own)."""
    import torch
    from paper_2512_16642_gb300 import egh

    torch.manual_seed(n)
    with egh.Context(4, 512, 10.0, 10.0, 0, 0.5, 1e-3, 100, np.zeros(n, np.int32),
                     np.arange(n, dtype=np.int32), np.array([5.0, 9.0]), precision=0) as ctx:
        buf = ctx.transform_buffer(n, 2)
        buf.normal_()
        buf.add_(0.5)
        ctx.import_green(buf)
        ctx.hessian(egh.EGH_MU_ABS, 0.0)
        Q = ctx.get_hessian(False).astype(np.complex128)
        mu = ctx.hessian(egh.EGH_MU_REL_MAXEIG, 0.25)
    assert mu == pytest.approx(oracle.mu_max_eig(Q, 0.25), rel=1e-11)


@pytest.mark.parametrize("n", [2, 161, 345, 441, 442, 461])
def test_condition_bound(n, tmp_path):
    """The bound 1.25 ||Q||_F / lambda_min from the power iteration on the inverse (rows of the inverse
    in shared memory to 441 receivers, then in part from L2), for Q = I - 0.95 u u^H, whose smallest
    eigenvalue 0.05 stands apart: the iteration has converged after a few steps, and what is left is the
    FP32 rounding of the inverse, the condition 20 times n 2^-24 at most."""
    rng = np.random.default_rng(n)
    u = rng.standard_normal((2, n)) + 1j * rng.standard_normal((2, n))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    Q = (np.eye(n) - 0.95 * u[:, :, None] * u[:, None, :].conj()).astype(np.complex64)
    with _line_ctx(n, 2, 100, 1) as ctx:
        _load_set(ctx, Q, tmp_path, mu=1e-30)
        got = ctx.get_refinement()[0]
    for k in range(2):
        q = Q[k].astype(np.complex128)
        want = 1.25 * np.linalg.norm(q) / np.linalg.eigvalsh(q)[0]
        assert abs(got[k] / want - 1) <= 20 * n * 2.0 ** -24, k


@pytest.mark.parametrize("n", [384, 385, 400, 461, 801, 1537])
def test_inverse_of_large_sets(n, tmp_path):
    """Mixed-precision solves (Q X = D, D the transform with Q = I) of sets whose columns reach past the
    groups that a warp of the inverse factor reads ahead (from 385 rows), of the column form of the
    factorisation (from 801) and of one column per warp (from 1537): backward error n u with u = 2^-24,
    times 2 for the product with the inverse and the correction."""
    import torch

    rng = np.random.default_rng(n)
    nt, ns = 200, 3
    A = rng.standard_normal((n, n + 4)) + 1j * rng.standard_normal((n, n + 4))
    Q = A @ A.conj().T / (n + 4) + 0.05 * np.eye(n)
    Q = (0.5 * (Q + Q.conj().T)).astype(np.complex64)[None]
    r = torch.from_numpy(rng.standard_normal((ns, n, nt)).astype(np.float32)).cuda()
    out = {}
    for name, M in (("D", np.eye(n, dtype=np.complex64)[None]), ("X", Q)):
        with _line_ctx(n, 1, nt, 1) as ctx:
            _load_set(ctx, M, tmp_path)
            x = torch.zeros((1, n, ns, 2), device="cuda")
            ctx.deblur_freq(r, x)
            torch.cuda.synchronize()
            out[name] = torch.view_as_complex(x).cpu().numpy()[0].astype(np.complex128)
    q = Q[0].astype(np.complex128)
    res = np.linalg.norm(out["D"] - q @ out["X"])
    assert res <= 2 * n * 2.0 ** -24 * np.linalg.eigvalsh(q)[-1] * np.linalg.norm(out["X"])


@pytest.mark.parametrize("nrec", [5, 40, 70, 97])
@pytest.mark.parametrize("nz,nx,gram_splits", [(9, 61, 0), (31, 61, 7), (40, 20, 3), (17, 130, 5)])
def test_gram_skips_only_zeros(nrec, nz, nx, gram_splits):
    """The FP32 Hessian of a context's own transforms leaves their padding columns out; imported ones
    count them.  The padding is zero, so both give the same bits, on grids whose rows are half padding
    and with point ranges that begin inside it."""
    import torch
    from paper_2512_16642_gb300 import egh

    rng = np.random.default_rng(nrec + nx)
    v = torch.from_numpy((2000.0 + 500.0 * rng.random((nz, nx))).astype(np.float32)).cuda()
    args = (nz, nx, 10.0, 10.0, 0, 0.5, 1e-3, 50, np.zeros(nrec, np.int32),
            (np.arange(nrec) % nx).astype(np.int32), np.array([12.0, 25.0]))
    with egh.Context(*args, gram_splits=gram_splits) as ctx:
        ctx.green(v)
        ctx.hessian(egh.EGH_MU_ABS, 0.0)
        own = ctx.get_hessian(False)
        buf = ctx.transform_buffer(nrec, 2)
        ctx.export_green(0, 2, buf)
    with egh.Context(*args, gram_splits=gram_splits) as ctx:
        ctx.import_green(buf)
        ctx.hessian(egh.EGH_MU_ABS, 0.0)
        assert np.array_equal(ctx.get_hessian(False), own)
    assert np.abs(own).max() > 0


@pytest.mark.parametrize("kw", [{}, {"batch_receivers": 4}])
@pytest.mark.parametrize("nt", [1, 2, 3, 40])
def test_modelling_of_few_levels(nt, kw):
    """Traces of egh_forward against the FP64 oracle: records of one to three levels (the first and last
    are recorded outside the steps), an odd number of sources in several batches, sources at the edges
    of row tiles and of 64-column tiles, two at one point, and a wavelet that is zero in the middle and
    at the end.  FP32 time stepping of 40 levels: 1e-4 as for the other modelling tests."""
    import torch
    from paper_2512_16642_gb300 import egh

    rng = np.random.default_rng(nt)
    nz, nx, ns = 30, 140, 3
    v = (2000.0 + 500.0 * rng.random((nz, nx))).astype(np.float32)
    src = [(0, 0), (8, 60), (9, 61), (11, 60), (12, 61), (20, 124), (21, 125), (29, 139), (13, 70), (13, 70),
           (5, 5), (6, 6), (7, 7), (8, 8), (9, 9), (10, 10), (11, 11), (12, 12), (15, 100)]
    iz, ix = (np.array([s[i] for s in src], np.int32) for i in (0, 1))
    rx = np.arange(0, nx, 6).astype(np.int32)
    rz = (np.arange(rx.size) % nz).astype(np.int32)
    wav = rng.standard_normal(nt).astype(np.float32)
    wav[2:5] = 0.0
    wav[10:13] = 0.0
    wav[30:] = 0.0
    with egh.Context(nz, nx, 10.0, 10.0, ns, 1e-3, 1e-3, nt, rz, rx, np.array([12.0]), **kw) as ctx:
        data = torch.full((iz.size, rx.size, nt), float("nan"), device="cuda")
        ctx.forward(torch.from_numpy(v).cuda(), iz, ix, wav, data)
        got = data.cpu().numpy()
    grid = oracle.Grid(v.astype(np.float64), 10.0, 10.0, ns, 1e-3)
    ref = oracle.forward_traces(grid, iz, ix, rz, rx, wav.astype(np.float64), 1e-3, workers=4)
    assert got.shape == ref.shape and np.all(np.isfinite(got))
    assert np.linalg.norm(got - ref) <= 1e-4 * np.linalg.norm(ref)
    assert np.all(got[..., 0] == 0.0)

"""Kernels at the sizes where they can go wrong: edges of tiles, remainders, smallest and largest
of a dispatch's range, against 64-bit references of the same operation.

Solves are judged by their backward error ||D - Q X|| / (||Q|| ||X||), which a stable FP32 solve
keeps at a small multiple of the unit roundoff (6e-8) whatever the condition of Q; 2e-6 leaves
room for the growth with the matrix size (n u at n = 33) and for the transform in front of it
(bf16x3, about 1e-5 of the right-hand side, does not enter: the residual is taken against the
spectra the library itself computed for a unit-diagonal set).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _hpd(rng, nf, n):
    A = rng.standard_normal((nf, n, n + 4)) + 1j * rng.standard_normal((nf, n, n + 4))
    Q = A @ A.conj().transpose(0, 2, 1) / (n + 4) + 0.05 * np.eye(n)
    return (0.5 * (Q + Q.conj().transpose(0, 2, 1))).astype(np.complex64)


def _line_ctx(n, nf, nt, precision):
    """A context on a small grid with n receivers (two may share a column when n is large)."""
    from paper_2512_16642_gb300 import egh

    nx = max(64, n)
    return egh.Context(4, nx, 10.0, 10.0, 0, 0.5, 1e-3, nt, np.zeros(n, np.int32),
                       np.arange(n, dtype=np.int32) % nx, np.linspace(5.0, 40.0, nf), precision=precision)


def _load_set(ctx, Q, tmp_path):
    """Puts given Hessians into a context through the set-file format (egh_save / egh_load)."""
    import json
    import struct

    nf, n, _ = Q.shape
    h = json.dumps({"format": "egh Hessian set", "version": 1, "nrec": n, "nfreq": nf,
                    "freq_hz": [float(f) for f in ctx.freqs], "dt": 1e-3, "nt": ctx.nt,
                    "precision": ctx.prec_for_test, "mu": 0.05, "rec_iz": [0] * n,
                    "rec_ix": [int(i) % max(64, n) for i in range(n)]}).encode()
    p = tmp_path / "set.bin"
    p.write_bytes(b"EGHQSET1" + struct.pack("<Q", len(h)) + h + Q.tobytes() + Q.tobytes())
    ctx.load(str(p))


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("n,ns", [(1, 1), (2, 3), (31, 16), (32, 17), (33, 4), (64, 5), (65, 33), (161, 57),
                                  (230, 1), (345, 40)])
def test_solve_backward_error(n, ns, precision, tmp_path):
    """X of egh_deblur_freq against the spectra D (the same transform with Q = I): Q X = D."""
    import torch

    rng = np.random.default_rng(100 * n + ns)
    nf, nt = 3, 200
    Q = _hpd(rng, nf, n)
    r = torch.from_numpy(rng.standard_normal((ns, n, nt)).astype(np.float32)).cuda()
    out = {}
    for name, M in (("D", np.broadcast_to(np.eye(n, dtype=np.complex64), Q.shape).copy()), ("X", Q)):
        with _line_ctx(n, nf, nt, precision) as ctx:
            ctx.prec_for_test = precision
            _load_set(ctx, M, tmp_path)
            x = torch.zeros((nf, n, ns, 2), device="cuda")
            ctx.deblur_freq(r, x)
            torch.cuda.synchronize()
            out[name] = torch.view_as_complex(x).cpu().numpy().astype(np.complex128)
    for k in range(nf):
        q = Q[k].astype(np.complex128)
        res = np.linalg.norm(out["D"][k] - q @ out["X"][k])
        assert res <= 2e-6 * np.linalg.norm(q, 2) * np.linalg.norm(out["X"][k]), (k, res)


@pytest.mark.parametrize("nf", [3, 16, 17, 33, 48, 49])
@pytest.mark.parametrize("n,ns,nt", [(1, 1, 64), (5, 1, 256), (127, 1, 388), (129, 1, 4000), (64, 5, 2052), (40, 60, 900),
                                     (7, 3, 2001)])
def test_forward_transform(n, ns, nt, nf, tmp_path):
    """Spectra of egh_deblur_freq with Q = I (the product with the identity is exact) against the
    64-bit transform: traces of one tile, a few tiles and many,
    one stage to many (block sums from scratch), every width of the component dimension, rows that are not a multiple of
    16 bytes.  The bf16 pairs carry 16 bits: 2^-17 per factor, 2e-5 of the spectra's norm with room
    for the dropped product."""
    import torch

    rng = np.random.default_rng(n + ns + nt + nf)
    r = rng.standard_normal((ns, n, nt)).astype(np.float32)
    with _line_ctx(n, nf, nt, 1) as ctx:
        ctx.prec_for_test = 1
        _load_set(ctx, np.broadcast_to(np.eye(n, dtype=np.complex64), (nf, n, n)).copy(), tmp_path)
        x = torch.zeros((nf, n, ns, 2), device="cuda")
        for _ in range(2):  # again on the same scratch
            ctx.deblur_freq(torch.from_numpy(r).cuda(), x)
        torch.cuda.synchronize()
        got = torch.view_as_complex(x).cpu().numpy()
        ph = 2 * np.pi * np.mod(ctx.freqs[:, None] * np.arange(nt)[None] * 1e-3, 1.0)
        many = torch.from_numpy(np.concatenate([r] * (-(-20000 // (n * ns))))).cuda() if n * ns < 200 else None
        if many is not None:  # the same traces among many others: the same bits
            y = torch.zeros((nf, n, many.shape[0], 2), device="cuda")
            ctx.deblur_freq(many, y)
            assert torch.equal(y[:, :, :ns], x) and torch.equal(y[:, :, -ns:], x)
    ref = np.einsum("kt,srt->krs", np.exp(-1j * ph), r.astype(np.float64), optimize=True)
    assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("nrec", [1, 16, 24, 33, 48, 49, 97])
@pytest.mark.parametrize("nx,nz,gram_splits", [(64, 3, 0), (60, 7, 1), (61, 40, 5), (130, 33, 0)])
def test_gram_fp32(nrec, nx, nz, gram_splits):
    """FP32 Hessians of imported transforms against the 64-bit Gram: one tile to several of either
    edge, last panels with few rows, point ranges that begin and end inside a grid row, zero
    padding columns.  FP32 products and sums over at most 4000 points with chains of at most 1024:
    random rounding stays below 1e-6 of the Hessian's norm."""
    import torch
    from paper_2512_16642_gb300 import egh

    rng = np.random.default_rng(nrec + nx)
    nf = 2
    ix = np.arange(nrec, dtype=np.int32) % nx
    with egh.Context(nz, nx, 10.0, 10.0, 0, 0.5, 1e-3, 100, np.zeros(nrec, np.int32), ix,
                     np.array([5.0, 9.0]), precision=0, gram_splits=gram_splits) as ctx:
        buf = ctx.transform_buffer(nrec, nf)
        px = ctx.stats()["pitch"]
        v = rng.standard_normal((nrec, nf, 2, nz, nx)).astype(np.float32)
        buf[..., : nz * px].unflatten(-1, (nz, px))[..., :nx] = torch.from_numpy(v).cuda()
        ctx.import_green(buf)
        ctx.hessian(egh.EGH_MU_ABS, 0.0)
        Q = ctx.get_hessian(False)
    g = (v[:, :, 0] + 1j * v[:, :, 1]).reshape(nrec, nf, -1).astype(np.complex128)
    for k in range(nf):
        H = g[:, k] @ g[:, k].conj().T
        assert np.linalg.norm(Q[k] - H) <= 1e-6 * np.linalg.norm(H), k


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nrec", [1, 7, 8, 9, 57, 63, 64, 65, 100, 129, 200])
def test_gram_of_whole_planes(nrec, precision):
    """Hessians of imported transforms sum over the whole planes, padding included, for every width of
    the last panel (one receiver, a multiple of eight, one less and one more) in the first or second
    half of a block.  Tensor cores: 2^-17 per factor of the bf16 pairs, 2e-5 of the norm with room for
    the dropped product; FP32 as above."""
    import torch
    from paper_2512_16642_gb300 import egh

    nz, nx, nf = 9, 70, 3
    torch.manual_seed(nrec)
    ix = np.arange(nrec, dtype=np.int32) % nx
    with egh.Context(nz, nx, 10.0, 10.0, 4, 0.5, 1e-3, 100, np.zeros(nrec, np.int32), ix,
                     np.array([5.0, 9.0, 11.0]), precision=precision) as ctx:
        buf = ctx.transform_buffer(nrec, nf)
        buf.normal_()
        ctx.import_green(buf)
        ctx.hessian(egh.EGH_MU_ABS, 0.0)
        Q = ctx.get_hessian(False)
    v = buf.cpu().numpy().astype(np.float64)
    for k in range(nf):
        g = v[:, k, 0] + 1j * v[:, k, 1]
        H = g @ g.conj().T
        assert np.linalg.norm(Q[k] - H) <= (1e-6, 2e-5)[precision] * np.linalg.norm(H), k


@pytest.mark.parametrize("nz,nx,nsponge,nrec,nt,decim,kw", [
    (12, 29, 10, 5, 77, 1, {"dft_chunk": 32}),     # 32 rows: four per block, an odd column count
    (26, 90, 5, 7, 70, 1, {}),                     # uneven rows, one chunk
    (101, 101, 20, 12, 150, 1, {"dft_chunk": 64}), # the small model's grid, several chunks
    (101, 101, 20, 3, 131, 4, {"dft_chunk": 32}),  # band-limited, decimated
    (37, 64, 0, 9, 100, 7, {"batch_receivers": 4, "dft_chunk": 32}),  # no sponge, ragged batches
    (215, 230, 20, 4, 60, 1, {}),                  # (few receivers on a larger grid: the per-step kernel)
    (215, 230, 20, 20, 60, 1, {}),                 # the largest slabs: coefficients from global memory
])
def test_cluster_solver_equals_per_step_kernel(nz, nx, nsponge, nrec, nt, decim, kw):
    """Small grids: the cluster solver's transforms are the per-step kernel's bit for bit (the same
    operations per point in the same order)."""
    import torch
    from paper_2512_16642_gb300 import egh

    rng = np.random.default_rng(nz + nx)
    v = torch.from_numpy((2000.0 + 500.0 * rng.random((nz, nx))).astype(np.float32)).cuda()
    ix = np.linspace(0, nx - 1, nrec).round().astype(np.int32)
    iz = (np.arange(nrec) * 3 % nz).astype(np.int32)
    t = np.arange(40) * 1e-3 - 0.02
    a = (np.pi * 30.0 * t) ** 2
    wav = ((1 - 2 * a) * np.exp(-a)).astype(np.float32)
    out = {}
    for fk in (0, 2):
        with egh.Context(nz, nx, 10.0, 10.0, nsponge, 1e-3 if nsponge else 0.5, 1e-3, nt, iz, ix,
                         np.array([12.0, 25.0]), fd_kernel=fk, **kw) as ctx:
            for _ in range(2):  # again on used slots
                if decim == 1:
                    ctx.green(v)
                else:
                    ctx.green_bandlimited(v, wav, decim)
            out[fk] = ctx.get_green()
            assert ctx.stats()["fd_kernel"] == (3 if fk == 0 and (nz, nrec) != (215, 4) else 2)
    assert np.array_equal(out[0], out[2])


@pytest.mark.parametrize("nf", [3, 33, 64])
@pytest.mark.parametrize("n,ns,nt,off", [(1, 1, 1, 0), (3, 1, 5, 1), (5, 3, 63, 2), (17, 2, 65, 3), (129, 1, 130, 0),
                                         (43, 3, 1021, 1), (64, 2, 514, 2)])
def test_ragged_rows(n, ns, nt, off, nf, tmp_path):
    """Traces that are not a multiple of four samples, in buffers that start 4, 8 or 12 bytes past a
    16-byte boundary: spectra and multipliers against the 64-bit transform and synthesis (Q = I).
    Two bf16-pair products in a row: 4e-5 of the multipliers' norm."""
    import torch

    rng = np.random.default_rng(n * ns + nt)
    r = rng.standard_normal((ns, n, nt)).astype(np.float32)
    flat = torch.full((off + r.size + 8,), float("nan"), device="cuda")  # (read past the rows shows)
    rd = flat[off: off + r.size].view(ns, n, nt)
    rd.copy_(torch.from_numpy(r))
    out = torch.full((off + r.size + 8,), 7.0, device="cuda")
    md = out[off: off + r.size].view(ns, n, nt)
    with _line_ctx(n, nf, max(nt, 2), 1) as ctx:
        ctx.prec_for_test = 1
        _load_set(ctx, np.broadcast_to(np.eye(n, dtype=np.complex64), (nf, n, n)).copy(), tmp_path)
        ctx.deblur(rd, md)
        torch.cuda.synchronize()
        f = ctx.freqs
    ph = 2 * np.pi * np.mod(f[:, None] * np.arange(nt)[None] * 1e-3, 1.0)
    X = np.einsum("kt,srt->krs", np.exp(-1j * ph), r.astype(np.float64), optimize=True)
    w = 2e-3 * np.gradient(f)
    ref = np.einsum("k,krs,kt->srt", w, X, np.exp(1j * ph), optimize=True).real
    assert np.linalg.norm(md.cpu().numpy() - ref) <= 4e-5 * np.linalg.norm(ref)
    assert bool((out[:off] == 7.0).all()) and bool((out[off + r.size:] == 7.0).all())

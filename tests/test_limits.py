"""What a call may rely on whatever other calls do: contexts of different sizes in different host
threads and in batches, calls under stream capture, and the digits of the smallest steps."""
import threading

import numpy as np
import pytest

from test_kernel_edges import _line_ctx

pytestmark = pytest.mark.gpu


def _load_set(ctx, Q, tmp_path, mu=0.05):
    """Puts given Hessians and their penalty into a mixed-precision context (the set-file format)."""
    import json
    import struct

    nf, n, _ = Q.shape
    h = json.dumps({"format": "egh Hessian set", "version": 1, "nrec": n, "nfreq": nf,
                    "freq_hz": [float(f) for f in ctx.freqs], "dt": 1e-3, "nt": ctx.nt, "precision": 1,
                    "mu": mu, "rec_iz": [0] * n, "rec_ix": [int(i) % max(64, n) for i in range(n)]}).encode()
    p = tmp_path / "set.bin"
    p.write_bytes(b"EGHQSET1" + struct.pack("<Q", len(h)) + h + Q.tobytes() + Q.tobytes())
    ctx.load(str(p))


def _in_threads(*work):
    """Runs the functions side by side; the first exception of any is raised."""
    errors = []
    start = threading.Barrier(len(work))

    def run(f):
        try:
            start.wait()
            f()
        except BaseException as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=run, args=(f,)) for f in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]


def _random_ctx(n, nf, precision):
    """A context whose transforms are random numbers: Hessians of n receivers over 4 x 512 points."""
    from paper_2512_16642_gb300 import egh

    ctx = egh.Context(4, 512, 10.0, 10.0, 0, 0.5, 1e-3, 100, np.zeros(n, np.int32),
                      np.arange(n, dtype=np.int32), np.linspace(5.0, 40.0, nf), precision=precision)
    buf = ctx.transform_buffer(n, nf)
    buf.normal_()
    ctx.import_green(buf)
    return ctx


def test_threads_with_contexts_of_different_sizes():
    """Distinct contexts are independent: two host threads build penalties and factors of 161 and 341
    receivers at the same time, again and again; each gets what it got alone."""
    import torch
    from paper_2512_16642_gb300 import egh

    torch.manual_seed(5)
    ctxs = [_random_ctx(n, 2, 1) for n in (161, 341)]
    try:
        alone = []
        for c in ctxs:
            mu = c.hessian(egh.EGH_MU_REL_MAXEIG, 1e-2)
            c.factor()
            alone.append((mu, c.get_hessian(True), c.get_refinement()[0]))

        def loop(c, want):
            for _ in range(200):
                assert c.hessian(egh.EGH_MU_REL_MAXEIG, 1e-2) == want[0]
                c.factor()
            assert np.array_equal(c.get_hessian(True), want[1])
            assert np.array_equal(c.get_refinement()[0], want[2])

        _in_threads(*(lambda c=c, w=w: loop(c, w) for c, w in zip(ctxs, alone)))
    finally:
        for c in ctxs:
            c.close()


def test_threads_with_grids_of_different_sizes():
    """As above for the Green stage of small grids and the creation of contexts beside it."""
    import torch
    from paper_2512_16642_gb300 import egh

    grids = [(101, 101), (60, 61), (101, 150)]

    def make(nz, nx):
        return egh.Context(nz, nx, 10.0, 10.0, 10, 1e-3, 1e-3, 40, np.zeros(4, np.int32),
                           np.arange(4, dtype=np.int32), np.array([12.0, 25.0]), dft_chunk=32)

    vel = [torch.full(g, 2000.0, device="cuda") for g in grids]
    alone = []
    for g, v in zip(grids, vel):
        with make(*g) as c:
            c.green(v)
            alone.append(c.get_green())
    torch.cuda.synchronize()

    def loop(i):
        for _ in range(8):
            with make(*grids[i]) as c:
                for _ in range(10):
                    c.green(vel[i])
                assert np.array_equal(c.get_green(), alone[i])

    _in_threads(*(lambda i=i: loop(i) for i in range(len(grids))))


def test_small_batch_after_a_large_one(tmp_path):
    """A batch of small matrices created after one of large matrices takes nothing from it."""
    from paper_2512_16642_gb300 import egh

    rng = np.random.default_rng(3)
    ctxs = []
    try:
        for n in (200, 9):
            A = rng.standard_normal((2, n, 2 * n)) + 1j * rng.standard_normal((2, n, 2 * n))
            Q = (A @ A.conj().transpose(0, 2, 1) / n + 0.1 * np.eye(n)).astype(np.complex64)
            c = _line_ctx(n, 2, 100, 1)
            ctxs.append(c)
            _load_set(c, Q, tmp_path)
        single = [c.get_hessian(True) for c in ctxs]
        with egh.Batch(ctxs[:1]) as big, egh.Batch(ctxs[1:]) as small:
            big.factor()
            small.factor()
        for c, L in zip(ctxs, single):
            assert np.array_equal(c.get_hessian(True), L)
    finally:
        for c in ctxs:
            c.close()


def test_capture_of_a_smaller_deblur(tmp_path):
    """After one call on device buffers, calls of fewer sources take no device memory (their workspaces
    stand), so that they can be captured: the replay gives the bits of the call."""
    import torch

    n, nf, nt = 129, 26, 2000
    torch.manual_seed(1)
    r = torch.randn((60, n, nt), device="cuda")
    big, one, again = torch.empty_like(r), torch.empty_like(r[:1]), torch.empty_like(r[:1])
    with _line_ctx(n, nf, nt, 1) as ctx:
        _load_set(ctx, np.broadcast_to(np.eye(n, dtype=np.complex64), (nf, n, n)).copy(), tmp_path)
        ctx.deblur(r, big)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, capture_error_mode="thread_local"):
            ctx.deblur(r[:1], again)
        g.replay()
        ctx.deblur(r[:1], one)
        torch.cuda.synchronize()
        assert torch.equal(one, big[:1]) and torch.equal(again, one)


@pytest.mark.parametrize("fd_kernel", [0, 2])
def test_transform_totals_below_the_normal_range(fd_kernel):
    """Sums over several chunks whose totals lie below 2^-126 lose nothing.  A medium so slow that the
    impulse stays where it is: u(t) = t u(1) with u(1) = 2^-133; at a quarter of the sampling rate the
    twiddles are 0 and +-1, so that every term and total is an integer times 2^-133 and exact."""
    import torch
    from paper_2512_16642_gb300 import egh

    nt = 160
    v = torch.full((40, 40), float(np.sqrt(2.0 ** -113) / 1e-3), device="cuda")
    with egh.Context(40, 40, 1024.0, 1024.0, 0, 0.5, 1e-3, nt, np.array([20], np.int32), np.array([7], np.int32),
                     np.array([250.0]), dft_chunk=32, fd_kernel=fd_kernel) as ctx:
        ctx.green(v)
        g = ctx.get_green()[0, 0]
    t = np.arange(nt)
    want = np.sum(t * (-1j) ** (t % 4))
    assert abs(want) < 2.0 ** 7
    got = g[20, 7].astype(np.complex128) * 2.0 ** 133
    assert got == want


def test_pivot_is_the_rounded_64_bit_root(tmp_path):
    """Mixed precision's pivots: L22 = float(sqrt(a - x^2)) of [[1, x], [x, a]], the difference and its
    root in 64 bits, for pairs whose root lies next to the middle between two floats."""
    pairs = [("0x1.09ed800000000p+1", "0x1.71f6b40000000p-13"), ("0x1.884f1e0000000p+1", "0x1.3b94ee0000000p-12"),
             ("0x1.6db68c0000000p+1", "0x1.d1c4960000000p-12"), ("0x1.81d2960000000p+0", "0x1.38d3c60000000p-13"),
             ("0x1.8000000000000p+1", "0x1.0000000000000p-12")]
    a, x = (np.array([float.fromhex(p[i]) for p in pairs]) for i in (0, 1))
    Q = np.zeros((len(pairs), 2, 2), np.complex64)
    Q[:, 0, 0], Q[:, 0, 1], Q[:, 1, 0], Q[:, 1, 1] = 1.0, x, x, a
    with _line_ctx(2, len(pairs), 100, 1) as ctx:
        _load_set(ctx, Q, tmp_path)
        L = ctx.get_hessian(True)
    assert np.array_equal(L[:, 1, 0].real, x.astype(np.float32))
    assert np.array_equal(L[:, 1, 1].real, np.sqrt(a - x * x).astype(np.float32))


@pytest.mark.parametrize("n,v", [(341, 0.32015), (461, 0.39017), (860, 0.5487)])
def test_frobenius_norm_of_the_condition_bound(n, v, tmp_path):
    """The condition bound ||Q||_F / mu (mu above the smallest eigenvalue's estimate) of a matrix whose
    entries are all equal but the diagonal ones, so that every partial sum rounds the same way: FP64
    sums of at most 2 n^2 / 256 terms, joined in a few steps, are off by at most half of
    (n^2 / 128 + 40) 2^-53, and the root and the quotient by two roundings."""
    Q = np.full((1, n, n), np.float32(v), np.complex64)
    Q[0, np.arange(n), np.arange(n)] = 1.0
    with _line_ctx(n, 1, 100, 1) as ctx:
        _load_set(ctx, Q, tmp_path, mu=16.0)
        got = ctx.get_refinement()[0][0]
    off = float(np.float32(v)) ** 2  # exact in 64 bits, as are its multiples below
    want = np.sqrt(n + n * (n - 1) * off) / 16.0
    assert abs(got / want - 1) <= (n * n / 128 + 40) / 2 * 2.0 ** -53 + 2.0 ** -51


@pytest.mark.parametrize("nz,nx,nrec,nf,solver", [(101, 101, 21, 5, 3), (151, 201, 12, 26, 3), (215, 230, 6, 26, 2),
                                                  (201, 201, 100, 60, 2), (231, 238, 24, 60, 2)])
def test_solver_of_a_small_grid(nz, nx, nrec, nf, solver):
    """The solver that is clearly the faster one is taken: with many frequencies the clusters leave the
    transform too few SMs."""
    from paper_2512_16642_gb300 import egh

    with egh.Context(nz, nx, 10.0, 10.0, 20, 1e-3, 1e-3, 100, np.zeros(nrec, np.int32),
                     np.arange(nrec, dtype=np.int32), np.linspace(3.0, 15.0, nf)) as ctx:
        assert ctx.stats()["fd_kernel"] == solver


def test_server_keeps_what_its_solves_read():
    """A mixed-precision set of a server holds its Hessians and the operand images of their inverses
    (48 KB per 128 rows x 32 columns), not the factors they were made from."""
    import torch
    from paper_2512_16642_gb300 import egh

    n, nf = 257, 40
    A = np.random.default_rng(1).standard_normal((n, 2 * n))
    Q = np.broadcast_to((A @ A.T / n + np.eye(n)).astype(np.complex64), (nf, n, n)).copy()
    with egh.Server(8 << 20, precision=egh.EGH_PREC_MIXED) as sv:
        f = np.linspace(2.0, 10.0, nf)
        sv.add_set(Q, f, 1e-3, 500, 500)  # (loads the kernels)
        free = torch.cuda.mem_get_info()[0]
        for _ in range(4):
            sv.add_set(Q, f, 1e-3, 500, 500)
        held = (free - torch.cuda.mem_get_info()[0]) / 4
    images = nf * -(-n // 128) * -(-n // 32) * (48 << 10)
    assert held <= Q.nbytes + images + (6 << 20)  # twiddle tables and the allocator's 2 MB blocks


@pytest.mark.parametrize("nz,nx,nrec,nt,batch", [(295, 496, 12, 400, 12), (600, 600, 15, 400, 8),
                                                 (351, 1701, 11, 400, 8), (295, 496, 20, 400, 16),
                                                 (295, 496, 20, 1403, 20)])
def test_batch_of_a_few_receivers(nz, nx, nrec, nt, batch):
    """One batch of all receivers is taken where it is clearly the faster choice and not where its levels
    leave L2, or where the transform of a short record, with no steps beside it, outweighs its steps (the
    other choice takes 1.07 to 1.27 times as long in each)."""
    import torch
    from paper_2512_16642_gb300 import egh

    with egh.Context(nz, nx, 10.0, 10.0, 20, 1e-3, 1e-3, nt, np.zeros(nrec, np.int32),
                     np.arange(nrec, dtype=np.int32), np.array([8.0])) as ctx:
        ctx.green(torch.full((nz, nx), 2000.0, device="cuda"))
        assert ctx.stats()["batch_receivers"] == batch


def test_threads_that_wait_for_the_device():
    """A host thread that waits for the device and one whose contexts run their first Green stages and
    batched factorisations (which build their graphs then) leave each other alone."""
    import torch
    from paper_2512_16642_gb300 import egh

    done = threading.Event()
    vel = torch.full((60, 300), 2000.0, device="cuda")

    def wait():
        while not done.is_set():
            torch.cuda.synchronize()

    def work():
        try:
            first = None
            for _ in range(8):
                ctxs = [egh.Context(60, 300, 10.0, 10.0, 10, 1e-3, 1e-3, 200, np.zeros(n, np.int32),
                                    np.arange(n, dtype=np.int32), np.array([10.0, 20.0]), fd_kernel=2,
                                    dft_chunk=64, precision=1, gram_splits=2) for n in (12, 33)]
                try:
                    for c in ctxs:
                        c.green(vel)
                        c.hessian(egh.EGH_MU_REL_MEANDIAG, 1e-2)
                    with egh.Batch(ctxs) as b:
                        b.factor()
                        b.factor()
                    out = [ctxs[0].get_green()] + [c.get_hessian(True) for c in ctxs]
                finally:
                    for c in ctxs:
                        c.close()
                first = first or out
                assert all(np.array_equal(a, w) for a, w in zip(out, first))
        finally:
            done.set()

    _in_threads(wait, work)

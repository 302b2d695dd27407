"""Inputs that take a kernel off its common path: columns that need no reflector, blocks rotated in
place, values near the ends of the FP32 range, planes that only just fit a block's shared memory."""
import numpy as np
import pytest

import workloads as W
from oracle import lobpcgf as olb

from ._helpers import gpu, make_pair, rel_err, to_dev

pytestmark = pytest.mark.gpu


def _rand(shape, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


# blocks of A on its diagonal: every block ends in two columns without a reflector and a 1 x 1 block
# is one more, so that one, two and three (and longer runs of) steps are left out between executed ones
@pytest.mark.parametrize("blocks", [(5, 1, 6, 1, 7), (40, 1, 39, 1, 1, 38), (2, 30, 2, 1, 64, 1, 1, 1, 29),
                                    (1,) * 33, (100, 1, 60, 1, 139)])
def test_rayleigh_ritz_decoupled_columns(blocks):
    torch = gpu()
    import paper_1211_1446_gb300 as P
    nz = n = sum(blocks)
    # one spectrum of even gaps dealt out to the blocks, so that no eigenvector is ill-conditioned
    lam_all = np.random.default_rng(49).permutation(np.linspace(-3.0, 4.0, nz))
    a, at = np.zeros((nz, nz), dtype=np.complex128), 0
    for i, b in enumerate(blocks):
        q = np.linalg.qr(_rand((b, b), 50 + i))[0]
        h = (q * lam_all[at:at + b]) @ q.conj().T
        a[at:at + b, at:at + b] = 0.5 * (h + h.conj().T)
        at += b
    s = np.eye(nz, dtype=np.complex128)
    lam_ref, _, _ = olb.rayleigh_ritz(a, s, n)
    # backward error of 2^-46 per operation and step of the double-float parts, |A| = 4: up to
    # 4 nz 2^-46 |A| in the eigenvalues, the same over the gap in the vectors
    tol = 4.0 * nz * 2.0 ** -46 * 4.0
    gap = 7.0 / (nz - 1)
    for _ in range(20):
        v = torch.empty((n, nz), dtype=torch.complex128, device="cuda")
        lam = torch.empty(n, dtype=torch.float64, device="cuda")
        info = torch.zeros(4, dtype=torch.int32, device="cuda")
        P.rayleigh_ritz(to_dev(a.T.copy(), torch.complex128), to_dev(s, torch.complex128), n, v, lam, info)
        torch.cuda.synchronize()
        assert info.cpu().numpy()[:3].tolist() == [0, nz, 0]
        lg, vg = lam.cpu().numpy(), v.cpu().numpy().T
        assert np.abs(lg - lam_ref).max() < tol
        assert np.abs(vg.conj().T @ vg - np.eye(n)).max() < tol / gap
        assert np.abs(a @ vg - vg * lg).max() < tol / gap


# up to 32 columns may be rotated into Z itself: around the 64 rows a block owns, the first columns
# and the last ones, with and without beta
@pytest.mark.parametrize("dtype", ["c64", "c128", "c128e"])
@pytest.mark.parametrize("rows,nz,n,at,beta", [(1, 2, 2, 0, 0.0), (63, 5, 2, 3, 0.0), (64, 36, 5, 0, 0.5), (65, 36, 17, 19, 0.0),
                                               (1500, 96, 32, 0, 0.0), (1500, 96, 32, 64, 2.0), (60000, 64, 31, 1, 0.0)])
def test_rotate_in_place(rows, nz, n, at, beta, dtype):
    torch = gpu()
    import paper_1211_1446_gb300 as P
    z0, w = _rand((nz, rows), 21), _rand((nz, n), 22)
    z = to_dev(z0, torch.complex64 if dtype == "c64" else torch.complex128)
    z0 = z.cpu().numpy().astype(np.complex128)
    P.rotate(z, to_dev(w.T.copy(), torch.complex128), n, z[at:at + n], beta=beta, emulated=dtype == "c128e")
    torch.cuda.synchronize()
    got = z.cpu().numpy()
    # rounding of nz + 2 products and sums each way: FP32, FP64, and the emulated form's 2^-48 of the
    # largest value of each column
    u = {"c64": 2.0 ** -24, "c128": 2.0 ** -53, "c128e": 2.0 ** -48}[dtype]
    size = lambda a: np.abs(a.real) + np.abs(a.imag)  # noqa: E731
    sz = size(z0) if dtype != "c128e" else np.broadcast_to(size(z0).max(axis=1, keepdims=True), z0.shape)
    bound = (2 * nz + 8) * u * (size(w).T @ sz + abs(beta) * sz[at:at + n])
    assert (np.abs(got[at:at + n] - (w.T @ z0 + beta * z0[at:at + n])) <= bound).all()
    keep = np.ones(nz, dtype=bool)
    keep[at:at + n] = False
    assert np.array_equal(got[keep], z0[keep].astype(got.dtype))


# H' is linear: a block scaled by a power of two gives the scaled result.  At 2^-100 the trailing parts
# of the double-float values lie below the smallest normal FP32 number, 2^-126, and still count.
@pytest.mark.parametrize("model", ["dks", "ksso"])
@pytest.mark.parametrize("power", [0, 60, 93, 100])
def test_emulated_h_small_scale(power, model):
    torch = gpu()
    nc = 4 if model == "dks" else 2
    wl, ctx, hop, q = make_pair("small", model=model, projectors=False)
    x = W.random_block(len(q), 3, 12, ncomp=nc)
    if model == "dks":
        x[:, 2:] = 0.0            # then the upper components of H' x are the local term alone
    xd = to_dev(x * 2.0 ** -power, torch.complex128)
    hx = torch.empty_like(xd)
    ctx.apply_H(0, xd, hx, emulated=True)
    torch.cuda.synchronize()
    # the bound of the unscaled block: the granularity 2^-149 of FP32 is 2^-49 of a block of 2^-100, no more
    # than the 2^-48 of a double-float step
    assert rel_err(hx.cpu().numpy()[:, :2] * 2.0 ** power, hop(x)[:, :2]) < 1e-11


# FP32 outputs of 1 to 5 groups of eight columns to a block, and of two and three blocks of them
@pytest.mark.parametrize("n", [7, 15, 23, 24, 25, 31, 32, 33, 39, 47, 56, 65, 81])
@pytest.mark.parametrize("rows", [3, 300])
def test_rotate_fp32_widths(rows, n):
    torch = gpu()
    import paper_1211_1446_gb300 as P
    nz = n + 10
    z, w, o = _rand((nz, rows), 31).astype(np.complex64), _rand((nz, n), 32), _rand((n, rows), 33).astype(np.complex64)
    out = to_dev(o, torch.complex64)
    P.rotate(to_dev(z, torch.complex64), to_dev(w.T.copy(), torch.complex128), n, out, beta=1.0)
    torch.cuda.synchronize()
    z, o = z.astype(np.complex128), o.astype(np.complex128)
    size = lambda a: np.abs(a.real) + np.abs(a.imag)  # noqa: E731
    # one rounding of W, two per product and sum, one of the update
    bound = (2 * nz + 6) * 2.0 ** -24 * (size(w).T @ size(z) + size(o))
    assert (np.abs(out.cpu().numpy() - (w.T @ z + o)) <= bound).all()


# grids of few lines (one or a few to a block) and of one line more or less than the blocks of a share
@pytest.mark.parametrize("grid", [(12, 12, 12), (14, 12, 15), (24, 25, 27), (32, 32, 36), (36, 42, 35), (12, 12, 256)])
def test_hxc_few_lines(grid):
    torch = gpu()
    import paper_1211_1446_gb300 as P
    from oracle import scf as oscf
    wl = W.make("small", grid=grid, ecut=1.0)
    ctx = P.Context.from_workload(wl)
    rho = np.random.default_rng(8).uniform(0.0, 0.1, grid)
    v = torch.empty(grid, dtype=torch.float64, device="cuda")
    eh, exc = ctx.hxc(to_dev(rho, torch.float64), v)
    want, eh0, exc0 = oscf.hxc(rho, wl.lattice, wl.volume)
    # at most 2 (p + q + 1) = 66 roundings of 2^-53 per axis and direction, six passes: 4.4e-14, and the
    # reference's own
    assert rel_err(v.cpu().numpy(), want) < 1e-13
    assert abs(eh - eh0) < 1e-12 * abs(eh0) and abs(exc - exc0) < 1e-12 * abs(exc0)


# the row kernels of the split plane FFT take 40 (complex128) or 81 (complex64) rows to a block here: last
# blocks of 1, 2, 3 and 4 rows, and a block that is not full
@pytest.mark.parametrize("grid", [(81, 100, 12), (84, 100, 12), (42, 100, 12), (27, 100, 12)])
@pytest.mark.parametrize("dtype", ["c64", "c128", "c128e"])
def test_split_plane_last_rows(grid, dtype):
    torch = gpu()
    from oracle import scf as oscf
    wl, ctx, hop, q = make_pair("small", grid=grid, ecut=4.0)
    ctx.set_tuning(64 << 20, 0, 1)
    x = W.random_block(len(q), 2, 13)
    xd = to_dev(x, torch.complex64 if dtype == "c64" else torch.complex128)
    hx = torch.empty_like(xd)
    ctx.apply_H(0, xd, hx, emulated=dtype == "c128e")
    torch.cuda.synchronize()
    assert rel_err(hx.cpu().numpy(), hop(x)) < (2e-6 if dtype == "c64" else 1e-11)   # the operator's other tests
    if dtype == "c128":
        rho = torch.zeros(grid, dtype=torch.float64, device="cuda")
        ctx.density(0, xd, [1.0, 0.5], rho)
        torch.cuda.synchronize()
        assert rel_err(rho.cpu().numpy(), oscf.density(x, ctx.basis(0), wl.grid, wl.volume, [1.0, 0.5])) < 1e-11


# planes whose data just fits a block's shared memory (227 KB), with room for the twiddles and without:
# one kernel; one row or column more: three
@pytest.mark.parametrize("grid,dtype,kernels", [((160, 180, 10), "c64", 1), ((168, 168, 10), "c64", 1),
                                                ((168, 175, 10), "c64", 3), ((120, 120, 10), "c128", 1),
                                                ((120, 120, 10), "c128e", 1), ((112, 125, 10), "c128e", 1),
                                                ((125, 112, 10), "c128e", 1), ((90, 160, 10), "c128", 1),
                                                ((120, 125, 10), "c128", 3), ((120, 125, 10), "c128e", 3)])
def test_plane_at_the_shared_memory_limit(grid, dtype, kernels):
    torch = gpu()
    import paper_1211_1446_gb300 as P
    wl, ctx, hop, q = make_pair("cubic", grid=grid, ecut=4.0)
    x = W.random_block(len(q), 1, 14)
    xd = to_dev(x, torch.complex64 if dtype == "c64" else torch.complex128)
    want = hop(x)
    for threads in (0, 64, 512):
        ctx.set_tuning(64 << 20, threads, 0)
        hx = torch.empty_like(xd)
        P.profile_enable(True)
        ctx.apply_H(0, xd, hx, emulated=dtype == "c128e")
        count = P.profile_read()["plane_fft_v" + ("_fp32" if dtype == "c64" else "")]["launches"]
        P.profile_enable(False)
        assert count == kernels
        assert rel_err(hx.cpu().numpy(), want) < (2e-6 if dtype == "c64" else 1e-11)   # the operator's other tests


# pencils at which the Cholesky (295) and the Householder reduction (309) leave the staged form
@pytest.mark.parametrize("nz", [294, 295, 308, 309])
def test_rayleigh_ritz_staging_limits(nz):
    torch = gpu()
    import paper_1211_1446_gb300 as P
    n = 20
    z = _rand((nz, nz + 16), 41)
    h = np.linspace(-3.0, 4.0, nz + 16)
    a, s = (z * h) @ z.conj().T, z @ z.conj().T
    lam_ref, _, info_ref = olb.rayleigh_ritz(a, s, n)
    v = torch.empty((n, nz), dtype=torch.complex128, device="cuda")
    lam = torch.empty(n, dtype=torch.float64, device="cuda")
    info = torch.zeros(4, dtype=torch.int32, device="cuda")
    P.rayleigh_ritz(to_dev(a.T.copy(), torch.complex128), to_dev(s.T.copy(), torch.complex128), n, v, lam, info)
    torch.cuda.synchronize()
    lam, v, info = lam.cpu().numpy(), v.cpu().numpy().T, info.cpu().numpy()
    assert bool(info[0]) == info_ref.svqb and info[1] == info_ref.rank and info[2] == 0
    # 2^-46 per operation of the double-float steps: nz 2^-46 |S^-1| |A|, |A| <= 4 |S|
    tol = 4.0 * nz * 2.0 ** -46 * np.linalg.cond(s)
    assert np.abs(lam - lam_ref).max() < 4.0 * tol
    assert np.abs(v.conj().T @ s @ v - np.eye(n)).max() < tol
    assert np.abs(a @ v - (s @ v) * lam).max() < 4.0 * tol * np.linalg.norm(s, 2) ** 0.5


# complex64 Gram matrices sum 32 rows in FP32 and the rest in double-float pairs: the error stays that of
# 32 rows however many there are (sums in FP32 throughout, or operands of fewer bits, are beyond it)
@pytest.mark.parametrize("rows,nz", [(32, 17), (33, 31), (2060, 33), (20000, 40), (65537, 24)])
def test_gram_fp32_folded_sums(rows, nz):
    torch = gpu()
    import paper_1211_1446_gb300 as P
    z, hz = (to_dev(_rand((nz, rows), s), torch.complex64) for s in (61, 62))
    a = torch.empty((nz, nz), dtype=torch.complex128, device="cuda")
    s = torch.empty_like(a)
    P.gram_hermitian(z, hz, a, s)
    torch.cuda.synchronize()
    z, hz = z.cpu().numpy().astype(np.complex128), hz.cpu().numpy().astype(np.complex128)
    size = lambda x: np.abs(x.real) + np.abs(x.imag)  # noqa: E731
    low = np.tril(np.ones((nz, nz), dtype=bool))
    for got, b in ((a, hz), (s, z)):
        err = np.abs(got.cpu().numpy().T - z.conj() @ b.T)
        # two roundings of 2^-24 for each of at most 32 products of a part, and 2^-46 for every fold
        bound = ((2 * min(rows, 32) + 4) * 2.0 ** -24 + (rows // 32 + 1) * 2.0 ** -46) * (size(z) @ size(b).T)
        assert (err <= bound)[low].all()
        # 64 steps of a part and chunk round independently by at most 2^-24 of a partial sum of RMS at most
        # 8: 64 2^-24 for a chunk, both parts and rows / 32 chunks: 16 2^-24 sqrt(rows) off the diagonal
        assert np.sqrt(np.mean(err[np.tril(low, -1)] ** 2)) < 16 * 2.0 ** -24 * np.sqrt(max(rows, 32))


# FP64 A^H B and its lower-triangle form with 12 and 16 blocks to an SM, last chunks of one row and of few
@pytest.mark.parametrize("rows,nz", [(1, 3), (33, 96), (2060, 96), (2049, 17), (20001, 40), (57419, 48)])
def test_gram_fp64_chunks(rows, nz):
    torch = gpu()
    import paper_1211_1446_gb300 as P
    z, hz = (to_dev(_rand((nz, rows), s), torch.complex128) for s in (71, 72))
    zn, hn = z.cpu().numpy(), hz.cpu().numpy()
    size = lambda x: np.abs(x.real) + np.abs(x.imag)  # noqa: E731
    low = np.tril(np.ones((nz, nz), dtype=bool))
    for f, where in ((P.gram, np.ones((nz, nz), dtype=bool)), (P.gram_hermitian, low)):
        a = torch.empty((nz, nz), dtype=torch.complex128, device="cuda")
        s = torch.empty_like(a)
        f(z, hz, a, s)
        torch.cuda.synchronize()
        for got, b in ((a, hn), (s, zn)):
            err = np.abs(got.cpu().numpy().T - zn.conj() @ b.T)
            # at most 2 rows + 4 roundings of 2^-53 on the way of any product, in the reference too
            assert (err <= 2 * (2 * rows + 4) * 2.0 ** -53 * (size(zn) @ size(b).T))[where].all()

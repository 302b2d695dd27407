"""Kernels at the sizes where their tiling can go wrong: one row or column more or less than a tile,
every output checked against an elementwise rounding bound or the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import lobpcgf as olb

from ._helpers import gpu, make_pair, rel_err, to_dev

pytestmark = pytest.mark.gpu


def _rand(shape, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def _cabs(a):
    """|Re| + |Im|: the product of two such sums bounds all four real products of a complex one."""
    return np.abs(a.real) + np.abs(a.imag)


# a complex dot product of length k in working precision u: at most 2 k + 4 roundings on the way of
# any of its real products (the split sums and their FP64 additions take no more)
def _bound(k, u, prod):
    return (2 * k + 4) * u * prod


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("rows,nz", [(4, 1), (31, 15), (32, 16), (33, 17), (63, 31), (64, 32), (65, 33),
                                     (257, 48), (1028, 65), (2060, 18)])
def test_gram_hermitian_edges(dtype, rows, nz):
    torch = gpu()
    import paper_1211_1446_gb300 as P
    dt, u = (torch.complex64, 2.0 ** -24) if dtype == "c64" else (torch.complex128, 2.0 ** -53)
    z, hz = (to_dev(_rand((nz, rows), s), dt) for s in (1, 2))
    a = torch.empty((nz, nz), dtype=torch.complex128, device="cuda")
    s = torch.empty_like(a)
    P.gram_hermitian(z, hz, a, s)
    torch.cuda.synchronize()
    z, hz = z.cpu().numpy().astype(np.complex128), hz.cpu().numpy().astype(np.complex128)
    low = np.tril(np.ones((nz, nz), dtype=bool))
    for got, b in ((a, hz), (s, z)):
        err = np.abs(got.cpu().numpy().T - z.conj() @ b.T)
        assert (err <= _bound(rows, u, _cabs(z) @ _cabs(b).T))[low].all()


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("rows,nz,n", [(1, 1, 1), (31, 15, 2), (32, 16, 4), (33, 17, 5), (255, 63, 8), (256, 64, 9),
                                       (257, 65, 16), (1500, 36, 17), (2296, 120, 41), (10000, 33, 40)])
def test_rotate_edges(dtype, rows, nz, n):
    torch = gpu()
    import paper_1211_1446_gb300 as P
    n = min(n, nz)
    dt, u = (torch.complex64, 2.0 ** -24) if dtype == "c64" else (torch.complex128, 2.0 ** -53)
    z, w = to_dev(_rand((nz, rows), 3), dt), _rand((nz, n), 4)
    out = torch.full((n, rows), float("nan"), dtype=dt, device="cuda")
    P.rotate(z, to_dev(w.T.copy(), torch.complex128), n, out)
    torch.cuda.synchronize()
    z = z.cpu().numpy().astype(np.complex128)
    err = np.abs(out.cpu().numpy() - (z.T @ w).T)
    # one rounding of W and one of the result more
    assert (err <= _bound(nz + 1, u, _cabs(w).T @ _cabs(z))).all()


@pytest.mark.parametrize("nz,n", [(4, 4), (16, 5), (17, 17), (33, 32), (127, 40), (128, 43), (129, 43), (257, 86),
                                  (385, 20)])
def test_rayleigh_ritz_edges(nz, n):
    """Pencils around the 128 rows a block's threads own once (and twice, and three times), and
    around multiples of the cluster's 16 blocks."""
    torch = gpu()
    import paper_1211_1446_gb300 as P
    z = _rand((nz, nz + 16), 5)
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
    # backward stable to 2^-46 per operation of the double-float steps: errors up to about
    # nz 2^-46 |S^-1| |A|, with |A| <= 4 |S|
    tol = 4.0 * nz * 2.0 ** -46 * np.linalg.cond(s)
    assert np.abs(lam - lam_ref).max() < 4.0 * tol
    assert np.abs(v.conj().T @ s @ v - np.eye(n)).max() < tol
    assert np.abs(a @ v - (s @ v) * lam).max() < 4.0 * tol * np.linalg.norm(s, 2) ** 0.5


# axis lengths whose passes merge differently: primes 2, 3, 5 and 7 alone and mixed, odd lengths,
# a short axis beside a long one
@pytest.mark.parametrize("grid", [(14, 15, 16), (25, 18, 27), (32, 35, 36), (20, 49, 21), (15, 28, 64), (30, 14, 125)])
@pytest.mark.parametrize("dtype", ["c64", "c128", "c128e"])
def test_apply_h_axes(grid, dtype):
    torch = gpu()
    wl, ctx, hop, q = make_pair("small", grid=grid, ecut=4.0)
    x = W.random_block(len(q), 3, 11)
    dt = torch.complex64 if dtype == "c64" else torch.complex128
    xd = to_dev(x, dt)
    hx = torch.empty_like(xd)
    ctx.apply_H(0, xd, hx, emulated=dtype == "c128e")
    torch.cuda.synchronize()
    # the bounds of the operator's other parity tests
    assert rel_err(hx.cpu().numpy(), hop(x)) < (2e-6 if dtype == "c64" else 1e-11)


# the transforms of the grid densities: axes of one factor, of two equal ones, of prime powers, and
# numbers of lines that a block's share does not divide
@pytest.mark.parametrize("grid", [(14, 15, 16), (25, 18, 49), (20, 21, 125), (30, 14, 128)])
def test_hxc_axes(grid):
    torch = gpu()
    import paper_1211_1446_gb300 as P
    from oracle import scf as oscf
    wl = W.make("small", grid=grid, ecut=4.0)
    ctx = P.Context.from_workload(wl)
    rho = np.random.default_rng(7).uniform(0.0, 0.1, grid)
    v = torch.empty(grid, dtype=torch.float64, device="cuda")
    eh, exc = ctx.hxc(to_dev(rho, torch.float64), v)
    want, eh0, exc0 = oscf.hxc(rho, wl.lattice, wl.volume)
    # at most 2 (p + q + 1) roundings per axis and direction: six passes of 40 roundings of 2^-53, twice
    # over for the reference, stay below 1e-13 of the largest value
    assert rel_err(v.cpu().numpy(), want) < 1e-12
    assert abs(eh - eh0) < 1e-11 * abs(eh0) and abs(exc - exc0) < 1e-11 * abs(exc0)

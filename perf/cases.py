"""Timed cases of the library: the calls a user's program makes, over the sizes it makes them at.

A program of this framework holds a Context (cell, grid, cutoff, potential, projectors) and either
asks it for a whole solve, or drives Algorithm 1 itself through the single-step entry points: H' on
a block of columns, the Gram matrices of Z = [X | Y | P], the Rayleigh-Ritz step on their pencil,
the rotation of the blocks, and, around the eigenproblem, the density and its potential.  The
kinds below are those calls; the systems are the ones of workloads.make: "small" and "cubic"
(seconds-sized checks, where a call is a handful of short launches), "dimer" (the flagship: 57,419
planewaves, 36 projector channels, blocks of 32 + 8 columns) and "layered" (39,771 planewaves on a
60 x 60 x 216 grid, 270 projector channels, blocks of up to 96 + 8 columns).

Types: "c64" complex64 blocks (the FP32 phase of the mixed mode), "c128e" complex128 blocks with
emulated FP64 (its refinement phase), "c128" complex128 blocks in native FP64 (the default mode).
"""
import functools
import math

import numpy as np
import torch

import paper_1211_1446_gb300 as P
import workloads as W

ITEM = {"c64": 8, "c128e": 16, "c128": 16}
DTYPE = {"c64": torch.complex64, "c128e": torch.complex128, "c128": torch.complex128}
ROWS_DIMER, ROWS_LAYERED = 4 * 57419, 4 * 39771


def listed():
    return [
        # the smallest call: H' on the 16 x 15 x 18 grid in the default (native FP64) mode, as a
        # small molecule's or a test's solve makes it; launches and latency count
        dict(name="hx_small_c128", kind="hx", system="small", n1=16, n2=15, n3=18, dtype="c128", nb=9),
        # H' of the dimer's block in the FP32 phase (three such calls per iteration)
        dict(name="hx_dimer_c64", kind="hx", system="dimer", n1=48, n2=48, n3=56, dtype="c64", nb=40),
        # and in the refinement phase
        dict(name="hx_dimer_c128e", kind="hx", system="dimer", n1=48, n2=48, n3=56, dtype="c128e", nb=40),
        # H' of the layered crystal's widest block: long third axis, 270 projector channels
        dict(name="hx_layered_c64", kind="hx", system="layered", n1=60, n2=60, n3=216, dtype="c64", nb=104),
        # Gram matrices of the dimer's Z = [X | Y | P], FP32 phase and refinement phase
        dict(name="gram_dimer_c64", kind="gram", rows=ROWS_DIMER, nz=120, dtype="c64"),
        dict(name="gram_dimer_c128e", kind="gram", rows=ROWS_DIMER, nz=120, dtype="c128e"),
        # rotation of the dimer's block to the new X, FP32 phase
        dict(name="rotate_dimer_c64", kind="rotate", rows=ROWS_DIMER, nz=120, n=40, dtype="c64"),
        # rotation of the layered crystal's widest block, refinement phase
        dict(name="rotate_layered_c128e", kind="rotate", rows=ROWS_LAYERED, nz=312, n=104, dtype="c128e"),
        # the pencil of one dimer iteration, both phases
        dict(name="rr_120_40", kind="rr", nz=120, n=40),
        # the grid work of one SCF iteration: density of the 20 occupied states, V_hxc
        dict(name="scf_dimer", kind="scf", system="dimer", n1=48, n2=48, n3=56, nb=20),
        # a whole solve in the default mode at the smallest size
        dict(name="solve_cubic", kind="solve", system="cubic", mode="fp64", nev=8, nbuf=4),
        # the flagship: a whole mixed-precision solve of the dimer
        dict(name="solve_dimer", kind="solve", system="dimer", mode="mixed", nev=32, nbuf=8),
    ]


def _smooth(n):
    for p in (2, 3, 5, 7):
        while n % p == 0:
            n //= p
    return n == 1


_AXES = [n for n in range(12, 257) if _smooth(n)]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _axis_near(rng, n):
    near = sorted(_AXES, key=lambda a: abs(a - n))[:3]
    return rng.choice(near)


def draw(rng):
    """One more call of the same kinds: other grids (every axis length the transforms take, not
    only equal ones), block widths down to one column, odd numbers of rows and of columns."""
    kind = rng.choice(["hx", "hx", "hx", "gram", "gram", "rotate", "rotate", "rr", "scf"])
    if kind in ("hx", "scf"):
        system = rng.choice(["small", "dimer", "dimer", "layered"]) if kind == "hx" else rng.choice(["small", "dimer"])
        if system == "small":
            n1, n2, n3 = (_axis_near(rng, rng.uniform(13, 24)) for _ in range(3))
        elif system == "dimer":
            n1 = _axis_near(rng, math.exp(rng.uniform(math.log(24), math.log(64))))
            n2, n3 = _axis_near(rng, n1), _axis_near(rng, 1.2 * n1)
        else:
            n1 = n2 = _axis_near(rng, rng.uniform(30, 64))
            n3 = _axis_near(rng, 3.6 * n1)
        case = dict(kind=kind, system=system, n1=n1, n2=n2, n3=n3)
        if kind == "scf":
            return dict(case, nb=_log_int(rng, 1, 32))
        dtype = rng.choice(["c64", "c64", "c128e", "c128e", "c128"])
        top = {"c64": 104, "c128e": 64, "c128": 16}[dtype]
        return dict(case, dtype=dtype, nb=_log_int(rng, 1, top))
    if kind == "rr":
        nz = _log_int(rng, 12, 312)
        return dict(kind="rr", nz=nz, n=max(1, min(nz, int(round(nz * rng.uniform(0.3, 0.6))))))
    dtype = rng.choice(["c64", "c64", "c128e", "c128e", "c128"])
    nz = _log_int(rng, 12, 120 if dtype == "c128" else 312)
    rows = 4 * _log_int(rng, 515, 57419)
    if kind == "gram":
        return dict(kind="gram", rows=rows, nz=nz, dtype=dtype)
    return dict(kind="rotate", rows=rows, nz=nz, n=max(1, int(round(nz * rng.uniform(0.1, 0.5)))), dtype=dtype)


# ------------------------------------------------------------------ systems
@functools.lru_cache(maxsize=16)
def _workload(system, grid=None):
    """The named workload; on another grid, with the largest cutoff whose sphere that grid holds
    (2 % below it), as a program picks grid and cutoff together."""
    if grid is None or (system, grid) in (("small", (16, 15, 18)), ("dimer", (48, 48, 56))):
        return W.make(system)
    one = [[0.0, 0.0, 0.0]]
    if system == "layered" and grid == (60, 60, 216):
        return W.make("layered", kfrac=one)
    lat = {"small": np.diag([7.0, 7.5, 8.0]), "dimer": np.diag([20.0, 20.0, 24.0])}.get(system)
    if lat is None:
        lat = np.array([[7.8, 0.0, 0.0], [-3.9, 7.8 * math.sqrt(3.0) / 2.0, 0.0], [0.0, 0.0, 28.0]])
    # |m_i| <= |G| |a_i| / (2 pi) has to stay within (N_i - 1) // 2; the layered crystal's grids
    # are twice as fine as the sphere needs (29 of 60 and 105 of 216 frequencies hold planewaves)
    g = min(((n - 1) // 2) * 2.0 * math.pi / np.linalg.norm(a) for n, a in zip(grid, lat))
    g *= 0.5 if system == "layered" else 0.98
    return W.make(system, grid=grid, ecut=0.5 * g * g * 0.97, kfrac=one)


def _system(case):
    grid = (case["n1"], case["n2"], case["n3"]) if "n1" in case else None
    return _workload(case["system"], grid)


@functools.lru_cache(maxsize=16)
def _sphere(system, grid):
    """Miller triples of the first k-point in lexicographic order and k + G, by their definition."""
    wl = _workload(system, grid)
    b = 2.0 * np.pi * np.linalg.inv(wl.lattice).T
    k = wl.kfrac[0] @ b
    gmax = math.sqrt(2.0 * wl.ecut_k[0]) + np.linalg.norm(k)
    lim = [int(gmax * np.linalg.norm(a) / (2 * np.pi)) + 1 for a in wl.lattice]
    m = np.stack(np.meshgrid(*[np.arange(-v, v + 1) for v in lim], indexing="ij"), axis=-1).reshape(-1, 3)
    q = k + m @ b
    keep = 0.5 * (q * q).sum(axis=1) <= wl.ecut_k[0]
    return m[keep], q[keep]


def _sphere_of(case):
    return _sphere(case["system"], (case["n1"], case["n2"], case["n3"]) if "n1" in case else None)


def _channels(wl):
    return sum(2 * (int(l) + 1) ** 2 for l in wl.lmax)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(shape, gen):
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), dtype=torch.float64, device="cuda", generator=gen)
                                 * math.sqrt(0.5))


def _columns(ctx, q, nb, gen):
    """nb four-spinors as a solve holds them: coefficients that fall off with the kinetic energy,
    normalised, with kinetically balanced small components."""
    ek = torch.from_numpy(0.5 * (q * q).sum(axis=1)).cuda()
    x = _normal((nb, 4, len(q)), gen) / (1.0 + (ek / (0.1 * ek.max())) ** 2)
    ctx.kinetic_balance(0, x)
    return x / torch.linalg.vector_norm(x.reshape(nb, -1), dim=1)[:, None, None]


# ------------------------------------------------------------------ inputs
def _z_block(rows, nz, dtype, gen):
    """[X | Y | P] of a running solve: X of norm 1, the corrections Y and P shorter."""
    n = max(1, nz // 3)
    scale = torch.ones(nz, dtype=torch.float64, device="cuda")
    scale[n:] = 0.1 ** torch.empty(nz - n, dtype=torch.float64, device="cuda").uniform_(0.0, 2.0, generator=gen)
    z = torch.empty((nz, rows), dtype=dtype, device="cuda")
    for j in range(0, nz, 32):                          # by parts: the float64 draws need not all live at once
        part = _normal((min(32, nz - j), rows), gen)
        z[j:j + 32] = part * (scale[j:j + 32, None] / math.sqrt(rows))
    return z


def _pencil(nz, n, gen):
    """A, S of one iteration: in an orthonormal basis the columns of Z are the n Ritz vectors with
    a small error and short corrections in general directions; the wanted end of the spectrum is
    below the rest."""
    eps = 1e-3
    z = torch.eye(nz, dtype=torch.complex128, device="cuda")
    z = z + eps / math.sqrt(nz) * _normal((nz, nz), gen)
    z[:, n:] = eps * (torch.eye(nz, dtype=torch.complex128, device="cuda")[:, n:]
                      + 0.3 / math.sqrt(nz) * _normal((nz, nz - n), gen))
    u = torch.rand(nz, dtype=torch.float64, device="cuda", generator=gen)
    j = torch.arange(nz, dtype=torch.float64, device="cuda")
    lam = torch.where(j < n, -12.0 + 10.0 * (j + 0.5 * u) / n, 0.5 + 20.0 * (j - n + 0.5 * u) / max(1, nz - n))
    a = z.conj().T @ (lam[:, None] * z)
    s = z.conj().T @ z
    return 0.5 * (a + a.conj().T), 0.5 * (s + s.conj().T)


def prepare(case, seed):
    gen = _gen(seed)
    kind = case["kind"]
    st = dict(case=case)
    if kind == "hx":
        _, q = _sphere_of(case)
        st["ctx"] = ctx = P.Context.from_workload(_system(case))
        st["x"] = _columns(ctx, q, case["nb"], gen).to(DTYPE[case["dtype"]]).contiguous()
        st["hx"] = torch.empty_like(st["x"])
    elif kind == "gram":
        rows, nz = case["rows"], case["nz"]
        st["z"] = _z_block(rows, nz, DTYPE[case["dtype"]], gen)
        # HZ = H Z of a diagonal H: the Gram matrix A is Hermitian, as it is for H'
        h = torch.rand(rows, dtype=torch.float64, device="cuda", generator=gen) * 30.0 - 10.0
        st["hz"] = torch.empty_like(st["z"])
        for j in range(0, nz, 32):
            st["hz"][j:j + 32] = st["z"][j:j + 32].to(torch.complex128) * h
        st["a"] = torch.empty((nz, nz), dtype=torch.complex128, device="cuda")
        st["s"] = torch.empty_like(st["a"])
    elif kind == "rotate":
        st["z"] = _z_block(case["rows"], case["nz"], DTYPE[case["dtype"]], gen)
        st["w"] = _normal((case["n"], case["nz"]), gen) / math.sqrt(case["nz"])
        st["out"] = torch.empty((case["n"], case["rows"]), dtype=st["z"].dtype, device="cuda")
    elif kind == "rr":
        nz, n = case["nz"], case["n"]
        a, s = _pencil(nz, n, gen)
        st["a"], st["s"] = a.T.contiguous(), s.T.contiguous()          # column-major for the library
        st["v"] = torch.empty((n, nz), dtype=torch.complex128, device="cuda")
        st["lam"] = torch.empty(n, dtype=torch.float64, device="cuda")
        st["info"] = torch.zeros(4, dtype=torch.int32, device="cuda")
    elif kind == "scf":
        _, q = _sphere_of(case)
        wl = _system(case)
        st["ctx"] = ctx = P.Context.from_workload(wl)
        st["x"] = _columns(ctx, q, case["nb"], gen).contiguous()
        st["occ"] = np.full(case["nb"], 1.0)
        st["rho"] = torch.empty(wl.grid, dtype=torch.float64, device="cuda")
        st["v"] = torch.empty_like(st["rho"])
    else:
        wl = _system(case)
        st["ctx"] = ctx = P.Context.from_workload(wl)
        st["x0"] = _normal((case["nev"] + case["nbuf"], 4, ctx.npw(0)), gen)
        st["x"] = torch.empty_like(st["x0"])
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "hx":
        st["ctx"].apply_H(0, st["x"], st["hx"], emulated=case["dtype"] == "c128e")
        return st["hx"]
    if kind == "gram":
        P.gram_hermitian(st["z"], st["hz"], st["a"], st["s"], emulated=case["dtype"] == "c128e")
        return st["a"], st["s"]
    if kind == "rotate":
        P.rotate(st["z"], st["w"], case["n"], st["out"], emulated=case["dtype"] == "c128e")
        return st["out"]
    if kind == "rr":
        P.rayleigh_ritz(st["a"], st["s"], case["n"], st["v"], st["lam"], st["info"])
        # an eigenvector is given up to a phase: a program that stores or compares them makes its
        # leading component (that of the old Ritz vector) real
        lead = torch.diagonal(st["v"])
        return st["lam"], st["v"] * torch.sgn(lead.conj())[:, None], st["info"][:3]
    if kind == "scf":
        st["rho"].zero_()
        st["ctx"].density(0, st["x"], st["occ"], st["rho"])
        e_h, e_xc = st["ctx"].hxc(st["rho"], st["v"])
        return st["rho"], st["v"], e_h, e_xc
    st["x"].copy_(st["x0"])
    mode = P.MODE_MIXED if case["mode"] == "mixed" else P.MODE_FP64
    lam, _, _ = st["ctx"].solve([st["x"]], case["nev"], tol=1e-6, mode=mode, nbuf=case["nbuf"])
    # the eigenvectors of a Kramers pair, and within the tolerance those of any close cluster, are
    # one basis of many: what is determined is the eigenvalues
    return lam[0]


# ------------------------------------------------------------------ necessary work
def work(case):
    kind = case["kind"]
    if kind in ("hx", "scf"):
        m, _ = _sphere_of(case)
        wl = _system(case)
        npw, ng, nb = len(m), wl.ng, case["nb"]
        fft = 5.0 * ng * math.log2(ng)
        if kind == "scf":
            return dict(bytes=4.0 * nb * npw * 16 + 2.0 * ng * 8, flops=4.0 * nb * (fft + 3.0 * ng) + 2 * fft)
        item, ch = ITEM[case["dtype"]], _channels(wl)
        return dict(bytes=8.0 * nb * npw * item + ng * item / 2 + ch * 2.0 * npw * item,
                    flops=4.0 * nb * (2 * fft + 2.0 * ng) + 2 * 8.0 * ch * 2 * nb * 2 * npw + 64.0 * nb * npw)
    if kind == "gram":
        rows, nz = case["rows"], case["nz"]
        return dict(bytes=2.0 * nz * rows * ITEM[case["dtype"]] + 2.0 * nz * nz * 16,
                    flops=2 * 8.0 * rows * nz * (nz + 1) / 2)
    if kind == "rotate":
        rows, nz, n = case["rows"], case["nz"], case["n"]
        return dict(bytes=(nz + n) * float(rows) * ITEM[case["dtype"]] + 16.0 * nz * n, flops=8.0 * rows * nz * n)
    if kind == "rr":
        nz, n = float(case["nz"]), float(case["n"])
        return dict(bytes=2 * 16.0 * nz * nz + 16.0 * nz * n, flops=8.0 * (11.0 / 6.0 * nz ** 3 + 1.5 * nz * nz * n))
    # a solve: the start block in, the vectors out; the arithmetic of the three initial filters and
    # of one iteration (the number of iterations is the method's)
    wl = _system(case)
    npw = len(_sphere_of(case)[0])
    n, rows = case["nev"] + case["nbuf"], 4.0 * npw
    h = 4.0 * n * (10.0 * wl.ng * math.log2(wl.ng) + 2.0 * wl.ng) + 2 * 8.0 * _channels(wl) * 2 * n * 2 * npw
    return dict(bytes=2.0 * 16 * n * rows, flops=9.0 * h + 2 * 8.0 * rows * 3 * n * (3 * n + 1) / 2
                + 4 * 8.0 * rows * 3 * n * n)


# ------------------------------------------------------------------ 64-bit values
def _lower(p):
    return torch.tril(p) + torch.tril(p, -1).conj().T


def _harmonics(l, u):
    """Y_lm(u), m = -l..l, as rows (Condon-Shortley phase)."""
    x, y, z = u[:, 0], u[:, 1], u[:, 2]
    xp, xm = torch.complex(x, y), torch.complex(x, -y)
    one = torch.ones_like(xp)
    c = lambda v: math.sqrt(v / math.pi)  # noqa: E731
    if l == 0:
        return torch.stack([c(1 / 4) * one])
    if l == 1:
        return torch.stack([c(3 / 8) * xm, c(3 / 4) * z * one, -c(3 / 8) * xp])
    return torch.stack([c(15 / 32) * xm * xm, c(15 / 8) * z * xm, c(5 / 16) * (3 * z * z - 1) * one,
                        -c(15 / 8) * z * xp, c(15 / 32) * xp * xp])


def _spin_orbit(l, d_hi, d_lo):
    """D_{l+1/2} P_{l+1/2} + D_{l-1/2} P_{l-1/2} on (m, spin), P_{l+-1/2} from L.sigma."""
    n = 2 * l + 1
    lz = torch.diag(torch.arange(-l, l + 1, dtype=torch.float64))
    up = torch.zeros((n, n), dtype=torch.float64)
    for i, m in enumerate(range(-l, l)):
        up[i + 1, i] = math.sqrt(l * (l + 1) - m * (m + 1))
    ls = torch.zeros((n, 2, n, 2), dtype=torch.float64)
    ls[:, 0, :, 0], ls[:, 1, :, 1] = lz, -lz
    ls[:, 0, :, 1], ls[:, 1, :, 0] = up.T, up            # L_- sigma_+, L_+ sigma_-
    ls = ls.reshape(2 * n, 2 * n)
    one = torch.eye(2 * n, dtype=torch.float64)
    return (d_hi * ((l + 1) * one + ls) + d_lo * (l * one - ls)) / n


def _apply_h64(wl, m, q, x):
    """H' x by plain 64-bit FFTs and products."""
    q = torch.from_numpy(q).cuda()
    c = wl.c
    cross = torch.complex(q[:, 0], -q[:, 1])             # q_x - i q_y
    y = torch.empty_like(x)
    y[:, 0] = c * (q[:, 2] * x[:, 2] + cross * x[:, 3])
    y[:, 1] = c * (cross.conj() * x[:, 2] - q[:, 2] * x[:, 3])
    y[:, 2] = c * (q[:, 2] * x[:, 0] + cross * x[:, 1]) - 2 * c * c * x[:, 2]
    y[:, 3] = c * (cross.conj() * x[:, 0] - q[:, 2] * x[:, 1]) - 2 * c * c * x[:, 3]
    grid = tuple(wl.grid)
    i = np.mod(m, np.asarray(grid))
    at = torch.from_numpy((i[:, 0] * grid[1] + i[:, 1]) * grid[2] + i[:, 2]).cuda()
    v = torch.from_numpy(np.ascontiguousarray(wl.v_r)).cuda()
    for b in range(x.shape[0]):
        g = torch.zeros((4, v.numel()), dtype=torch.complex128, device="cuda")
        g[:, at] = x[b]
        g = torch.fft.fftn(torch.fft.ifftn(g.reshape((4,) + grid), dim=(1, 2, 3)) * v, dim=(1, 2, 3))
        y[b] += g.reshape(4, -1)[:, at]
    qn = torch.linalg.vector_norm(q, dim=1)
    u = torch.where((qn > 0)[:, None], q / qn.clamp_min(1e-300)[:, None],
                    torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device="cuda"))
    xs = x.reshape(-1, 2, x.shape[2])                    # two-spinors
    ys = y.reshape(-1, 2, x.shape[2])
    for s in range(wl.nsite):
        r = torch.from_numpy(wl.pos[s]).cuda()
        wave = torch.exp(-1j * (q @ r)) / math.sqrt(wl.volume)
        for l in range(int(wl.lmax[s]) + 1):
            rl = float(wl.rl[s, l])
            norm = math.sqrt(2.0 * (2.0 * math.pi) ** 3 * rl ** (2 * l + 3) / math.gamma(l + 1.5))
            f = _harmonics(l, u) * (norm * qn ** l * torch.exp(-0.5 * (qn * rl) ** 2) * wave)
            mat = _spin_orbit(l, float(wl.d[s, l, 0]), float(wl.d[s, l, 1])).to(torch.complex128).cuda()
            z = torch.einsum("mp,bsp->bms", f.conj(), xs).reshape(len(xs), -1)
            z = (z @ mat.T).reshape(len(xs), 2 * l + 1, 2)
            ys += torch.einsum("mp,bms->bsp", f, z)
    return y


def _hxc64(rho, wl):
    """Hartree potential, PZ81 LDA and their energies from the formulas."""
    grid = tuple(wl.grid)
    b = 2.0 * np.pi * np.linalg.inv(wl.lattice).T
    mm = np.stack(np.meshgrid(*[np.fft.fftfreq(n, 1.0 / n) for n in grid], indexing="ij"), axis=-1)
    g2 = torch.from_numpy(((mm @ b) ** 2).sum(axis=-1)).cuda()
    vg = torch.where(g2 > 0, 4.0 * math.pi * torch.fft.fftn(rho) / g2.clamp_min(1e-300), torch.zeros_like(g2) + 0j)
    vh = torch.fft.ifftn(vg).real
    on = rho > 1e-30
    rs = (3.0 / (4.0 * math.pi * torch.where(on, rho, torch.ones_like(rho)))) ** (1.0 / 3.0)
    ex = -0.75 * (9.0 / (4.0 * math.pi ** 2)) ** (1.0 / 3.0) / rs
    lr, sq = torch.log(rs), torch.sqrt(rs)
    ec1 = 0.0311 * lr - 0.048 + 0.0020 * rs * lr - 0.0116 * rs
    vc1 = ec1 - rs / 3.0 * (0.0311 / rs + 0.0020 * lr + 0.0020 - 0.0116)
    den = 1.0 + 1.0529 * sq + 0.3334 * rs
    ec2 = -0.1423 / den
    vc2 = ec2 - rs / 3.0 * (0.1423 * (0.5 * 1.0529 / sq + 0.3334) / den ** 2)
    eps = torch.where(on, ex + torch.where(rs < 1, ec1, ec2), torch.zeros_like(rho))
    vxc = torch.where(on, 4.0 / 3.0 * ex + torch.where(rs < 1, vc1, vc2), torch.zeros_like(rho))
    dv = wl.volume / rho.numel()
    return vh + vxc, 0.5 * dv * float((rho * vh).sum()), dv * float((rho.clamp_min(0.0) * eps).sum())


def _dense64(wl, m, q):
    """The dense H' of a system without projectors, index comp * npw + pw."""
    npw = len(m)
    vh = np.fft.fftn(wl.v_r) / wl.v_r.size
    dm = np.mod(m[:, None, :] - m[None, :, :], np.asarray(wl.grid))
    v = vh[dm[..., 0], dm[..., 1], dm[..., 2]]
    h = np.zeros((4, npw, 4, npw), dtype=np.complex128)
    i = np.arange(npw)
    for a in range(4):
        h[a, :, a, :] += v
    for a, b, t in ((0, 2, q[:, 2]), (0, 3, q[:, 0] - 1j * q[:, 1]), (1, 2, q[:, 0] + 1j * q[:, 1]), (1, 3, -q[:, 2])):
        h[a, i, b, i] += wl.c * t
        h[b, i, a, i] += wl.c * np.conj(t)
    for a in (2, 3):
        h[a, i, a, i] -= 2.0 * wl.c ** 2
    return h.reshape(4 * npw, 4 * npw)


def exact(case, seed):
    kind = case["kind"]
    if kind == "hx":
        m, q = _sphere_of(case)
        return _apply_h64(_system(case), m, q, prepare(case, seed)["x"].to(torch.complex128))
    if kind == "gram":
        st = prepare(case, seed)
        z, hz = (st[k].to(torch.complex128) for k in ("z", "hz"))
        # the library's matrices are column-major: row j of the tensor is column j of Z^H HZ
        return tuple(_lower(z.conj() @ w.T).T.contiguous() for w in (hz, z))
    if kind == "rotate":
        st = prepare(case, seed)
        return st["w"] @ st["z"].to(torch.complex128)
    if kind == "rr":
        st = prepare(case, seed)
        a, s = st["a"].T, st["s"].T
        d = torch.rsqrt(torch.diagonal(s).real)
        low = torch.linalg.cholesky(d[:, None] * s * d[None, :])
        t = torch.linalg.solve_triangular(low, (d[:, None] * a * d[None, :]).to(torch.complex128), upper=False)
        t = torch.linalg.solve_triangular(low, t.conj().T.contiguous(), upper=False)
        lam, c = torch.linalg.eigh(0.5 * (t + t.conj().T))
        n = case["n"]
        v = (d[:, None] * torch.linalg.solve_triangular(low.conj().T, c[:, :n], upper=True)).T
        return lam[:n], v * torch.sgn(torch.diagonal(v).conj())[:, None], None
    if kind == "scf":
        wl = _system(case)
        m, _ = _sphere_of(case)
        x = prepare(case, seed)["x"]
        grid = tuple(wl.grid)
        i = np.mod(m, np.asarray(grid))
        at = torch.from_numpy((i[:, 0] * grid[1] + i[:, 1]) * grid[2] + i[:, 2]).cuda()
        rho = torch.zeros(grid, dtype=torch.float64, device="cuda")
        for b in range(x.shape[0]):
            g = torch.zeros((4, wl.ng), dtype=torch.complex128, device="cuda")
            g[:, at] = x[b]
            psi = torch.fft.ifftn(g.reshape((4,) + grid), dim=(1, 2, 3)) * wl.ng
            rho += (psi.real ** 2 + psi.imag ** 2).sum(dim=0) / wl.volume
        v, e_h, e_xc = _hxc64(rho, wl)
        return rho, v, e_h, e_xc
    if case["system"] != "cubic":
        return None                                       # 57,419 planewaves: no dense spectrum
    wl = _system(case)
    m, q = _sphere_of(case)
    lam = np.linalg.eigvalsh(_dense64(wl, m, q))
    return lam[lam > -wl.c ** 2][: case["nev"]]

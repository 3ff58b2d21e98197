"""The performance cases: what a user of this library has it do, through its public calls.

A pass is what a program does with one nonlinear eigenvalue problem in hand: rsrr_sample (resolvent
samples on a contour), one of the projections, rsrr_solve (eigenpairs inside the contour).  The
families are those of the repository's workloads and tests, with sizes from its configurations:

  gun     T = K - zM + i sqrt(z) W1 - sqrt(s2^2 - z) W2, the gun-like square-root NEP
  qep     T = K + zC + z^2 M, the damped quadratic NEP
  delay   T = -zI + K + A1 exp(-tau z), the time-delay NEP with a random 5 % coupling A1
  string  the loaded string, T = T1 + z/(z-1) e_n e_n^T - z T3 (tridiagonal)
  tz      a distributed-delay NEP known only by its values (callback), reduced by Chebyshev
          interpolation

K is the 5-point Laplacian on an nx x ny grid of a 1 x 0.8 domain (index ix * ny + iy, so the
half-bandwidth is ny): on a square its eigenvalues come in equal pairs, whose eigenvectors no two
computations agree on.  Contours cross the real axis, or pass between the eigenvalues, where the
predicted spectrum leaves a gap, as a user who counts eigenvalues places them.
"""
import functools
import math

import numpy as np
import torch

import paper_1510_07522_gb300 as rs

ASPECT = 0.8       # the domain is 1 x ASPECT
SIGMA2 = 108.8     # second branch point of the gun-like NEP is SIGMA2^2
DELTA = 1e-14      # truncation level of the projection
TOL = 1e-10        # backward error every sample has to meet
C64 = rs.RSRR_C64_IR | rs.RSRR_REFINE_FULL


# ---- the cases -------------------------------------------------------------------------------
def listed():
    return [
        # one small request served from scratch: handle made, solved and closed (a server's
        # smallest request; launches, synchronisations and host work)
        dict(name="request_144", family="gun", nx=12, ny=12, N=16, L=8, mode="fp64", NS=500, K=2,
             shape="circle", lo=118.0, hi=400.0, once=True),
        # the paper's small gun-type problem in FP64 on a handle kept between passes
        dict(name="gun_900_fp64", family="gun", nx=30, ny=30, N=32, L=16, mode="fp64", NS=500, K=2,
             shape="circle", lo=118.0, hi=400.0, once=False),
        # the same problem on a rectangle with Gauss-Legendre points, mixed precision, the
        # moment scheme: the paper's other contour and its other projection
        dict(name="rect_moments_900", family="gun", nx=30, ny=30, N=36, L=4, mode="c64", NS=500, K=2,
             shape="rectangle", lo=118.0, hi=335.0, once=False, moments=18),
        # the benchmark workload's matrices (n = 40000, band 200) with a contour that encloses
        # eigenpairs: the largest ordinary run, mixed precision
        dict(name="qep_40000", family="qep", nx=200, ny=200, N=64, L=32, mode="c64", NS=500, K=2, m=10),
        # a mid-size run with odd sizes everywhere: band, points and probing columns
        dict(name="qep_9991_odd", family="qep", nx=103, ny=97, N=31, L=13, mode="c64", NS=500, K=2, m=8),
        # plain FP64 sampling of a mid-size problem (no mixed precision)
        dict(name="qep_3840_fp64", family="qep", nx=64, ny=60, N=32, L=16, mode="fp64", NS=500, K=2, m=8),
        # a band wider than the tensor-core factor takes (250, as the 400 x 250 gun-like problem)
        # with that problem's contour on half its points
        dict(name="gun_60000_wide", family="gun", nx=240, ny=250, N=32, L=24, mode="c64", NS=500, K=2,
             shape="circle", lo=38.0, hi=500.0, once=False),
        # one time-delay problem whose coupling leaves no band: dense LU per point
        dict(name="delay_1600_dense", family="delay", nx=40, ny=40, N=32, L=8, mode="c64", NS=500, K=2,
             k0=3, m=8, band=-1),
        # the same kind with only the grid's band factored and GMRES on the full matrix
        dict(name="delay_2475_gmres", family="delay", nx=45, ny=55, N=32, L=8, mode="c64", NS=500, K=2,
             k0=4, m=10, band=55),
        # samples of a batch of uneven time-delay problems in one call, read back by the caller
        dict(name="batch_6_samples", family="batch", sides="20,26,31,36,41,24", N=32, L=8, mode="c64"),
        # the paper's loaded string: tridiagonal, one probing column, many points, K = 8
        dict(name="string_5000", family="string", n=5000, N=100, L=1, mode="fp64", NS=1000, K=8),
        # T known by its values: callback at the points, Chebyshev interpolant of degree 16
        dict(name="tz_cheb_272", family="tz", nx=17, ny=16, N=48, L=4, mode="c64", NS=500, K=2, d=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    f = rng.choice(["gun", "gun", "rect", "qep", "qep", "qep64", "wide", "dense", "gmres", "batch", "string", "tz"])
    if f == "gun":
        nx, ny, N = rng.randint(16, 36), rng.randint(16, 36), rng.randint(16, 34)
        return dict(family="gun", nx=nx, ny=ny, N=N, L=max(6, min(18, int(0.57 * nx * ny / N))),
                    mode=rng.choice(["fp64", "c64"]), NS=500, K=2, shape="circle", lo=118.0, hi=400.0,
                    once=nx * ny < 360)
    if f == "rect":
        N = 2 * rng.randint(15, 22)
        return dict(family="gun", nx=rng.randint(18, 34), ny=rng.randint(18, 34), N=N, L=rng.randint(4, 7),
                    mode=rng.choice(["fp64", "c64"]), NS=500, K=2, shape="rectangle", lo=118.0, hi=335.0,
                    once=False, moments=rng.randint(14, 20))
    if f == "qep":
        return dict(family="qep", nx=_log(rng, 40, 190), ny=_log(rng, 40, 190), N=rng.randint(24, 56),
                    L=rng.randint(8, 28), mode="c64", NS=500, K=2, m=rng.randint(6, 11))
    if f == "qep64":
        return dict(family="qep", nx=_log(rng, 24, 70), ny=_log(rng, 24, 64), N=rng.randint(20, 36),
                    L=rng.randint(8, 18), mode="fp64", NS=500, K=2, m=rng.randint(6, 9))
    if f == "wide":
        return dict(family="gun", nx=rng.randint(228, 250), ny=rng.randint(228, 250), N=rng.randint(24, 31),
                    L=rng.randint(14, 24), mode="c64", NS=500, K=2, shape="circle", lo=38.0, hi=500.0, once=False)
    if f == "dense":
        return dict(family="delay", nx=rng.randint(18, 40), ny=rng.randint(18, 40), N=rng.randint(24, 36),
                    L=rng.randint(6, 10), mode=rng.choice(["c64", "c64", "fp64"]), NS=500, K=2,
                    k0=rng.randint(3, 6), m=rng.randint(5, 10), band=-1)
    if f == "gmres":
        nx, ny = rng.randint(24, 48), rng.randint(24, 52)
        return dict(family="delay", nx=nx, ny=ny, N=rng.randint(24, 34), L=rng.randint(6, 9), mode="c64",
                    NS=500, K=2, k0=rng.randint(3, 6), m=rng.randint(5, 10), band=ny)
    if f == "batch":
        return dict(family="batch", sides=",".join(str(rng.randint(18, 40)) for _ in range(rng.randint(3, 7))),
                    N=rng.randint(20, 34), L=rng.randint(6, 9), mode="c64")
    if f == "string":
        return dict(family="string", n=_log(rng, 600, 6000), N=rng.randint(90, 110), L=1, mode="fp64", NS=1000, K=8)
    nx = rng.randint(13, 18)
    return dict(family="tz", nx=nx, ny=nx - 1, N=rng.randint(44, 56), L=rng.randint(5, 7),
                mode=rng.choice(["fp64", "c64"]), NS=500, K=2, d=rng.randint(15, 20))


# ---- matrices on one sparsity pattern ------------------------------------------------------------
def _laplacian_1d(n, h):
    return (np.diag(np.full(n, 2.0)) - np.diag(np.ones(n - 1), 1) - np.diag(np.ones(n - 1), -1)) / h ** 2


def _grid(nx, ny):
    """(rows, cols, K values) of the 5-point Laplacian, entries sorted by row, then column."""
    hx, hy = 1.0 / (nx + 1), ASPECT / (ny + 1)
    i = np.arange(nx * ny).reshape(nx, ny)
    r, c, v = [i.ravel()], [i.ravel()], [np.full(nx * ny, 2.0 / hx ** 2 + 2.0 / hy ** 2)]
    for a, b, w in ((i[:-1], i[1:], -1.0 / hx ** 2), (i[:, :-1], i[:, 1:], -1.0 / hy ** 2)):
        r += [a.ravel(), b.ravel()]
        c += [b.ravel(), a.ravel()]
        v += [np.full(a.size, w)] * 2
    r, c, v = np.concatenate(r), np.concatenate(c), np.concatenate(v)
    o = np.lexsort((c, r))
    return r[o], c[o], v[o]


def _csr(n, rows, cols):
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(rows, minlength=n), out=rowptr[1:])
    return rowptr, cols.astype(np.int32)


def _probe(n, L, rng):
    U = rng.standard_normal((L, n, 2))
    return np.asfortranarray(((U[..., 0] + 1j * U[..., 1]) / math.sqrt(2.0)).T)


def _levels(nx, ny):
    """Eigenvalues of K, ascending."""
    lx = np.linalg.eigvalsh(_laplacian_1d(nx, 1.0 / (nx + 1)))
    ly = np.linalg.eigvalsh(_laplacian_1d(ny, ASPECT / (ny + 1)))
    return np.sort((lx[:, None] + ly[None, :]).ravel())


def _gap_near(x, levels, slack=0.15):
    """The middle of the widest gap of `levels` whose middle lies within slack * x of x."""
    mid, wid = 0.5 * (levels[1:] + levels[:-1]), np.diff(levels)
    wid = np.where(np.abs(mid - x) <= slack * x, wid, 0.0)
    return float(mid[np.argmax(wid)])


@functools.lru_cache(maxsize=None)
def _gun_ends(nx, ny, lo, hi):
    """Where the contour crosses the real axis: in gaps of the spectrum predicted with the mean
    mass and the square-root terms frozen at the centre (then the operator separates in x and y)."""
    z0 = 0.5 * (lo + hi)
    Ax = _laplacian_1d(nx, 1.0 / (nx + 1)).astype(complex)
    Ax[0, 0] += 1j * np.sqrt(z0)
    Ax[-1, -1] -= np.sqrt(SIGMA2 ** 2 - z0)
    lx = np.linalg.eigvals(Ax).real
    ly = np.linalg.eigvalsh(_laplacian_1d(ny, ASPECT / (ny + 1)))
    lev = np.sort((lx[:, None] + ly[None, :]).ravel()) / 1.05
    return _gap_near(lo, lev), _gap_near(hi, lev)


@functools.lru_cache(maxsize=None)
def _qep_ellipse(nx, ny, m):
    """An ellipse around the m lowest upper-branch eigenvalues (predicted with the mean mass),
    scaled so that no eigenvalue lies near it."""
    mu = _levels(nx, ny) / 1.05
    c = 0.02 + 0.05 * mu
    s = np.sqrt(4 * mu - c * c + 0j)
    z = (-c + 1j * s) / 2
    w = z[:m]
    re_lo, re_hi = w.real.min() - 0.5, w.real.max() + 0.5
    im_lo, im_hi = 0.5 * w.imag.min(), 0.5 * (w.imag.max() + z[m].imag)
    g = complex(0.5 * (re_lo + re_hi), 0.5 * (im_lo + im_hi))
    a, b = 0.8 * (re_hi - re_lo), 0.5 * (im_hi - im_lo)
    allz = np.concatenate([z, (-c - 1j * s) / 2])
    rho = np.abs((allz.real - g.real) / a + 1j * (allz.imag - g.imag) / b)
    best = max(np.linspace(0.92, 1.12, 41), key=lambda t: np.min(np.abs(rho / t - 1)))
    return g, float(a * best), float(b * best)


def _gun(case, rng):
    nx, ny = case["nx"], case["ny"]
    n = nx * ny
    rows, cols, kv = _grid(nx, ny)
    d = rows == cols
    ix = rows // ny
    vals = np.zeros((4, rows.size), dtype=np.complex128)
    vals[0] = kv
    vals[1, d] = -(1.0 + 0.1 * rng.random(n))
    vals[2, d & (ix == 0)] = 1.0
    vals[3, d & (ix == nx - 1)] = 1.0
    fns = [(rs.F_CONST, []), (rs.F_Z, []), (rs.F_ISQRT_SHIFT, [0.0, 0.0]), (rs.F_ISQRT_SHIFT, [SIGMA2 ** 2, 1.0])]
    lo, hi = _gun_ends(nx, ny, case["lo"], case["hi"])
    c, r = 0.5 * (lo + hi), 0.5 * (hi - lo)
    if case["shape"] == "rectangle":
        # a long rectangle about the axis, as the paper's gun example has, 2 N / 3 points on the long sides
        contour = (complex(c, 20.0), r, 25.0, rs.RSRR_CONTOUR_RECTANGLE, case["N"] // 3)
    else:
        contour = (complex(c), r, r, rs.RSRR_CONTOUR_ELLIPSE, 0)
    return n, rows, cols, vals, fns, contour


def _qep(case, rng):
    nx, ny = case["nx"], case["ny"]
    n = nx * ny
    rows, cols, kv = _grid(nx, ny)
    M = np.zeros(rows.size)
    M[rows == cols] = 1.0 + 0.1 * rng.random(n)
    vals = np.stack([kv, 0.05 * kv + 0.02 * M, M]).astype(np.complex128)
    g, a, b = _qep_ellipse(nx, ny, case["m"])
    return n, rows, cols, vals, [(rs.F_CONST, []), (rs.F_Z, []), (rs.F_Z2, [])], (g, a, b, rs.RSRR_CONTOUR_ELLIPSE, 0)


def _delay(nx, ny, k0, m, rng):
    n = nx * ny
    tau = rng.uniform(0.5, 2.0)
    kr, kc, kv = _grid(nx, ny)
    cnt = rng.binomial(n, 0.05, size=n)
    ar = np.repeat(np.arange(n), cnt)
    ac = rng.integers(0, n, ar.size)
    ak = np.unique(ar * n + ac)
    ak = ak[ak // n != ak % n]
    av = rng.uniform(-1.0, 1.0, ak.size)
    diag = 1.0 + np.bincount(ak // n, weights=np.abs(av), minlength=n)   # strictly dominant rows
    kk = kr * n + kc
    keys = np.union1d(kk, ak)
    rows, cols = keys // n, keys % n
    vals = np.zeros((3, keys.size), dtype=np.complex128)
    vals[0, rows == cols] = -1.0
    vals[1, np.searchsorted(keys, kk)] = kv
    vals[2, np.searchsorted(keys, ak)] = av
    vals[2, rows == cols] = diag
    lev = _levels(nx, ny)
    # the widest of three neighbouring gaps at either end
    i, j = (max(range(q - 1, q + 2), key=lambda t: lev[t + 1] - lev[t]) for q in (k0 - 1, k0 + m - 1))
    lo, hi = float(0.5 * (lev[i] + lev[i + 1])), float(0.5 * (lev[j] + lev[j + 1]))
    r = 0.5 * (hi - lo)
    fns = [(rs.F_Z, []), (rs.F_CONST, []), (rs.F_EXP_DELAY, [tau])]
    return n, rows, cols, vals, fns, (complex(0.5 * (lo + hi)), r, r, rs.RSRR_CONTOUR_ELLIPSE, 0)


def _string(case):
    n = case["n"]
    i = np.arange(n)
    rows = np.concatenate([i, i[:-1], i[1:]])
    cols = np.concatenate([i, i[1:], i[:-1]])
    vals = np.zeros((3, rows.size), dtype=np.complex128)
    vals[0] = np.where(rows == cols, 2.0 * n, -float(n))
    vals[0, n - 1] = n
    vals[1, n - 1] = 1.0
    vals[2] = -np.where(rows == cols, 4.0, 1.0) / (6.0 * n)
    vals[2, n - 1] = -2.0 / (6.0 * n)
    o = np.lexsort((cols, rows))
    fns = [(rs.F_CONST, []), (rs.F_RATIONAL, [1.0, -1.0]), (rs.F_Z, [])]
    return n, rows[o], cols[o], vals[:, o], fns, (5001.5 + 0j, 4998.5, 249.925, rs.RSRR_CONTOUR_ELLIPSE, 0)


@functools.lru_cache(maxsize=None)
def _tz_data(nx, ny):
    """T(z)_ij = K_ij - z d_ij + B_ij exp(-tau_ij z), K unscaled, and the contour: a flat ellipse
    about an interval of the real axis whose ends lie where T(x) (real symmetric) is far from singular."""
    n = nx * ny
    rows, cols, kv = _grid(nx, ny)
    kv = np.where(rows == cols, 4.0, -1.0)
    rng = np.random.default_rng([5, nx, ny])
    _, inv = np.unique(np.minimum(rows, cols) * n + np.maximum(rows, cols), return_inverse=True)
    off = rows != cols
    b = np.where(off, 0.3 * rng.uniform(-1.0, 1.0, inv.max() + 1)[inv], 0.0)
    tau = rng.uniform(0.5, 2.0, inv.max() + 1)[inv]

    def clear(x):
        T = np.zeros((n, n))
        T[rows, cols] = kv - x * (~off) + b * np.exp(-tau * x)
        return np.min(np.abs(np.linalg.eigvalsh(T)))
    lo, hi = (max(np.linspace(x - 0.1, x + 0.1, 15), key=clear) for x in (0.98, 2.0))
    contour = (complex(0.5 * (lo + hi)), 0.5 * (hi - lo), 0.1, rs.RSRR_CONTOUR_ELLIPSE, 0)
    return n, rows, cols, kv, ~off, b, tau, contour


def _problem(case, seed):
    """(n, rows, cols, vals, fns, contour, U) of a case other than batch and tz."""
    rng = np.random.default_rng([17, seed])
    f = case["family"]
    p = _gun(case, rng) if f == "gun" else _qep(case, rng) if f == "qep" else _string(case) if f == "string" \
        else _delay(case["nx"], case["ny"], case["k0"], case["m"], rng)
    return p + (_probe(p[0], case["L"], rng),)


def _batch_problems(case, seed):
    out = []
    for i, s in enumerate(int(x) for x in case["sides"].split(",")):
        rng = np.random.default_rng([19, seed, i])
        p = _delay(s, s, 3 + i % 4, 5 + i % 5, rng)
        out.append(p + (_probe(p[0], case["L"], rng),))
    return out


def _open(p):
    rowptr, colind = _csr(p[0], p[1], p[2])
    return rowptr, colind, p[3], p[4]


# ---- prepare and run ----------------------------------------------------------------------------
def prepare(case, seed):
    prec = C64 if case["mode"] == "c64" else rs.RSRR_FP64
    if case["family"] == "batch":
        ps = _batch_problems(case, seed)
        return dict(case=case, prec=prec, handles=[rs.Nep(p[0], *_open(p)) for p in ps], contours=[p[5] for p in ps],
                    U=[p[6] for p in ps])
    if case["family"] == "tz":
        n, rows, cols, kv, dg, b, tau, contour = _tz_data(case["nx"], case["ny"])
        rowptr, colind = _csr(n, rows, cols)
        h = rs.Nep.from_tz(n, rowptr, colind, lambda z: kv - z * dg + b * np.exp(-tau * z))
        return dict(case=case, prec=prec, h=h, contour=contour, U=_probe(n, case["L"], np.random.default_rng([17, seed])))
    p = _problem(case, seed)
    s = dict(case=case, prec=prec, n=p[0], csr=_open(p), contour=p[5], U=p[6], h=None)
    if not case.get("once"):
        banded = case.get("band", -1) >= 0   # iterate with the factor of the grid's own band
        s["h"] = rs.Nep(s["n"], *s["csr"], rs.RSRR_NATURAL_ORDER if banded else 0)
        if banded:
            s["h"].set_band_preconditioner(case["band"])
    return s


def _fix_phase(V, U):
    """Unit eigenvectors are free up to a phase: make their inner products with the first probing column real."""
    t = U[:, 0].conj() @ V
    return V * (np.abs(t) / t)


def run(s):
    case = s["case"]
    if case["family"] == "batch":
        k = len(s["handles"])
        rs.sample_batch(s["handles"], s["contours"], [case["N"]] * k, [case["L"]] * k, s["U"], s["prec"], TOL, 20)
        return [h.samples() for h in s["handles"]]
    h = s["h"] or rs.Nep(s["n"], *s["csr"])
    g, a, b, shape, side = s["contour"]
    h.sample(g, a, b, case["N"], case["L"], s["U"], s["prec"], TOL, 60, shape=shape, side_nodes=side)
    if case["family"] == "tz":
        h.project_chebyshev(case["d"], g.real - a, g.real + a, DELTA)
    elif case.get("moments"):
        h.project_moments(case["moments"], DELTA)
    else:
        h.project(DELTA)
    sigma = h.sigma()
    lam, V, _ = h.solve(case["NS"], case["K"], 1e3, 128, True)
    if case.get("once"):
        h.close()
    return dict(lam=lam, V=_fix_phase(V, s["U"]), sigma=sigma)


# ---- what a pass cannot do without ------------------------------------------------------------------
def _sizes(case):
    """(n, half-bandwidth or -1, stored entries, terms)"""
    f = case["family"]
    if f == "string":
        return case["n"], 1, 3 * case["n"], 3
    n = case["nx"] * case["ny"]
    if f == "delay":
        return n, case["band"], int(0.05 * n * n) + 6 * n, 3
    return n, case["ny"], 5 * n, 4 if f == "gun" else 3 if f == "qep" else case["N"] + case["d"]


def work(case):
    """Inputs read and outputs written once; flops of the factorisations and solves of every point, of a
    basis of rank k of the samples (k about 250 on these problems), of A_i's projections, of the
    reduced problem's inverses at the quadrature points and of one bidiagonalisation."""
    if case["family"] == "batch":
        b = f = 0.0
        for s in (int(x) for x in case["sides"].split(",")):
            n = s * s
            b += 3 * 16 * 0.05 * n * n + 16.0 * n * case["L"] * (1 + case["N"])
            f += case["N"] * (8.0 / 3.0 * n ** 3 + 8.0 * n * n * case["L"])
        return dict(bytes=b, flops=f)
    n, band, nnz, J = _sizes(case)
    N, L = case["N"], case["L"]
    if band < 0:
        flops = N * (8.0 / 3.0 * n ** 3 + 8.0 * n * n * L)
    else:
        flops = N * (16.0 * n * band * band + 24.0 * n * band * L)
    m = case["moments"] * L if case.get("moments") else N * L
    k = min(n, m, 250)
    D = case["K"] * k
    flops += 8.0 * n * m * k + 8.0 * n * k * k * min(J, 17) + 8.0 * case["NS"] * k ** 3 + 32.0 / 3.0 * D ** 3
    return dict(bytes=16.0 * nnz * J + 4.0 * nnz + 16.0 * n * L + 16.0 * n * 16 + 8.0 * min(n, m), flops=flops)


# ---- the same results in 64 bits by plain torch ---------------------------------------------------------
def _coef(fns, z):
    """f_i(z) and f_i'(z) for the points z: two arrays [points, terms]."""
    z = np.asarray(z, dtype=np.complex128)
    f, d = [], []
    for kind, p in fns:
        if kind == rs.F_CONST:
            f.append(np.ones_like(z)), d.append(np.zeros_like(z))
        elif kind == rs.F_Z:
            f.append(z), d.append(np.ones_like(z))
        elif kind == rs.F_Z2:
            f.append(z * z), d.append(2 * z)
        elif kind == rs.F_EXP_DELAY:
            f.append(np.exp(-p[0] * z)), d.append(-p[0] * np.exp(-p[0] * z))
        elif kind == rs.F_RATIONAL:
            f.append(p[0] * z / (z + p[1])), d.append(p[0] * p[1] / (z + p[1]) ** 2)
        elif p[1] == 0.0:
            r = np.sqrt(z - p[0])
            f.append(1j * r), d.append(0.5j / r)
        else:
            r = np.sqrt(p[0] - z)
            f.append(-r), d.append(0.5 / r)
    return np.stack(f, 1), np.stack(d, 1)


class _Solver:
    """T(z_k) X = B for several points at once on the GPU in complex128: block tridiagonal elimination
    (blocks of the half-bandwidth) with one step of iterative refinement, or dense LU."""

    def __init__(self, n, rows, cols, block):
        self.n, self.b = n, block
        self.rows, self.cols = (torch.as_tensor(x, device="cuda", dtype=torch.int64) for x in (rows, cols))

    def mul(self, v, X):   # v [B, nnz], X [B, n, L]
        Y = torch.zeros_like(X)
        for k in range(X.shape[0]):
            Y[k].index_add_(0, self.rows, v[k][:, None] * X[k][self.cols])
        return Y

    def solve(self, v, B):   # v [points, nnz], B [points, n, L] -> X
        if self.b == 0:
            out = []
            for k in range(v.shape[0]):
                T = torch.zeros(self.n, self.n, dtype=torch.complex128, device="cuda")
                T[self.rows, self.cols] = v[k]
                out.append(torch.linalg.solve(T, B[k]))
            return torch.stack(out)
        n, b, P = self.n, self.b, v.shape[0]
        nb = -(-n // b)
        D, Lo, Up = (torch.zeros(nb, P, b, b, dtype=torch.complex128, device="cuda") for _ in range(3))
        br, bc, r, c = self.rows // b, self.cols // b, self.rows % b, self.cols % b
        for M, off in ((D, 0), (Lo, 1), (Up, -1)):
            at = br - bc == off
            M[br[at], :, r[at], c[at]] = v[:, at].T
        for i in range(n, nb * b):
            D[i // b, :, i % b, i % b] = 1.0
        G, C = [], []
        S = D[0]
        for i in range(nb):
            G.append(torch.linalg.inv(S))
            if i + 1 < nb:
                C.append(G[i] @ Up[i])
                S = D[i + 1] - Lo[i + 1] @ C[i]

        def sweep(R):
            R = torch.nn.functional.pad(R, (0, 0, 0, nb * b - n)).reshape(P, nb, b, -1)
            y = []
            for i in range(nb):
                y.append(G[i] @ (R[:, i] - Lo[i] @ y[i - 1] if i else R[:, 0]))
            for i in range(nb - 2, -1, -1):
                y[i] = y[i] - C[i] @ y[i + 1]
            return torch.stack(y, 1).reshape(P, nb * b, -1)[:, :n]
        X = sweep(B)
        return X + sweep(B - self.mul(v, X))


def _nodes(contour, N):
    """Points and weights of (1 / 2 pi i) oint dz for the contour's rule."""
    g, a, b, shape, side = contour
    if shape == rs.RSRR_CONTOUR_ELLIPSE:
        t = 2 * np.pi * (np.arange(N) + 0.5) / N
        return g + a * np.cos(t) + 1j * b * np.sin(t), (-a * np.sin(t) + 1j * b * np.cos(t)) / (1j * N)
    z, w = [], []
    corner = [g - a - 1j * b, g + a - 1j * b, g + a + 1j * b, g - a + 1j * b]
    for k, m in enumerate((side, N // 2 - side) * 2):
        x, q = np.polynomial.legendre.leggauss(m)
        d = (corner[(k + 1) % 4] - corner[k]) / 2
        z.append(corner[k] + d * (x + 1)), w.append(q * d / (2j * np.pi))
    return np.concatenate(z), np.concatenate(w)


def _inside(contour, z):
    g, a, b, shape, _ = contour
    x, y = (z.real - g.real) / a, (z.imag - g.imag) / b
    return x * x + y * y < 1 if shape == rs.RSRR_CONTOUR_ELLIPSE else (np.abs(x) < 1) & (np.abs(y) < 1)


def _eigenpairs(S, vals_at, dvals_at, contour, nodes, guess=72):
    """All eigenpairs inside the contour: contour moments of T^{-1} on random vectors, then inverse
    iteration with the Rayleigh functional of the nonlinear problem until it stands still."""
    g, a, b, shape, _ = contour
    z, w = _nodes(contour[:4] + (nodes * 3 // 10,), nodes)
    rnd = torch.Generator(device="cuda").manual_seed(3)
    R = torch.randn(1, S.n, guess, dtype=torch.complex128, device="cuda", generator=rnd)
    A0 = A1 = 0
    for k in range(0, z.size, 20):
        X = S.solve(vals_at(z[k:k + 20]), R.expand(min(20, z.size - k), -1, -1))
        wk, zk = (torch.as_tensor(q[k:k + 20], device="cuda").reshape(-1, 1, 1) for q in (w, (z - g) / max(a, b)))
        A0, A1 = A0 + (wk * X).sum(0), A1 + (wk * zk * X).sum(0)
    Q, s, Wh = torch.linalg.svd(A0, full_matrices=False)
    r = int((s > 1e-7 * s[0]).sum())
    core = (Q[:, :r].conj().T @ A1 @ Wh[:r].conj().T) / s[:r]
    lam, y = torch.linalg.eig(core)
    lam, V = lam.cpu().numpy() * max(a, b) + g, Q[:, :r] @ y
    near = [t for t in range(r) if np.isfinite(lam[t]) and _inside((g, 1.05 * a, 1.05 * b, shape, 0), lam[t:t + 1])[0]]
    lam, V = lam[near], V[:, near].T[:, :, None].contiguous()
    for _ in range(5):
        V = S.solve(vals_at(lam), S.mul(dvals_at(lam), V))
        V = V / torch.linalg.norm(V, dim=1, keepdim=True)
        left = V.conj() if S.b == 0 else V   # the banded ones are complex symmetric: v^T is the left vector
        step = (left * S.mul(vals_at(lam), V)).sum((1, 2)) / (left * S.mul(dvals_at(lam), V)).sum((1, 2))
        step = step.cpu().numpy()
        lam = lam - step
    out = []
    for t in range(lam.size):
        if abs(step[t]) < 1e-9 * abs(lam[t]) and _inside(contour, lam[t:t + 1])[0] and \
                all(abs(lam[t] - q) > 1e-9 * abs(q) for q, _ in out):
            out.append((lam[t], V[t, :, 0].cpu().numpy()))
    out.sort(key=lambda e: abs(e[0]))
    return np.array([e[0] for e in out]), np.stack([e[1] for e in out], 1) if out else np.zeros((S.n, 0))


def exact(case, seed):
    if case["family"] in ("gun", "qep") and case["nx"] * case["ny"] ** 3 > 1.7e9:
        return None   # the eliminations below would take more than 20 s
    cuda = lambda x: torch.as_tensor(np.ascontiguousarray(x), device="cuda")  # noqa: E731
    if case["family"] == "batch":
        out = []
        for n, rows, cols, vals, fns, contour, U in _batch_problems(case, seed):
            S, z = _Solver(n, rows, cols, 0), _nodes(contour, case["N"])[0]
            X = S.solve(cuda(_coef(fns, z)[0] @ vals), cuda(U).expand(z.size, -1, -1))
            out.append(np.asfortranarray(X.permute(1, 0, 2).reshape(n, -1).cpu().numpy()))
        return out
    if case["family"] == "tz":
        n, rows, cols, kv, dg, b, tau, contour = _tz_data(case["nx"], case["ny"])
        U = _probe(n, case["L"], np.random.default_rng([17, seed]))
        vals_at = lambda z: cuda(np.stack([kv - x * dg + b * np.exp(-tau * x) for x in z]))  # noqa: E731
        dvals_at = lambda z: cuda(np.stack([-1.0 * dg - tau * b * np.exp(-tau * x) for x in z]).astype(complex))  # noqa: E731
        S = _Solver(n, rows, cols, case["ny"])
    else:
        n, rows, cols, vals, fns, contour, U = _problem(case, seed)
        vd = cuda(vals)
        vals_at = lambda z: cuda(_coef(fns, z)[0]) @ vd  # noqa: E731
        dvals_at = lambda z: cuda(_coef(fns, z)[1]) @ vd  # noqa: E731
        S = _Solver(n, rows, cols, 50 if case["family"] == "string" else 0 if case["family"] == "delay" else case["ny"])
    lam, V = _eigenpairs(S, vals_at, dvals_at, contour, dict(string=400, qep=48).get(case["family"], 80))
    sigma = None
    if n * case["N"] * case["L"] <= 1.2e7:   # larger: the SVD of the samples takes too long
        z, w = _nodes(contour, case["N"])
        X = torch.cat([S.solve(vals_at(z[k:k + 8]), cuda(U).expand(len(z[k:k + 8]), -1, -1)) for k in range(0, z.size, 8)])
        if case.get("moments"):
            zeta = (z - contour[0]) / max(contour[1], contour[2])
            W = cuda(w[:, None] * zeta[:, None] ** np.arange(case["moments"]))
            X = torch.einsum("ia,inl->anl", W, X)
        sigma = torch.linalg.svdvals(X.permute(1, 0, 2).reshape(n, -1).cpu()).numpy()
    return dict(lam=lam, V=_fix_phase(V, U), sigma=sigma)

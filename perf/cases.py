"""The work that users of this package have it do, as measurable cases.

A user fixes fields: a field in device memory is loaded into a context, relaxed
to its tolerance and read back (the ``fix`` cases, over the sizes, gauges,
algorithms and link storages in use); a user with a driver of their own issues
sweeps and reads the estimate (``sweep``), or polishes a field that is nearly
fixed (``polish``); a field is measured (``measure``) or only goes in and out of
a context (``io``); and a stream of jobs goes through the server (``serve``).

Every case is a dict of plain values; ``prepare`` makes its inputs from a seed
on the GPU, ``run`` is one pass through the public entry points, ``exact`` the
same pass in 64 bits with torch alone.  Fields are held as ``m[r][c]``, nine
complex tensors of the lattice's shape, while they are made and in ``exact``.
"""
import math
import time

import numpy as np
import torch

from paper_1305_3440_gb300 import lgt

GAUGES = {"landau": lgt.LGT_LANDAU, "coulomb": lgt.LGT_COULOMB, "mag": lgt.LGT_MAG}
BULKS = {"fp64": lgt.LGT_FP64, "fp32_18": lgt.LGT_FP32_18, "fp32_12": lgt.LGT_FP32_12}
AXIS = {0: 0, 1: 3, 2: 2, 3: 1}  # tensor axis of direction mu (t, x1, x2, x3)
SUBGROUPS = ((0, 1), (0, 2), (1, 2))
REAL = 8  # bytes


def _case(name, kind, dims, **kw):
    d = dict(kind=kind, nt=dims[0], n3=dims[1], n2=dims[2], n1=dims[3], gauge="landau", algo="or",
             bulk="fp32_12", omega=1.7, late=0.0, p=0.8, eps=0.5, tol=1e-14, sweeps=0, jobs=0)
    d.update(kw)
    if name:
        d["name"] = name
    return d


def listed():
    return [
        # One small field to full precision: nothing but launches and latency.
        _case("fix_8", "fix", (8, 8, 8, 8), eps=0.3),
        # A Coulomb job of the served sizes, with the omega schedule its stream uses.
        _case("fix_coulomb_16x32", "fix", (32, 16, 16, 16), gauge="coulomb", late=1.1, tol=1e-12),
        # Uneven extents, links stored whole in FP32.
        _case("fix_ragged", "fix", (14, 10, 12, 18), bulk="fp32_18", eps=0.4),
        # Every sweep in FP64, for users who want no FP32 phase.
        _case("fix_fp64", "fix", (12, 12, 12, 12), bulk="fp64", eps=0.4),
        # The headline: 32^4 Landau from rough to theta < 1e-14.
        _case("fix_32", "fix", (32, 32, 32, 32)),
        # Sweeps of the two production lattices, a driver's chunk of 20 and its check; the
        # second by stochastic relaxation.
        _case("sweep_coulomb_48x96", "sweep", (96, 48, 48, 48), gauge="coulomb", sweeps=20),
        _case("sweep_sr_64", "sweep", (64, 64, 64, 64), algo="sr", p=0.9, sweeps=20),
        # The third gauge, whose update is quadratic in g.
        _case("sweep_mag_24", "sweep", (24, 24, 24, 24), gauge="mag", sweeps=20),
        # The sweeps after promotion, on a field that is nearly fixed.
        _case("polish_32", "polish", (32, 32, 32, 32), omega=1.3, sweeps=20),
        # F, theta and plaquette, from a context and straight from a caller's buffer.
        _case("measure_32", "measure", (32, 32, 32, 32), bulk="fp64"),
        # A field into a context and out again (what every job pays beside its sweeps).
        _case("io_odd", "io", (36, 24, 28, 20)),
        # A burst of small and middling jobs through the server, host memory to host memory.
        _case("serve_burst", "serve", (16, 16, 16, 16), jobs=12, late=1.1, tol=1e-12),
    ]


def _dims(rng, lo, hi, shortest=4):
    """Four even extents whose volume is near exp(U(log lo, log hi)), unevenly split."""
    side = math.exp(rng.uniform(math.log(lo), math.log(hi))) ** 0.25
    out = [max(shortest, 2 * round(side * math.exp(rng.uniform(-0.45, 0.45)) / 2)) for _ in range(4)]
    while math.prod(out) > hi:
        out[out.index(max(out))] -= 2
    return tuple(out)


def draw(rng):
    kind = rng.choice(["fix", "fix", "fix", "sweep", "sweep", "sweep", "polish", "measure", "io", "serve"])
    eps = round(rng.uniform(0.3, 0.6), 3)
    if kind == "fix":
        bulk = rng.choice(["fp32_12", "fp32_12", "fp32_18", "fp64"])
        dims = _dims(rng, 8**4, 12**4 if bulk == "fp64" else 24**4)
        # a whole stochastic relaxation in FP32 leaves the constant rotation of its field at
        # 1e-4 or so: in FP32 it is drawn as sweeps
        algo = rng.choice(["or", "sr"]) if bulk == "fp64" else "or"
        return _case(None, kind, dims, gauge=rng.choice(["landau", "coulomb"]), algo=algo, bulk=bulk, eps=eps,
                     omega=round(rng.uniform(1.5, 1.7), 2), late=rng.choice([0.0, 1.1]) if algo == "or" else 0.0,
                     tol=rng.choice([1e-12, 1e-14]))
    if kind == "sweep":
        bulk = rng.choice(["fp32_12", "fp32_12", "fp32_12", "fp32_18", "fp64"])
        dims = _dims(rng, 8**4, 24**4 if bulk == "fp64" else 56**4)
        return _case(None, kind, dims, gauge=rng.choice(["landau", "landau", "coulomb", "coulomb", "mag"]),
                     algo=rng.choice(["or", "or", "sr"]), bulk=bulk, eps=eps, omega=round(rng.uniform(1.1, 1.8), 2),
                     sweeps=rng.randrange(5, 21))
    if kind == "polish":
        return _case(None, kind, _dims(rng, 8**4, 48**4), gauge=rng.choice(["landau", "coulomb"]),
                     algo=rng.choice(["or", "or", "sr"]), omega=round(rng.uniform(1.1, 1.5), 2),
                     sweeps=rng.randrange(5, 21))
    if kind == "measure":
        return _case(None, kind, _dims(rng, 8**4, 48**4), bulk=rng.choice(["fp64", "fp64", "fp32_12"]), eps=eps)
    if kind == "io":
        return _case(None, kind, _dims(rng, 8**4, 48**4), bulk=rng.choice(["fp32_12", "fp32_18", "fp64"]), eps=eps)
    side = rng.choice([8, 10, 12, 14, 16])
    return _case(None, kind, (side,) * 4, jobs=rng.randrange(2, 13), late=1.1, tol=1e-12)


# ------------------------------------------------------------ complex 3x3 fields
def _dims_of(case):
    return case["nt"], case["n3"], case["n2"], case["n1"]


def _mul(a, b):
    out = []
    for r in range(3):
        row = []
        for c in range(3):
            x = a[r][0] * b[0][c]
            x.addcmul_(a[r][1], b[1][c])
            row.append(x.addcmul_(a[r][2], b[2][c]))
        out.append(row)
    return out


def _dag(a):
    return [[a[c][r].conj().resolve_conj() for c in range(3)] for r in range(3)]


def _roll(a, mu, s):
    """The field at x + s mu."""
    return [[a[r][c].roll(-s, AXIS[mu]) for c in range(3)] for r in range(3)]


def _one(like):
    return [[torch.full_like(like, float(r == c)) for c in range(3)] for r in range(3)]


def _normal(gen, dims):
    return torch.randn(dims, generator=gen, device="cuda", dtype=torch.complex128) * math.sqrt(2)


def _su3(rows):
    """The SU(3) matrices of two rows: Gram-Schmidt, row 2 = conj(row 0 x row 1)."""
    def unit(v):
        n = (v[0].abs() ** 2 + v[1].abs() ** 2 + v[2].abs() ** 2).rsqrt()
        return [x * n for x in v]
    a = unit(rows[0])
    b = rows[1]
    for _ in range(2):  # twice: orthogonal to rounding
        s = a[0].conj() * b[0] + a[1].conj() * b[1] + a[2].conj() * b[2]
        b = unit([y - s * x for x, y in zip(a, b)])
    c = [(a[(k + 1) % 3] * b[(k + 2) % 3] - a[(k + 2) % 3] * b[(k + 1) % 3]).conj().resolve_conj() for k in range(3)]
    return [a, b, c]


def _near_one(gen, dims, eps):
    """SU(3) matrices at about exp(i eps sum_a r_a lambda_a / 2) with normal r_a."""
    z = [[_normal(gen, dims) for _ in range(3)] for _ in range(2)]
    off = 0.5 * eps  # an off-diagonal entry of i eps H: normal re and im of that width
    rows = [[(0.5j * eps * 1.15) * z[0][0].real + 1.0, off * z[0][1], off * z[0][2]],
            [0, (0.5j * eps * 1.15) * z[1][1].real + 1.0, off * z[1][2]]]
    rows[1][0] = -rows[0][1].conj()
    return _su3(rows)


def _store(u, out, mu):
    for r in range(3):
        for c in range(3):
            out[..., mu, r, c] = u[r][c]


def _field(case, seed, dims=None):
    """Links (complex128 on the GPU, public layout).  Fluctuations of width eps about
    one under a Haar-random gauge transformation: what a Monte Carlo hands over.
    The polish case instead has a constant background (stationary in Landau and
    Coulomb gauge) with violations of about 1e-4, as a promoted field has; sweeps that
    are given out without fixing start from a smooth field, as one is after its first
    relaxation (from a random one FP32 rounding, and stochastic relaxation anyhow, ends
    on another trajectory)."""
    dims = dims or _dims_of(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    near = case["kind"] == "polish"
    out = torch.empty(dims + (4, 3, 3), dtype=torch.complex128, device="cuda")
    if near or case["kind"] == "sweep":
        h = _near_one(gen, dims, 1e-4 if near else 0.4)
    else:
        h = _su3([[_normal(gen, dims) for _ in range(3)] for _ in range(2)])
    for mu in range(4):
        u = _near_one(gen, dims, 1e-4 if near else case["eps"])
        if near:
            u = _mul([[x.reshape(1, 1, 1, 1) for x in row] for row in _near_one(gen, (1,), 0.3)], u)
        _store(_mul(_mul(h, u), _dag(_roll(h, mu, 1))), out, mu)
    return out


def _load(links):
    return [[[links[..., mu, r, c].contiguous() for c in range(3)] for r in range(3)] for mu in range(4)]


# ------------------------------------------------------------------- the package
class _Context:
    """A context that frees its device memory with its last reference."""

    def __init__(self, params, links):
        self.h = lgt.lgt_create(params, links)

    def __del__(self):
        lgt.lgt_destroy(self.h)


class _Server:
    def __init__(self, budget):
        self.h = lgt.lgt_server_create(budget)

    def __del__(self):
        lgt.lgt_server_destroy(self.h)


def _params(case, dims=None, **kw):
    d = dict(dims=dims or _dims_of(case), gauge=GAUGES[case["gauge"]], bulk=BULKS[case["bulk"]], omega=case["omega"],
             algo=lgt.LGT_SR if case["algo"] == "sr" else lgt.LGT_OR, p=case["p"], seed=77, theta_tol=case["tol"],
             max_sweeps=40000, polish_algo=lgt.LGT_POLISH_OR if case["algo"] == "sr" else lgt.LGT_POLISH_SAME)
    if case["late"]:
        d.update(omega_late=case["late"], theta_omega=1e-2)
    d.update(kw)
    return lgt.lgt_params_default(**d)


def _jobs(case):
    """The served burst: sizes around the case's side, both gauges, both tolerances."""
    side = case["nt"]
    out = []
    for k in range(case["jobs"]):
        n = max(4, side - 2 * (k % 4))
        out.append(((2 * n if k % 3 == 2 else n, n, n, n), "coulomb" if k % 2 else "landau",
                    1e-14 if k % 4 == 1 else 1e-12, 0.3 + 0.03 * k))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        jobs = []
        for k, (dims, gauge, tol, eps) in enumerate(_jobs(case)):
            c = dict(case, gauge=gauge, tol=tol, eps=eps)
            U = _field(c, 1000 * int(seed) + k, dims).cpu().numpy()
            jobs.append((_params(c, dims), U, np.empty_like(U)))
        return {"case": case, "server": _Server(64 << 30), "jobs": jobs}
    links = _field(case, seed)
    torch.cuda.synchronize()
    extra = {"omega_polish": 0.0, "polish_algo": lgt.LGT_POLISH_SAME} if kind == "polish" else {}
    state = {"case": case, "ctx": _Context(_params(case, **extra), links)}
    if kind == "polish":
        lgt.lgt_promote(state["ctx"].h)
    if kind in ("fix", "io", "measure"):
        state["links"] = links
    if kind == "measure":
        state["sums"] = torch.empty(8 + 2 * case["nt"], dtype=torch.float64, device="cuda")
    else:
        state["out"] = torch.empty_like(links)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "serve":
        srv = state["server"].h
        ids = {lgt.lgt_submit(srv, p, U): k for k, (p, U, _) in enumerate(state["jobs"])}
        done = {}
        while ids:
            for jid, k in list(ids.items()):
                st, res = lgt.lgt_poll(srv, jid, state["jobs"][k][2])
                if st != lgt.LGT_EAGAIN:
                    # a fixed field is defined up to a constant rotation, which the FP32 phase
                    # leaves at FP32 accuracy: kept in single precision, as configurations are
                    done[k] = [int(st), res.F, res.plaquette, state["jobs"][k][2].astype(np.complex64)]
                    del ids[jid]
            if ids:
                time.sleep(0.0002)
        return [done[k] for k in sorted(done)]
    ctx = state["ctx"].h
    if kind == "fix":
        lgt.lgt_load(ctx, state["links"])
        st, res = lgt.lgt_fix(ctx)
        lgt.lgt_get_links(ctx, out=state["out"])
        out = state["out"] if case["bulk"] == "fp64" else state["out"].to(torch.complex64)  # as in serve
        return [int(st), res.F, res.plaquette, out]
    if kind == "sweep":
        lgt.lgt_sweep(ctx, case["sweeps"])
        F, theta, _, _ = lgt.lgt_estimate(ctx, case["nt"])
        lgt.lgt_get_working_links(ctx, out=state["out"])
        # the working links of an FP32 context are FP32 values
        return [F, theta, state["out"] if case["bulk"] == "fp64" else state["out"].to(torch.complex64)]
    if kind == "polish":
        lgt.lgt_sweep(ctx, case["sweeps"])
        lgt.lgt_get_links(ctx, out=state["out"])
        return [state["out"]]
    if kind == "measure":
        F, theta, plaq = lgt.lgt_measure(ctx)
        F_t, theta_t = lgt.lgt_measure_slices(ctx, case["nt"])
        lgt.lgt_measure_noalloc(_dims_of(case), state["links"], state["sums"])
        # the context's field is FP32 where its bulk is: its plaquette and F carry that rounding
        m = np.array([F, theta, plaq])
        if case["bulk"] != "fp64":
            m, F_t, theta_t = m.astype(np.float32), F_t.astype(np.float32), theta_t.astype(np.float32)
        return [m, F_t, theta_t, state["sums"]]
    lgt.lgt_load(ctx, state["links"])
    lgt.lgt_get_links(ctx, out=state["out"])
    return [state["out"]]


# ------------------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    vol = math.prod(_dims_of(case))
    field = vol * 4 * 18 * REAL  # a field in the public layout
    stored = vol * 4 * (18 * REAL if case["bulk"] == "fp64" else (12 if case["bulk"] == "fp32_12" else 18) * 4)
    update = 6000 if case["gauge"] == "mag" else (1800 if case["gauge"] == "coulomb" else 2300)
    if kind == "serve":
        b = f = 0
        for dims, gauge, _, _ in _jobs(case):
            v = math.prod(dims)
            b += v * 4 * 18 * (REAL + REAL + 4)
            f += 2300 * v * 3 * v**0.47
        return {"bytes": b, "flops": f}
    if kind == "fix":  # a fixed field's sweeps grow about as its extent to the power 1.9
        return {"bytes": 2 * field + (field // 2 if case["bulk"] != "fp64" else 0),
                "flops": update * vol * (2.2 if case["late"] else 5.0) * vol**0.47}
    if kind == "sweep":  # the stored field read and written once, and given out in its own precision
        return {"bytes": 2 * stored + field // (1 if case["bulk"] == "fp64" else 2),
                "flops": update * vol * case["sweeps"]}
    if kind == "polish":
        return {"bytes": 2 * field, "flops": 2300 * vol * case["sweeps"]}
    if kind == "measure":
        return {"bytes": 2 * stored + field, "flops": 3 * 3000 * vol}
    return {"bytes": 2 * field, "flops": 600 * vol}


# ------------------------------------------------------------- the same in 64 bits
def _parity(dims):
    t, a, b, c = (torch.arange(n, device="cuda") for n in dims)
    return (t[:, None, None, None] + a[None, :, None, None] + b[None, None, :, None] + c[None, None, None, :]) & 1


def _umulhi(a, b):
    """High and low 32 bits of the product of a 32-bit constant and int64 words."""
    lo, hi = a * (b & 0xFFFF), a * (b >> 16)
    return (hi + (lo >> 16)) >> 16, (a * b) & 0xFFFFFFFF


def _philox(ctr, key):
    k0, k1 = key
    for _ in range(10):
        ha, la = _umulhi(0xD2511F53, ctr[0])
        hb, lb = _umulhi(0xCD9E8D57, ctr[2])
        ctr = [hb ^ ctr[1] ^ k0, lb, ha ^ ctr[3] ^ k1, la]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return ctr


def _gather(U, first):
    K = None
    for mu in range(first, 4):
        b = _dag(_roll(U[mu], mu, -1))
        if K is None:
            K = [[U[mu][r][c] + b[r][c] for c in range(3)] for r in range(3)]
        else:
            for r in range(3):
                for c in range(3):
                    K[r][c] += U[mu][r][c]
                    K[r][c] += b[r][c]
    return K


def _violation(K):
    """tr Delta^2, Delta the traceless part of (K - K^dagger) / (2i)."""
    d = [K[a][a].imag for a in range(3)]
    tr = (d[0] + d[1] + d[2]) / 3
    s = sum((x - tr) ** 2 for x in d)
    for a in range(3):
        for b in range(a + 1, 3):
            s = s + 0.5 * (K[a][b] - K[b][a].conj()).abs() ** 2
    return s


def _mag_X(U):
    X = None
    for mu in range(4):
        w = _roll(U[mu], mu, -1)
        part = [[U[mu][r][c] * U[mu][c][c].conj() - w[r][r].conj() * w[r][c] for c in range(3)] for r in range(3)]
        X = part if X is None else [[X[r][c] + part[r][c] for c in range(3)] for r in range(3)]
    return X


def _relaxed(r, case, square):
    """Overrelaxation to first order, or the square where `square` says so."""
    if case["algo"] == "or":
        w = case["omega"]
        r = [(1 - w) + w * r[0]] + [w * x for x in r[1:]]
        n = (r[0] ** 2 + r[1] ** 2 + r[2] ** 2 + r[3] ** 2).rsqrt()
        return [x * n for x in r]
    sq = [r[0] ** 2 - (r[1] ** 2 + r[2] ** 2 + r[3] ** 2)] + [2 * r[0] * x for x in r[1:]]
    return [torch.where(square, a, b) for a, b in zip(sq, r)]


def _rotate(r, i, j, m):
    a, b = torch.complex(r[0], r[3]), torch.complex(r[2], r[1])
    for c in range(3):
        x, y = m[i][c], m[j][c]
        m[i][c], m[j][c] = a * x + b * y, a.conj() * y - b.conj() * x


def _update(case, U, K, draws):
    """g(x) of every site: three subgroup steps."""
    g = _one(U[0][0][0])
    thr = math.floor(case["p"] * 4294967296.0)
    for s, (i, j) in enumerate(SUBGROUPS):
        square = None if draws is None else draws[s] < thr
        if case["gauge"] == "mag":
            v = [0.0, 0.0, 0.0]

            def add(a, b, sign):
                z = a.conj() * b
                v[0] = v[0] + sign * 2 * z.real
                v[1] = v[1] + sign * 2 * z.imag
                v[2] = v[2] + sign * (a.abs() ** 2 - b.abs() ** 2)
            gd = _dag(g)
            for mu in range(4):
                f, b = _mul(g, U[mu]), _mul(_roll(U[mu], mu, -1), gd)
                add(f[i][i], f[j][i], 1)
                add(f[i][j], f[j][j], -1)
                add(b[i][i].conj(), b[i][j].conj(), 1)
                add(b[j][i].conj(), b[j][j].conj(), -1)
            a = (v[0] ** 2 + v[1] ** 2 + v[2] ** 2).sqrt() + v[2]
            n = (a * a + v[0] ** 2 + v[1] ** 2).rsqrt()
            r = [a * n, -v[1] * n, v[0] * n, torch.zeros_like(a)]
        else:
            q = [K[i][i].real + K[j][j].real, K[i][j].imag + K[j][i].imag, K[i][j].real - K[j][i].real,
                 K[i][i].imag - K[j][j].imag]
            n = (q[0] ** 2 + q[1] ** 2 + q[2] ** 2 + q[3] ** 2).rsqrt()
            r = [q[0] * n, -q[1] * n, -q[2] * n, -q[3] * n]
        r = _relaxed(r, case, square)
        if case["gauge"] != "mag":
            _rotate(r, i, j, K)
        _rotate(r, i, j, g)
    return g


def _sweep(case, U, n, sweep0=0):
    """n sweeps in place; (F, theta) as the sweeps' own estimate gives them."""
    dims = _dims_of(case)
    par = _parity(dims)
    first = 1 if case["gauge"] == "coulomb" else 0
    vol = math.prod(dims)
    site = torch.arange(vol, device="cuda").reshape(dims)
    F = theta = 0.0
    for k in range(n):
        sums = torch.zeros(dims[0], dtype=torch.float64, device="cuda")
        for p in range(2):
            K = _gather(U, first)
            on = par == p
            viol = _violation(_mag_X(U) if case["gauge"] == "mag" else K)
            sums += torch.where(on, viol, torch.zeros_like(viol)).sum((1, 2, 3))
            if p == 0:
                if case["gauge"] == "mag":
                    F = float(sum((U[mu][a][a].abs() ** 2).sum() for mu in range(4) for a in range(3))) / (12 * vol)
                else:
                    F = float(sum(U[mu][a][a].real.sum() for mu in range(first, 4) for a in range(3)))
                    F /= 3 * (4 - first) * vol
            draws = None
            if case["algo"] == "sr":
                word = [site & 0xFFFFFFFF, site >> 32, torch.full_like(site, sweep0 + k),
                        torch.full_like(site, 0x53524C58)]
                draws = _philox(word, (77, 0))
            g = _update(case, U, K, draws)
            one = _one(U[0][0][0][:1, :1, :1, :1])
            g = [[torch.where(on, g[r][c], one[r][c]) for c in range(3)] for r in range(3)]
            for mu in range(4):
                U[mu] = _mul(_mul(g, U[mu]), _dag(_roll(g, mu, 1)))
        vs = vol // dims[0]
        theta = float(sums.max()) / (3 * vs) if case["gauge"] == "coulomb" else float(sums.sum()) / (3 * vol)
    return F, theta


def _measured(U, dims):
    """F, theta, plaquette (Landau) and the timeslices' F_t, theta_t (Coulomb)."""
    vol, nt = math.prod(dims), dims[0]
    vs = vol // nt

    def delta(first):
        D = None
        for mu in range(first, 4):
            b = _roll(U[mu], mu, -1)
            part = [[U[mu][r][c] - b[r][c] for c in range(3)] for r in range(3)]
            D = part if D is None else [[D[r][c] + part[r][c] for c in range(3)] for r in range(3)]
        # A = traceless part of (U - U^dagger) / 2i is linear in U: halve the anti-Hermitian part
        return _violation([[0.5 * (D[r][c] - D[c][r].conj()) for c in range(3)] for r in range(3)])
    tr = [sum(U[mu][a][a].real for a in range(3)) for mu in range(4)]
    plaq = 0.0
    for mu in range(4):
        for nu in range(mu + 1, 4):
            A, B = _mul(U[mu], _roll(U[nu], mu, 1)), _mul(U[nu], _roll(U[mu], nu, 1))
            plaq += float(sum((A[r][c] * B[r][c].conj()).real.sum() for r in range(3) for c in range(3)))
    F = float(sum(x.sum() for x in tr)) / (12 * vol)
    theta = float(delta(0).sum()) / (3 * vol)
    F_t = sum(tr[1:]).sum((1, 2, 3)) / (9 * vs)
    theta_t = delta(1).sum((1, 2, 3)) / (3 * vs)
    return F, theta, plaq / (18 * vol), F_t, theta_t


def exact(case, seed):
    kind = case["kind"]
    vol = math.prod(_dims_of(case))
    if kind == "serve" or (kind == "fix" and (vol > 9000 or case["late"] or case["algo"] == "sr")):
        return None  # hundreds to thousands of sweeps: minutes in torch
    links = _field(case, seed)
    if kind == "io":
        return [links]
    U = _load(links)
    if kind == "fix":
        # to a theta at which F has its last digits; the links themselves depend on
        # where the sweeps stop
        for k in range(200):
            if _sweep(case, U, 10, 10 * k)[1] < 1e-15:
                break
        F, _, plaq, F_t, _ = _measured(U, _dims_of(case))
        return [0, float(F_t.mean()) if case["gauge"] == "coulomb" else F, plaq, None]
    if kind == "measure":
        F, theta, plaq, F_t, theta_t = _measured(U, _dims_of(case))
        head = [F, theta, plaq, float(F_t.mean()), float(theta_t.max()), float(theta_t.mean()), 0.0, 0.0]
        sums = torch.cat([torch.tensor(head, dtype=torch.float64, device="cuda"), F_t, theta_t])
        return [np.array([F, theta, plaq]), F_t, theta_t, sums]
    F, theta = _sweep(case, U, case["sweeps"])
    out = links
    for mu in range(4):
        _store(U[mu], out, mu)
    return [out] if kind == "polish" else [F, theta, out]

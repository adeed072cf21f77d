"""The marcher's work as its users have it done, as cases that can be timed and checked.

Every case goes through the Python binding of the C ABI: plans made once (``prepare``), then per
pass the starters set, the march (alone, batched, or through the serving loop) and the whole
results read back, as ``bench.py`` and the serving loop do.  Fields start as a sum of the guide's
propagating modes (within 30 degrees of horizontal) with random complex amplitudes: the field of a
guide some way down range, which fills the whole depth.  ``exact`` marches the same inputs in
complex128 with plain torch (the product form of the Pade propagator, the Neumann series with
its stop rule, library FFTs).
"""
import math

import numpy as np
import torch

from paper_2511_03343_gb300 import inputs, sssp

C0 = inputs.C0_DEFAULT


def _march(name, N, count, steps, fmin, fmax, **kw):
    c = dict(name=name, kind="march", N=N, count=count, steps=steps, fmin=float(fmin), fmax=float(fmax), H=5000.0,
             dr=25.0, order=6, terms=12, tol=1e-10, env="munk", bc="dirichlet", op="spectral", tl_every=0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: the isovelocity guide at its own sizes, a TL row every step, where
        # launches and host calls count
        _march("iso_n255", 255, 1, 100, 100, 100, H=100.0, dr=5.0, order=4, terms=0, env="iso", tl_every=1),
        # one user, one solve of the batch's grid
        _march("munk_n1023", 1023, 1, 100, 150, 150, tl_every=10),
        # the headline: 256 solves over the frequencies of the batched workload that the grid resolves
        _march("batch256_n1023", 1023, 256, 160, 60, 250, tl_every=20),
        # a ragged number of mid-size solves with an absorbing bottom layer (complex n^2)
        _march("absorb37_n2047", 2047, 37, 40, 60, 200, env="absorb", tl_every=10),
        # the single full-size Munk march
        _march("munk_n4095", 4095, 1, 100, 50, 50, dr=50.0, tl_every=20),
        # the range-dependent march: a profile node per step, [8/8]
        _march("eddy_n16383", 16383, 1, 40, 250, 250, order=8, env="eddy", tl_every=20),
        # the largest grid, a full device of solves (the memory-bound batch)
        _march("batch152_n65535", 65535, 152, 2, 100, 1000, order=4),
        # sizes of the serving mix in one batched call, uneven step counts
        dict(name="mix45", kind="mix", sizes="255,511,1023,4095,8191", count=45, steps=40, H=5000.0, order=6,
             terms=12, tol=1e-10, tl_every=10),
        # rigid boundaries (the cosine transform), a small batch
        _march("neumann24_n1025", 1025, 24, 60, 60, 300, bc="neumann", tl_every=10),
        # the finite-difference comparison operator
        _march("fd16_n1023", 1023, 16, 200, 30, 60, op="fd3", tl_every=20),
        # the transform alone, batched, fields resident on the device
        dict(name="dst4096_n1023", kind="dst", N=1023, count=4096),
        # the serving loop: requests of mixed sizes from submission to the results on the host
        dict(name="serve30", kind="serve", sizes="255,1023,4095", count=30, steps=60, chunk=20, H=5000.0,
             order=6, terms=12, tol=1e-10, tl_every=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _band(N):
    """Frequencies a 5000 m guide of N points resolves."""
    top = min(1000.0, 0.15 * (N + 1))
    return 0.5 * top, top


def _step_and_order(N, order):
    """Range step and Pade order whose Neumann series converges on the Munk guide at _band(N)
    (short steps at a high order diverge on coarse grids)."""
    return (100.0, min(order, 4)) if N < 400 else (50.0 if N < 800 else 25.0, min(order, 6))


def draw(rng):
    kind = rng.choice(["march", "march", "march", "march", "mix", "bc", "fd", "dst", "serve"])
    order, tl = rng.randint(4, 8), rng.choice([0, 7, 10])
    if kind == "dst":
        N = 2 ** rng.randint(7, 16) - 1
        return dict(kind="dst", N=N, count=max(1, min(_log_int(rng, 3, 9000), (1 << 23) // N)))
    if kind == "mix":
        sizes = rng.sample([255, 511, 1023, 2047, 4095, 8191, 16383], 3)
        return dict(kind="mix", sizes=",".join(str(n) for n in sorted(sizes)), count=_log_int(rng, 3, 60),
                    steps=rng.randint(10, 40), H=5000.0, order=min(order, 6), terms=rng.choice([4, 8, 12]),
                    tol=1e-10, tl_every=tl)
    if kind == "serve":
        sizes = rng.sample([255, 511, 1023, 2047, 4095, 8191], 3)
        return dict(kind="serve", sizes=",".join(str(n) for n in sorted(sizes)), count=_log_int(rng, 3, 40),
                    steps=rng.randint(20, 60), chunk=rng.randint(7, 30), H=5000.0, order=min(order, 6),
                    terms=12, tol=1e-10, tl_every=tl)
    if kind == "fd":
        N = 2 ** rng.randint(6, 10) - 1
        lo, hi = _band(N)
        c = _march("", N, _log_int(rng, 1, 24), rng.randint(20, 200), 0.1 * lo, 0.3 * hi, op="fd3", order=order,
                   tl_every=tl)
    elif kind == "bc":
        q = rng.randint(6, 11)
        bc = rng.choice(["neumann", "periodic"])
        N = 2 ** q + 1 if bc == "neumann" else 2 ** (q + 1)
        lo, hi = _band(N)
        dr, order = _step_and_order(N, order)
        c = _march("", N, _log_int(rng, 1, 60), rng.randint(10, 60), lo, hi, bc=bc, dr=dr, order=order, tl_every=tl)
    else:
        q = rng.randint(6, 16)
        N = 2 ** q - 1
        lo, hi = _band(N)
        many = {16: 60, 15: 40, 14: 40, 13: 60, 12: 200}.get(q, 400)
        steps = {16: 2, 15: 4, 14: 8, 13: 16, 12: 30}.get(q, 100)
        env = rng.choice(["munk", "munk", "eddy", "absorb"])
        count = 1 if rng.random() < 0.3 else _log_int(rng, 2, many)
        dr, order = _step_and_order(N, order)
        c = _march("", N, count, rng.randint(max(1, steps // 3), steps), lo, hi, dr=dr, order=order, env=env,
                   terms=rng.choice([4, 8, 12, 12]), tl_every=tl if steps > 10 else rng.choice([0, 1]))
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------
# the problems of a case
# ------------------------------------------------------------------------------------------------
def _problems(case):
    """The solves of a case, as dicts: grid, frequency, step count and profile kind."""
    kind = case["kind"]
    if kind == "march":
        c = case["count"]
        f = [case["fmin"]] if c == 1 else [case["fmin"] + (case["fmax"] - case["fmin"]) * i / (c - 1) for i in range(c)]
        return [dict(N=case["N"], freq=x, steps=case["steps"], env=case["env"], bc=case["bc"], op=case["op"],
                     dr=case["dr"], order=case["order"]) for x in f]
    sizes = [int(n) for n in case["sizes"].split(",")]
    out = []
    for i in range(case["count"]):
        N = sizes[i % len(sizes)]
        lo, hi = _band(N)
        x = (i * 0.6180339887498949) % 1.0
        # a small grid marches more steps than a large one, no two solves equally far
        steps = max(1, int(case["steps"] * (0.5 + 0.5 * x) * (2 if N < 1024 else 1)))
        dr, order = _step_and_order(N, case["order"])
        out.append(dict(N=N, freq=lo + (hi - lo) * x, steps=steps, env="munk", bc="dirichlet", op="spectral", dr=dr,
                        order=order))
    return out


def _n2_rows(case, p):
    """(ranges, rows): the profile nodes of one solve, float64 or complex128."""
    z = inputs.depth_grid(p["N"], case["H"], p["bc"])
    if p["env"] == "iso":
        return [0.0], np.ones((1, p["N"]))
    c = inputs.munk_c(z)
    if p["env"] == "eddy":  # a node per step, the eddy inside the marched range
        dr, span = p["dr"], p["steps"] * p["dr"]
        r = [n * dr for n in range(p["steps"])]
        rows = [inputs.n2_from_c(c + inputs.gaussian_eddy_dc(x + 0.5 * dr, z, -18.0, r0=0.5 * span, Lr=0.4 * span))
                for x in r]
        return r, np.stack(rows)
    n2 = inputs.n2_from_c(c)[None]
    if p["env"] == "absorb":
        za = 0.8 * case["H"]
        n2 = n2 + 0.002j * np.clip((z - za) / (case["H"] - za), 0.0, None) ** 2
    return [0.0], n2


def _k0(p):
    return 2.0 * math.pi * p["freq"] / C0


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _fields(case, problems, seed):
    """The starters, one complex64 tensor per solve: random amplitudes on the propagating modes."""
    g = torch.Generator().manual_seed(int(seed))
    out = []
    for p in problems:
        N, bc = p["N"], p["bc"]
        top = max(3, int(math.sin(math.radians(30.0)) * _k0(p) * case["H"] / math.pi))
        M = max(2, min(top, int(0.6 * (N // 2 if bc == "periodic" else N))))
        a = torch.view_as_complex(torch.randn(M, 2, generator=g, dtype=torch.float64))
        a = (a / math.sqrt(M)).to(_dev())
        if bc == "periodic":
            s = torch.zeros(N, dtype=torch.complex128, device=a.device)
            s[1:M // 2 + 1] = a[:M // 2]
            s[N - (M - M // 2):] = a[M // 2:]
            u = torch.fft.ifft(s) * N
        elif bc == "neumann":
            K = N - 1
            s = torch.zeros(2 * K, dtype=torch.complex128, device=a.device)
            s[1:M + 1] = a
            u = (torch.fft.fft(s) + torch.fft.ifft(s) * (2 * K))[:N] * 0.5
        else:
            s = torch.zeros(2 * (N + 1), dtype=torch.complex128, device=a.device)
            s[1:M + 1] = a
            u = ((torch.fft.ifft(s) * (2 * (N + 1)) - torch.fft.fft(s)) / 2j)[1:N + 1]
        out.append(u.to(torch.complex64).contiguous())
    return out


# ------------------------------------------------------------------------------------------------
# prepare / run
# ------------------------------------------------------------------------------------------------
class _State:
    pass


def _plan(case, p):
    pl = sssp.Plan(p["N"], case["H"], _k0(p), p["dr"], p["order"], case["terms"], case["tol"], bc=p["bc"])
    pl.set_output(case["tl_every"])
    if p["op"] != "spectral":
        pl.set_operator(p["op"])
    if case["terms"] > 1 or p["op"] != "spectral":
        r, rows = _n2_rows(case, p)
        pl.set_profile_nodes(list(zip(r, rows)))
    return pl


def prepare(case, seed):
    s = _State()
    s.case = case
    if case["kind"] == "dst":
        g = torch.Generator(device=_dev()).manual_seed(int(seed))
        s.x = torch.randn(case["count"], case["N"], generator=g, dtype=torch.complex64, device=_dev())
        s.out = torch.empty_like(s.x)
        s.plan = sssp.Plan(case["N"], 5000.0, 0.4, 25.0, 4)
        return s
    s.problems = _problems(case)
    s.u0 = _fields(case, s.problems, seed)
    if case["kind"] == "serve":
        s.solves = []
        for p, u in zip(s.problems, s.u0):
            v = inputs.Solve("munk", p["N"], case["H"], p["freq"], p["dr"], p["steps"], p["order"], case["terms"],
                             case["tol"], 0.0)
            r, rows = _n2_rows(case, p)
            v.profiles = list(zip(r, rows))
            v.u0 = u.cpu().numpy()
            s.solves.append(v)
        return s
    s.plans = [_plan(case, p) for p in s.problems]
    s.steps = [p["steps"] for p in s.problems]
    # results: one field and one block of TL rows per size, the rows in pinned host memory
    s.fields, s.tl, at = {}, {}, {}
    for N in sorted({p["N"] for p in s.problems}):
        mine = [p for p in s.problems if p["N"] == N]
        s.fields[N] = torch.empty(len(mine), N, dtype=torch.complex64, device=_dev())
        rows = [p["steps"] // case["tl_every"] if case["tl_every"] else 0 for p in mine]
        s.tl[N] = torch.empty(sum(rows), N, dtype=torch.float32, pin_memory=torch.cuda.is_available())
        at[N] = [0, 0]
    s.where = []
    for p in s.problems:
        N, k = p["N"], (p["steps"] // case["tl_every"] if case["tl_every"] else 0)
        i, row = at[N]
        s.where.append((s.fields[N][i], s.tl[N][row:row + k] if k else None))
        at[N] = [i + 1, row + k]
    return s


def run(s):
    case = s.case
    if case["kind"] == "dst":
        return s.plan.dst1_batch(s.x, s.out)
    if case["kind"] == "serve":
        srv = sssp.Server(hbm_budget_bytes=20_000_000_000, max_live=512, chunk_steps=case["chunk"])
        ids = [srv.submit(v, tl_every=case["tl_every"], admit=sssp.ADMIT_MINIMAX_C0) for v in s.solves]
        live = queued = 1
        while live or queued:
            live, queued, _ = srv.step()
        got = [srv.take(i) for i in ids]
        srv.close()
        out = {}
        for v, (f, tl) in zip(s.solves, got):
            o = out.setdefault(str(v.N), {"field": [], "tl": []})
            o["field"].append(f)
            o["tl"].append(tl)
        return {n: {"field": np.stack(o["field"]), "tl": np.concatenate(o["tl"])} for n, o in out.items()}
    for pl, u in zip(s.plans, s.u0):
        pl.set_field(u)
    if len(s.plans) == 1:
        s.plans[0].march(s.steps[0])
    elif len(set(s.steps)) == 1:
        sssp.march_batch(s.plans, s.steps[0])
    else:
        sssp.march_batch_steps(s.plans, s.steps)
    for pl, (f, tl) in zip(s.plans, s.where):
        pl.read_field(f)
        if tl is not None:
            pl.read_tl(tl)
    return {str(N): {"field": s.fields[N], "tl": s.tl[N]} for N in s.fields}


# ------------------------------------------------------------------------------------------------
# work: each input read once, each output written once; the transforms of the Neumann series
# ------------------------------------------------------------------------------------------------
def work(case):
    if case["kind"] == "dst":
        L = case["N"] + 1
        return {"bytes": 16.0 * case["N"] * case["count"], "flops": case["count"] * 5.0 * L * math.log2(L)}
    b = fl = 0.0
    for p in _problems(case):
        N, steps = p["N"], p["steps"]
        L = 2 * (N - 1) if p["bc"] == "neumann" else (N if p["bc"] == "periodic" else N + 1)
        rows = steps // case["tl_every"] if case["tl_every"] else 0
        nodes = steps if p["env"] == "eddy" else 1
        b += 16.0 * N + 4.0 * N * rows + 4.0 * N * nodes * (2 if p["env"] == "absorb" else 1) + 32.0 * L * p["order"]
        if p["op"] == "fd3":  # per stage: right-hand side, two sweeps, multiply-add of complex values
            fl += steps * p["order"] * N * 40.0
            continue
        # a stage of c terms takes 2 c - 2 transforms; the stop rule ends most series at about
        # three quarters of the cap (99 of 133 transforms a step on the Munk workload)
        c = max(2.0, 0.8 * case["terms"])
        t = rows + 1 + (steps * p["order"] * (2.0 * c - 2.0) if case["terms"] > 1 else 0.0)
        fl += t * (5.0 * L * math.log2(L) + 10.0 * L) + (steps * L * 16.0 if case["terms"] <= 1 else 0.0)
    return {"bytes": b, "flops": fl}


# ------------------------------------------------------------------------------------------------
# the same in 64 bits
# ------------------------------------------------------------------------------------------------
def _pade(sigma, p):
    """(b, a): [p/p] Pade factors of exp(i sigma (sqrt(1 + X) - 1)) at X = 0 (Baker's system)."""
    s = [1.0]
    for k in range(1, 2 * p + 1):
        s.append(s[-1] * (-0.5 - (k - 1)) / k)  # (1 + X)^(-1/2)
    g = [1.0 + 0j]
    for n in range(2 * p):  # g' = (i sigma/2) (1 + X)^(-1/2) g
        g.append(0.5j * sigma * sum(s[k] * g[n - k] for k in range(n + 1)) / (n + 1))
    A = np.array([[g[p + i - j] if p + i - j >= 0 else 0.0 for j in range(1, p + 1)] for i in range(1, p + 1)])
    q = np.concatenate([[1.0], np.linalg.solve(A, -np.array([g[p + i] for i in range(1, p + 1)]))])
    b = -1.0 / np.roots(q[::-1])
    b = b[np.argsort(b.real)]
    return b, np.conj(b)


def _to_spec(x, bc):
    if bc == "periodic":
        return torch.fft.fft(x)
    L = x.shape[1] + 1
    z = torch.zeros(x.shape[0], 2 * L, dtype=torch.complex128, device=x.device)
    z[:, 1:L] = x
    z[:, L + 1:] = -x.flip(1)
    return 0.5j * torch.fft.fft(z)[:, 1:L]


def _to_depth(X, bc):
    return torch.fft.ifft(X) if bc == "periodic" else _to_spec(X, bc) * (2.0 / (X.shape[1] + 1))


def _exact_march(case, u0, k0s, rows, ranges, steps, dr, order, bc):
    """(fields, TL rows) of solves of one size and step count: u0 (B, N), rows (B, nodes, N)."""
    dev = _dev()
    H, N = case["H"], u0.shape[1]
    if bc == "neumann":  # the even extension to [0, 2H], periodic
        u0 = torch.cat([u0, u0[:, 1:-1].flip(1)], 1)
        rows = torch.cat([rows, rows[:, :, 1:-1].flip(2)], 2)
        H, bc = 2.0 * H, "periodic"
    n = u0.shape[1]
    k0 = torch.tensor(k0s, dtype=torch.float64, device=dev)[:, None]
    if bc == "periodic":
        m = torch.arange(n, dtype=torch.float64, device=dev)
        kz = 2.0 * math.pi * torch.where(m <= n // 2, m, m - n) / H
    else:
        kz = math.pi * torch.arange(1, n + 1, dtype=torch.float64, device=dev) / H
    lam = -(kz[None] / k0) ** 2
    ab = [_pade(k * dr, order) for k in k0s]
    b = torch.tensor(np.array([x[0] for x in ab]), device=dev)
    a = torch.tensor(np.array([x[1] for x in ab]), device=dev)
    U = _to_spec(u0.to(torch.complex128), bc)
    tl = []
    for s in range(steps):
        if case["terms"] <= 1:
            for j in range(order):
                U = U * (1.0 + a[:, j:j + 1] * lam) / (1.0 + b[:, j:j + 1] * lam)
        else:
            mid, node = (s + 0.5) * dr, 0
            while node + 1 < len(ranges) and ranges[node + 1] <= mid:
                node += 1
            V = rows[:, node] - 1.0
            for j in range(order):
                bj, aj = b[:, j:j + 1], a[:, j:j + 1]
                inv = 1.0 / (1.0 + bj * lam)
                t = inv * U
                w = t.clone()
                on = torch.ones(len(k0s), 1, dtype=torch.bool, device=dev)
                for m in range(1, case["terms"]):
                    t = -bj * inv * _to_spec(V * _to_depth(t, bc), bc)
                    w = torch.where(on, w + t, w)
                    if m == case["terms"] - 1:
                        break
                    nt, nw = t.abs().square().sum(1, True), w.abs().square().sum(1, True)
                    on = on & ~(nt <= case["tol"] ** 2 * nw)
                    if not bool(on.any()):
                        break
                U = (aj / bj) * U + (1.0 - aj / bj) * w
        if case["tl_every"] and (s + 1) % case["tl_every"] == 0:
            u = _to_depth(U, bc)[:, :N]
            tl.append(-20.0 * torch.log10(u.abs()) + 10.0 * math.log10((s + 1) * dr))
    u = _to_depth(U, bc)[:, :N] * torch.exp(1j * k0 * steps * dr)
    return u, torch.stack(tl, 1) if tl else torch.empty(len(k0s), 0, N, dtype=torch.float64, device=dev)


def _exact_fd(case, u0, k0s, rows, steps, dr, order):
    """The three-point operator by its eigenvectors: u_n = Q R(x)^n Q^T u_0."""
    dev, N = _dev(), u0.shape[1]
    h = case["H"] / (N + 1)
    fields, tls = [], []
    for i, k in enumerate(k0s):
        X = torch.diag(rows[i, 0].real - 1.0 - 2.0 / (k * h) ** 2)
        off = torch.full((N - 1,), 1.0 / (k * h) ** 2, dtype=torch.float64, device=dev)
        x, Q = torch.linalg.eigh(X + torch.diag(off, 1) + torch.diag(off, -1))
        b, a = _pade(k * dr, order)
        R = torch.ones(N, dtype=torch.complex128, device=dev)
        for j in range(order):
            R = R * (1.0 + a[j] * x) / (1.0 + b[j] * x)
        Q = Q.to(torch.complex128)
        c, tl = Q.T @ u0[i].to(torch.complex128), []
        for s in range(steps):
            c = c * R
            if case["tl_every"] and (s + 1) % case["tl_every"] == 0:
                tl.append(-20.0 * torch.log10((Q @ c).abs()) + 10.0 * math.log10((s + 1) * dr))
        fields.append((Q @ c) * np.exp(1j * k * steps * dr))
        tls.append(torch.stack(tl) if tl else torch.empty(0, N, dtype=torch.float64, device=dev))
    return torch.stack(fields), torch.stack(tls)


def exact(case, seed):
    dev = _dev()
    if case["kind"] == "dst":
        g = torch.Generator(device=dev).manual_seed(int(seed))
        x = torch.randn(case["count"], case["N"], generator=g, dtype=torch.complex64, device=dev)
        return _to_spec(x.to(torch.complex128), "dirichlet")
    problems = _problems(case)
    u0 = _fields(case, problems, seed)
    groups = {}
    for i, p in enumerate(problems):
        groups.setdefault((p["N"], p["steps"]), []).append(i)
    field, tl = [None] * len(problems), [None] * len(problems)
    for (N, steps), ids in groups.items():
        most = max(1, (1 << 24) // (N + 1))
        for at in range(0, len(ids), most):
            part = ids[at:at + most]
            p0 = problems[part[0]]
            k0s = [_k0(problems[i]) for i in part]
            ranges, n2 = _n2_rows(case, p0)  # the profile does not depend on the frequency
            rows = torch.from_numpy(np.ascontiguousarray(n2)).to(dev)[None].expand(len(part), -1, -1)
            scale = 1.0
            if case["kind"] == "serve":  # the minimax reference sound speed of the admission
                scale = 2.0 / (n2.real.min() + n2.real.max())
                rows, k0s = rows * scale, [k / math.sqrt(scale) for k in k0s]
            u = torch.stack([u0[i] for i in part])
            if p0["op"] == "fd3":
                f, t = _exact_fd(case, u, k0s, rows, steps, p0["dr"], p0["order"])
            else:
                f, t = _exact_march(case, u, k0s, rows, ranges, steps, p0["dr"], p0["order"], p0["bc"])
            for k, i in enumerate(part):
                field[i], tl[i] = f[k], t[k]
    out = {}
    for N in sorted({p["N"] for p in problems}):
        ids = [i for i, p in enumerate(problems) if p["N"] == N]
        out[str(N)] = {"field": torch.stack([field[i] for i in ids]), "tl": torch.cat([tl[i] for i in ids])}
    return out

"""The work this framework does for its users, as timed cases.

Each case is one call sequence a user's program makes on fiber-network RVEs:
damped dynamic relaxation of one network, of a batch, of an FE2 macro step, of
a stream of serving requests. The networks are the synthetic stand-ins the
benchmark uses (uniform nodes in the unit cube, 4 nearest neighbours, a fixed
boundary band of 0.05, lognormal or unit rigidities, F = I + 0.02 sym N(0,1)).
Full solves take 2e4 to 1e6 iterations; the cases bound them (`iters`), as the
benchmark's experiment shapes do, with the double-float lead at a tenth of the
iterations (about its share of a full mixed solve) unless `lead` is -1, the
default rule.
"""
import math

import numpy as np
import torch

import paper_2305_07030_gb300 as fe2

_DEV = "cuda" if torch.cuda.is_available() else "cpu"
_STATUS = {v: k for k, v in fe2.RVE_STATUS.items()}
_BASE = {"call": "device", "precision": "mixed", "count": 1, "lo": 512, "hi": 512, "ea": "lognormal",
         "iters": 2000, "lead": 0, "tol": 0.0, "init": "affine", "energy": 0}


def _case(name=None, **kw):
    c = dict(_BASE, **kw)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # one 512-node network (unit rigidities) solved to tol 1e-8 from host arrays: the
        # smallest whole solve, bound by the latency of an iteration
        _case("solve512_mixed", call="host", ea="unit", iters=100000, lead=-1, tol=1e-8),
        # a few tiny networks for a few iterations: launches and host work count
        _case("tiny_mixed", call="host", count=8, lo=37, hi=200, iters=100, lead=-1, tol=1e-8),
        # one FE2 macro step: 64 Gauss points of a 2 x 2 x 2 hex mesh, an affine solve of the
        # last state's F, then a warm restart at the next F, stresses read back after each
        _case("fe2_step_mixed", call="step", count=64, lo=300, hi=900, iters=1000, lead=-1, tol=1e-8),
        # the benchmark's batch: 64 networks of 5000 nodes
        _case("rve5000x64_mixed", count=64, lo=5000, hi=5000, iters=4000),
        # many networks of one cluster CTA each
        _case("rve1000x256_mixed", count=256, lo=1000, hi=1000, iters=2000),
        # uneven batch, 1k to 33k nodes: several launch classes at once
        _case("uneven1k33k_mixed", count=24, lo=1000, hi=33000, iters=2000),
        # large networks: the biggest clusters, kinetic energy tracked
        _case("rve20000x8_mixed", count=8, lo=20000, hi=20000, iters=1000, energy=1),
        # serving: micro-batches submitted as they come and polled until all are back
        _case("serve_mixed", call="serve", count=32, lo=1000, hi=8000, iters=1000, lead=-1, tol=1e-8),
        # the bit-exact FP64 mode: one small network, the field read back
        _case("rve512_fp64", call="host", precision="fp64", ea="unit", iters=1000),
        # FP64 batch of small networks (one CTA each) with the energy balance
        _case("small200x300_fp64", call="host", precision="fp64", count=300, lo=200, hi=1000, iters=200,
              energy=2),
        # FP64 batch of 5000-node networks on thread-block clusters
        _case("rve5000x32_fp64", precision="fp64", count=32, lo=5000, hi=5000, iters=300),
        # the allocation-free call on a caller's own device buffers
        _case("noalloc700_fp64", call="noalloc", precision="fp64", lo=700, hi=700, iters=500),
    ]


def draw(rng):
    """A case of the same ranges; node-iterations bounded by the largest listed one's time."""
    def logu(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["device", "device", "host", "step", "serve", "fp64", "fp64", "noalloc"])
    if kind == "noalloc":
        n = logu(40, 4000)
        return _case(call="noalloc", precision="fp64", lo=n, hi=n, ea=rng.choice(["unit", "lognormal"]),
                     iters=min(logu(50, 2000), 400000 // n + 20))
    if kind == "fp64":
        lo = logu(37, 12000)
        hi = max(lo, min(20000, int(lo * rng.uniform(1.0, 4.0))))
        count = min(logu(1, 300), 320000 // hi + 1)
        # from u = 0 the transient amplifies rounding: a few iterations only
        init = rng.choice(["affine", "affine", "reference"])
        return _case(call=rng.choice(["device", "host"]), precision="fp64", count=count, lo=lo, hi=hi,
                     iters=min(logu(20, 1000 if init == "affine" else 100), 40000000 // (count * hi) + 20,
                               2000000 // hi + 20),
                     energy=rng.choice([0, 1, 2]), init=init)
    lo = logu(37, 20000) if kind != "serve" else logu(300, 8000)
    hi = max(lo, min(33000, int(lo * rng.uniform(1.0, 6.0))))
    count = max(2, min(logu(1, 256), 320000 // hi + 1))
    iters = min(logu(50, 4000), 600000000 // (count * hi) + 50, 20000000 // hi + 50)
    return _case(call=kind, count=count, lo=lo, hi=hi, iters=iters, ea=rng.choice(["unit", "lognormal"]),
                 lead=rng.choice([0, 0, -1]), tol=rng.choice([0.0, 1e-8]), energy=rng.choice([0, 0, 1]))


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------

class _Net:
    def __init__(self, X, elems, EA, fixed):
        self.X, self.elems, self.EA, self.fixed, self.V0 = X, elems, EA, fixed, 1.0


def _sizes(case):
    """Node counts: the midpoints of `count` equal strata of log-U(lo, hi)."""
    k, lo, hi = case["count"], case["lo"], case["hi"]
    return [int(round(lo * (hi / lo) ** ((i + 0.5) / k))) for i in range(k)]


def _edges(X):
    """Undirected 4-nearest-neighbour edges, a < b, in lexicographic order."""
    n = X.shape[0]
    Xd = torch.as_tensor(X, device=_DEV)
    near = []
    for s in range(0, n, 4096):
        d2 = ((Xd[s:s + 4096, None, 0] - Xd[None, :, 0]) ** 2 + (Xd[s:s + 4096, None, 1] - Xd[None, :, 1]) ** 2
              + (Xd[s:s + 4096, None, 2] - Xd[None, :, 2]) ** 2)
        near.append(d2.topk(5, dim=1, largest=False).indices)
    near = torch.cat(near)
    i = torch.arange(n, device=near.device)[:, None].expand(n, 5)
    keep = near != i
    lo, hi = torch.minimum(i, near)[keep], torch.maximum(i, near)[keep]
    key = torch.unique(lo * n + hi).cpu().numpy()
    return np.stack([key // n, key % n], axis=1).astype(np.int32)


def _inputs(case, seed):
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    nets, F, F2 = [], [], []
    for n in _sizes(case):
        X = rng.random((n, 3))
        elems = _edges(X)
        EA = np.ones(len(elems)) if case["ea"] == "unit" else rng.lognormal(0.0, 0.3, len(elems))
        fixed = (np.minimum(X, 1.0 - X).min(axis=1) <= 0.05).astype(np.uint8)
        nets.append(_Net(X, elems, EA, fixed))
        G = rng.standard_normal((3, 3))
        F.append(np.eye(3) + 0.01 * (G + G.T))
        F2.append(np.diag([1.005, 1.0, 1.0]) @ F[-1])
    return nets, np.array(F), np.array(F2)


def _opts(case):
    o = dict(precision=case["precision"], tol=case["tol"], max_iter=case["iters"], init=case["init"],
             kinetic_energy="balance" if case["energy"] == 2 else bool(case["energy"]))
    if case["precision"] == "mixed" and case["lead"] >= 0:
        o["lead_iters"] = max(1, case["iters"] // 10)
    return o


# ----------------------------------------------------------------------------
# the calls
# ----------------------------------------------------------------------------

def prepare(case, seed):
    nets, F, F2 = _inputs(case, seed)
    s = {"call": case["call"], "opts": _opts(case), "F": F, "F2": F2, "energy": case["energy"] == 2,
         "field": case["call"] == "host"}
    if case["call"] == "noalloc":
        net = nets[0]

        def dev(a):
            return torch.as_tensor(np.ascontiguousarray(a), device="cuda")

        s.update(n=len(net.X), E=len(net.elems),
                 inputs=[dev(net.X), dev(net.elems), dev(net.EA), dev(net.fixed), dev(F[0])],
                 u=torch.zeros(len(net.X), 3, dtype=torch.float64, device="cuda"),
                 out=[torch.zeros(3, 3, dtype=torch.float64, device="cuda"),
                      torch.zeros(1, dtype=torch.int64, device="cuda"),
                      torch.zeros(1, dtype=torch.float64, device="cuda"),
                      torch.zeros(1, dtype=torch.int32, device="cuda")])
        return s
    s["batch"] = fe2.Batch(nets)
    P = len(nets)
    if case["call"] == "device":
        s["F_dev"] = torch.as_tensor(F.reshape(-1), device="cuda")
        s["out"] = [torch.zeros(P, 3, 3, dtype=torch.float64, device="cuda"),
                    torch.zeros(P, dtype=torch.int64, device="cuda"),
                    torch.zeros(P, dtype=torch.float64, device="cuda"),
                    torch.zeros(P, dtype=torch.int32, device="cuda")]
    if case["call"] == "serve":
        # micro-batches of up to 8 requests, strided over the sizes
        k = max(1, -(-P // 8))
        s["micro"] = [np.arange(j, P, k, dtype=np.int32) for j in range(k)]
    return s


def _plain(r):
    return [r["sigma"], r["iters"], r["rel_res"], np.array([_STATUS[x] for x in r["status"]], np.int32)]


def run(s):
    o = s["opts"]
    if s["call"] == "noalloc":
        sig, it, rel, st = s["out"]
        fe2.rve_solve_noalloc(s["n"], s["E"], *s["inputs"], s["u"], sig, it, rel, st,
                              stream=torch.cuda.current_stream(), **o)
        return [sig, it, rel, st, s["u"]]
    b = s["batch"]
    if s["call"] == "device":
        st = torch.cuda.current_stream()
        b.solve_dev(s["F_dev"], stream=st, **o)
        sig, it, rel, code = s["out"]
        b.results_dev(sigma_dev=sig, iters_dev=it, rel_dev=rel, status_dev=code, stream=st)
        return s["out"]
    if s["call"] == "host":
        b.solve(s["F"], **o)
        out = _plain(b.stress())
        if s["energy"]:
            e = b.energy()
            out += [e["kinetic"], e["internal_work"], e["external_work"]]
        return out + [b.displacement()]
    if s["call"] == "step":
        b.solve(s["F"], **o)
        first = _plain(b.stress())
        b.solve(s["F2"], **dict(o, init="warm"))
        return first + _plain(b.stress())
    # serving loop: submit while slots are free, poll until every request is back
    P = len(s["F"])
    out = [np.zeros((P, 3, 3)), np.zeros(P, np.int64), np.zeros(P), np.zeros(P, np.int32)]
    todo, back = list(s["micro"]), 0
    while back < P:
        while todo and b.submit(todo[0], s["F"][todo[0]], **o) is not None:
            todo.pop(0)
        r = b.poll()
        back += len(r["ids"])
        for a, v in zip(out, _plain(r)):
            a[r["ids"]] = v
    return out


def work(case):
    """Operations of the relaxation itself (per element and iteration 13 add / multiply, 2
    divisions, a square root and the two nodal sums; per node 40), each input read once and
    each result written once. About 2.5 elements per node; 6e4 iterations for a whole solve."""
    n = sum(_sizes(case))
    it = case["iters"] if case["iters"] < 50000 else 60000
    passes = 2 if case["call"] == "step" else 1
    return {"bytes": passes * (n * (24 + 1 + 24) + 2.5 * n * 16.0 + 160 * case["count"]),
            "flops": passes * it * n * (2.5 * 22 + 40.0)}


# ----------------------------------------------------------------------------
# the same relaxation in plain 64-bit torch
# ----------------------------------------------------------------------------

class _Relax64:
    def __init__(self, nets):
        t = dict(dtype=torch.float64, device=_DEV)
        off = np.concatenate([[0], np.cumsum([len(n.X) for n in nets])])
        self.P, self.off = len(nets), off
        self.X = torch.as_tensor(np.concatenate([n.X for n in nets]), **t)
        el = np.concatenate([n.elems.astype(np.int64) + o for n, o in zip(nets, off)])
        N, E = len(self.X), len(el)
        self.a, self.b = (torch.as_tensor(el[:, k], device=_DEV) for k in (0, 1))
        self.EA = torch.as_tensor(np.concatenate([n.EA for n in nets]), **t)
        self.rve = torch.as_tensor(np.repeat(np.arange(self.P), np.diff(off)), device=_DEV)
        self.erve = self.rve[self.a]
        d = self.X[self.b] - self.X[self.a]
        self.L = (d * d).sum(1).sqrt()
        deg = np.bincount(el.reshape(-1), minlength=N)
        # each node's elements, padded to the longest row with a zero force
        ends = np.concatenate([el[:, 0], el[:, 1]])
        order = np.argsort(ends, kind="stable")
        start = np.concatenate([[0], np.cumsum(deg)])
        rows = np.full((N, max(1, deg.max(initial=0))), 2 * E)
        rows[ends[order], np.arange(2 * E) - start[ends[order]]] = order
        self.rows = torch.as_tensor(rows, device=_DEV)
        half = self.EA / self.L / 2  # half an element's mass, rho A L / 2 with rho A = EA / L^2
        self.m = torch.zeros(N, **t).index_add_(0, self.a, half).index_add_(0, self.b, half)
        fixed = np.concatenate([n.fixed for n in nets]) != 0
        self.free = torch.as_tensor((~fixed & (deg > 0)).astype(np.float64)[:, None], device=_DEV)
        self.minv = self.free / torch.where(self.m > 0, self.m, torch.ones_like(self.m))[:, None]
        # critical step: min over elements of L sqrt(rho A / EA)
        dt = torch.full((self.P,), math.inf, **t)
        dt.scatter_reduce_(0, self.erve, self.L * (1 / self.L ** 2).sqrt(), "amin")
        self.dt = 0.9 * dt[self.rve][:, None]
        c = 0.002 * (512.0 / np.diff(off)) ** (1.0 / 3.0)
        self.c = torch.as_tensor(c, device=_DEV)[self.rve][:, None]

    def force(self, u):
        x = self.X + u
        d = x[self.b] - x[self.a]
        l = (d * d).sum(1).sqrt()
        self.q, self.d = self.EA * (l / self.L - 1) / l, d
        f = self.q[:, None] * d
        return torch.cat([f, -f, f.new_zeros(1, 3)])[self.rows].sum(1)

    def per_rve(self, v, rve=None):
        return torch.zeros((self.P,) + v.shape[1:], dtype=v.dtype, device=v.device).index_add_(
            0, self.rve if rve is None else rve, v)

    def solve(self, F, tol, max_iter, init, warm=None):
        Fd = torch.as_tensor(F, device=_DEV)
        uaff = torch.einsum("nij,nj->ni", Fd[self.rve], self.X) - self.X
        u = uaff.clone() if init == "affine" else uaff * (1 - self.free) + (0 if warm is None else warm * self.free)
        fa = self.per_rve((self.force(uaff) ** 2).sum(1)).sqrt()
        g = self.force(u)
        fref = torch.maximum(fa, self.per_rve((g ** 2).sum(1)).sqrt())
        a, v, fd = g * self.minv, torch.zeros_like(u), torch.zeros_like(u)
        w = torch.zeros(self.P, 2, dtype=torch.float64, device=_DEV)
        res, its = torch.zeros_like(fref), torch.zeros(self.P, dtype=torch.int64, device=_DEV)
        done, u_end, k_end, w_end = its > 0, u.clone(), torch.zeros_like(fref), w.clone()
        sig = torch.zeros(self.P, 3, 3, dtype=torch.float64, device=_DEV)

        def step():
            v.add_(self.dt / 2 * a)
            du = self.dt * v * self.free
            u.add_(du)
            gn = self.force(u)
            fn = -self.c * self.m[:, None] * v * self.free
            w.add_(torch.stack([-self.per_rve((du * (g + gn)).sum(1)) / 2, self.per_rve((du * (fd + fn)).sum(1)) / 2], 1))
            g.copy_(gn)
            fd.copy_(fn)
            a.copy_((g + fd) * self.minv)
            v.add_(self.dt / 2 * a)
            r = self.per_rve(((g * self.free) ** 2).sum(1)).sqrt()
            s = self.per_rve((self.q[:, None, None] * self.d[:, :, None] * self.d[:, None, :]), self.erve)
            live = ~done
            its.add_(live.to(torch.int64))
            res.copy_(torch.where(live, r, res))
            sig.copy_(torch.where(live[:, None, None], s, sig))
            u_end.copy_(torch.where(live[self.rve][:, None], u, u_end))
            k_end.copy_(torch.where(live, self.per_rve(self.m * (v ** 2 * self.free).sum(1)) / 2, k_end))
            w_end.copy_(torch.where(live[:, None], w, w_end))
            done.logical_or_(r <= tol * fref)

        todo = max_iter
        if _DEV == "cuda" and max_iter > 50:
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                for _ in range(3):
                    step()
            torch.cuda.current_stream().wait_stream(side)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                step()
            todo -= 3
            for k in range(todo):
                graph.replay()
                if k % 500 == 499 and bool(done.all()):
                    break
        else:
            for _ in range(todo):
                step()
        V = torch.linalg.det(Fd)
        zero = fref > 0
        rel = torch.where(zero, res / torch.where(zero, fref, torch.ones_like(fref)), res)
        return sig / V[:, None, None], rel, u_end, [k_end, w_end[:, 0], w_end[:, 1]]


def exact(case, seed):
    nets, F, F2 = _inputs(case, seed)
    R = _Relax64(nets)
    sig, rel, u, energy = R.solve(F, case["tol"], case["iters"], case["init"])
    if case["call"] == "noalloc":
        return [sig[0], None, rel, None, u]
    out = [sig, None, rel, None]
    if case["call"] == "host":
        return out + (energy if case["energy"] == 2 else []) + [u]
    if case["call"] == "step":
        sig, rel, _, _ = R.solve(F2, case["tol"], case["iters"], "warm", u)
        return out + [sig, None, rel, None]
    return out

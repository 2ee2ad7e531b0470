"""What the PRIEST library is asked to do by the programs that use it: one case
per way of calling it, each through the C ABI as the binding exposes it.

  projections  the batched projection of caller-given samples (Sec. III-A):
               device buffers (priest_project_device), many problems at once
               (priest_project_batch), the allocation-free form
               (priest_project_noalloc)
  solves       Alg. 1 whole: device buffers (priest_plan_device), host buffers
               (priest_plan_z), a batch of uneven problems through host buffers
               (priest_plan_batch_host), a burst of requests to the serving
               loop (priest_submit / priest_wait)

Scenes, sample counts and iteration counts are those of the workloads module,
the tests and the benchmark, or lie between them.  The FP32 mode's results
carry FP32 precision in FP64 buffers; the program keeps them as float32.
"""
import math

import numpy as np
import torch

from paper_2309_08235_gb300 import priest as P
from paper_2309_08235_gb300 import workloads as W

FP64, FP32, MIXED = P.PRIEST_FP64_CHECK, P.PRIEST_FP32, P.PRIEST_MIXED_BF16
NV = W.DEGREE + 1


# ---- the cases ----------------------------------------------------------------

def _project(**k):
    c = {"call": "project", "scene": "clutter", "n_static": 90, "n_dyn": 10, "n_p": 100, "horizon": 8.0, "N": 1000,
         "K": 100, "precision": FP32, "warm": False, "bounds": False, "mask": 7}
    c.update(k)
    return c


def _solve(**k):
    c = {"call": "solve", "scene": "p2p2d", "n_static": 50, "n_dyn": 0, "n_p": 100, "horizon": 8.0, "N": 110, "K": 50,
         "L": 13, "n_elite": 20, "n_proj": 80, "precision": FP32, "host": False, "bounds": False, "mask": 7}
    c.update(k)
    return c


def listed():
    return [
        # a real-time loop's call: a few samples, coarse time stamps, no device
        # allocation; latency is all that counts
        _project(name="noalloc_loop", call="noalloc", scene="small", n_static=8, n_dyn=0, n_p=50, horizon=5.0, N=32,
                 K=20),
        # a replan at the paper's sample count with the multipliers of the plan before
        _project(name="project_replan", scene="p2p2d", n_static=50, n_dyn=0, N=110, K=50, warm=True),
        # the 2-D clutter scene of the benchmark, one CEM iteration's projection
        _project(name="project_clutter"),
        # odd sizes everywhere, a dense scene with moving obstacles, warm multipliers
        _project(name="project_ragged", n_static=333, n_dyn=38, n_p=77, horizon=6.16, N=777, K=45, warm=True),
        # the 3-D ellipsoid scene of the benchmark in its mixed precision mode
        _project(name="project_ellipsoids", scene="ellipsoids", n_static=200, n_dyn=0, n_p=150, horizon=10.0, N=2000,
                 precision=MIXED),
        # workspace rows and the paper's four boundary rows per axis (seven free coefficients)
        _project(name="project_bounds", bounds=True, mask=1),
        # the FP64 mode on the small 2-D scene: results checked against a reference
        _project(name="project_fp64", scene="small", n_static=20, n_dyn=0, horizon=5.0, N=200, K=50, precision=FP64),
        # many robots' samples projected together: uneven problems, one launch
        {"name": "project_batch", "call": "project_batch", "n": 64, "mix": 11, "K": 60},
        # one robot's plan at the paper's settings (110 samples, 13 CEM iterations), device buffers
        _solve(name="solve_p2p2d"),
        # the 2-D clutter solve of the benchmark through host buffers, result read back
        _solve(name="solve_clutter_host", scene="clutter", n_static=90, n_dyn=10, N=1000, K=100, L=5, n_elite=100,
               n_proj=727, host=True),
        # the benchmark's headline: 256 uneven problems end to end through host buffers
        {"name": "solve_batch_host", "call": "solve_batch", "n": 256, "mix": 1, "K": 60, "L": 3},
        # a burst of requests of mixed sizes (2-D and 3-D) to the serving loop
        {"name": "serve_burst", "call": "serve", "n": 32, "mix": 3, "K": 60, "L": 3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over the ranges the listed ones span."""
    call = rng.choice(["noalloc", "project", "project", "project", "solve", "solve", "project_batch", "solve_batch",
                       "serve"])
    if call in ("project_batch", "solve_batch", "serve"):
        c = {"call": call, "n": _log_int(rng, 2, 96 if call != "serve" else 24), "mix": rng.randrange(1 << 20),
             "K": _log_int(rng, 20, 60)}
        if call != "project_batch":
            c["L"] = rng.randrange(2, 4)
        return c
    scene = rng.choice(["clutter", "clutter", "p2p2d", "ellipsoids", "p2p3d", "dynamic", "small"])
    n_obs = _log_int(rng, 10, 400) if scene in ("clutter", "ellipsoids") else _log_int(rng, 8, 60)
    n_dyn = n_obs // 10 if scene == "clutter" else n_obs if scene == "dynamic" else 0
    n_p = rng.randrange(64, 161) if scene in ("ellipsoids", "p2p3d") else rng.randrange(40, 161)
    k = {"scene": scene, "n_static": n_obs - n_dyn, "n_dyn": n_dyn, "n_p": n_p, "horizon": round(0.08 * n_p, 2)}
    if call == "solve":
        N = _log_int(rng, 64, 2048)
        k.update(N=N, K=_log_int(rng, 20, 100), L=rng.randrange(2, 9), n_elite=max(1, N // 10),
                 n_proj=max(1, 80 * N // 110), host=rng.random() < 0.4)
        return _solve(**k)
    if call == "noalloc":
        return _project(call="noalloc", **dict(k, N=_log_int(rng, 16, 256), K=_log_int(rng, 10, 60)))
    k.update(N=_log_int(rng, 16, 2048), K=_log_int(rng, 20, 100), warm=rng.random() < 0.4)
    p = rng.random()
    if scene == "clutter" and p < 0.2:
        k.update(bounds=True, mask=1)
    elif p < 0.3:
        k.update(precision=MIXED)
    elif p < 0.4:
        k.update(precision=FP64, N=min(k["N"], 256), K=min(k["K"], 50))
    return _project(**k)


# ---- inputs -------------------------------------------------------------------

def _scene(c, seed):
    s, ns, nd = c["scene"], c["n_static"], c["n_dyn"]
    if s == "clutter":
        p = W.scene_clutter_2d(seed=seed, n_static=ns, n_dyn=nd, n_p=c["n_p"], horizon=c["horizon"])
    elif s == "ellipsoids":
        p = W.scene_ellipsoids_3d(seed=seed, n_obs=ns, n_p=c["n_p"], horizon=c["horizon"])
    elif s == "p2p2d":
        p = W.scene_p2p_2d(seed=seed, n_obs=ns, n_p=c["n_p"], horizon=c["horizon"])
    elif s == "p2p3d":
        p = W.scene_p2p_3d(seed=seed, n_obs=ns, n_p=c["n_p"], horizon=c["horizon"])
    elif s == "dynamic":
        p = W.scene_dynamic_2d(seed=seed, n_obs=nd, n_p=c["n_p"], horizon=c["horizon"])
    else:
        p = W.scene_small_2d(seed=seed, n_obs=ns, n_p=c["n_p"], horizon=c["horizon"])
    if c["bounds"]:
        p.update(use_bounds=True, smin=np.zeros(2), smax=np.full(2, 30.0))
    p["bc_final_mask"] = c["mask"]
    return p


def _cem(c, dims):
    return W.cem_settings(c.get("N", 256), c["K"], c.get("L", 1), n_proj=c.get("n_proj"), n_elite=c.get("n_elite"),
                          dims=dims)


def _mix(c):
    """The sizes of a batch or burst: (dims, n_obs, N, n_p) per problem, the
    benchmark's ranges; fixed by the case, not by the seed."""
    rng = np.random.default_rng(10_000 + c["mix"])
    out = []
    for _ in range(c["n"]):
        n_obs = int(round(math.exp(rng.uniform(math.log(10), math.log(400)))))
        N = int(rng.choice([256, 512, 1024, 2048]))
        n_p = int(rng.choice([60, 100, 150]))
        d3 = c["call"] == "serve" and rng.random() < 0.2
        out.append((3 if d3 else 2, n_obs, N, n_p))
    return out


def _mix_problems(c, seed):
    out = []
    for k, (dims, n_obs, N, n_p) in enumerate(_mix(c)):
        s = (seed * 1009 + k) & 0x7FFFFFFF
        if dims == 3:
            p = W.scene_ellipsoids_3d(seed=s, n_obs=n_obs, n_p=n_p, horizon=0.08 * n_p)
        else:
            nd = n_obs // 10
            p = W.scene_clutter_2d(seed=s, n_static=n_obs - nd, n_dyn=nd, n_p=n_p, horizon=0.08 * n_p)
        out.append((p, N))
    return out


def _mean(p):
    """Straight-line coefficients: the mean that samples are drawn around."""
    b0, bf = np.asarray(p["b0"])[:, 0], np.asarray(p["bf"])[:, 0]
    return np.concatenate([np.linspace(b0[a], bf[a], NV) for a in range(p["dims"])])


def _normals(seed, *shape):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _samples(p, N, seed):
    std = W.INIT_STD_2D if p["dims"] == 2 else W.INIT_STD_3D
    return torch.as_tensor(_mean(p), device="cuda") + std * _normals(seed, N, p["dims"] * NV)


_stream = None


def stream():
    """The program's one CUDA stream, which its contexts run on."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


class State:
    """Context, loaded problems and buffers of one program."""

    def __init__(self, case):
        self.case, self.ctx, self.handles = case, None, []

    def context(self, p, cem, precision=FP32, **over):
        self.ctx = P.Context(p, cem, precision=precision, stream=stream().cuda_stream, **over)
        return self.ctx.h

    def load(self, p, cem=None):
        s, _keep = P.make_problem(p, cem, per_problem_shape=cem is not None)
        h = P.priest_load(self.ctx.h, s)
        self.handles.append(h)
        return h

    def __del__(self):
        if self.ctx is not None and self.ctx.h:
            for h in self.handles:
                P.priest_unload(self.ctx.h, h)
            self.ctx.close()


def prepare(case, seed):
    st = State(case)
    call = case["call"]
    if call in ("noalloc", "project"):
        p = _scene(case, seed)
        D, N = p["dims"] * NV, case["N"]
        st.xi = _samples(p, N, seed)
        st.lam0 = 0.05 * _normals(seed + 1, N, D) if case["warm"] else None
        st.lam = torch.empty_like(st.xi) if case["warm"] else None
        st.xb = torch.empty_like(st.xi)
        st.score = torch.empty(2, N, device="cuda", dtype=torch.float64)  # r, c_1
        st.ptrs = (st.xi.data_ptr(), st.lam.data_ptr() if case["warm"] else 0, st.xb.data_ptr(),
                   st.score[0].data_ptr(), st.score[1].data_ptr())
        if call == "noalloc":
            st.cfg = P.make_config(p, _cem(case, p["dims"]), case["precision"])
            st.prob, st.keep = P.make_problem(p)
        else:
            st.context(p, _cem(case, p["dims"]), case["precision"])
            st.h = st.load(p)
    elif call == "solve":
        p = _scene(case, seed)
        cem = _cem(case, p["dims"])
        st.context(p, cem, case["precision"])
        z = _normals(seed, case["L"], case["N"], p["dims"] * NV)
        if case["host"]:
            st.z = z.cpu().pin_memory().numpy()
            st.prob, st.keep = P.make_problem(p)
            st.res = P.priest_result()
        else:
            st.z = z
            st.h = st.load(p, cem)
            st.out = torch.zeros(p["dims"] * NV + 4, device="cuda", dtype=torch.float64)
    elif call == "project_batch":
        probs = _mix_problems(case, seed)
        st.context(probs[0][0], W.cem_settings(256, case["K"], 1))
        st.rows = [N for _, N in probs]
        total = sum(st.rows)
        xi = [_samples(p, N, seed + k) for k, (p, N) in enumerate(probs)]
        st.xi = torch.cat(xi)
        st.xb = torch.empty_like(st.xi)
        st.score = torch.empty(2, total, device="cuda", dtype=torch.float64)
        off = np.concatenate([[0], np.cumsum(st.rows)])[:-1]
        row = 8 * 2 * NV
        st.ptrs = [[st.xi.data_ptr() + row * int(o) for o in off], None,
                   [st.xb.data_ptr() + row * int(o) for o in off],
                   [st.score[0].data_ptr() + 8 * int(o) for o in off],
                   [st.score[1].data_ptr() + 8 * int(o) for o in off]]
        for p, N in probs:
            st.load(p, W.cem_settings(N, case["K"], 1))
    elif call == "solve_batch":
        probs = _mix_problems(case, seed)
        st.context(probs[0][0], W.cem_settings(256, case["K"], case["L"]))
        structs = [P.make_problem(p, W.cem_settings(N, case["K"], case["L"]), per_problem_shape=True)
                   for p, N in probs]
        st.keep = [k for _, k in structs]
        st.probs = P.priest_problem_array([s for s, _ in structs])
        sizes = [case["L"] * N * 2 * NV for _, N in probs]
        st.z = torch.empty(sum(sizes), dtype=torch.float64, pin_memory=True)
        st.z.copy_(_normals(seed, sum(sizes)))
        off = np.concatenate([[0], np.cumsum(sizes)])[:-1]
        st.zp = P.pointer_array([st.z.data_ptr() + 8 * int(o) for o in off])
        st.res = (P.priest_result * len(probs))()
    else:
        probs = _mix_problems(case, seed)
        st.context(probs[0][0], W.cem_settings(256, case["K"], case["L"]))
        st.reqs = [P.make_problem(p, W.cem_settings(N, case["K"], case["L"], dims=p["dims"]),
                                  seed=seed * 7919 + k, per_problem_shape=True) for k, (p, N) in enumerate(probs)]
        st.res = [P.priest_result() for _ in probs]
    torch.cuda.synchronize()
    return st


# ---- one pass -----------------------------------------------------------------

def _results(results):
    """Host results as arrays: best coefficients, final means, (r, c_1, c_aug)."""
    xb = np.array([r.xi_best[:] for r in results], dtype=np.float32)
    mu = np.array([r.mu[:] for r in results], dtype=np.float32)
    sc = np.array([[r.resid, r.cost, r.c_aug] for r in results], dtype=np.float32)
    return {"best": xb, "mu": mu, "score": sc}


def run(st):
    c = st.case
    call = c["call"]
    if call in ("noalloc", "project", "project_batch"):
        with torch.cuda.stream(stream()):
            if call == "project_batch":
                P.priest_project_batch(st.ctx.h, st.handles, st.rows, *st.ptrs)
                return {"xi_bar": st.xb.float(), "score": st.score.float()}
            if c["warm"]:
                st.lam.copy_(st.lam0)
            if call == "project":
                P.priest_project_device(st.ctx.h, st.h, c["N"], *st.ptrs)
            else:
                s = P.priest_project_noalloc(st.cfg, st.prob, c["N"], *st.ptrs, stream=stream().cuda_stream)
                if s != P.PRIEST_OK:
                    raise P.PriestError(s, "priest_project_noalloc")
            out = [st.xb, st.score] + ([st.lam] if c["warm"] else [])
            if c["precision"] != FP64:
                out = [x.float() for x in out]
            return dict(zip(("xi_bar", "score", "lam"), out))
    if call == "solve":
        if c["host"]:
            P.priest_plan_z(st.ctx.h, st.prob, None, None, st.z, st.res)
            return _results([st.res])
        with torch.cuda.stream(stream()):
            P.priest_plan_device(st.ctx.h, st.h, st.z.data_ptr(), st.out.data_ptr())
            return st.out.float()
    if call == "solve_batch":
        P.priest_plan_batch_host(st.ctx.h, st.probs, st.zp, st.res)
        return _results(st.res)
    tickets = [P.priest_submit(st.ctx.h, s) for s, _ in st.reqs]
    for t, r in zip(tickets, st.res):
        P.priest_wait(st.ctx.h, t, r)
    return _results(st.res)


# ---- work ---------------------------------------------------------------------

def _iter_flops(dims, nf, n_p):
    """One sample's iteration without the pair tests: trajectory (position,
    velocity, acceleration) and its transpose on the free columns, norms and
    residual rows per time stamp, the shared-inverse step."""
    return 2 * (2 * 3 * dims * n_p * nf) + 12 * dims * n_p + 4 * dims * nf * nf


def _project_work(dims, nf, n_p, n_obs, N, K, warm):
    D = dims * NV
    return {"bytes": 8 * (N * (D * (4 if warm else 2) + 2) + n_obs * (2 * dims + 2)),
            "flops": N * (K * _iter_flops(dims, nf, n_p) + n_p * n_obs * (3 * dims + 2))}  # each pair looked at once


def work(case):
    call = case["call"]
    if call in ("noalloc", "project", "solve"):
        dims = 3 if case["scene"] in ("ellipsoids", "p2p3d") else 2
        nf = NV - 3 - {7: 3, 3: 2, 1: 1, 0: 0}[case["mask"]]
        w = _project_work(dims, nf, case["n_p"], case["n_static"] + case["n_dyn"], case["N"], case["K"],
                          case.get("warm", False))
        if call == "solve":
            D = dims * NV
            w = {"bytes": 8 * (case["L"] * case["N"] * D + D + 4),
                 "flops": case["L"] * (w["flops"] + case["N"] * D * D + case["n_elite"] * 2 * D * D + D ** 3 / 3)}
        return w
    L = case.get("L", 1)
    total = {"bytes": 0.0, "flops": 0.0}
    for dims, n_obs, N, n_p in _mix(case):
        w = _project_work(dims, 5, n_p, n_obs, N, case["K"], False)
        D = dims * NV
        if call == "project_batch":
            total["bytes"] += w["bytes"]
            total["flops"] += w["flops"]
        else:
            draws = 0 if call == "serve" else L * N * D
            total["bytes"] += 8 * (draws + n_obs * (2 * dims + 2) + 2 * D + 4)
            total["flops"] += L * (w["flops"] + N * D * D + (N // 10) * 2 * D * D + D ** 3 / 3)
    return total


# ---- the same results in plain 64-bit torch -----------------------------------

def _basis(n, n_p, horizon):
    """Bernstein values and derivatives: three n_p x (n + 1) matrices."""
    tau = torch.arange(n_p, device="cuda", dtype=torch.float64) / (n_p - 1)

    def bern(m, j):
        return math.comb(m, j) * tau ** j * (1 - tau) ** (m - j) if 0 <= j <= m else torch.zeros_like(tau)

    b = torch.stack([bern(n, j) for j in range(n + 1)], 1)
    d = torch.stack([n * (bern(n - 1, j - 1) - bern(n - 1, j)) for j in range(n + 1)], 1) / horizon
    dd = torch.stack([n * (n - 1) * (bern(n - 2, j - 2) - 2 * bern(n - 2, j - 1) + bern(n - 2, j))
                      for j in range(n + 1)], 1) / horizon ** 2
    return b, d, dd


class _Ref:
    """The projection (Sec. III-A, alternating minimisation) and Alg. 1 in 64 bits."""

    def __init__(self, p):
        t = lambda x: torch.as_tensor(np.asarray(x, dtype=float), device="cuda")  # noqa: E731
        self.p, self.dims, n = p, p["dims"], W.DEGREE
        Th = p["horizon"]
        self.B = _basis(n, p["n_p"], Th)
        self.center, self.vel, self.semi = t(p["center"]), t(p["vel"]), t(p["semi"])
        self.tt = torch.arange(p["n_p"], device="cuda", dtype=torch.float64) * Th / (p["n_p"] - 1)
        b0, bf, mask = t(p["b0"]), t(p["bf"]), p["bc_final_mask"]
        cB = torch.zeros(self.dims, NV, device="cuda", dtype=torch.float64)
        cB[:, 0] = b0[:, 0]
        cB[:, 1] = cB[:, 0] + Th * b0[:, 1] / n
        cB[:, 2] = 2 * cB[:, 1] - cB[:, 0] + Th * Th * b0[:, 2] / (n * (n - 1))
        hi = NV
        if mask & 1:
            cB[:, n] = bf[:, 0]
            hi = n
        if mask & 2:
            cB[:, n - 1] = cB[:, n] - Th * bf[:, 1] / n
            hi = n - 1
        if mask & 4:
            cB[:, n - 2] = 2 * cB[:, n - 1] - cB[:, n] + Th * Th * bf[:, 2] / (n * (n - 1))
            hi = n - 2
        self.cB, self.free = cB, slice(3, hi)
        rho = p["rho"]
        F = [b[:, self.free] for b in self.B]
        wP = p["n_obs"] + (2 if p["use_bounds"] else 0)
        H = torch.eye(hi - 3, device="cuda", dtype=torch.float64) + rho * (
            wP * F[0].T @ F[0] + F[1].T @ F[1] + F[2].T @ F[2])
        self.Winv = torch.linalg.inv(H)

    def _rows(self, c, sums):
        """Residual rows of the N x dims x NV coefficients: per time stamp
        (position, velocity, acceleration rows), or r^2 and c_1."""
        p, dims = self.p, self.dims
        pos, vel, acc = (torch.einsum("tj,naj->nta", b, c) for b in self.B)

        def ball(x, m):
            s = x.norm(dim=2, keepdim=True)
            return torch.where(s > m, x * (1 - m / s.clamp_min(1e-300)), torch.zeros_like(x))

        rv, ra = ball(vel, p["vmax"]), ball(acc, p["amax"])
        rp = torch.zeros_like(pos)
        sq = rv.square().sum((1, 2)) + ra.square().sum((1, 2))
        ax = torch.ones(p["n_obs"], dims, device="cuda", dtype=torch.float64) * self.semi[:, :1]
        if dims == 3:
            ax[:, 2] = self.semi[:, 1]
        for j0 in range(0, p["n_obs"], 50):
            j = slice(j0, j0 + 50)
            o = self.center[j] + self.tt[:, None, None] * self.vel[j]  # n_p x obstacles x dims
            d = pos[:, :, None, :] - o
            q = (d / ax[j]).square().sum(3)
            w = torch.where(q < 1, 1 - q.clamp_min(1e-300).rsqrt(), torch.zeros_like(q))
            if sums:
                sq = sq + (w.square() * d.square().sum(3)).sum((1, 2))
            else:
                rp = rp + torch.einsum("nto,ntoa->nta", w, d)
        if p["use_bounds"]:
            lo, hi = (torch.as_tensor(np.asarray(p[k], dtype=float)[:dims], device="cuda") for k in ("smin", "smax"))
            up, dn = (pos - hi).clamp_min(0), (lo - pos).clamp_min(0)
            rp = rp + up - dn
            sq = sq + up.square().sum((1, 2)) + dn.square().sum((1, 2))
        if not sums:
            return rp, rv, ra
        a2 = acc.square().sum(2)
        cost = a2
        if p.get("cost_kind", 0) == 1:
            cr = torch.linalg.cross(*(torch.nn.functional.pad(x, (0, 3 - dims)) for x in (vel, acc)), dim=2)
            kap2 = cr.square().sum(2) / (vel.square().sum(2) + p["curv_eps"] ** 2) ** 3
            s, g = (torch.as_tensor(np.asarray(p[k], dtype=float)[:, 0], device="cuda") for k in ("b0", "bf"))
            ln = (g - s).norm()
            u = (g - s) / ln
            along = ((pos - s) @ u).clamp(0, float(ln))
            dist2 = (pos - s - along[..., None] * u).square().sum(2)
            cost = p["w_acc"] * a2 + p["w_curv"] * kap2 + p["w_path"] * dist2
        return sq.sqrt(), cost.sum(1)

    def project(self, xi, K, lam=None):
        """xi, lam: N x D.  (xi_bar, lam, r, c_1)."""
        N = xi.shape[0]
        out = [self._project(xi[i:i + 512], K, None if lam is None else lam[i:i + 512]) for i in range(0, N, 512)]
        return [torch.cat(x) for x in zip(*out)]

    def _project(self, xi, K, lam):
        N, dims, f, rho = xi.shape[0], self.dims, self.free, self.p["rho"]
        x = xi.reshape(N, dims, NV)
        lam = torch.zeros_like(x) if lam is None else lam.reshape(N, dims, NV).clone()
        c = self.cB.expand(N, dims, NV).clone()
        c[:, :, f] = x[:, :, f]
        for _ in range(K):
            g = sum(torch.einsum("tj,nta->naj", b, r) for b, r in zip(self.B, self._rows(c, False)))
            lam = lam - rho * g
            u = x[:, :, f] + lam[:, :, f] - rho * g[:, :, f] - c[:, :, f]
            c[:, :, f] += u @ self.Winv.T
        r, c1 = self._rows(c, True)
        return c.reshape(N, -1), lam.reshape(N, -1), r, c1

    def solve(self, z, K, cem):
        """Alg. 1 with the draws z (L x N x D)."""
        p, D = self.p, self.dims * NV
        mu = torch.as_tensor(_mean(p), device="cuda")
        eye = torch.eye(D, device="cuda", dtype=torch.float64)
        cov = cem["init_std"] ** 2 * eye
        for zl in z:
            chol = torch.linalg.cholesky(cov + cem["chol_eps"] * cov.trace() / D * eye)
            xb, _, r, c1 = self.project(mu + zl @ chol.T, K)
            caug = c1 + r
            keep = torch.argsort(r, stable=True)[:cem["n_proj"]].sort().values
            el = keep[torch.argsort(caug[keep], stable=True)][:cem["n_elite"]]
            w = torch.exp(-(caug[el] - caug[el[0]]) / cem["gamma"])
            w = w / w.sum()
            s = cem["sigma_lr"]
            mu = (1 - s) * mu + s * (w @ xb[el])
            d = xb[el] - mu
            cov = (1 - s) * cov + s * torch.einsum("m,mi,mj->ij", w, d, d)
        b = el[0]
        return xb[b], mu, r[b], c1[b], caug[b], b


def exact(case, seed):
    """What run() returns, in 64 bits.  The batch, the burst and the solves of
    many samples take too long this way; the projections they are made of are
    covered by the other cases."""
    call = case["call"]
    if call in ("noalloc", "project"):
        p = _scene(case, seed)
        xi = _samples(p, case["N"], seed)
        lam = 0.05 * _normals(seed + 1, *xi.shape) if case["warm"] else None
        xb, lam, r, c1 = _Ref(p).project(xi, case["K"], lam)
        out = {"xi_bar": xb, "score": torch.stack([r, c1])}
        if case["warm"]:
            out["lam"] = lam
        return out
    if call == "project_batch":
        if sum(N for _, _, N, _ in _mix(case)) * case["K"] > 5_000_000:
            return None
        got = [_Ref(p).project(_samples(p, N, seed + k), case["K"])
               for k, (p, N) in enumerate(_mix_problems(case, seed))]
        return {"xi_bar": torch.cat([g[0] for g in got]),
                "score": torch.stack([torch.cat([g[2] for g in got]), torch.cat([g[3] for g in got])])}
    if call == "solve" and case["N"] * case["K"] * case["L"] * case["n_p"] <= 60_000_000:
        p = _scene(case, seed)
        D = p["dims"] * NV
        z = _normals(seed, case["L"], case["N"], D)
        xb, mu, r, c1, caug, i = _Ref(p).solve(z, case["K"], _cem(case, p["dims"]))
        if not case["host"]:
            return torch.cat([xb, torch.stack([r, c1, caug, i.double()])])
        pad = torch.nn.functional.pad
        return {"best": pad(xb, (0, P.MAX_D - D))[None], "mu": pad(mu, (0, P.MAX_D - D))[None],
                "score": torch.stack([r, c1, caug])[None]}
    return None
